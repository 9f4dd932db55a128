// coop.cu -- the order of cooperative launches (coop.h).
#include "coop.h"

#include <mutex>

namespace pcg {
namespace {

constexpr int MAX_DEVICES = 64;
std::mutex g_coop_mu;
cudaEvent_t g_coop_last[MAX_DEVICES] = {};  // end of the last scope on each device

}  // namespace

CoopOrder::CoopOrder(cudaStream_t st) : st_(st), dev_(0) {
    g_coop_mu.lock();
    if (cudaGetDevice(&dev_) != cudaSuccess || dev_ < 0 || dev_ >= MAX_DEVICES) dev_ = 0;
    cudaEvent_t& e = g_coop_last[dev_];
    if (!e) {
        if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) {
            cudaGetLastError();
            e = nullptr;
        }
    } else {
        cudaStreamWaitEvent(st_, e, 0);
    }
}

CoopOrder::~CoopOrder() {
    if (g_coop_last[dev_]) cudaEventRecord(g_coop_last[dev_], st_);
    g_coop_mu.unlock();
}

cudaError_t coop_launch(const void* kernel, dim3 grid, dim3 block, void** params, size_t smem,
                        cudaStream_t st) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusActive)
        return cudaLaunchCooperativeKernel(kernel, grid, block, params, smem, st);
    CoopOrder order(st);
    return cudaLaunchCooperativeKernel(kernel, grid, block, params, smem, st);
}

}  // namespace pcg
