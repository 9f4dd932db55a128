"""One-time set-up of the kernels that need more shared memory than a launch gets by default belongs
to each device of the process, not to the first that ran them.  The library's own launch code is
linked against a stand-in for the CUDA runtime with two devices, which records on which device a
kernel's attribute was set before it was launched there (no GPU)."""
import os
import subprocess

from paper_1410_1942_gb300 import build

FAKE = r"""
#include <cstring>
#include <map>
#include <utility>

#include <cuda_runtime_api.h>

int dev = 0, launches = 0, refused = 0;
static std::map<std::pair<int, const void*>, size_t> allowed;  // (device, kernel) -> shared bytes

static cudaError_t launch(const void* f, size_t smem) {
    ++launches;
    auto it = allowed.find({dev, f});
    if (smem > 48 * 1024 && (it == allowed.end() || it->second < smem)) {
        ++refused;
        return cudaErrorInvalidValue;
    }
    return cudaSuccess;
}

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = dev; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaPeekAtLastError() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) allowed[{dev, f}] = (size_t)v;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
    return launch(f, c->dynamicSmemBytes);
}
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3, dim3, void**, size_t smem, cudaStream_t) {
    return launch(f, smem);
}
cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void**, size_t smem, cudaStream_t) {
    return launch(f, smem);
}
cudaError_t cudaMalloc(void** p, size_t n) { *p = new char[n]; return cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) { *p = new char[n]; return cudaSuccess; }
cudaError_t cudaFree(void*) { return cudaSuccess; }
cudaError_t cudaFreeHost(void*) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
    *s = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
// registration of the kernels and the <<<>>> launches
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaInitModule(void**) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, cudaStream_t) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* n, void* s) {
    *g = dim3(1); *b = dim3(1); *n = 0; memset(s, 0, sizeof(cudaStream_t));
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(const void** k, const void* f) { *k = f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(const void* f, dim3, dim3, void**, size_t smem, cudaStream_t) {
    return launch(f, smem);
}
}
"""

MAIN = r"""
#include <cstdio>
#include "kernels.h"
#include "mg.h"
#include "mg_tma.h"
#include "march.h"
#include "resident.h"

using namespace pcg;

// what the linked objects need of the rest of the library
namespace pcg {
std::atomic<unsigned long long> g_kernel_launches{0};
int quad_kc(const Dims&, int) { return 8; }
bool march_encode_box(CUtensorMap*, const void*, bool, const Dims&, int, int) { return true; }
}  // namespace pcg
extern int dev, launches, refused;  // of the stand-in

int main() {
    Dims d{};
    d.nx = 64; d.ny = 48; d.nz = 32; d.sxy = d.nx * d.ny; d.n = d.sxy * d.nz;
    for (dev = 0; dev < 2; ++dev) {
        Scalars sc{};
        FineMaps maps{};
        Dims dc = d;
        dc.nx = 32; dc.ny = 24; dc.nz = 16; dc.sxy = dc.nx * dc.ny; dc.n = dc.sxy * dc.nz;
        launch_fine_a(maps, d, true, nullptr, &sc, nullptr, nullptr);
        launch_fine_b(maps, d, true, nullptr, nullptr, nullptr, 1.f, &sc, nullptr, nullptr);
        launch_fine_restrict(maps, d, dc, 2, nullptr, nullptr, nullptr, 1.f, &sc, nullptr);
        launch_fine_smooth(maps, d, dc, 1, nullptr, 1.f, 1.f, nullptr, &sc, nullptr, -1, nullptr);
        Dims f = d;  // (its bottom levels in FP64 take more than a launch gets by default)
        f.nx = 256; f.ny = 128; f.nz = 128; f.sxy = f.nx * f.ny; f.n = f.sxy * f.nz;
        MgHier m{};
        mg_plan(f, &m);
        mg_alloc(&m, true);
        mg_apply<double, CoefFaces64>(&m, f, 8, CoefFaces64{}, (double*)nullptr, (double*)nullptr,
                                      nullptr, nullptr);
        for (bool dbl : {false, true}) {
            Dims s = d;
            s.nx = 128; s.ny = s.nz = 64; s.sxy = s.nx * s.ny; s.n = s.sxy * s.nz;
            ResPlan plan{};
            ResSolve rs{};
            rs.d = s;
            rs.active = 1;
            if (res_plan_build(&plan, &rs, 1, dbl, nullptr) != 0) return 2;
            launch_res(plan, dbl ? RES_FACES64 : RES_ETA32, &rs, 1, nullptr);
        }
    }
    printf("launches %d refused %d\n", launches, refused);
    return refused ? 1 : 0;
}
"""


def test_kernels_with_much_shared_memory_run_on_a_second_device(tmp_path):
    objs = [os.path.join(build.BUILD, n + ".o") for n in ("mg_tma", "mg", "resident", "coop", "alloc")]
    build.build(force=not all(map(os.path.exists, objs)))
    fake, main, exe = (str(tmp_path / n) for n in ("fake.cpp", "main.cu", "two"))
    for path, text in ((fake, FAKE), (main, MAIN)):
        with open(path, "w") as f:
            f.write(text)
    for path in (fake, main):
        subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I",
                        build.CSRC, "-I", os.path.join(build.ROOT, "include"), "-c", path, "-o",
                        path + ".o"], check=True)
    subprocess.run(["g++", fake + ".o", main + ".o", *objs, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
    launched, refused = (int(r.stdout.split()[q]) for q in (1, 3))
    assert refused == 0 and launched >= 2 * (4 + 1 + 2)
