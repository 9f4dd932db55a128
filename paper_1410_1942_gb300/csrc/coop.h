// coop.h -- cooperative launches one after another.
//
// A cooperative kernel whose CTAs wait for each other needs all of them resident.  Two such
// grids in flight on different streams (two handles solved by two threads) could each hold part
// of the SMs and wait for the rest until their deadlines.  Every cooperative launch of the library
// therefore waits, on its stream, for the one before it on the device: an event recorded after
// each launch, under a lock.  Kernels of that kind fill the GPU, so nothing is lost by it.
#pragma once

#include <cuda_runtime.h>

namespace pcg {

// Scope around a launch on st that contains cooperative kernels (a graph of them, say): the
// constructor locks and makes st wait for the previous such scope, the destructor records its
// end and unlocks.
class CoopOrder {
public:
    explicit CoopOrder(cudaStream_t st);
    ~CoopOrder();
    CoopOrder(const CoopOrder&) = delete;
    CoopOrder& operator=(const CoopOrder&) = delete;

private:
    cudaStream_t st_;
    int dev_;
};

// One cooperative launch, ordered as above (on a stream being captured: recorded as it is, the
// graph's launch is to be ordered).
cudaError_t coop_launch(const void* kernel, dim3 grid, dim3 block, void** params, size_t smem,
                        cudaStream_t st);

}  // namespace pcg
