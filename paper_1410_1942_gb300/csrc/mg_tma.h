// mg_tma.h -- the fine-level passes of the multigrid PCG on TMA-staged planes (mg_tma.cu).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include "internal.cuh"

namespace pcg {

// Tensor maps of a handle's fine-level arrays (host copies, passed by value to the launches), for
// the FP32 V-cycle on the rho/2 operator.
struct FineMaps {
    bool on = false;
    bool bf16 = false;
    int withhold = 0;  // testing aid (fine_maps_withhold): the pass whose planes stay incomplete
    const float *z = nullptr, *pa = nullptr, *pb = nullptr, *x0 = nullptr, *r = nullptr, *x = nullptr;
    // halo boxes of z, both p buffers, x0 and rho/2; centre boxes of r and x
    CUtensorMap mz, mpa, mpb, mx0, meta, mr, mx, mshort;
};

// Whether the passes serve a grid: rows of whole 32 bytes, no wrap, no stored faces, aggregates of
// 2 x 2 cells in x-y.
bool fine_maps_fit(const Dims& d);
// Encodes the maps; false if that fails.
bool fine_maps_build(FineMaps* m, const Dims& d, const void* eta, bool bf16, const float* z,
                     const float* pa, const float* pb, const float* x0, const float* r,
                     const float* x);

// Testing aid: the boxes that one pass (1 phase A, 2 phase B, 3 restriction, 4 smoothing; 0: none)
// loads of its field are a row short, so that its waits for the full planes run out.
bool fine_maps_withhold(FineMaps* m, const Dims& d, int pass);

// The passes (launched with programmatic stream serialization): phase A, phase B, the finest
// restriction and the finest post-smoothing, as k_cg_a, k_mg_cg_b, k_mg_restrict and k_mg_smooth.
void launch_fine_a(const FineMaps& m, const Dims& d, bool in_a, float* p_out, Scalars* sc,
                   double* part, cudaStream_t st);
void launch_fine_b(const FineMaps& m, const Dims& d, bool p_a, float* x, float* r, float* x0,
                   float omega, Scalars* sc, double* part, cudaStream_t st);
void launch_fine_restrict(const FineMaps& m, const Dims& d, const Dims& dc, int fz,
                          const float* cdiag, float* rc, float* xc, float omega, const Scalars* sc,
                          cudaStream_t st);
void launch_fine_smooth(const FineMaps& m, const Dims& d, const Dims& dc, int sz, const float* e,
                        float alpha, float omega, float* y, Scalars* sc, double* part, int mode,
                        cudaStream_t st);

}  // namespace pcg
