// resident.h -- host interface of the on-chip PCG (resident.cu): inner solves whose whole state
// fits the registers and shared memory of the GPU.
#pragma once

#include <vector>

#include <cuda_runtime.h>

#include "internal.cuh"

namespace pcg {

// Coefficient source of a launch: rho/2 in FP32 or BF16, stored FP32 faces (cut cells), or the
// FP64 faces (FP64 arithmetic throughout).
enum ResKind { RES_ETA32 = 0, RES_ETA16 = 1, RES_FACES32 = 2, RES_FACES64 = 3 };

// One solve as the device sees it, copied there before every launch.  FP32 kinds: r = the FP32
// right side, x = the correction (written).  RES_FACES64: r = the FP64 residual, x = the FP64
// iterate (the correction is added).
struct ResSolve {
    Dims d;
    const void* c[4];  // rho/2; or bx, by, bz, diag
    const void* r;
    void* x;
    Scalars* sc;   // in: rr (and bb); out: iter, rr, rz, done
    int ctas;      // boxes of the solve (res_plan_build)
    // controls of the launch
    int active;    // 0: skipped; its scalars come back CONVERGED with 0 iterations
    double tol2;   // stop when r.r <= tol2 (b.b for RES_FACES64, else r0.r0)
    int max_iter;
    unsigned tag0;  // the solve's sweeps carry the tags tag0 + 1, tag0 + 2, ... (res_tags)
};

// One box of a solve held by one CTA.
struct ResTask {
    int solve;
    int x0, y0, z0, bx, by, bz;
    int rank;    // among the solve's boxes
    int src[6];  // word offset of the facing values in the neighbour's outbox (-x, +x, -y, +y,
                 // -z, +z); -1: no neighbour
};

struct ResArgs {
    const ResSolve* solves;
    const ResTask* tasks;
    const int* cta_task;  // CTA c runs tasks [cta_task[c], cta_task[c + 1]) in order
    void* sums;           // reduction records per solve and parity
    void* outbox;         // halo words, `box_words` per CTA and parity
    int box_words;
    int extra;            // > 0: wait for one box more than there are (a testing aid)
    int* error;           // set to 1 once a wait has run out
    int nsolves;
    unsigned long long wait_ns;  // a wait without progress in the launch gives up after this
};

constexpr unsigned long long RES_WAIT_NS = 1000ull * 1000ull * 1000ull;  // 1 s
constexpr int RES_MAX_CTAS = 159;  // boxes of one solve (one more reduction word for the test aid)

struct ResPlan {
    int ncta = 0, nsolves = 0, ntasks = 0, box_words = 0;
    int depth = 0;  // planes per thread of the kernel: 2, 4, 8 or 16
    size_t smem = 0;  // dynamic shared memory of the launch
    bool dbl = false;
    int extra = 0;
    unsigned long long wait_ns = RES_WAIT_NS;
    unsigned next_tag = 0;
    // one device allocation, carved into:
    void* mem = nullptr;
    size_t cap = 0;
    ResSolve* solves = nullptr;
    ResTask* tasks = nullptr;
    int* cta_task = nullptr;
    int* error = nullptr;
    void* words = nullptr;  // the tagged words: sums, then outbox
    size_t words_bytes = 0;
    void* sums = nullptr;
    void* outbox = nullptr;
};

// Whether a grid fits on chip (one box per SM at most), in FP32 or FP64.
bool res_supported(const Dims& d, bool dbl);
// Device bytes of the plan of one solve of this grid.
size_t res_plan_bytes(const Dims& d, bool dbl);
size_t res_plan_held(const ResPlan& p);
// Boxes and schedule of the solves (one precision), whose `ctas` it sets; device arrays allocated
// or reused, copied on st and synchronised.  0, -1 (a solve does not fit) or -2 (no memory).
int res_plan_build(ResPlan* p, ResSolve* solves, int n, bool dbl, cudaStream_t st);
void res_plan_free(ResPlan* p);
// Tags for the next launch (max_iter set): fills tag0, and clears the words first when the tags
// would wrap around.  0, or -1 when the clearing fails.
int res_tags(ResPlan* p, ResSolve* solves, int n, cudaStream_t st);
// One cooperative launch over the plan: `solves` (n, pinned host memory) copied to the device,
// then the kernel.  0, or -1 when the launch is refused.
int launch_res(const ResPlan& p, ResKind kind, const ResSolve* solves, int n, cudaStream_t st);

}  // namespace pcg
