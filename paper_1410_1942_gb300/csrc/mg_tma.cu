// mg_tma.cu -- the fine-level passes of the multigrid PCG on the rho/2 operator, with x-y planes
// staged in shared memory by TMA.
//
// The passes are those of the quad kernels (plane_tile.cuh: k_cg_a_q, k_mg_cg_b_q,
// k_mg_restrict_q, k_mg_smooth_q), which load planes through registers one or two ahead and, at three
// blocks per SM, keep too few bytes in flight: phase A, the restriction and the smoothing ran at
// 55-75 % of the copy bandwidth on a grid far larger than the L2, and at 2.6-3.3 TB/s on one that
// half fits it.  Here a producer warp issues the halo and centre boxes of the planes to come into a
// ring of four stages, and eight consumer warps march the tile's 64 x 16 columns with 2 x 2 cells per
// thread: planes k - 1, k, k + 1 of the own cells in registers, the neighbour strips from the stage of
// plane k.  No barrier joins the warps; a stage is handed over by its full and empty mbarriers.  Tiles
// may be ragged in x and y (the boxes' parts outside the grid read as zero, block_edges knows the
// walls), so every grid with nx % 8 == 0 takes these passes, not only those of whole 64-cell tiles.
// Per cell the arithmetic is that of the quad kernels, in the same order.
//
// us on 1024x512x256, quad kernels / here: phase A 405 / 346 (16 B a cell: 6.2 TB/s), phase B 571 /
// 570 (28 B: 6.6 TB/s), restriction 362 / 305 (5.7 TB/s), smoothing 555 / 427 (5.2 TB/s, bound by
// issue); the solve 396 / 355 ms.  Grids not of whole 64-cell tiles took slower passes before: a
// server's step of 16 uneven grids 41.2 / 26.8 ms.
#include "mg_tma.h"

#include <algorithm>
#include <atomic>

#include "kernels.h"
#include "march_dev.cuh"
#include "plane_tile.cuh"

namespace pcg {
namespace {

constexpr int FX = 2, FY = 2, FT = 8;             // cells per thread, consumer warps
constexpr int FW = 32 * FX, FH = FY * FT;         // tile
constexpr int FNS = 4;                            // stages
constexpr int FTHREADS = 32 * (FT + 1);
constexpr int FBLOCKS = 3;                        // resident blocks per SM (register budget)

enum { PASS_A, PASS_B, PASS_RESTRICT, PASS_SMOOTH };

// Stage of a pass: NF halo boxes of the stencil field's parts, the halo box of rho/2, NC centre
// boxes.
template <int PASS, typename E>
struct FGeo {
    static constexpr int NF = PASS == PASS_A ? 2 : 1;
    static constexpr int NC = PASS == PASS_A ? 0 : PASS == PASS_B ? 2 : 1;
    static constexpr int VW = FW + 8, H = FH + 2;
    static constexpr int EOFF = EtaX<E>::OFF, EW = FW + 2 * EOFF;
    static constexpr int VB = VW * H * 4, EB = EW * H * (int)sizeof(E), CB = FW * FH * 4;
    static constexpr int ETA = NF * align128(VB), C = ETA + align128(EB);
    static constexpr int STAGE = C + NC * align128(CB);
    static constexpr int TX_HALO = NF * VB + EB, TX = TX_HALO + NC * CB;
    static constexpr int SMEM = FNS * STAGE;
};

struct FineArgs {
    Dims d, dc;
    int kc;         // planes per block (even)
    int fz, sz;     // restriction, smoothing: the aggregates' factor and shift along z
    int mode;       // smoothing: as k_mg_smooth
    float alpha, omega;
    const float* e;      // smoothing: the coarse correction
    const float* cdiag;  // restriction
    float *o0, *o1, *o2; // outputs: A p; B x, r, x0; restriction rc, xc; smoothing y
    Scalars* sc;
    double* partials;
};

template <int PASS, typename E>
__global__ void __launch_bounds__(FTHREADS, FBLOCKS)
k_fine(const __grid_constant__ CUtensorMap mf0, const __grid_constant__ CUtensorMap mf1,
       const __grid_constant__ CUtensorMap meta, const __grid_constant__ CUtensorMap mc0,
       const __grid_constant__ CUtensorMap mc1, const FineArgs a) {
    using G = FGeo<PASS, E>;
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ __align__(8) uint64_t full[FNS];
    __shared__ __align__(8) uint64_t empty[FNS];
    __shared__ double red[64];
    __shared__ volatile int s_fail;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        for (int s = 0; s < FNS; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], FT);
        }
        fence_mbar_init();
        s_fail = 0;
    }
    pdl_entry();
    // (one answer for the whole block: a block of this grid whose wait runs out sets `done` meanwhile,
    // and threads that left by themselves would be missing at the barriers below)
    if (__syncthreads_or(a.sc && a.sc->done)) return;
    const Dims d = a.d;
    const int x0 = blockIdx.x * FW, y0 = blockIdx.y * FH;
    const int k0 = blockIdx.z * a.kc, k1 = min(d.nz, k0 + a.kc);
    float acc = 0.f;
    int issued = 0;  // planes issued (the producer)
    if (warp == FT) {
        if (lane == 0) {
            // planes k0 - 1 .. k1; the centre boxes of the planes computed
            const int L = k1 - k0;
            for (int q = 0; q < L + 2; ++q) {
                const int st = q % FNS, k = k0 - 1 + q;
                if (q >= FNS && !mbar_wait_or(&empty[st], ((q / FNS) - 1) & 1, &s_fail)) {
                    s_fail = 1;
                    break;
                }
                issued = q + 1;
                unsigned char* dst = sm + st * G::STAGE;
                const bool centre = G::NC > 0 && q > 0 && q <= L;
                mbar_arrive_expect_tx(&full[st], centre ? G::TX : G::TX_HALO);
                tma_load_3d(dst, &mf0, &full[st], x0 - 4, y0 - 1, k);
                if (G::NF > 1) tma_load_3d(dst + align128(G::VB), &mf1, &full[st], x0 - 4, y0 - 1, k);
                tma_load_3d(dst + G::ETA, &meta, &full[st], x0 - G::EOFF, y0 - 1, k);
                if (centre) {
                    tma_load_3d(dst + G::C, &mc0, &full[st], x0, y0, k);
                    if (G::NC > 1) tma_load_3d(dst + G::C + align128(G::CB), &mc1, &full[st], x0, y0, k);
                }
            }
        }
    } else {
        const int i0 = x0 + FX * lane, j0 = y0 + FY * warp;
        const int r0 = 1 + FY * warp, cv = 4 + FX * lane, ce = G::EOFF + FX * lane, cc = FX * lane;
        const unsigned edges = block_edges<FX, FY>(d, i0, j0);
        const float be = PASS == PASS_A ? (float)a.sc->beta : 0.f;
        const float al = PASS == PASS_B ? (float)a.sc->alpha : a.alpha;
        const bool in0 = i0 < d.nx && j0 < d.ny, in1 = i0 < d.nx && j0 + 1 < d.ny;
        // smoothing: the coarse correction at the block's parent and its four neighbours, of the
        // coarse plane in use (ev) and the next (en)
        float ev[5], en[5];
        const Dims dc = a.dc;
        const int I = i0 >> 1, J = j0 >> 1;
        auto parents = [&](int K, float (&o)[5]) {
            if constexpr (PASS == PASS_SMOOTH) {
                const int n = min(max(K, 0), dc.nz - 1) * dc.sxy;
                const int Ic = min(I, dc.nx - 1), Jc = min(J, dc.ny - 1);
                o[0] = a.e[n + Ic + dc.nx * Jc];
                o[1] = a.e[n + max(Ic - 1, 0) + dc.nx * Jc];
                o[2] = a.e[n + min(Ic + 1, dc.nx - 1) + dc.nx * Jc];
                o[3] = a.e[n + Ic + dc.nx * max(Jc - 1, 0)];
                o[4] = a.e[n + Ic + dc.nx * min(Jc + 1, dc.ny - 1)];
            }
        };
        auto stage = [&](int q) { return sm + (q % FNS) * G::STAGE; };
        auto acquire = [&](int q) {
            if (s_fail) return false;
            if (!mbar_wait_or(&full[q % FNS], (q / FNS) & 1, &s_fail)) {
                s_fail = 1;
                return false;
            }
            return true;
        };
        auto release = [&](int q) {
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[q % FNS]);
        };
        // the stencil field of the own cells of stage q (pe: their parent's correction)
        auto field = [&](int q, float pe, float (&o)[FY][FX]) {
            const float* S = (const float*)stage(q);
            load_centre<FX, FY>(S, G::VW, r0, cv, o);
            if constexpr (PASS == PASS_A) {
                float b[FY][FX];
                load_centre<FX, FY>((const float*)(stage(q) + align128(G::VB)), G::VW, r0, cv, b);
#pragma unroll
                for (int y = 0; y < FY; ++y)
#pragma unroll
                    for (int x = 0; x < FX; ++x) o[y][x] = o[y][x] + be * b[y][x];
            }
            if constexpr (PASS == PASS_SMOOTH) {
#pragma unroll
                for (int y = 0; y < FY; ++y)
#pragma unroll
                    for (int x = 0; x < FX; ++x) o[y][x] = o[y][x] + al * pe;
            }
        };
        auto eta_of = [&](int q) { return (const E*)(stage(q) + G::ETA); };
        float um[FY][FX], uc[FY][FX], em[FY][FX], ec[FY][FX], wzl[FY][FX];
        if constexpr (PASS == PASS_SMOOTH) {
            parents((k0 - 1) >> a.sz, en);
            parents(k0 >> a.sz, ev);
        }
        bool ok = acquire(0);
        if (ok) {
            field(0, PASS == PASS_SMOOTH && k0 > 0 ? en[0] : 0.f, um);  // (below the grid: 0)
            load_centre<FX, FY>(eta_of(0), G::EW, r0, ce, em);
        }
        release(0);
        ok = acquire(1);
        if (ok) {
            field(1, PASS == PASS_SMOOTH ? ev[0] : 0.f, uc);
            load_centre<FX, FY>(eta_of(1), G::EW, r0, ce, ec);
#pragma unroll
            for (int y = 0; y < FY; ++y)
#pragma unroll
                for (int x = 0; x < FX; ++x)
                    wzl[y][x] = (k0 > 0 || (d.walls & 16)) ? rcp_approx(ec[y][x] + em[y][x]) : 0.f;
        }
        if constexpr (PASS == PASS_SMOOTH) parents((k0 >> a.sz) + 1, en);
        float rs = 0.f;  // restriction: the aggregate's sum so far
        for (int k = k0; k < k1; ++k) {
            const int qc = 1 + k - k0, qn = qc + 1;
            ok = acquire(qn);
            if (ok) {
                const unsigned char* S = stage(qc);
                // smoothing: plane k + 1 has the next parents when it starts an aggregate
                const bool next = PASS == PASS_SMOOTH && ((k + 1) >> a.sz) != (k >> a.sz);
                float up[FY][FX], ep[FY][FX];
                field(qn, PASS == PASS_SMOOTH ? (next ? en[0] : ev[0]) : 0.f, up);
                load_centre<FX, FY>(eta_of(qn), G::EW, r0, ce, ep);
                float vxm[FY], vxp[FY], vym[FX], vyp[FX];
                load_halo<FX, FY>((const float*)S, G::VW, r0, cv, vxm, vxp, vym, vyp);
                if constexpr (PASS == PASS_A) {
                    float bxm[FY], bxp[FY], bym[FX], byp[FX];
                    load_halo<FX, FY>((const float*)(S + align128(G::VB)), G::VW, r0, cv, bxm, bxp, bym,
                                      byp);
#pragma unroll
                    for (int y = 0; y < FY; ++y) {
                        vxm[y] = vxm[y] + be * bxm[y];
                        vxp[y] = vxp[y] + be * bxp[y];
                    }
#pragma unroll
                    for (int x = 0; x < FX; ++x) {
                        vym[x] = vym[x] + be * bym[x];
                        vyp[x] = vyp[x] + be * byp[x];
                    }
                }
                if constexpr (PASS == PASS_SMOOTH) {
                    // (beyond the grid the field stays 0, as at a wall)
                    const float exm = i0 > 0 ? ev[1] : 0.f, exp_ = i0 + FX < d.nx ? ev[2] : 0.f;
                    const float eym = j0 > 0 ? ev[3] : 0.f, eyp = j0 + FY < d.ny ? ev[4] : 0.f;
#pragma unroll
                    for (int y = 0; y < FY; ++y) {
                        vxm[y] = vxm[y] + al * exm;
                        vxp[y] = vxp[y] + al * exp_;
                    }
#pragma unroll
                    for (int x = 0; x < FX; ++x) {
                        vym[x] = vym[x] + al * eym;
                        vyp[x] = vyp[x] + al * eyp;
                    }
                    if (!in1) {  // an odd last row: what lies above it is the wall
#pragma unroll
                        for (int x = 0; x < FX; ++x) {
                            uc[1][x] = 0.f;
                            up[1][x] = 0.f;
                        }
                    }
                    if (k + 1 == d.nz) {  // and above the top
#pragma unroll
                        for (int y = 0; y < FY; ++y)
#pragma unroll
                            for (int x = 0; x < FX; ++x) up[y][x] = 0.f;
                    }
                }
                float exm[FY], exq[FY], eym[FX], eyp[FX];
                load_halo<FX, FY>(eta_of(qc), G::EW, r0, ce, exm, exq, eym, eyp);
                float qv[FY][FX], D[FY][FX];
                stencil<FX, FY>(d, edges, k, uc, vxm, vxp, vym, vyp, um, up, ec, exm, exq, eym, eyp, ep,
                                wzl, qv, D);
                const float* C0 = (const float*)(S + G::C);
                const size_t c = (size_t)i0 + (size_t)d.nx * (j0 + (size_t)d.ny * k);
                if constexpr (PASS == PASS_A) {
#pragma unroll
                    for (int y = 0; y < FY; ++y)
                        if (y == 0 ? in0 : in1) {
#pragma unroll
                            for (int x = 0; x < FX; ++x) acc += uc[y][x] * qv[y][x];
                            st_row<FX>(a.o0 + c + (size_t)y * d.nx, uc[y]);
                        }
                } else if constexpr (PASS == PASS_B) {
                    const float* C1 = (const float*)(S + G::C + align128(G::CB));
                    float xo[FY][FX], ro[FY][FX];
                    load_centre<FX, FY>(C0, FW, FY * warp, cc, xo);
                    load_centre<FX, FY>(C1, FW, FY * warp, cc, ro);
#pragma unroll
                    for (int y = 0; y < FY; ++y)
                        if (y == 0 ? in0 : in1) {
                            float xn[FX], rn[FX], zn[FX];
#pragma unroll
                            for (int x = 0; x < FX; ++x) {
                                xn[x] = xo[y][x] + al * uc[y][x];
                                rn[x] = ro[y][x] - al * qv[y][x];
                                zn[x] = div_refined(a.omega * rn[x], D[y][x]);
                                acc += rn[x] * rn[x];
                            }
                            st_row<FX>(a.o0 + c + (size_t)y * d.nx, xn);
                            st_row<FX>(a.o1 + c + (size_t)y * d.nx, rn);
                            st_row<FX>(a.o2 + c + (size_t)y * d.nx, zn);
                        }
                } else if constexpr (PASS == PASS_RESTRICT) {
                    float ro[FY][FX];
                    load_centre<FX, FY>(C0, FW, FY * warp, cc, ro);
#pragma unroll
                    for (int y = 0; y < FY; ++y)
                        if (y == 0 ? in0 : in1) {
#pragma unroll
                            for (int x = 0; x < FX; ++x) rs += ro[y][x] - qv[y][x];
                        }
                    if (a.fz == 1 || (k & 1) || k + 1 == d.nz) {
                        if (in0) {
                            const int Ic = I + dc.nx * (J + dc.ny * (a.fz == 1 ? k : k >> 1));
                            a.o0[Ic] = rs;
                            a.o1[Ic] = a.omega * rs / a.cdiag[Ic];
                        }
                        rs = 0.f;
                    }
                } else {
                    float ro[FY][FX];
                    load_centre<FX, FY>(C0, FW, FY * warp, cc, ro);
#pragma unroll
                    for (int y = 0; y < FY; ++y)
                        if (y == 0 ? in0 : in1) {
                            float yn[FX];
#pragma unroll
                            for (int x = 0; x < FX; ++x) {
                                yn[x] = uc[y][x] + div_refined(a.omega * (ro[y][x] - qv[y][x]), D[y][x]);
                                acc += ro[y][x] * yn[x];
                            }
                            st_row<FX>(a.o0 + c + (size_t)y * d.nx, yn);
                        }
                    if (next) {
#pragma unroll
                        for (int q = 0; q < 5; ++q) ev[q] = en[q];
                        parents(((k + 1) >> a.sz) + 1, en);
                    }
                }
#pragma unroll
                for (int y = 0; y < FY; ++y)
#pragma unroll
                    for (int x = 0; x < FX; ++x) {
                        um[y][x] = uc[y][x];
                        uc[y][x] = up[y][x];
                        ec[y][x] = ep[y][x];
                    }
            }
            release(qc);
        }
    }
    __syncthreads();
    if (s_fail) {
        // a wait ran out: the copies in flight land before the block ends, the solve stops
        if (warp == FT && lane == 0)
            for (int q = max(0, issued - FNS); q < issued; ++q)
                (void)mbar_wait(&full[q % FNS], (q / FNS) & 1);
        if (tid == 0 && a.sc) atomicExch(&a.sc->done, (int)TIMEDOUT);
        __syncthreads();
    }
    if constexpr (PASS == PASS_RESTRICT) return;
    if (!a.sc || (PASS == PASS_SMOOTH && a.mode < 0)) return;
    double v[1] = {(double)acc}, tot[1];
    if (!grid_sum<1>(v, a.partials, &a.sc->ticket, tot, red) || tid != 0) return;
    Scalars* sc = a.sc;
    if (*(volatile int*)&sc->done == TIMEDOUT) return;
    if constexpr (PASS == PASS_A) {
        if (!(tot[0] > 0.0) || !isfinite(tot[0])) {
            sc->done = BREAKDOWN;
        } else {
            sc->pq = tot[0];
            sc->alpha = sc->rz / tot[0];
        }
    } else if constexpr (PASS == PASS_B) {
        sc->rr = tot[0];
    } else if constexpr (PASS == PASS_SMOOTH) {
        cg_next(sc, tot[0], a.mode);
    }
}

// z-chunk: even, one wave of resident blocks if the grid allows it (quad_kc's rule).
int fine_kc(const Dims& d) {
    static const int sms = [] {
        int dev = 0, n = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
            cudaGetLastError();
            n = 152;
        }
        return n;
    }();
    const long long tiles = (long long)((d.nx + FW - 1) / FW) * ((d.ny + FH - 1) / FH);
    const long long slots = (long long)sms * FBLOCKS;
    long long kc = 64, best = -1;
    for (long long k = 2; k <= 64; k += 2) {
        const long long blocks = tiles * ((d.nz + k - 1) / k);
        const long long t = ((blocks + slots - 1) / slots) * (k + 3);
        if (blocks <= 4096 && (best < 0 || t < best)) { best = t; kc = k; }
        if (k >= d.nz) break;
    }
    return (int)kc;
}

dim3 fine_grid(const Dims& d, int kc) {
    return dim3((d.nx + FW - 1) / FW, (d.ny + FH - 1) / FH, (d.nz + kc - 1) / kc);
}

template <int PASS>
void launch(const FineMaps& m, const CUtensorMap& field, const CUtensorMap& f1, const CUtensorMap& c0,
            const CUtensorMap& c1, FineArgs a, cudaStream_t st) {
    const CUtensorMap& f0 = m.withhold == PASS + 1 ? m.mshort : field;
    static OncePerDevice once;
    once.run([] {
        cudaFuncSetAttribute(k_fine<PASS, float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             FGeo<PASS, float>::SMEM);
        cudaFuncSetAttribute(k_fine<PASS, __nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             FGeo<PASS, __nv_bfloat16>::SMEM);
        cudaGetLastError();
    });
    a.kc = fine_kc(a.d);
    const dim3 grid = fine_grid(a.d, a.kc);
    if (m.bf16)
        launch_pdl(k_fine<PASS, __nv_bfloat16>, grid, dim3(FTHREADS), FGeo<PASS, __nv_bfloat16>::SMEM,
                   st, f0, f1, m.meta, c0, c1, a);
    else
        launch_pdl(k_fine<PASS, float>, grid, dim3(FTHREADS), FGeo<PASS, float>::SMEM, st, f0, f1,
                   m.meta, c0, c1, a);
    g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
}

}  // namespace

bool fine_maps_fit(const Dims& d) {
    return d.nx % 8 == 0 && d.ny >= 2 && !(d.walls & (PERIODIC_X | CUT_CELLS));
}

bool fine_maps_build(FineMaps* m, const Dims& d, const void* eta, bool bf16, const float* z,
                     const float* pa, const float* pb, const float* x0, const float* r,
                     const float* x) {
    *m = FineMaps{};
    m->bf16 = bf16;
    m->z = z; m->pa = pa; m->pb = pb; m->x0 = x0; m->r = r; m->x = x;
    const int eoff = bf16 ? 8 : 4;
    m->on = march_encode_box(&m->mz, z, false, d, FW + 8, FH + 2) &&
            march_encode_box(&m->mpa, pa, false, d, FW + 8, FH + 2) &&
            march_encode_box(&m->mpb, pb, false, d, FW + 8, FH + 2) &&
            march_encode_box(&m->mx0, x0, false, d, FW + 8, FH + 2) &&
            march_encode_box(&m->meta, eta, bf16, d, FW + 2 * eoff, FH + 2) &&
            march_encode_box(&m->mr, r, false, d, FW, FH) &&
            march_encode_box(&m->mx, x, false, d, FW, FH);
    return m->on;
}

bool fine_maps_withhold(FineMaps* m, const Dims& d, int pass) {
    if (pass && !march_encode_box(&m->mshort, m->z, false, d, FW + 8, FH + 1)) return false;
    m->withhold = pass;
    return true;
}

void launch_fine_a(const FineMaps& m, const Dims& d, bool in_a, float* p_out, Scalars* sc,
                   double* part, cudaStream_t st) {
    FineArgs a{};
    a.d = d;
    a.o0 = p_out;
    a.sc = sc;
    a.partials = part;
    launch<PASS_A>(m, m.mz, in_a ? m.mpa : m.mpb, m.mr, m.mx, a, st);
}

void launch_fine_b(const FineMaps& m, const Dims& d, bool p_a, float* x, float* r, float* x0,
                   float omega, Scalars* sc, double* part, cudaStream_t st) {
    FineArgs a{};
    a.d = d;
    a.omega = omega;
    a.o0 = x;
    a.o1 = r;
    a.o2 = x0;
    a.sc = sc;
    a.partials = part;
    launch<PASS_B>(m, p_a ? m.mpa : m.mpb, m.mz, m.mx, m.mr, a, st);
}

void launch_fine_restrict(const FineMaps& m, const Dims& d, const Dims& dc, int fz,
                          const float* cdiag, float* rc, float* xc, float omega, const Scalars* sc,
                          cudaStream_t st) {
    FineArgs a{};
    a.d = d;
    a.dc = dc;
    a.fz = fz;
    a.omega = omega;
    a.cdiag = cdiag;
    a.o0 = rc;
    a.o1 = xc;
    a.sc = const_cast<Scalars*>(sc);
    launch<PASS_RESTRICT>(m, m.mx0, m.mz, m.mr, m.mx, a, st);
}

void launch_fine_smooth(const FineMaps& m, const Dims& d, const Dims& dc, int sz, const float* e,
                        float alpha, float omega, float* y, Scalars* sc, double* part, int mode,
                        cudaStream_t st) {
    FineArgs a{};
    a.d = d;
    a.dc = dc;
    a.sz = sz;
    a.e = e;
    a.alpha = alpha;
    a.omega = omega;
    a.o0 = y;
    a.sc = sc;
    a.partials = part;
    a.mode = mode;
    launch<PASS_SMOOTH>(m, m.mx0, m.mz, m.mr, m.mx, a, st);
}

}  // namespace pcg
