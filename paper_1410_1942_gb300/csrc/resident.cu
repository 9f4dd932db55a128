// resident.cu -- Jacobi-preconditioned CG with the whole state of a solve on chip.
//
// A grid whose boxes, one an SM, fit the registers and shared memory is held there: on 152 SMs every
// ship-tank shape (width and depth 0.35 to 0.75 of the length) of up to 0.8 million cells in FP32 and
// 0.5 million in FP64, half of them at 1.0 and 0.55 million, and only shapes that are nearly whole
// boxes up to 1.2 and 0.6 million.  One CTA of 512 threads per SM holds a box of the grid for a whole
// inner solve: a thread owns one x-y column of the box (up to 16 planes in FP32, 8 in FP64) with
// x, p, s^ and w^ in registers; u with a one-cell halo, the three low faces and the diagonal lie
// in shared memory.  The recurrences are the Chronopoulos-Gear form of march1.cu (one reduction
// an iteration).  Nothing is streamed from memory between the first and the last sweep; per
// iteration a CTA exchanges
//   * its three partial sums, and
//   * the w^ of its box's surface cells (the neighbours keep u and s^ of their halo cells by the
//     same recurrences, with the same explicit fused multiply-adds, so both sides hold the same
//     bits).
// Both travel as words that carry the sweep's tag beside the value, stored and loaded whole
// (8 or 16 bytes): a reader polls the word until the tag is the one it waits for.  That is the
// grid barrier: no counter, no fence, one trip through the L2 instead of the three of an atomic
// barrier followed by reading the partial sums.  Words alternate between two buffers by the
// sweep's parity: a CTA writes sweep m + 2 only after every CTA's sums of sweep m + 1, which each
// wrote after it had read sweep m.  Tags are never used twice (ResPlan::next_tag).
//
// In FP64 the operator is scaled to a unit diagonal, D^-1/2 A D^-1/2, once at the start: the
// preconditioned recurrences without a second diagonal array and with one multiplication less
// per cell (the FP64 pipe, two lanes a clock per SM, bounds that kernel); the residual norm that
// stops it is still that of r.  In FP32 the diagonal stays the sum of its own faces: a scaled
// operator would lose the exact weighted-Laplacian rows that keep refinement fast.
//
// What bounds it: FP32, per iteration about 2.4 us of exchange (reduction in the CTA, one trip of
// the words, decision) and 0.3 us per plane of a box (shared-memory loads: eleven a cell); FP64,
// the FP64 pipe (fifteen operations a cell) and the exchange's FP64 additions.  Measured against the
// streamed and column kernels it replaces, us per iteration: FP32 64x48x32 3.5 against 8.3,
// 128x64x64 4.3 against 11.4, 160x96x80 6.7 (182 Gcell-iterations/s) against 15.1, odd 123x55x43
// 4.4 against 34.7; FP64 32^3 7.1 against 18.3, 128x64x64 22.4 against 63 (a solve's time over its
// iterations; inside the launches alone 2.96, 3.93, 6.61, 3.84, 7.2 and 21.8).
//
// The scalars of the FP32 recurrences (alpha, beta, the denominator, the stopping test) are
// float-float, about 2^-44, formed by every thread.  Formed in FP64 by one lane they gave bit for bit
// the same pressure on 120 of 120 random grids, at 0.8 to 2 us more an iteration.
//
// Several solves share one launch: the host gives each a set of CTAs and every CTA a list of
// boxes ordered by one global order of the solves, so no two CTAs wait for each other's later
// solves.  All waits are bounded (RES_WAIT_NS without progress anywhere in the launch) and end the
// launch with the error flag set.
#include "resident.h"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>

#include "alloc.h"
#include "coop.h"
#include "kernels.h"
#include "march_dev.cuh"

namespace pcg {
namespace {

constexpr int RES_T = 512;
constexpr int RES_W = RES_T / 32;
constexpr int RANKS = 160;               // boxes of a solve at most: 5 warps poll their sums

// Most planes per thread (the kernels come for up to 2, 4, 8 and 16 planes: the unrolled code of
// the shallow ones stays in the instruction cache, whose misses cost a box of few planes more than
// its arithmetic), and halo cells per thread of a kernel for up to M planes.
template <typename V> struct ResCfg;
template <> struct ResCfg<float> { static constexpr int M = 16; };
template <> struct ResCfg<double> { static constexpr int M = 8; };
// FP32 boxes are at most FIX_X x FIX_Y cells in x-y and lie in shared memory and in the outbox as
// if they were that large: a thread's addresses then differ by compile-time constants, and the
// sweep's instructions per cell halve (computed addresses were half of them).  FP64, bound by its
// pipe, keeps the pitch of the box and with it any shape of up to 512 columns.
constexpr int FIX_X = 32, FIX_Y = RES_T / FIX_X;
constexpr int halo_slots(int M) { return M > 8 ? 5 : M > 4 ? 4 : 3; }
constexpr int depth_class(int bz) { return bz <= 2 ? 2 : bz <= 4 ? 4 : bz <= 8 ? 8 : 16; }

// A 16-byte word stored and loaded whole.
struct alignas(16) Word {
    unsigned long long v, tag;
};

__device__ __forceinline__ void st_word(Word* p, unsigned long long v, unsigned long long tag) {
    asm volatile("{ .reg .b128 t; mov.b128 t, {%1, %2}; st.relaxed.gpu.global.b128 [%0], t; }" ::"l"(p),
                 "l"(v), "l"(tag)
                 : "memory");
}
__device__ __forceinline__ Word ld_word(const Word* p) {
    Word w;
    asm volatile("{ .reg .b128 t; ld.relaxed.gpu.global.b128 t, [%2]; mov.b128 {%0, %1}, t; }"
                 : "=l"(w.v), "=l"(w.tag)
                 : "l"(p)
                 : "memory");
    return w;
}

// Halo words: a float and a 32-bit tag in 8 bytes, or a double and the tag in 16.
template <typename V> struct Halo;
template <> struct Halo<float> {
    using W = unsigned long long;
    static __device__ __forceinline__ void put(W* p, float v, unsigned tag) {
        const W w = ((W)tag << 32) | __float_as_uint(v);
        asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
    }
    static __device__ __forceinline__ bool get(const W* p, unsigned tag, float& v) {
        W w;
        asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
        v = __uint_as_float((unsigned)w);
        return (unsigned)(w >> 32) == tag;
    }
};
template <> struct Halo<double> {
    using W = Word;
    static __device__ __forceinline__ void put(W* p, double v, unsigned tag) {
        st_word(p, (unsigned long long)__double_as_longlong(v), tag);
    }
    static __device__ __forceinline__ bool get(const W* p, unsigned tag, double& v) {
        const Word w = ld_word(p);
        v = __longlong_as_double((long long)w.v);
        return w.tag == tag;
    }
};

// Sums: float-float for FP32 (march_dev.cuh), doubles for FP64.  The three sums of a box travel
// in a record of whole 32-byte sectors (one in FP32: gamma, delta.hi and the tag; delta.lo, rho and
// the tag; two in FP64: a double and the tag each), which neighbouring lanes store in one
// instruction.  A polled sector written twice, by two CTAs or by two stores of one, made the
// exchange of 152 CTAs take 5600 to 11000 cycles instead of 2340.
template <typename V> struct Sum;
template <> struct Sum<float> {
    using T = ff;
    static constexpr int WORDS = 2, STRIDE = 2, TAG_AT = 3;  // (tag_of's 32 bits of a word)
    static __device__ __forceinline__ ff of(float v) { return ff{v, 0.f}; }
    static __device__ __forceinline__ ff add(ff a, ff b) { return ff_add(a, b); }
    static __device__ __forceinline__ ff shfl(ff v, int m) {
        return ff{__shfl_xor_sync(0xffffffffu, v.hi, m), __shfl_xor_sync(0xffffffffu, v.lo, m)};
    }
    static __device__ __forceinline__ unsigned long long pair(float lo, float hi) {
        return ((unsigned long long)__float_as_uint(hi) << 32) | __float_as_uint(lo);
    }
    // word `lane` of the record
    static __device__ __forceinline__ void put(Word* p, int lane, ff g, ff d, ff r, unsigned tag) {
        const unsigned long long a = lane ? pair(d.lo, r.hi) : pair(g.hi, g.lo);
        st_word(p + lane, a, pair(lane ? r.lo : d.hi, __uint_as_float(tag)));
    }
    static __device__ __forceinline__ ff from_lane(ff v, int l) {
        return ff{__shfl_sync(0xffffffffu, v.hi, l), __shfl_sync(0xffffffffu, v.lo, l)};
    }
    static __device__ __forceinline__ unsigned tag_of(const Word& w) { return (unsigned)(w.tag >> 32); }
    static __device__ __forceinline__ void get(const Word (&w)[WORDS], ff& g, ff& d, ff& r) {
        g = ff{__uint_as_float((unsigned)w[0].v), __uint_as_float((unsigned)(w[0].v >> 32))};
        d = ff{__uint_as_float((unsigned)w[0].tag), __uint_as_float((unsigned)w[1].v)};
        r = ff{__uint_as_float((unsigned)(w[1].v >> 32)), __uint_as_float((unsigned)w[1].tag)};
    }
};
template <> struct Sum<double> {
    using T = double;
    static constexpr int WORDS = 3, STRIDE = 4, TAG_AT = 2;
    static __device__ __forceinline__ double of(double v) { return v; }
    static __device__ __forceinline__ double add(double a, double b) { return a + b; }
    static __device__ __forceinline__ double shfl(double v, int m) {
        return __shfl_xor_sync(0xffffffffu, v, m);
    }
    static __device__ __forceinline__ void put(Word* p, int lane, double g, double d, double r,
                                               unsigned tag) {
        const double v = lane == 0 ? g : lane == 1 ? d : r;
        st_word(p + lane, (unsigned long long)__double_as_longlong(v), tag);
    }
    static __device__ __forceinline__ double from_lane(double v, int l) {
        return __shfl_sync(0xffffffffu, v, l);
    }
    static __device__ __forceinline__ unsigned tag_of(const Word& w) { return (unsigned)w.tag; }
    static __device__ __forceinline__ void get(const Word (&w)[WORDS], double& g, double& d, double& r) {
        g = __longlong_as_double((long long)w[0].v);
        d = __longlong_as_double((long long)w[1].v);
        r = __longlong_as_double((long long)w[2].v);
    }
};

// Warp sums of three values with six additions instead of fifteen: the first two steps also
// split the values over the lanes.  Lane 0 ends with a's sum, lane 8 with b's, lane 16 with c's.
template <typename V>
__device__ __forceinline__ typename Sum<V>::T warp_sum3(typename Sum<V>::T a,
                                                        typename Sum<V>::T b,
                                                        typename Sum<V>::T c, int lane) {
    using S = Sum<V>;
    using T = typename S::T;
    const bool h4 = lane & 16, h3 = lane & 8;
    const T zero = S::of((V)0);
    T k0 = h4 ? c : a, k1 = h4 ? zero : b;
    k0 = S::add(k0, S::shfl(h4 ? a : c, 16));
    k1 = S::add(k1, S::shfl(h4 ? b : zero, 16));
    T r = h3 ? k1 : k0;
    const T o = h3 ? k0 : k1;
    r = S::add(r, S::shfl(o, 8));
    r = S::add(r, S::shfl(r, 4));
    r = S::add(r, S::shfl(r, 2));
    r = S::add(r, S::shfl(r, 1));
    return r;
}

// Float-float product and quotient (Dekker's, with fused multiply-adds for the exact product;
// the quotient by one correction step), about 2^-44 relative.
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, e));
    const float h = __fadd_rn(p, e);
    return ff{h, __fsub_rn(e, __fsub_rn(h, p))};
}
__device__ __forceinline__ ff ff_div(ff a, ff b) {
    const float y = rcp_approx(b.hi);
    const float q = __fmul_rn(a.hi, y);
    float r = __fmaf_rn(-q, b.hi, a.hi);  // exact
    r = __fadd_rn(r, __fmaf_rn(-q, b.lo, a.lo));
    const float q2 = __fmul_rn(r, y);
    const float h = __fadd_rn(q, q2);
    return ff{h, __fsub_rn(q2, __fsub_rn(h, q))};
}

__device__ __forceinline__ bool ff_le(ff a, ff b) {
    return a.hi < b.hi || (a.hi == b.hi && a.lo <= b.lo);
}

template <typename Coef> __device__ __forceinline__ Coef coef_of(const ResSolve& s);
template <> __device__ __forceinline__ CoefEta<float> coef_of(const ResSolve& s) {
    return CoefEta<float>{(const float*)s.c[0]};
}
template <> __device__ __forceinline__ CoefEta<__nv_bfloat16> coef_of(const ResSolve& s) {
    return CoefEta<__nv_bfloat16>{(const __nv_bfloat16*)s.c[0]};
}
template <> __device__ __forceinline__ CoefFaces32 coef_of(const ResSolve& s) {
    return CoefFaces32{(const float*)s.c[0], (const float*)s.c[1], (const float*)s.c[2],
                       (const float*)s.c[3]};
}
template <> __device__ __forceinline__ CoefFaces64 coef_of(const ResSolve& s) {
    return CoefFaces64{(const double*)s.c[0], (const double*)s.c[1], (const double*)s.c[2],
                       (const double*)s.c[3], nullptr};
}

// 1/D (FP32: r -> u) or D^-1/2 (FP64: r -> u of the scaled system)
__device__ __forceinline__ float inv_of(float D) { return rcp_approx(D); }
__device__ __forceinline__ double inv_of(double D) { return 1.0 / sqrt(D); }

__device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return __fma_rn(a, b, c); }

// Bounded poll bookkeeping: false once the deadline has passed or another CTA has given up.
struct Deadline {
    unsigned spins = 0, seen = 0;
    unsigned long long t0 = 0;
    __device__ __forceinline__ bool more(int* error, unsigned long long limit) {
        if (__builtin_expect((++spins & 63u) != 0, 1)) return true;
        if (*(volatile int*)error) return false;
        const unsigned long long t = globaltimer();
        if (!t0) t0 = t;
        if (__builtin_expect(t - t0 <= limit, 1)) return true;
        atomicExch(error, 1);
        return false;
    }
    // The wait for a box's sums: the box may belong to a CTA that is still in an earlier solve of its
    // list, which is no fault however long it takes.  It gives up only when no solve of the launch
    // has begun a sweep during the second half of the limit, as the tags of their first boxes' sums
    // tell.  The iteration caps bound the whole.
    template <typename V>
    __device__ __forceinline__ bool more_queued(const ResArgs& a, unsigned long long limit) {
        if (__builtin_expect((++spins & 63u) != 0, 1)) return true;
        if (*(volatile int*)a.error) return false;
        const unsigned long long t = globaltimer();
        if (!t0) t0 = t;
        if (__builtin_expect(t - t0 <= limit / 2, 1)) return true;
        unsigned now = 1;
#pragma unroll 1
        for (int q = 0; q < 2 * a.nsolves; ++q)  // both parities
            now += ((const volatile unsigned*)a.sums)[4 * (size_t)RANKS * Sum<V>::STRIDE * q +
                                                      Sum<V>::TAG_AT];
        if (seen && now == seen) {
            atomicExch(a.error, 1);
            return false;
        }
        seen = now;
        t0 = t;
        return true;
    }
};

// The words of an outbox: faces -x, +x (wy x pz each), -y, +y (wx x pz), -z, +z (wx x wy).
struct OutFaces {
    int xp, ym, yp, zm, zp, words;
    __host__ __device__ OutFaces(int wx, int wy, int pz)
        : xp(wy * pz), ym(2 * wy * pz), yp(ym + wx * pz), zm(ym + 2 * wx * pz), zp(zm + wx * wy),
          words(zm + 2 * wx * wy) {}
};

template <typename V, typename Coef, int M>
__global__ void __launch_bounds__(RES_T, 1) k_res(ResArgs a) {
    using S = Sum<V>;
    using T = typename S::T;
    using HW = Halo<V>;
    constexpr int HQ = halo_slots(M);
    constexpr bool DBL = std::is_same<V, double>::value;
    constexpr bool FIX = !DBL;
    // deep FP32 boxes pass the words of their x and y faces through shared memory, so that all
    // threads store them: by the columns at the edges alone, plane after plane, they took as long as
    // the sweep (4000 of 18000 cycles at 32 x 16 x 16 cells)
    constexpr bool STAGE = FIX && M > 4;
    constexpr int STG = STAGE ? 2 * M * (FIX_X + FIX_Y) : 1;
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ float stage[STG];  // the outbox's x and y faces
    __shared__ T red[RES_W][3];
    __shared__ T tot[RANKS / 32][3];
    __shared__ double s_dec[2];
    __shared__ ff s_stop;  // FP32: stop when r.r is at most this
    __shared__ int s_state, s_iter;
    // A wait that ran out: for a sum, written before the decision's barrier and read after it; for a
    // halo word, written after that barrier and read after the sweep's last one.  One flag for
    // both could be set by a late halo poll while slower warps still read it after the decision,
    // and part of the CTA would leave while the rest waits at a barrier.
    __shared__ volatile int s_fail, s_late;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        s_fail = 0;
        s_late = 0;
    }
    for (int it = a.cta_task[blockIdx.x]; it < a.cta_task[blockIdx.x + 1]; ++it) {
        const ResTask& tk = a.tasks[it];
        const ResSolve& sv = a.solves[tk.solve];
        if (!sv.active) {
            if (tk.rank == 0 && tid == 0) {
                sv.sc->done = CONVERGED;
                sv.sc->iter = 0;
            }
            continue;
        }
        __syncthreads();  // the shared arrays of the last box are no longer read
        const Dims d = sv.d;
        const int bx = tk.bx, by = tk.by, bz = tk.bz;
        const int sx = FIX ? FIX_X + 2 : bx + 2, sxy = FIX ? (FIX_X + 2) * (FIX_Y + 2) : sx * (by + 2);
        const int pz = FIX ? M : bz;                               // planes laid out
        const int wx = FIX ? FIX_X : bx, wy = FIX ? FIX_Y : by;    // columns laid out
        // u: all planes with halo; faces and D: the planes 1 .. bz (fz one more), addressed with
        // the same index (their pointers start one plane early)
        V* const u = reinterpret_cast<V*>(dyn);
        V* const fx = u + sxy * (pz + 2) - sxy;
        V* const fy = fx + sxy * pz;
        V* const fz = fy + sxy * pz;
        V* const Ds = fz + sxy * (pz + 1);
        for (int q = tid; q < sxy * (5 * pz + 3); q += RES_T) u[q] = (V)0;
        __syncthreads();
        const int ti = tid % wx, tj = tid / wx;
        const bool act = ti < bx && tj < by;
        const int li = act ? ti : 0, lj = act ? tj : 0;
        const int gi = tk.x0 + li, gj = tk.y0 + lj;
        const int o = (li + 1) + sx * (lj + 1) + sxy;  // plane m of the column: o + m sxy
        const int c0 = gi + d.nx * (gj + d.ny * tk.z0);
        const Coef coef = coef_of<Coef>(sv);
        const bool per = d.walls & PERIODIC_X;
        // FP32: r scaled by a power of two so that its norm is near one (sums of squares of a
        // small residual would leave the FP32 range); x is scaled back
        V scale = (V)1, unscale = (V)1;
        if (!DBL) {
            const double rr = sv.sc->rr;
            if (rr > 0.0 && isfinite(rr)) {
                const int e = max(-120, min(120, ilogb(rr) / 2));
                scale = (V)scalbnf(1.f, -e);
                unscale = (V)scalbnf(1.f, e);
            }
        }
        const V* const rg = reinterpret_cast<const V*>(sv.r);
        V x[M], p[M], s[M], w[M];
#pragma unroll
        for (int m = 0; m < M; ++m) { x[m] = (V)0; p[m] = (V)0; s[m] = (V)0; w[m] = (V)0; }
        if (act)
            for (int m = 0; m < bz; ++m) {
                const int c = c0 + m * d.sxy, q = o + m * sxy, gk = tk.z0 + m;
                Stencil<V> st;
                coef.weights(d, c, gi, gj, gk, st);
                fx[q] = (gi > 0 || per) ? st.xm : (V)0;
                if (li == bx - 1) fx[q + 1] = (gi + 1 < d.nx || per) ? st.xp : (V)0;
                fy[q] = gj > 0 ? st.ym : (V)0;
                if (lj == by - 1) fy[q + sx] = gj + 1 < d.ny ? st.yp : (V)0;
                fz[q] = gk > 0 ? st.zm : (V)0;
                if (m == bz - 1) fz[q + sxy] = gk + 1 < d.nz ? st.zp : (V)0;
                Ds[q] = st.D;
                u[q] = DBL ? inv_of(st.D) : rg[c] * scale * inv_of(st.D);
            }
        // the halo cells of this thread: shared index, outbox word, s^ of the cell
        int hoff[HQ], hsrc[HQ];
        unsigned has = 0;  // bit q: slot q holds a cell
        V hs[HQ], hr[HQ];
        {
            const int nyz = by * bz, nxz = bx * bz, nxy = bx * by;
            const int nh = 2 * (nyz + nxz + nxy);
#pragma unroll
            for (int q = 0; q < HQ; ++q) {
                hoff[q] = 0;
                hsrc[q] = 0;
                hs[q] = (V)0;
                hr[q] = (V)0;
                int h = tid + q * RES_T;
                if (h >= nh) continue;
                int f, i, j, k;
                if (h < 2 * nyz) {
                    f = h >= nyz;
                    h -= f * nyz;
                    j = h % by; k = h / by; i = f ? bx : -1;
                    h = j + wy * k;
                } else if ((h -= 2 * nyz) < 2 * nxz) {
                    f = h >= nxz;
                    h -= f * nxz;
                    i = h % bx; k = h / bx; j = f ? by : -1;
                    h = i + wx * k;
                    f += 2;
                } else {
                    h -= 2 * nxz;
                    f = h >= nxy;
                    h -= f * nxy;
                    i = h % bx; j = h / bx; k = f ? bz : -1;
                    h = i + wx * j;
                    f += 4;
                }
                if (tk.src[f] < 0) continue;
                hoff[q] = (i + 1) + sx * (j + 1) + sxy * (k + 1);
                hsrc[q] = tk.src[f] + h;
                has |= 1u << q;
                int ci = tk.x0 + i;
                if (ci < 0) ci += d.nx;
                else if (ci >= d.nx) ci -= d.nx;
                const int cj = tk.y0 + j, ck = tk.z0 + k;
                const int c = ci + d.nx * (cj + d.ny * ck);
                Stencil<V> st;
                coef.weights(d, c, ci, cj, ck, st);
                if (DBL) {
                    hr[q] = rg[c];
                    u[hoff[q]] = inv_of(st.D);
                } else {
                    u[hoff[q]] = rg[c] * scale * inv_of(st.D);
                }
            }
        }
        __syncthreads();
        if (DBL) {
            // u holds D^-1/2: scale the faces (the product of the two square roots first, so that
            // the two boxes of a shared face round it alike), then u = D^-1/2 r
            if (act)
                for (int m = 0; m < bz; ++m) {
                    const int q = o + m * sxy;
                    fx[q] *= u[q] * u[q - 1];
                    if (li == bx - 1) fx[q + 1] *= u[q] * u[q + 1];
                    fy[q] *= u[q] * u[q - sx];
                    if (lj == by - 1) fy[q + sx] *= u[q] * u[q + sx];
                    fz[q] *= u[q] * u[q - sxy];
                    if (m == bz - 1) fz[q + sxy] *= u[q] * u[q + sxy];
                }
            __syncthreads();
            if (act)
                for (int m = 0; m < bz; ++m) u[o + m * sxy] *= rg[c0 + m * d.sxy];
#pragma unroll
            for (int q = 0; q < HQ; ++q)
                if (has & (1u << q)) u[hoff[q]] *= hr[q];
            __syncthreads();
        }
        Word* const sums = reinterpret_cast<Word*>(a.sums) +
                           (size_t)2 * RANKS * S::STRIDE * tk.solve;
        typename HW::W* const boxes = reinterpret_cast<typename HW::W*>(a.outbox);
        const size_t half = (size_t)gridDim.x * a.box_words;  // words of one parity
        typename HW::W* const mine = boxes + (size_t)blockIdx.x * a.box_words;
        // own outbox (a box one cell wide keeps one face of the two): a column at the box's edge in
        // x or y has its words at stride wy or wx
        const OutFaces of(wx, wy, pz);
        const int oxp = of.xp, oym = of.ym, oyp = of.yp, ozm = of.zm, ozp = of.zp;
        const int px = !act ? -1 : li == 0 ? lj : li == bx - 1 ? oxp + lj : -1;
        const int py = !act ? -1 : lj == 0 ? oym + li : lj == by - 1 ? oyp + li : -1;
        const int nwait = sv.ctas + (a.extra > 0 ? 1 : 0);
        // scalars: in FP32 every thread holds them (float-float); in FP64 warp 0 decides
        T gam = S::of((V)0), den = S::of((V)0);
        V al = (V)0, be = (V)0;
        bool first = true;
        int iter = 0, state = RUNNING;
        double rr_out = 0.0, rz_out = 0.0;
        unsigned tag = sv.tag0;
        const double tol2 = sv.tol2;
        const int max_iter = sv.max_iter;
        if (DBL && tid == 0) s_iter = 0;
        for (;;) {
            ++tag;
            const unsigned par = tag & 1u;
            // w^ = M^-1 A u and the three sums
            V sg = (V)0, sd = (V)0, sr = (V)0;
            typename HW::W* const out = mine + par * half;
            if (act) {
                V um = u[o - sxy], uc = u[o], fzl = fz[o], wl = (V)0;
                // two planes at a time: their chains overlap (FP32; an odd last plane's twin has
                // its q and so its sums zeroed)
                constexpr int STEP = DBL ? 1 : 2;
#pragma unroll
                for (int m0 = 0; m0 < M; m0 += STEP) {
                    if (m0 < bz) {
#pragma unroll
                        for (int m = m0; m < m0 + STEP; ++m) {
                            const int q = o + m * sxy;
                            const V up = u[q + sxy], fzh = fz[q + sxy];
                            V t = fx[q] * u[q - 1];
                            t = fma_(fx[q + 1], u[q + 1], t);
                            t = fma_(fy[q], u[q - sx], t);
                            t = fma_(fy[q + sx], u[q + sx], t);
                            t = fma_(fzl, um, t);
                            t = fma_(fzh, up, t);
                            if (DBL) {
                                wl = uc - t;
                                sg = fma_(uc, uc, sg);
                                sd = fma_(wl, uc, sd);
                                sr = fma_(Ds[q] * uc, uc, sr);
                                w[m] = wl;
                            } else {
                                const V D = Ds[q];
                                const V du = D * uc;
                                V qv = fma_(D, uc, -t);
                                const bool in = m == m0 || m < bz;
                                if (!in) qv = (V)0;
                                w[m] = qv * (V)inv_of(D);
                                if (in) wl = w[m];
                                sg = fma_(du, uc, sg);
                                sd = fma_(qv, uc, sd);
                                sr = fma_(du, du, sr);
                            }
                            um = uc;
                            uc = up;
                            fzl = fzh;
                        }
                    }
                }
                // the surface cells of the box, for the neighbours' halos
                HW::put(out + ozm + tid, w[0], tag);
                if (bz > 1) HW::put(out + ozp + tid, wl, tag);
                if (px >= 0) {
#pragma unroll
                    for (int m = 0; m < M; ++m) {
                        if constexpr (STAGE) stage[px + wy * m] = (float)w[m];
                        else if (m < bz) HW::put(out + px + wy * m, w[m], tag);
                    }
                }
                if (py >= 0) {
#pragma unroll
                    for (int m = 0; m < M; ++m) {
                        if constexpr (STAGE) stage[py + wx * m] = (float)w[m];
                        else if (m < bz) HW::put(out + py + wx * m, w[m], tag);
                    }
                }
            }
            if (FIX ? warp < by : 32 * warp < bx * by) {
                const T v = warp_sum3<V>(S::of(sg), S::of(sd), S::of(sr), lane);
                if ((lane & 7) == 0 && lane < 24) red[warp][lane >> 3] = v;
            } else if (lane < 3) {
                red[warp][lane] = S::of((V)0);
            }
            __syncthreads();
            if constexpr (STAGE)
                for (int q = tid; q < STG; q += RES_T) HW::put(out + q, (V)stage[q], tag);
            Word* const sw = sums + par * RANKS * S::STRIDE;
            if (warp == 0) {
                // lanes 8 v .. 8 v + 7 add value v of the sixteen warps
                const int v = min(lane >> 3, 2), b = lane & 7;
                T t = S::add(red[b][v], red[b + 8][v]);
                t = S::add(t, S::shfl(t, 4));
                t = S::add(t, S::shfl(t, 2));
                t = S::add(t, S::shfl(t, 1));
                const T tg = S::from_lane(t, 0), td = S::from_lane(t, 8), tr = S::from_lane(t, 16);
                if (lane < S::WORDS) S::put(sw + tk.rank * S::STRIDE, lane, tg, td, tr, tag);
            }
            // x of the sweep before, in the shadow of the exchange
            if (act) {
#pragma unroll
                for (int m = 0; m < M; ++m)
                    if (m < bz) x[m] = fma_(al, p[m], x[m]);
            }
            // The neighbours' halo words: the warps that do not poll sums try for them meanwhile, the
            // others after their sums.  What is late then is polled after the decision: only then
            // is it certain that the neighbour stays in the solve and does not write over them.
            V hw[HQ];
            unsigned late = has;
            auto get_halo = [&](unsigned which) {
                unsigned miss = 0;
#pragma unroll
                for (int q = 0; q < HQ; ++q)
                    if ((which & (1u << q)) && !HW::get(boxes + par * half + hsrc[q], tag, hw[q]))
                        miss |= 1u << q;
                return miss;
            };
#pragma unroll
            for (int q = 0; q < HQ; ++q) hw[q] = (V)0;
            if (warp == 0 || 32 * (warp - 1) >= nwait)
                for (int t = 0; t < 3 && late; ++t) late = get_halo(late);
            // the sums of every box: one lane of warps 1 .. 5 each, added per warp
            if (warp >= 1 && 32 * (warp - 1) < nwait) {
                const int rank = tid - 32;
                T t0 = S::of((V)0), t1 = t0, t2 = t0;
                if (rank < nwait) {
                    const Word* const wv = sw + rank * S::STRIDE;
                    Word wd[S::WORDS];
                    Deadline dl;
                    for (;;) {
                        bool all = true;
#pragma unroll
                        for (int q = 0; q < S::WORDS; ++q) wd[q] = ld_word(wv + q);
#pragma unroll
                        for (int q = 0; q < S::WORDS; ++q) all = all && S::tag_of(wd[q]) == tag;
                        if (all) break;
                        if (!dl.more_queued<V>(a, a.wait_ns)) { s_fail = 1; break; }
                    }
                    S::get(wd, t0, t1, t2);
                }
                __syncwarp();
                const T t = warp_sum3<V>(t0, t1, t2, lane);
                if ((lane & 7) == 0 && lane < 24) tot[warp - 1][lane >> 3] = t;
            }
            __syncthreads();
            if (s_fail) { state = TIMEDOUT; break; }
            // (in flight during the decision)
            if (late) late = get_halo(late);
            if constexpr (!DBL) {
                ff g = tot[0][0], dl = tot[0][1], r = tot[0][2];
                const ff stop_at = s_stop;  // (set by the first decision)
                for (int q = 1; 32 * q < nwait; ++q) {
                    g = ff_add(g, tot[q][0]);
                    dl = ff_add(dl, tot[q][1]);
                    r = ff_add(r, tot[q][2]);
                }
                rr_out = r.hi;
                rz_out = g.hi;
                if (!isfinite(g.hi) || !isfinite(dl.hi) || !isfinite(r.hi) || g.hi < 0.f) {
                    if (!first) ++iter;
                    state = BREAKDOWN;
                } else if (first) {
                    first = false;
                    const float th = (float)tol2;
                    const ff stop = ff_mul(ff{th, (float)(tol2 - (double)th)}, r);
                    if (tid == 0) s_stop = stop;
                    gam = g;
                    if (ff_le(r, stop)) state = CONVERGED;
                    else if (!(dl.hi > 0.f)) state = BREAKDOWN;
                    else {
                        den = dl;
                        al = ff_div(g, dl).hi;
                        be = 0.f;
                    }
                } else {
                    ++iter;
                    if (ff_le(r, stop_at)) state = CONVERGED;
                    else if (iter >= max_iter) state = CAPPED;
                    else {
                        // beta = gamma'/gamma, alpha = gamma' / (delta' - beta^2 den)
                        const ff b = ff_div(g, gam);
                        const ff bd = ff_mul(ff_mul(b, b), den);
                        const ff dn = ff_add(dl, ff{-bd.hi, -bd.lo});
                        if (!(dn.hi > 0.f) || !isfinite(dn.hi)) state = BREAKDOWN;
                        else {
                            be = b.hi;
                            al = ff_div(g, dn).hi;
                            gam = g;
                            den = dn;
                        }
                    }
                }
            } else {
                if (warp == 0) {
                    double t = 0.0;
                    if (lane < 3)
                        for (int q = 0; 32 * q < nwait; ++q) t += tot[q][lane];
                    const double g = __shfl_sync(0xffffffffu, t, 0);
                    const double dl = __shfl_sync(0xffffffffu, t, 1);
                    const double r = __shfl_sync(0xffffffffu, t, 2);
                    if (lane == 0) {
                        int st = RUNNING;
                        double na = 0.0, nb = 0.0;
                        const double ginv = 1.0 / g;  // for the next decision: overlaps the rest
                        if (!isfinite(g) || !isfinite(dl) || !isfinite(r) || g < 0.0) {
                            if (!first) s_iter += 1;
                            st = BREAKDOWN;
                        } else if (first) {
                            gam = ginv;
                            if (r <= tol2 * sv.sc->bb) st = CONVERGED;
                            else if (!(dl > 0.0)) st = BREAKDOWN;
                            else {
                                den = dl;
                                na = g / dl;
                            }
                        } else {
                            s_iter += 1;
                            if (r <= tol2 * sv.sc->bb) st = CONVERGED;
                            else if (s_iter >= max_iter) st = CAPPED;
                            else {
                                nb = g * gam;  // (gam: 1/gamma of the sweep before)
                                const double dn = fma(-nb * nb, den, dl);
                                if (!(dn > 0.0) || !isfinite(dn)) st = BREAKDOWN;
                                else {
                                    na = g / dn;
                                    gam = ginv;
                                    den = dn;
                                }
                            }
                        }
                        rr_out = r;
                        rz_out = g;
                        s_dec[0] = na;
                        s_dec[1] = nb;
                        s_state = st;
                    }
                }
                first = false;
                __syncthreads();
                al = s_dec[0];
                be = s_dec[1];
                state = s_state;
            }
            if (state != RUNNING) break;
            // p, s^, u of the own cells and u, s^ of the halo cells
            if (act) {
                constexpr int STEP = M < 4 ? M : DBL ? 2 : 4;  // planes whose loads overlap
#pragma unroll
                for (int m0 = 0; m0 < M; m0 += STEP) {
                    if (m0 < bz) {
                        V uo[STEP];
#pragma unroll
                        for (int e = 0; e < STEP; ++e) uo[e] = m0 + e < bz ? u[o + (m0 + e) * sxy] : (V)0;
#pragma unroll
                        for (int e = 0; e < STEP; ++e) {
                            const int m = m0 + e;
                            p[m] = fma_(be, p[m], uo[e]);
                            s[m] = fma_(be, s[m], w[m]);
                            uo[e] = fma_(-al, s[m], uo[e]);
                        }
#pragma unroll
                        for (int e = 0; e < STEP; ++e)
                            if (m0 + e < bz) u[o + (m0 + e) * sxy] = uo[e];
                    }
                }
            }
            if (late) {
                Deadline dl;
                while ((late = get_halo(late)) != 0)
                    if (!dl.more(a.error, a.wait_ns)) { s_late = 1; break; }
            }
#pragma unroll
            for (int q = 0; q < HQ; ++q) {
                if (has & (1u << q)) {
                    hs[q] = fma_(be, hs[q], hw[q]);
                    u[hoff[q]] = fma_(-al, hs[q], u[hoff[q]]);
                }
            }
            __syncthreads();
            if (s_late) { state = TIMEDOUT; break; }
        }
        // the correction and the scalars
        V* const xg = reinterpret_cast<V*>(sv.x);
        if (act) {
#pragma unroll
            for (int m = 0; m < M; ++m)
                if (m < bz) {
                    const int c = c0 + m * d.sxy;
                    if (DBL) xg[c] = fma_(inv_of(Ds[o + m * sxy]), x[m], xg[c]);
                    else xg[c] = x[m] * unscale;
                }
        }
        if (tk.rank == 0 && tid == 0) {
            const double us = (double)unscale * (double)unscale;
            sv.sc->iter = DBL ? s_iter : iter;
            sv.sc->rr = rr_out * us;
            sv.sc->rz = rz_out * us;
            sv.sc->done = state;
        }
        if (state == TIMEDOUT) {
            // this CTA's remaining solves never started: they end the same way
            for (int q = it + 1; q < a.cta_task[blockIdx.x + 1]; ++q)
                if (a.tasks[q].rank == 0 && tid == 0 && a.solves[a.tasks[q].solve].active) {
                    a.solves[a.tasks[q].solve].sc->iter = 0;
                    a.solves[a.tasks[q].solve].sc->done = TIMEDOUT;
                }
            return;
        }
    }
}

// ------------------------------------------------------------------ host side
constexpr size_t SMEM_MAX = 227 * 1024 - 2048;  // dynamic, beside the static arrays
constexpr size_t smem_fix(int depth) {  // an FP32 box of the kernel for `depth` planes
    return sizeof(float) * (FIX_X + 2) * (FIX_Y + 2) * (5 * (size_t)depth + 3);
}
static_assert(smem_fix(ResCfg<float>::M) + 4 * 2 * ResCfg<float>::M * (FIX_X + FIX_Y) <= SMEM_MAX,
              "the deepest FP32 box and its staging fit");

int sm_count() {
    static const int n = [] {
        int dev = 0, m = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&m, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            m = 0;
        }
        return m;
    }();
    return n;
}

inline int ceil_div(int a, int b) { return (a + b - 1) / b; }

struct Tiling {
    int tx = 0, ty = 0, tz = 0;
    double time = 0.0;  // estimated SM cycles of an iteration
    int ctas() const { return tx * ty * tz; }
};

// The split of a grid into at most `most` boxes with the least estimated time of an iteration.
// In SM cycles: 6000 for the exchange (polling, reductions, decision), 4 per box polled, 250 per
// plane (a thread's chain through one), per 32 cells 20 (FP32: shared-memory loads) or 240 (FP64:
// the FP64 pipe), per halo cell 1.
// throughput: the split of least time x boxes instead (many solves that queue for the SMs).
Tiling choose_tiling(const Dims& d, bool dbl, int most, bool throughput) {
    const int M = dbl ? ResCfg<double>::M : ResCfg<float>::M;
    const size_t es = dbl ? 8 : 4;
    most = std::min(most, RES_MAX_CTAS);
    Tiling best;
    double least = 0.0;
    int last_bx = 0;
    for (int tx = 1; tx <= std::min(d.nx, most); ++tx) {
        const int bx = ceil_div(d.nx, tx);
        if (bx == last_bx) continue;  // the same boxes, one of them empty or smaller
        last_bx = bx;
        int last_by = 0;
        for (int ty = 1; ty <= std::min(d.ny, most / tx); ++ty) {
            const int by = ceil_div(d.ny, ty);
            if (by == last_by) continue;
            last_by = by;
            if (dbl ? bx * by > RES_T : bx > FIX_X || by > FIX_Y) continue;
            int last_bz = 0;
            for (int tz = ceil_div(d.nz, M); tz <= std::min(d.nz, most / (tx * ty)); ++tz) {
                const int bz = ceil_div(d.nz, tz);
                if (bz == last_bz) continue;
                last_bz = bz;
                const int nh = 2 * (by * bz + bx * bz + bx * by);
                if (nh > halo_slots(depth_class(bz)) * RES_T) continue;
                if (dbl && es * (size_t)(bx + 2) * (by + 2) * (5 * bz + 3) > SMEM_MAX) continue;
                const int n = tx * ty * tz;
                const double t = 6000.0 + 4.0 * n + 250.0 * bz +
                                 (dbl ? ceil_div(bx * by, 32) * bz * 240.0 : by * bz * 20.0) + 1.0 * nh;
                const double k = throughput ? t * n : t;
                if (!best.tx || k < least) {
                    least = k;
                    best.tx = tx;
                    best.ty = ty;
                    best.tz = tz;
                    best.time = t;
                }
            }
        }
    }
    return best;
}

// Low end of part q of n cells cut into t nearly equal parts (the first n % t one longer).
inline int part_lo(int n, int t, int q) { return q * (n / t) + std::min(q, n % t); }

struct Built {
    std::vector<ResTask> tasks;  // grouped by CTA
    std::vector<int> cta_task;
    std::vector<int> ctas;       // boxes per solve
    int box_words = 0, depth = 0;
};

// Boxes and schedule.  One solve: the tiling of least time.  Several: tilings of least SM time,
// solves in decreasing order of work, each on the CTAs that come free first.
bool build(const Dims* d, int n, bool dbl, Built* out) {
    const int sms = std::min(sm_count(), RES_MAX_CTAS);
    if (sms <= 0) return false;
    std::vector<Tiling> tl(n);
    // iterations grow with the longest side
    auto len = [&](int q) { return (double)std::max(d[q].nx, std::max(d[q].ny, d[q].nz)); };
    for (int pass = 0; pass < 2; ++pass) {
        long long all = 0;
        for (int q = 0; q < n; ++q) {
            tl[q] = choose_tiling(d[q], dbl, sms, n > 1 && pass == 1);
            if (!tl[q].tx) return false;
            all += tl[q].ctas();
        }
        if (n == 1 || all <= sms) break;  // every solve at its fastest, all at once
    }
    if (n > 1) {
        // few solves that do not fill the GPU at their least SM time: widen the largest boxes
        for (;;) {
            long long all = 0;
            for (auto& t : tl) all += t.ctas();
            if (all >= sms) break;
            int slow = 0;
            for (int q = 1; q < n; ++q)
                if (tl[q].time * len(q) > tl[slow].time * len(slow)) slow = q;
            Tiling t = choose_tiling(d[slow], dbl, tl[slow].ctas() + (int)(sms - all), false);
            if (!t.tx || t.ctas() <= tl[slow].ctas()) break;
            if (t.time >= tl[slow].time) break;
            tl[slow] = t;
        }
    }
    out->depth = 2;
    for (int q = 0; q < n; ++q)
        out->depth = std::max(out->depth, depth_class(ceil_div(d[q].nz, tl[q].tz)));
    const int depth = out->depth;
    std::vector<int> order(n);
    std::vector<double> work(n);
    for (int q = 0; q < n; ++q) {
        order[q] = q;
        work[q] = len(q) * tl[q].time;
    }
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
        return work[a] * tl[a].ctas() > work[b] * tl[b].ctas();
    });
    std::vector<double> free_at(sms, 0.0);
    std::vector<std::vector<ResTask>> lists(sms);
    out->ctas.assign(n, 0);
    int words = dbl ? 0 : OutFaces(FIX_X, FIX_Y, depth).words, used = 0;
    for (int q : order) {
        const Tiling& t = tl[q];
        const int G = t.ctas();
        std::vector<int> c(sms);
        for (int i = 0; i < sms; ++i) c[i] = i;
        std::stable_sort(c.begin(), c.end(), [&](int a, int b) { return free_at[a] < free_at[b]; });
        c.resize(G);
        std::sort(c.begin(), c.end());
        double start = 0.0;
        for (int i : c) start = std::max(start, free_at[i]);
        for (int i : c) free_at[i] = start + work[q];
        out->ctas[q] = G;
        const bool per = d[q].walls & PERIODIC_X;
        for (int kz = 0; kz < t.tz; ++kz)
            for (int jy = 0; jy < t.ty; ++jy)
                for (int ix = 0; ix < t.tx; ++ix) {
                    ResTask k{};
                    k.solve = q;
                    k.x0 = part_lo(d[q].nx, t.tx, ix);
                    k.y0 = part_lo(d[q].ny, t.ty, jy);
                    k.z0 = part_lo(d[q].nz, t.tz, kz);
                    k.bx = part_lo(d[q].nx, t.tx, ix + 1) - k.x0;
                    k.by = part_lo(d[q].ny, t.ty, jy + 1) - k.y0;
                    k.bz = part_lo(d[q].nz, t.tz, kz + 1) - k.z0;
                    k.rank = ix + t.tx * (jy + t.ty * kz);
                    for (int f = 0; f < 6; ++f) {
                        int nx = ix, ny = jy, nz = kz;
                        (f < 2 ? nx : f < 4 ? ny : nz) += (f & 1) ? 1 : -1;
                        if (per && f < 2) nx = (nx + t.tx) % t.tx;
                        k.src[f] = (nx < 0 || ny < 0 || nz < 0 || nx >= t.tx || ny >= t.ty || nz >= t.tz)
                                       ? -1
                                       : nx + t.tx * (ny + t.ty * nz);  // rank; word offset below
                    }
                    lists[c[k.rank]].push_back(k);
                    if (dbl) words = std::max(words, OutFaces(k.bx, k.by, k.bz).words);
                }
        for (int i : c) {
            ResTask& k = lists[i].back();
            for (int f = 0; f < 6; ++f) {
                if (k.src[f] < 0) continue;
                const int r = k.src[f];
                const ResTask& b = lists[c[r]].back();
                // the neighbour's outbox: its face opposite to f
                const OutFaces of = dbl ? OutFaces(b.bx, b.by, b.bz) : OutFaces(FIX_X, FIX_Y, depth);
                const int off[6] = {b.bx > 1 ? of.xp : 0,     0,     b.by > 1 ? of.yp : of.ym, of.ym,
                                    b.bz > 1 ? of.zp : of.zm, of.zm};
                // (the CTA's outbox offset is added once box_words is known)
                k.src[f] = off[f] + (c[r] << 16);
            }
        }
        used = std::max(used, c.back() + 1);
    }
    out->box_words = words;
    out->tasks.clear();
    out->cta_task.clear();
    for (int i = 0; i < used; ++i) {
        out->cta_task.push_back((int)out->tasks.size());
        for (ResTask k : lists[i]) {
            for (int f = 0; f < 6; ++f)
                if (k.src[f] >= 0) k.src[f] = (k.src[f] >> 16) * words + (k.src[f] & 0xffff);
            out->tasks.push_back(k);
        }
    }
    out->cta_task.push_back((int)out->tasks.size());
    return true;
}

size_t bytes_sums(int nsolves, bool dbl) {
    return sizeof(Word) * 2 * RANKS * (size_t)nsolves * (dbl ? Sum<double>::STRIDE : Sum<float>::STRIDE);
}
size_t bytes_out(const Built& b, bool dbl) {
    return (dbl ? 16 : 8) * 2 * (size_t)b.box_words * (b.cta_task.size() - 1);
}

// The parts of a plan's allocation.
struct Parts {
    size_t solves, tasks, cta, error, sums, outbox, bytes;
    Parts(const Built& b, int n, bool dbl) {
        size_t at = 0;
        auto take = [&](size_t bytes) {
            const size_t p = at;
            at += (bytes + 255) & ~(size_t)255;
            return p;
        };
        solves = take(sizeof(ResSolve) * n);
        tasks = take(sizeof(ResTask) * b.tasks.size());
        cta = take(sizeof(int) * b.cta_task.size());
        error = take(sizeof(int));
        sums = take(bytes_sums(n, dbl));
        outbox = take(bytes_out(b, dbl));
        bytes = at;
    }
};

template <typename V, typename Coef>
const void* kernel_for(int depth) {
    switch (depth) {
        case 2: return (const void*)k_res<V, Coef, 2>;
        case 4: return (const void*)k_res<V, Coef, 4>;
        case 8: return (const void*)k_res<V, Coef, 8>;
        default: return (const void*)k_res<V, Coef, ResCfg<V>::M>;
    }
}
const void* kernel_of(ResKind kind, int depth) {
    switch (kind) {
        case RES_ETA32: return kernel_for<float, CoefEta<float>>(depth);
        case RES_ETA16: return kernel_for<float, CoefEta<__nv_bfloat16>>(depth);
        case RES_FACES32: return kernel_for<float, CoefFaces32>(depth);
        default: return kernel_for<double, CoefFaces64>(depth);
    }
}

}  // namespace

bool res_supported(const Dims& d, bool dbl) {
    return sm_count() > 0 && choose_tiling(d, dbl, std::min(sm_count(), RES_MAX_CTAS), false).tx > 0;
}

size_t res_plan_bytes(const Dims& d, bool dbl) {
    Built b;
    return build(&d, 1, dbl, &b) ? Parts(b, 1, dbl).bytes : 0;
}

size_t res_plan_held(const ResPlan& p) { return p.cap; }

void res_plan_free(ResPlan* p) {
    if (p->mem) lib_free(p->mem);
    *p = ResPlan{};
}

int res_plan_build(ResPlan* p, ResSolve* solves, int n, bool dbl, cudaStream_t st) {
    std::vector<Dims> d(n);
    for (int q = 0; q < n; ++q) d[q] = solves[q].d;
    Built b;
    if (!build(d.data(), n, dbl, &b)) return -1;
    for (int q = 0; q < n; ++q) solves[q].ctas = b.ctas[q];
    const Parts at(b, n, dbl);
    if (at.bytes > p->cap) {
        res_plan_free(p);
        if (lib_malloc(&p->mem, at.bytes) != cudaSuccess) {
            cudaGetLastError();
            *p = ResPlan{};
            return -2;
        }
        p->cap = at.bytes;
    }
    char* const m = (char*)p->mem;
    p->solves = (ResSolve*)(m + at.solves);
    p->tasks = (ResTask*)(m + at.tasks);
    p->cta_task = (int*)(m + at.cta);
    p->error = (int*)(m + at.error);
    p->sums = m + at.sums;
    p->outbox = m + at.outbox;
    p->words = p->sums;
    p->words_bytes = at.bytes - at.sums;
    const bool ok =
        cudaMemcpyAsync(p->tasks, b.tasks.data(), sizeof(ResTask) * b.tasks.size(),
                        cudaMemcpyHostToDevice, st) == cudaSuccess &&
        cudaMemcpyAsync(p->cta_task, b.cta_task.data(), sizeof(int) * b.cta_task.size(),
                        cudaMemcpyHostToDevice, st) == cudaSuccess &&
        cudaMemsetAsync(p->words, 0, p->words_bytes, st) == cudaSuccess &&
        cudaStreamSynchronize(st) == cudaSuccess;  // the host vectors go out of scope
    if (!ok) {
        cudaGetLastError();
        res_plan_free(p);
        return -2;
    }
    p->ncta = (int)b.cta_task.size() - 1;
    p->nsolves = n;
    p->ntasks = (int)b.tasks.size();
    p->box_words = b.box_words;
    p->depth = b.depth;
    p->smem = smem_fix(b.depth);
    if (dbl) {
        p->smem = 0;
        for (const ResTask& k : b.tasks)
            p->smem = std::max(p->smem, sizeof(double) * (k.bx + 2) * (k.by + 2) * (5 * (size_t)k.bz + 3));
    }
    p->dbl = dbl;
    p->next_tag = 0;
    return 0;
}

int res_tags(ResPlan* p, ResSolve* solves, int n, cudaStream_t st) {
    // (a cap beyond the tags of one launch ends that launch early, and the solve goes on)
    const unsigned most = 0xf0000000u / (unsigned)n - 4u;
    unsigned long long need = 0;
    for (int q = 0; q < n; ++q) {
        solves[q].max_iter = (int)std::min((unsigned)solves[q].max_iter, most);
        need += (unsigned long long)solves[q].max_iter + 4;
    }
    if (p->next_tag + need >= 0xffffffffull) {
        if (cudaMemsetAsync(p->words, 0, p->words_bytes, st) != cudaSuccess) return -1;
        p->next_tag = 0;
    }
    for (int q = 0; q < n; ++q) {
        solves[q].tag0 = p->next_tag;
        p->next_tag += (unsigned)solves[q].max_iter + 4u;
    }
    return 0;
}

int launch_res(const ResPlan& p, ResKind kind, const ResSolve* solves, int n, cudaStream_t st) {
    static OncePerDevice once;
    once.run([] {
        for (int q = 0; q < 4; ++q)
            for (int depth : {2, 4, 8, 16})
                cudaFuncSetAttribute(kernel_of((ResKind)q, depth),
                                     cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(q == RES_FACES64 ? SMEM_MAX : smem_fix(depth)));
        cudaGetLastError();
    });
    ResArgs a{p.solves, p.tasks, p.cta_task, p.sums, p.outbox, p.box_words, p.extra, p.error, p.nsolves,
              p.wait_ns};
    void* params[] = {&a};
    if (cudaMemcpyAsync(p.solves, solves, sizeof(ResSolve) * n, cudaMemcpyHostToDevice, st) !=
            cudaSuccess ||
        cudaMemsetAsync(p.error, 0, sizeof(int), st) != cudaSuccess)
        return -1;
    const cudaError_t e =
        coop_launch(kernel_of(kind, p.depth), dim3(p.ncta), dim3(RES_T), params, p.smem, st);
    g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    return 0;
}

}  // namespace pcg
