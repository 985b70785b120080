// The persistent solver kernel and its launches (solve.cu has the host side and
// what the solver does).  Instantiated by format and flow in solve_*.cu, so that
// the builds run side by side.
#pragma once

#include <type_traits>

#include "vcycle.cuh"

namespace mvgd {
namespace solver {

constexpr int kCh = 256;   // rows per tile: one per thread, 8 slices of 32
constexpr int kThreads = 256;
constexpr int kChan = 2;     // reduced channels a step of the row-scaled flows
constexpr int kChanAmg = 5;  // ... of the multigrid flow (B takes five dot products)
__host__ __device__ constexpr int chan_count(bool amg) { return amg ? kChanAmg : kChan; }
constexpr int kRedSlots = 3;
constexpr int kMaxReq = 1024;
// Tiles up to which a step's partials are summed by a warp an entry instead of
// by the whole block entry after entry (arrive_and_finalize).  At 11 tiles the
// block-wide sum took about 6 us in FP64 (it adds batches of 16 whether or not
// there are that many tiles, on a pipe of one DADD a warp in 16 clocks); with
// the tile butterflies above, FP64 reducing steps went from 9.5 to 7.5 us there
// (2,562 rows), and B from 22 to 15 us at 28 tiles with four right-hand sides.
// Above this count a lane's chain of additions is the longer one.
constexpr int kFinWarpTiles = 512;
constexpr long long kStageWaitLimit = 1ll << 24;  // polls of an mbarrier: far beyond any copy's landing time

enum Phase : int { P_PRE_A = 0, P_A = 1, P_PRE_B = 2, P_B = 3, P_C = 4, P_COUNT = 5 };
enum Mode : int { M_RESTART = 0, M_INNER = 1, M_SKIP = 2, M_DONE = 3 };

__host__ __device__ constexpr int red_slot(int ph) { return ph == P_A ? 0 : (ph == P_B ? 1 : 2); }

struct RhsState {
    double rho, alpha, omega, beta;
    double fnorm, relres, scale, target;
    double rnorm, rmin;
    int mode, pp, iters, inner_iters, outer, status, discard, stall;
    int best_flag;   // the last iteration reached a new smallest inner residual: copy x to x_best
    int fold_best;   // on restart, fold x_best (not x) into u
    int since_best;  // inner iterations since the smallest residual last dropped by 1%
    int pending;     // multigrid flow: the last step's x += alpha ph + omega sh is still to apply
};

// Right-hand sides of the request (or group) in a kernel of width QT.
#define MVGD_NQ(P) (QT == 1 ? 1 : (P).nq)

// One request: an operator, its right-hand sides and all solver state.
struct Prob {
    int64_t n;
    int k, Q, prec, precond;
    double sigma;
    const int32_t* col;
    const void* val;
    const float* val_lo;
    const int32_t* order;
    double* f;         // stored order [n][Q]
    double* u;         // stored order [n][Q]
    void* x;
    void* xb;          // FP32 path: the inner iterate with the smallest residual so far
    void* r;
    void* rh;
    void* p[2];
    void* v[2];
    void* s;
    void* t;
    double* r64;
    void* invd;        // [n] VT: 1 / (sigma + sum_s |w_s|), the left scaling (precond == 1)
    RhsState* st;      // [Q]
    void* part;        // [kRedSlots][channels][nchunk][Q] tile partials (Part<MIXED>: F2 or double)
    unsigned* arrive;  // [groups][kRedSlots]
    int nchunk;
    int nq;            // right-hand sides a block works on: Q, or one group of them (see ReqTable::groups)
    // multigrid right preconditioning (precond == 2); amg == nullptr otherwise
    const AmgHeader* amg;
    int amg_levels;
    int q0;            // first right-hand side of the group (0: all of them)
    void* ph;                    // [n][Q] VT: M^-1 p
    void* sh;                    // [n][Q] VT: M^-1 s
    float* vy[kAmgMaxLevels];    // per level [n_l][Q]: pre-smoothed y_l = d_l b_l
    float* vr[kAmgMaxLevels];    //                     residual r_l
    float* vb[kAmgMaxLevels];    //                     right-hand side b_l (l >= 1)
    float* vx[kAmgMaxLevels];    //                     correction x_l (l >= 1)
    double rtol, inner_rtol;
    int maxit, inner_maxit, max_outer, pad2;
};

constexpr int kTraceMax = 1 << 16;

struct Ctl {
    GridBarrier bar;
    int* err;
    int* active;     // right-hand sides not DONE
    int* nrestart;   // right-hand sides in RESTART
    int* stop;
    const int* cancel;
    long long limit;
    unsigned long long* trace;  // where each step's end time is recorded (mvgd_trace_enable), or null
    unsigned* trace_n;
    int withhold;    // test control: block 0 leaves its first barrier arrival out
};

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// step code: Krylov phase ph (0..4), or 0x1000 | side << 8 | kind << 4 | level for a V-cycle step
__device__ __forceinline__ void trace_step(const Ctl& ctl, unsigned code) {
    if (!ctl.trace || blockIdx.x != 0 || threadIdx.x != 0) return;
    const unsigned i = *ctl.trace_n;
    *ctl.trace_n = i + 1;
    ctl.trace[i % kTraceMax] = ((unsigned long long)code << 48) | (global_ns() & 0xffffffffffffull);
}

__device__ __forceinline__ void load_state(RhsState& dst, const RhsState* src) {
    const unsigned long long* s = reinterpret_cast<const unsigned long long*>(src);
    unsigned long long* d = reinterpret_cast<unsigned long long*>(&dst);
#pragma unroll
    for (int w = 0; w < (int)(sizeof(RhsState) / 8); w++) d[w] = __ldcg(s + w);
}

// ------------------------------------------------------------------------------
// Row work
// ------------------------------------------------------------------------------

// PRE_A / PRE_B / C and the RESTART steps: elementwise on row r.
template <bool MIXED, int QT>
__device__ __forceinline__ void elementwise_row(const Prob& P, int64_t r, int ph, const RhsState* S,
                                                const bool (&inner)[QT], const bool (&restart)[QT],
                                                F2 (&af)[kChan][QT]) {
    using VT = typename std::conditional<MIXED, float, double>::type;
    const int Q = P.Q;
#pragma unroll
    for (int q = 0; q < QT; q++) {
        const int64_t e = r * Q + q;
        if (ph == P_PRE_A) {
            if (MIXED && restart[q] && S[q].outer > 0 && !S[q].discard)
                P.u[e] += S[q].scale * (double)static_cast<const VT*>(S[q].fold_best ? P.xb : P.x)[e];
            if (!MIXED && inner[q]) {
                VT* pv = static_cast<VT*>(P.p[0]);
                const VT* vv = static_cast<const VT*>(P.v[0]);
                const VT* rv = static_cast<const VT*>(P.r);
                pv[e] = rv[e] + (VT)S[q].beta * (pv[e] - (VT)S[q].omega * vv[e]);
            }
        } else if (ph == P_PRE_B) {
            if (!MIXED && inner[q]) {
                const VT* vv = static_cast<const VT*>(P.v[0]);
                const VT* rv = static_cast<const VT*>(P.r);
                static_cast<VT*>(P.s)[e] = rv[e] - (VT)S[q].alpha * vv[e];
            }
        } else if (ph == P_C) {
            if (inner[q]) {
                const VT* pv = static_cast<const VT*>(P.p[S[q].pp]);
                VT* X = static_cast<VT*>(P.x);
                const VT sv = static_cast<const VT*>(P.s)[e], tv = static_cast<const VT*>(P.t)[e];
                const VT al = (VT)S[q].alpha, om = (VT)S[q].omega;
                X[e] = X[e] + al * pv[e] + om * sv;
                const VT rn = sv - om * tv;
                static_cast<VT*>(P.r)[e] = rn;
                const VT rhv = static_cast<const VT*>(P.rh)[e];
                f2_add_prod(af[0][q], (float)rhv, (float)rn);
                f2_add_prod(af[1][q], (float)rn, (float)rn);
            }
        }
    }
}

// FP64 partials of the FP64 steps (C of the plain path) go through a double
// accumulator so that nothing is rounded to FP32.
template <int QT>
__device__ __forceinline__ void c_row_f64(const Prob& P, int64_t r, const RhsState* S, const bool (&inner)[QT],
                                          double (&ad)[kChan][QT]) {
    const int Q = P.Q;
#pragma unroll
    for (int q = 0; q < QT; q++) {
        if (!inner[q]) continue;
        const int64_t e = r * Q + q;
        const double* pv = static_cast<const double*>(P.p[0]);
        double* X = static_cast<double*>(P.x);
        const double sv = static_cast<const double*>(P.s)[e], tv = static_cast<const double*>(P.t)[e];
        X[e] = X[e] + S[q].alpha * pv[e] + S[q].omega * sv;
        const double rn = sv - S[q].omega * tv;
        static_cast<double*>(P.r)[e] = rn;
        ad[0][q] += static_cast<const double*>(P.rh)[e] * rn;
        ad[1][q] += rn * rn;
    }
}

__host__ __device__ constexpr int pow2_at_least(int x) { return x <= 1 ? 1 : 2 * pow2_at_least((x + 1) / 2); }

// Tile partials and their sums: F2 (double-float on the FP32 pipe) in the
// FP32 flow, double in the FP64 one.  One SM sums a request's thousands of
// partials in each reducing step.  GB300's FP64 rate (1.25 TFLOP/s nominal)
// is about two FP64 lanes a clock an SM, a warp instruction every 16 clocks,
// with 63 clocks of latency (measured), so in FP64 that sum alone took about
// 1 us a channel at 1M rows; F2 additions (eight FP32 operations) take a
// fraction of it with about 48 bits.  The F2
// range is FP32's: the FP32 flow's squared residual norms stay below 3.4e38
// (||f|| below about 1.8e19) or the step reports a non-finite residual.
template <bool MIXED>
using Part = typename std::conditional<MIXED, F2, double>::type;
__device__ __forceinline__ double part_value(F2 a) { return f2_to_double(a); }
__device__ __forceinline__ double part_value(double a) { return a; }
template <typename PT>
__device__ __forceinline__ PT part_zero() {
    if constexpr (std::is_same<PT, F2>::value) {
        F2 z;
        z.hi = 0.0f;
        z.lo = 0.0f;
        return z;
    } else {
        return 0.0;
    }
}
template <typename PT>
__device__ __forceinline__ PT part_from(double x) {
    if constexpr (std::is_same<PT, F2>::value) {
        F2 z;
        z.hi = __double2float_rn(x);
        z.lo = __double2float_rn(x - (double)z.hi);
        return z;
    } else {
        return x;
    }
}
__device__ __forceinline__ F2 part_warp_sum(F2 v) { return warp_sum_f2(v); }
__device__ __forceinline__ double part_warp_sum(double v) { return warp_sum(v); }
__device__ __forceinline__ F2 part_load(const F2* p) {
    const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
    F2 z;
    z.hi = v.x;
    z.lo = v.y;
    return z;
}
__device__ __forceinline__ double part_load(const double* p) { return __ldcg(p); }

// A warp's partials of its slice of a tile, channels 0 .. NCH-1 of every
// right-hand side, into out[ch * QT + q]: in the FP32 flow the F2 products
// summed over the warp, plus the FP64 ones where there are any (`with64`); in
// the FP64 flow the FP64 ones.  The values go through the shared butterfly at
// most 32 at a time.  In FP64 that is what bounds the step on a small system:
// a DADD takes the SM's FP64 pipe 16 clocks a warp, so 5 channels in separate
// butterflies (25 DADDs a warp, 9 here) held a tile's 8 warps for 1.5 us, and
// 8 right-hand sides (200 against about 45) for 12 us.
template <bool MIXED, int QT, int NC, int NCH>
__device__ __forceinline__ void tile_partials(const F2 (&af)[NC][QT], const double (&ad)[NC][QT], bool with64,
                                              int lane, Part<MIXED>* out) {
    constexpr int N = NCH * QT;
    auto group = [&](auto width, int e0) {  // values e0 .. e0 + E - 1 (those past N are zeros)
        constexpr int E = decltype(width)::value;
        int chan;
        double tot64 = 0.0;
        if (!MIXED || with64) {
            double v[E];
#pragma unroll
            for (int e = 0; e < E; e++) v[e] = e0 + e < N ? ad[(e0 + e) / QT][(e0 + e) % QT] : 0.0;
            tot64 = warp_sum_multi<E>(v, lane, chan);
        }
        Part<MIXED> tot = part_from<Part<MIXED>>(tot64);
        if constexpr (MIXED) {
            F2 v[E];
#pragma unroll
            for (int e = 0; e < E; e++) v[e] = e0 + e < N ? af[(e0 + e) / QT][(e0 + e) % QT] : part_zero<F2>();
            const F2 t = warp_sum_multi<E>(v, lane, chan);
            tot = with64 ? f2_add(t, tot) : t;
        }
        if ((lane & (32 / E - 1)) == 0 && e0 + chan < N) out[e0 + chan] = tot;
    };
    constexpr int kHead = N > 32 ? 32 : pow2_at_least(N);
    group(std::integral_constant<int, kHead>{}, 0);
    if constexpr (N > 32) group(std::integral_constant<int, pow2_at_least(N - 32)>{}, 32);
    static_assert(N <= 64, "two groups hold every channel of every right-hand side");
}

template <typename VT>
__host__ __device__ constexpr size_t stage_bytes_per_warp(int kmax) {
    return (size_t)kSlice * kmax * sizeof(int) + (size_t)kSlice * (kmax + 1) * sizeof(VT);
}

// Per-warp staging of operator slices.  A slice -- 32 rows' k column slots
// and k+1 weight slots, each 32 consecutive words in the sliced layout, so two
// contiguous runs -- arrives in the warp's shared memory by two bulk
// asynchronous copies issued by lane 0 and completing on one of the warp's
// mbarriers.  With two buffers the slice of the warp's next tile is requested
// before the current one is used, so the operator keeps streaming while the
// warp gathers and reduces.  The evict-first hint keeps the small, reused
// Krylov vectors in L2 while the operator streams past.
// Its state is two registers, kept for the whole launch: what the launch's
// shape fixes (buffer sizes and addresses, the L2 policy) is formed where it is
// used, because the steps between the copies are short of registers.
template <typename VT>
struct Stager {
    int next_c;    // tile whose slice was requested ahead (-1: none), in buffer next_b
    int have;      // one buffer: the slice it holds, 2 c + (FP64 weights), or -1
    uint32_t st;   // bits 0, 1: parity of buffer b's next completion; 2, 3: a copy into buffer b has not
                   // been waited for; 4: next_b; 5: a copy missed its wait, nothing more is issued
    static __device__ __forceinline__ uint32_t bytes(int kmax) { return (uint32_t)stage_bytes_per_warp<VT>(kmax); }
    static __device__ __forceinline__ unsigned char* buffer(int kmax, int nbuf, int b) {
        extern __shared__ __align__(16) unsigned char stage_smem[];
        return stage_smem + ((threadIdx.x >> 5) * nbuf + b) * bytes(kmax);
    }
    static __device__ __forceinline__ int* col(int kmax, int nbuf, int b) {
        return reinterpret_cast<int*>(buffer(kmax, nbuf, b));
    }
    static __device__ __forceinline__ void* val(int kmax, int nbuf, int b) {
        return buffer(kmax, nbuf, b) + kSlice * kmax * sizeof(int);
    }
    __device__ __forceinline__ bool ok() const { return (st & 32u) == 0; }

    __device__ __forceinline__ void issue(int kmax, int nbuf, uint64_t* bar, int b, const int32_t* colsrc,
                                          const void* valsrc, int esize, int k, int64_t slice) {
        __syncwarp();  // every lane has consumed what buffer b held
        if (!ok()) return;  // after a missed wait the warp issues nothing more
        st |= 4u << b;
        if (lane_id() == 0) {
            const uint32_t cb = (uint32_t)(kSlice * k * 4), vb = (uint32_t)(kSlice * (k + 1) * esize);
            const uint64_t pol = l2_evict_first_policy();
            mbar_expect_tx(&bar[b], cb + vb);
            bulk_g2s(col(kmax, nbuf, b), colsrc + slice * (int64_t)(kSlice * k), cb, &bar[b], pol);
            bulk_g2s(val(kmax, nbuf, b),
                     static_cast<const char*>(valsrc) + slice * (int64_t)(kSlice * (k + 1)) * esize, vb, &bar[b],
                     pol);
        }
    }

    // The buffer holding tile c's slice: requested now unless it was requested
    // ahead; then, with two buffers, requests tile c2's slice ahead (c2 < 0: none).
    __device__ __forceinline__ int acquire(int kmax, int nbuf, uint64_t* bar, int c, int64_t slice, int c2,
                                           int64_t slice2, const int32_t* colsrc, const void* valsrc, int esize, int k,
                                           int* err) {
        int b = (st >> 4) & 1u;
        if (next_c >= 0 && next_c != c) {  // a slice requested ahead for a tile not taken: let it land first
            wait(bar, b, err);
            next_c = -1;
        }
        if (next_c != c) {
            b = (st & 4u) ? 1 : 0;
            // the slice the buffer holds already (the warp's only one on a small system; the
            // last of the previous step on a large one, see `rev`): nothing to request
            const int want = 2 * c + (esize == 8);
            if (nbuf != 1 || have != want) issue(kmax, nbuf, bar, b, colsrc, valsrc, esize, k, slice);
            have = want;
        }
        next_c = -1;
        if (nbuf == 2 && c2 >= 0) {
            next_c = c2;
            st = (st & ~16u) | (b == 0 ? 16u : 0u);
            issue(kmax, nbuf, bar, b ^ 1, colsrc, valsrc, esize, k, slice2);
        }
        return b;
    }

    // Warp-collective bounded wait for buffer b.  A copy that missed its wait
    // stays marked busy with its parity unchanged, so drain() waits for it
    // again before the block's shared memory is released.
    __device__ __forceinline__ bool wait(uint64_t* bar, int b, int* err) {
        if (!ok()) return false;  // nothing was issued since the first miss
        if (!(st & (4u << b))) return true;  // it landed in an earlier step
        const bool landed = __all_sync(0xffffffffu, mbar_wait(&bar[b], (st >> b) & 1u, kStageWaitLimit));
        if (landed) {
            st = (st ^ (1u << b)) & ~(4u << b);
        } else {
            st |= 32u;
            if (lane_id() == 0) atomicCAS(err, 0, (int)MVGD_ETIMEOUT);
        }
        return ok();
    }

    // Before the block's shared memory goes away: bounded waits for every copy
    // still in flight (landed or not, each buffer's wait ends within its limit).
    __device__ void drain(uint64_t* bar) {
        for (int b = 0; b < 2; b++)
            if (st & (4u << b)) mbar_wait(&bar[b], (st >> b) & 1u, kStageWaitLimit);
    }
};

// A / B for INNER right-hand sides: one operator application each, reading
// the row's columns and weights from the warp's staged slice.  Called by every
// lane of a staged warp (`valid`: the lane's row exists); the row's own loads
// are issued before `landed()` waits for the slice, so they overlap the copy.
template <bool MIXED, int QT, typename Landed>
__device__ __forceinline__ void spmv_row(const Prob& P, int64_t r, bool valid, int ph, const RhsState* S,
                                         const bool (&on)[QT], const float (&c1)[QT], const float (&c2)[QT],
                                         F2 (&af)[kChan][QT], double (&ad)[kChan][QT], const int* colS,
                                         const typename std::conditional<MIXED, float, double>::type* valS,
                                         Landed&& landed) {
    using VT = typename std::conditional<MIXED, float, double>::type;
    const int Q = P.Q, k = P.k;
    const int lane = (int)(r % kSlice);
    const VT sig = (VT)P.sigma;
    const VT invd = (valid && P.precond) ? static_cast<const VT*>(P.invd)[r] : (VT)1;
    // vectors written by other blocks during this kernel: plain (coherent) loads
    const VT* R = static_cast<const VT*>(P.r);
    const VT* RH = static_cast<const VT*>(P.rh);
    const VT* src[QT];
    const VT* vold[QT];
    VT si[QT], acc[QT];
#pragma unroll
    for (int q = 0; q < QT; q++) {
        acc[q] = (VT)0;
        si[q] = (VT)0;
        src[q] = nullptr;
        vold[q] = nullptr;
        if (!on[q]) continue;
        const int64_t e = r * Q + q;
        if (MIXED) {
            vold[q] = static_cast<const VT*>(P.v[S[q].pp]);
            src[q] = static_cast<const VT*>(P.p[S[q].pp]);
            if (valid)
                si[q] = (ph == P_A) ? R[e] + (VT)c1[q] * (src[q][e] - (VT)c2[q] * vold[q][e])
                                    : R[e] - (VT)c1[q] * vold[q][e];
        } else {
            src[q] = static_cast<const VT*>(ph == P_A ? P.p[0] : P.s);
            if (valid) si[q] = src[q][e];
        }
    }
    if (!landed() || !valid) return;  // landed() is warp-collective: every lane calls it
    const VT w0 = valS[lane];
#pragma unroll 8
    for (int sl = 0; sl < k; sl++) {
        const int64_t j = colS[sl * kSlice + lane];
        const VT w = valS[(sl + 1) * kSlice + lane];
#pragma unroll
        for (int q = 0; q < QT; q++) {
            if (!on[q]) continue;
            const int64_t e = j * Q + q;
            if (MIXED) {
                const VT sj = (ph == P_A) ? R[e] + (VT)c1[q] * (src[q][e] - (VT)c2[q] * vold[q][e])
                                          : R[e] - (VT)c1[q] * vold[q][e];
                acc[q] = fmaf(w, sj - si[q], acc[q]);
            } else {
                acc[q] = fma(w, src[q][e], acc[q]);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < QT; q++) {
        if (!on[q]) continue;
        const int64_t e = r * Q + q;
        const VT lx = MIXED ? acc[q] : acc[q] + w0 * si[q];
        const VT res = invd * (sig * si[q] - lx);
        if (ph == P_A) {
            const int np = MIXED ? (S[q].pp ^ 1) : 0;
            if (MIXED) static_cast<VT*>(P.p[np])[e] = si[q];
            // the previous iteration reached a new best residual: keep its iterate
            if (MIXED && S[q].best_flag) static_cast<VT*>(P.xb)[e] = static_cast<const VT*>(P.x)[e];
            static_cast<VT*>(P.v[np])[e] = res;
            if (MIXED) f2_add_prod(af[0][q], (float)RH[e], (float)res);
            else ad[0][q] += (double)(RH[e] * res);
        } else {
            if (MIXED) static_cast<VT*>(P.s)[e] = si[q];
            static_cast<VT*>(P.t)[e] = res;
            if (MIXED) {
                f2_add_prod(af[0][q], (float)res, (float)si[q]);
                f2_add_prod(af[1][q], (float)res, (float)res);
            } else {
                ad[0][q] += (double)(res * si[q]);
                ad[1][q] += (double)(res * res);
            }
        }
    }
}

// RESTART steps: in A the FP64 true residual, in the step that ends the
// iteration (C of the row-scaled flows, B of the multigrid flow) the restart of
// the Krylov vectors.
template <bool MIXED, int QT, int NC>
__device__ __forceinline__ void restart_row(const Prob& P, int64_t r, int ph, const RhsState* S, const bool (&on)[QT],
                                            double (&ad)[NC][QT]) {
    using VT = typename std::conditional<MIXED, float, double>::type;
    const int Q = P.Q, k = P.k, m = k + 1;
    const int64_t vb = (r / kSlice) * (int64_t)(kSlice * m) + (r % kSlice);
    const int64_t cb = (r / kSlice) * (int64_t)(kSlice * k) + (r % kSlice);
    if (ph == P_A) {
        double w0;
        if (MIXED) w0 = (double)static_cast<const float*>(P.val)[vb] + (double)P.val_lo[vb];
        else w0 = static_cast<const double*>(P.val)[vb];
        double acc[QT], ui[QT];
#pragma unroll
        for (int q = 0; q < QT; q++) {
            ui[q] = on[q] ? P.u[r * Q + q] : 0.0;
            acc[q] = w0 * ui[q];
        }
#pragma unroll 4
        for (int sl = 0; sl < k; sl++) {
            const int64_t j = P.col[cb + (int64_t)sl * kSlice];
            const int64_t e = vb + (int64_t)(sl + 1) * kSlice;
            double w;
            if (MIXED) w = (double)static_cast<const float*>(P.val)[e] + (double)P.val_lo[e];
            else w = static_cast<const double*>(P.val)[e];
#pragma unroll
            for (int q = 0; q < QT; q++)
                if (on[q]) acc[q] = fma(w, P.u[j * Q + q], acc[q]);
        }
#pragma unroll
        for (int q = 0; q < QT; q++) {
            if (!on[q]) continue;
            const int64_t e = r * Q + q;
            const double fv = P.f[e];
            const double res = fv - (P.sigma * ui[q] - acc[q]);
            P.r64[e] = res;
            ad[0][q] += res * res;
            ad[1][q] += fv * fv;
        }
        return;
    }
    // the iteration's last step: restart the Krylov vectors
    const double invd = P.precond ? (double)static_cast<const VT*>(P.invd)[r] : 1.0;
#pragma unroll
    for (int q = 0; q < QT; q++) {
        if (!on[q]) continue;
        const int64_t e = r * Q + q;
        double rv = invd * P.r64[e];
        if (MIXED) rv /= S[q].scale;
        const VT rr = (VT)rv;
        static_cast<VT*>(P.r)[e] = rr;
        // shadow residual: r itself; after a refinement step that did not lower the
        // residual, a deterministic relative perturbation of up to +-50% sends the
        // retry down a different Krylov path ((rh, r) stays positive)
        VT rhv = rr;
        if (S[q].stall > 0) {
            uint32_t hsh = (uint32_t)(e + P.q0) * 2654435761u ^ (uint32_t)S[q].outer * 40503u;
            hsh ^= hsh >> 16; hsh *= 0x7feb352du; hsh ^= hsh >> 15; hsh *= 0x846ca68bu; hsh ^= hsh >> 16;
            const double u01 = (double)hsh * (1.0 / 4294967296.0);
            rhv = (VT)(rv * (1.0 + (u01 - 0.5)));
        }
        static_cast<VT*>(P.rh)[e] = rhv;
        static_cast<VT*>(P.p[0])[e] = (VT)0;
        static_cast<VT*>(P.v[0])[e] = (VT)0;
        if (MIXED) {
            static_cast<VT*>(P.p[1])[e] = (VT)0;
            static_cast<VT*>(P.v[1])[e] = (VT)0;
            static_cast<VT*>(P.x)[e] = (VT)0;
            static_cast<VT*>(P.xb)[e] = (VT)0;
        }
        ad[0][q] += (double)rr * (double)rr;
    }
}

// ------------------------------------------------------------------------------
// Multigrid-preconditioned flow (precond == 2).  Right preconditioning:
//   p = r + beta (p - omega v);  ph = M^-1 p;  v = A ph;  alpha = rho / (rh, v)
//   s = r - alpha v;             sh = M^-1 s;  t = A sh;  omega = (t, s) / (t, t)
//   x += alpha ph + omega sh;    r = s - omega t
// with M^-1 one V-cycle.  p and s are materialised (the cycle reads them at
// other rows), with their pre-smoothed FP32 copies y_0 = d_0 p for level 0.
// An iteration has six grid steps, PRE_A, (cycle), A, PRE_B, (cycle), B: the
// new residual's two dot products follow from those of s and t,
//   (rh, r) = (rh, s) - omega (rh, t),
//   (r, r)  = (s, s) - 2 omega (t, s) + omega^2 (t, t),
// so B takes all five and r = s - omega t is formed by the next PRE_A, row by
// row, with no step (and no grid barrier) of its own.
// ------------------------------------------------------------------------------
template <bool MIXED, int QT>
__device__ __forceinline__ void amg_pre_row(const Prob& P, int64_t r, int ph, const RhsState* S,
                                            const bool (&inner)[QT], const bool (&restart)[QT]) {
    using VT = typename std::conditional<MIXED, float, double>::type;
    const int Q = P.Q;
    const float d0 = P.amg->lv[0].dinv[r];
    VT* pv = static_cast<VT*>(P.p[0]);
    const VT* vv = static_cast<const VT*>(P.v[0]);
    VT* rv = static_cast<VT*>(P.r);
#pragma unroll
    for (int q = 0; q < QT; q++) {
        const int64_t e = r * Q + q;
        if (q >= MVGD_NQ(P)) break;
        if (ph == P_PRE_A) {
            VT rn = (VT)0;
            if (S[q].pending) {
                // the last iteration's step (alpha, omega still hold its values): its
                // residual r = s - omega t and its iterate x += alpha ph + omega sh
                const VT om = (VT)S[q].omega;
                rn = static_cast<const VT*>(P.s)[e] - om * static_cast<const VT*>(P.t)[e];
                rv[e] = rn;
                VT* X = static_cast<VT*>(P.x);
                X[e] = X[e] + (VT)S[q].alpha * static_cast<const VT*>(P.ph)[e] + om * static_cast<const VT*>(P.sh)[e];
            }
            if (MIXED && restart[q] && S[q].outer > 0 && !S[q].discard)
                P.u[e] += S[q].scale * (double)static_cast<const VT*>(S[q].fold_best ? P.xb : P.x)[e];
            if (inner[q]) {
                if (!S[q].pending) rn = rv[e];
                const VT nv = rn + (VT)S[q].beta * (pv[e] - (VT)S[q].omega * vv[e]);
                pv[e] = nv;
                P.vy[0][e] = d0 * (float)nv;
            }
        } else if (inner[q]) {
            const VT nv = rv[e] - (VT)S[q].alpha * vv[e];
            static_cast<VT*>(P.s)[e] = nv;
            P.vy[0][e] = d0 * (float)nv;
        }
    }
}

// PRE_A / PRE_B of NT rows at once (rows r[k], k < n, of up to NT tiles of one
// request; `ok[k]`: the row exists), for right-hand sides that are INNER or
// have a pending step (no RESTART in the request: its fold goes row by row).
// Every operand of every row is loaded before any is used, so a block's tiles
// cost one memory round trip a group instead of one a tile; each row's
// arithmetic is that of amg_pre_row.
template <bool MIXED, int QT, int NT>
__device__ __forceinline__ void amg_pre_rows(const Prob& P, const int64_t (&r)[NT], const bool (&ok)[NT], int ph,
                                             const RhsState* S, const bool (&inner)[QT]) {
    using VT = typename std::conditional<MIXED, float, double>::type;
    const int Q = P.Q;
    const float* dinv = P.amg->lv[0].dinv;
    VT* pv = static_cast<VT*>(P.p[0]);
    const VT* vv = static_cast<const VT*>(P.v[0]);
    VT* rv = static_cast<VT*>(P.r);
    // PRE_A: a = s, b = t, x, h1 = ph, h2 = sh (a pending step) or a = r; c = p, w = v.
    // PRE_B: a = r, w = v.
    float d0[NT];
    VT a[NT][QT], b[NT][QT], c[NT][QT], w[NT][QT], x[NT][QT], h1[NT][QT], h2[NT][QT];
#pragma unroll
    for (int k = 0; k < NT; k++) {
        d0[k] = ok[k] ? dinv[r[k]] : 0.0f;
#pragma unroll
        for (int q = 0; q < QT; q++) {
            a[k][q] = b[k][q] = c[k][q] = w[k][q] = x[k][q] = h1[k][q] = h2[k][q] = (VT)0;
            if (!ok[k] || q >= MVGD_NQ(P)) continue;
            const int64_t e = r[k] * Q + q;
            if (ph == P_PRE_A && S[q].pending) {
                a[k][q] = static_cast<const VT*>(P.s)[e];
                b[k][q] = static_cast<const VT*>(P.t)[e];
                x[k][q] = static_cast<const VT*>(P.x)[e];
                h1[k][q] = static_cast<const VT*>(P.ph)[e];
                h2[k][q] = static_cast<const VT*>(P.sh)[e];
            } else if (inner[q]) {
                a[k][q] = rv[e];
            }
            if (inner[q]) {
                w[k][q] = vv[e];
                if (ph == P_PRE_A) c[k][q] = pv[e];
            }
        }
    }
#pragma unroll
    for (int k = 0; k < NT; k++) {
        if (!ok[k]) continue;
#pragma unroll
        for (int q = 0; q < QT; q++) {
            if (q >= MVGD_NQ(P)) break;
            const int64_t e = r[k] * Q + q;
            if (ph == P_PRE_A) {
                VT rn = a[k][q];
                if (S[q].pending) {
                    const VT om = (VT)S[q].omega;
                    rn = a[k][q] - om * b[k][q];
                    rv[e] = rn;
                    static_cast<VT*>(P.x)[e] = x[k][q] + (VT)S[q].alpha * h1[k][q] + om * h2[k][q];
                }
                if (inner[q]) {
                    const VT nv = rn + (VT)S[q].beta * (c[k][q] - (VT)S[q].omega * w[k][q]);
                    pv[e] = nv;
                    P.vy[0][e] = d0[k] * (float)nv;
                }
            } else if (inner[q]) {
                const VT nv = a[k][q] - (VT)S[q].alpha * w[k][q];
                static_cast<VT*>(P.s)[e] = nv;
                P.vy[0][e] = d0[k] * (float)nv;
            }
        }
    }
}

// A: v = A ph and (rh, v); B: t = A sh and (t, s), (t, t), (rh, s), (rh, t),
// (s, s); from the staged slice (every lane of the warp calls).
template <bool MIXED, int QT, typename Landed>
__device__ __forceinline__ void amg_spmv_row(const Prob& P, int64_t r, bool valid, int ph, const RhsState* S,
                                             const bool (&on)[QT], F2 (&af)[kChanAmg][QT],
                                             double (&ad)[kChanAmg][QT], const int* colS,
                                             const typename std::conditional<MIXED, float, double>::type* valS,
                                             Landed&& landed) {
    using VT = typename std::conditional<MIXED, float, double>::type;
    const int Q = P.Q, k = P.k;
    const int lane = (int)(r % kSlice);
    const VT sig = (VT)P.sigma;
    const VT* src = static_cast<const VT*>(ph == P_A ? P.ph : P.sh);
    VT si[QT], acc[QT];
#pragma unroll
    for (int q = 0; q < QT; q++) {
        acc[q] = (VT)0;
        si[q] = (on[q] && valid) ? src[r * Q + q] : (VT)0;
    }
    if (!landed() || !valid) return;  // warp-collective
    const VT w0 = valS[lane];
#pragma unroll 8
    for (int sl = 0; sl < k; sl++) {
        const int64_t j = colS[sl * kSlice + lane];
        const VT w = valS[(sl + 1) * kSlice + lane];
        VT xj[QT];
        load_row<QT>(src, j, Q, xj);  // every right-hand side of neighbour j at once
#pragma unroll
        for (int q = 0; q < QT; q++) {
            if (!on[q]) continue;
            // FP32: difference form (rows of L sum to zero), as in the plain flow
            if (MIXED) acc[q] = fmaf(w, xj[q] - si[q], acc[q]);
            else acc[q] = fma(w, xj[q], acc[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < QT; q++) {
        if (!on[q]) continue;
        const int64_t e = r * Q + q;
        const VT lx = MIXED ? acc[q] : acc[q] + w0 * si[q];
        const VT res = sig * si[q] - lx;
        const VT rhv = static_cast<const VT*>(P.rh)[e];
        if (ph == P_A) {
            static_cast<VT*>(P.v[0])[e] = res;
            if (MIXED && S[q].best_flag) static_cast<VT*>(P.xb)[e] = static_cast<const VT*>(P.x)[e];
            if (MIXED) f2_add_prod(af[0][q], (float)rhv, (float)res);
            else ad[0][q] += (double)(rhv * res);
        } else {
            static_cast<VT*>(P.t)[e] = res;
            const VT sv = static_cast<const VT*>(P.s)[e];
            if (MIXED) {
                f2_add_prod(af[0][q], (float)res, (float)sv);
                f2_add_prod(af[1][q], (float)res, (float)res);
                f2_add_prod(af[2][q], (float)rhv, (float)sv);
                f2_add_prod(af[3][q], (float)rhv, (float)res);
                f2_add_prod(af[4][q], (float)sv, (float)sv);
            } else {
                ad[0][q] += (double)(res * sv);
                ad[1][q] += (double)(res * res);
                ad[2][q] += (double)(rhv * sv);
                ad[3][q] += (double)(rhv * res);
                ad[4][q] += (double)(sv * sv);
            }
        }
    }
}

// ------------------------------------------------------------------------------
// State transitions (run by the block that finishes a request's phase)
// ------------------------------------------------------------------------------
// c[] holds the step's reduced channels for this right-hand side.  The step
// that ends an iteration is C in the row-scaled flows and B in the multigrid
// flow, whose B also yields the new residual's (rh, r) and (r, r).
// `count`: this call keeps the launch's counts of running and restarting right-
// hand sides (false where other blocks form the same transition).
template <bool MIXED, bool AMG>
__device__ void advance(const Prob& P, int ph, RhsState& T, const double* c, const Ctl& ctl, bool count) {
    const int ph_end = AMG ? P_B : P_C;
    if (ph == P_A) T.pending = 0;  // applied by PRE_A of this iteration
    switch (T.mode) {
        case M_INNER:
            if (ph == P_A) {
                const double a = c[0];
                if (MIXED) T.pp ^= 1;
                if (!(fabs(a) > 0.0) || !isfinite(a)) T.mode = M_SKIP;
                else T.alpha = T.rho / a;
            } else if (ph == P_B || ph == P_C) {
                double a = c[0], b = c[1];  // C: (rh, r) and (r, r)
                if (ph == P_B) {
                    T.omega = (b > 0.0 && isfinite(a) && isfinite(b)) ? a / b : 0.0;
                    if (!AMG) break;
                    const double om = T.omega, ts = a, tt = b;
                    a = c[2] - om * c[3];
                    b = c[4] - 2.0 * om * ts + om * om * tt;
                    if (b < 0.0) b = 0.0;  // rounding of a near-cancellation
                }
                T.iters++;
                T.inner_iters++;
                const double rn = sqrt(b);
                T.rnorm = rn;
                const bool finite = isfinite(rn) && isfinite(a);
                // multigrid flow: x moves by this step only if it stayed finite
                T.pending = finite ? 1 : 0;
                // FP32 path: remember the iterate with the smallest residual; an
                // inner solve that stagnates or starts to diverge ends there and
                // hands back that best iterate instead of its last one
                const bool improved = finite && rn < T.rmin;
                if (improved) {
                    T.since_best = (rn < 0.99 * T.rmin) ? 0 : T.since_best + 1;
                    T.rmin = rn;
                } else {
                    T.since_best++;
                }
                T.best_flag = improved ? 1 : 0;
                const bool diverging = MIXED && finite && rn > 1e4 * T.rmin;
                const bool stagnating = MIXED && T.since_best > 200 && 2 * T.since_best > T.inner_iters;
                bool restart = !finite || diverging || stagnating || rn <= T.target || T.iters >= P.maxit ||
                               T.omega == 0.0 || a == 0.0 || (MIXED && T.inner_iters >= P.inner_maxit);
                if (restart) {
                    // x_best only ever holds finite iterates with smaller residuals (or
                    // the zero start), so folding it is always safe
                    T.discard = 0;
                    T.fold_best = improved ? 0 : 1;  // the current iterate is the best one iff it just improved
                    T.best_flag = 0;
                    T.mode = M_RESTART;
                    if (count) atomicAdd(ctl.nrestart, 1);
                } else {
                    T.beta = (a / T.rho) * (T.alpha / T.omega);
                    T.rho = a;
                }
            }
            break;
        case M_SKIP:
            if (ph == ph_end) {
                T.mode = M_RESTART;
                T.discard = 0;
                if (count) atomicAdd(ctl.nrestart, 1);
            }
            break;
        case M_RESTART:
            if (ph == P_A) {
                const double a = c[0], b = c[1];
                if (T.fnorm < 0) {
                    const double fn = sqrt(b);
                    T.fnorm = fn > 0 ? fn : 1.0;
                }
                const double rn = sqrt(a);
                const double rel = rn / T.fnorm;
                if (T.outer > 0 && !(rel < T.relres)) T.stall++;
                else T.stall = 0;
                T.relres = rel;
                if (!isfinite(rn)) {
                    T.mode = M_DONE;
                    T.status = MVGD_ENONFINITE;
                } else if (rel <= P.rtol) {
                    T.mode = M_DONE;
                    T.status = MVGD_OK;
                } else if (T.iters >= P.maxit) {
                    T.mode = M_DONE;
                    T.status = MVGD_ENOCONV;
                } else if (T.outer >= P.max_outer || T.stall >= 4) {
                    T.mode = M_DONE;
                    T.status = MVGD_EBREAKDOWN;
                } else {
                    T.scale = rn;
                }
                if (T.mode == M_DONE && count) {
                    atomicSub(ctl.active, 1);
                    atomicSub(ctl.nrestart, 1);
                }
            } else if (ph == ph_end) {
                const double a = c[0];
                const double rn = sqrt(a);
                T.rho = a;
                T.alpha = 1.0;
                T.omega = 1.0;
                T.beta = 0.0;
                T.pp = 0;
                T.rmin = rn;
                T.rnorm = rn;
                double red = 0.5 * P.rtol / T.relres;
                if (MIXED) red = fmax(P.inner_rtol, red);
                T.target = red * rn;
                T.outer++;
                T.inner_iters = 0;
                T.discard = 0;
                T.best_flag = 0;
                T.fold_best = 0;
                T.since_best = 0;
                T.mode = M_INNER;
                if (count) atomicSub(ctl.nrestart, 1);
            }
            break;
        default:
            break;
    }
}

// Work units of one kind of step: request i's are chunk_base[i] .. chunk_base[i + 1] - 1.
struct ChunkTable {
    const int* chunk_base;  // [count + 1] (several requests)
    int nchunks, pad;
};

// How a launch's blocks find their units.
enum Sharing : int {
    S_SINGLE = 0,  // one request: every gridDim-th unit
    S_LOCAL = 1,   // the same, with few tiles: every block keeps the states itself (local_advance)
    S_LISTED = 2   // several requests: a run of the running ones' units (Units)
};

// A launch of one request may cut its right-hand sides into `groups` of `gq`
// each: block b then works on group b % groups alone, as block b / groups of
// gridDim / groups (the grid is a multiple of `groups`).  A right-hand side's
// arithmetic does not depend on the others of its request, so neither do the
// results.  Unit counts are a group's.
struct ReqTable {
    const Prob* const* prob;       // [count]
    ChunkTable fine;               // kCh-row tiles of level 0 (every Krylov phase; V-cycle level 0)
    ChunkTable lvl[kAmgMaxLevels]; // [l], 1 <= l < mlev: kThreads / amg_group(n_l)-row units of level l
    ChunkTable coarse;             // groups of coarse_rows rows of every coarsest level
    int mlev;                      // largest (levels - 1) among the requests
    int nreq;                      // requests in the launch (1: every unit is request 0's, no lookups)
    int groups, gq;                // right-hand-side groups (1 with several requests)
    int sharing;                   // Sharing
    int act;                       // S_LISTED: the list of running requests is kept
    int ntab;                      // tables in use: fine, lvl[1 .. ntab-2] and coarse
    int coarse_rows;               // rows of a coarsest-level unit (a warp each, at most 8)
    int G[kAmgMaxLevels];          // [l], l >= 1: amg_group of the launch's rows at level l (see amg_lanes)
};

// The block's place among those that share its units.
__device__ __forceinline__ int block_place(const ReqTable& tab) {
    return tab.groups == 1 ? (int)blockIdx.x : (int)blockIdx.x / tab.groups;
}
__device__ __forceinline__ int block_count(const ReqTable& tab) {
    return tab.groups == 1 ? (int)gridDim.x : (int)gridDim.x / tab.groups;
}

// Several requests (S_LISTED).  A block that takes every gridDim-th unit of a step
// meets another request at almost every unit, and each change costs a descriptor and
// state load and, in reducing steps, an arrival: 4 us and more a tile with 32 clouds.
// A run of consecutive units meets one or two requests.  But requests finish at
// different times, and a fixed run of a finished request's units would leave its block
// idle.  So the blocks keep the list of running requests in shared memory, with the
// prefix of their unit counts per table, and cut the running units into equal runs;
// the list is formed anew when the launch's count of running right-hand sides changes.
// Two steps keep the stride, for a run of the dearest request's units would hold up the
// rest: the coarsest solves (a row costs its request's nc) and an A with restarts in it
// (a restart's FP64 residual is several inner steps): 48 -> 38 and 168 -> 116 us.
// 32 clouds of 2,000 .. 65,536 points, four right-hand sides, FP32 flow: an iteration
// 805 -> 624 us (B 134 -> 84, the level-0 steps 68 and 55 -> 51 and 39).
//   act[j]: running request j;  pre[t][j]: running units of table t before it (pre[t][na]:
//   all of them).
// Where that would take more than kActBytes (some 400 requests) the runs are cut from
// all requests' units, finished or not, by the tables themselves.
__host__ __device__ constexpr size_t act_bytes(int count, int ntab) { return sizeof(int) * (size_t)(count + 1) * (1 + ntab); }
constexpr size_t kActBytes = 8 << 10;

// A block's units of one step.
struct Units {
    int lo, step, cnt;  // units lo, lo + step, ... (cnt of them; S_LISTED: of the running ones)
    int cur;            // S_LISTED: place in the list of the unit taken last
    const int* pre;     // S_LISTED: the list's unit counts
};

// The sums of a step's tile partials (nch channels) of a request of few tiles, into
// tot[channel * QT + q]: a warp an entry, tiles across its lanes.  Block-wide.
template <bool MIXED, int QT, int NC>
__device__ __forceinline__ void sum_few_tiles(const Prob& P, int slot, int nch, double (&tot)[NC * QT]) {
    using PT = Part<MIXED>;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int kPerWarp = (NC * QT + kThreads / 32 - 1) / (kThreads / 32);
    constexpr int kEnt = kPerWarp > 4 ? 4 : kPerWarp;  // entries a warp takes at once
    constexpr int kDeep = kEnt >= 4 ? 2 : 4;  // tiles of an entry in flight a lane
    const int nchunk = P.nchunk, Q = P.Q, nq = MVGD_NQ(P), E = nch * nq;
    const PT* part = static_cast<const PT*>(P.part) + (int64_t)slot * NC * nchunk * Q;
    for (int e0 = wid; e0 < E; e0 += kEnt * (kThreads / 32)) {  // warp-uniform
        PT acc[kEnt];
#pragma unroll
        for (int u = 0; u < kEnt; u++) acc[u] = part_zero<PT>();
        for (int l0 = lane; l0 - lane < nchunk; l0 += 32 * kDeep) {
            PT v[kEnt][kDeep];
#pragma unroll
            for (int u = 0; u < kEnt; u++) {
                const int e = e0 + u * (kThreads / 32);
#pragma unroll
                for (int d = 0; d < kDeep; d++) {
                    const int l = l0 + 32 * d;
                    v[u][d] = e < E && l < nchunk ? part_load(part + ((int64_t)(e / nq) * nchunk + l) * Q + e % nq)
                                                  : part_zero<PT>();
                }
            }
#pragma unroll
            for (int u = 0; u < kEnt; u++)
#pragma unroll
                for (int d = 0; d < kDeep; d++)
                    if (l0 - lane + 32 * d < nchunk) acc[u] = part_add(acc[u], v[u][d]);
        }
#pragma unroll
        for (int u = 0; u < kEnt; u++) {
            const int e = e0 + u * (kThreads / 32);
            if (e >= E) break;  // warp-uniform
            const PT t = part_warp_sum(acc[u]);
            if (lane == 0) tot[(e / nq) * QT + e % nq] = part_value(t);
        }
    }
}

// This block has finished `cnt` tiles of request P in a reducing phase: publish
// them (one fence and one atomic per block and request), and if they were the
// request's last tiles, sum all its tile partials and advance the per-RHS state.
// The sum's order depends on the tile count alone: thread t takes tiles t,
// t + 256, ... in batches of kFinBatch whose loads are all issued before any
// is added, each batch summed as a balanced pairwise tree, the batches in
// order; then a butterfly over the warp and a pairwise tree over the 8 warps.
// The dependent chain is log-depth and costs one L2 round trip a batch; the
// additions are F2 in the FP32 flow (see Part).
template <bool MIXED, int QT, bool AMG>
__device__ __forceinline__ void arrive_and_finalize(const Prob& P, int ph, int slot, int cnt, const RhsState* S,
                                                    Part<MIXED> (&fin)[kThreads / 32][chan_count(AMG) * QT],
                                                    double (&tot)[chan_count(AMG) * QT], int* last, const Ctl& ctl) {
    constexpr int NC = chan_count(AMG);
    using PT = Part<MIXED>;
    const int nch = (AMG && ph == P_B) ? kChanAmg : kChan;  // the channels this step reduces
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    // the block's partial stores precede the barrier; thread 0's fence releases
    // them (cumulatively) with the arrival, and on the last arrival its second
    // fence orders every block's partials before the loads below
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        const bool lst = atomicAdd(&P.arrive[slot], (unsigned)cnt) + (unsigned)cnt == (unsigned)P.nchunk;
        if (lst) __threadfence();
        *last = lst;
    }
    __syncthreads();
    if (*last && P.nchunk <= kFinWarpTiles) {
        sum_few_tiles<MIXED, QT, NC>(P, slot, nch, tot);
    } else if (*last) {
        // tiles a batch: a tree over 16 is the sum of two trees over 8, loaded one
        // after the other (16 doubles of two entries would not fit the registers)
        constexpr int kFinBatch = (QT == 1 && !MIXED) ? 16 : 8;
        const int nchunk = P.nchunk, Q = P.Q, nq = MVGD_NQ(P);
        // two channels (or right-hand sides) at a time: 16 loads in flight
#pragma unroll
        for (int e0 = 0; e0 < NC * QT; e0 += 2) {
            const int e1 = e0 + 1;
            const bool on0 = e0 / QT < nch && e0 % QT < nq;                   // step-uniform
            const bool on1 = e1 < NC * QT && e1 / QT < nch && e1 % QT < nq;  // step-uniform
            PT acc0 = part_zero<PT>(), acc1 = part_zero<PT>();
            if (on0 || on1) {
                const PT* part = static_cast<const PT*>(P.part);
                const PT* b0 = &part[((int64_t)slot * NC + e0 / QT) * nchunk * Q + e0 % QT];
                const PT* b1 = &part[((int64_t)slot * NC + e1 / QT) * nchunk * Q + e1 % QT];
                for (int l0 = tid; l0 < nchunk; l0 += kThreads * kFinBatch) {
                    PT t0 = part_zero<PT>(), t1 = part_zero<PT>();
#pragma unroll 1
                    for (int h = 0; h < kFinBatch; h += 8) {
                        PT v0[8], v1[8];
#pragma unroll
                        for (int u = 0; u < 8; u++) {
                            const int l = l0 + (h + u) * kThreads;
                            v0[u] = on0 && l < nchunk ? part_load(b0 + (int64_t)l * Q) : part_zero<PT>();
                            v1[u] = on1 && l < nchunk ? part_load(b1 + (int64_t)l * Q) : part_zero<PT>();
                        }
#pragma unroll
                        for (int w = 1; w < 8; w <<= 1)
#pragma unroll
                            for (int u = 0; u < 8; u += 2 * w) {
                                v0[u] = part_add(v0[u], v0[u + w]);
                                v1[u] = part_add(v1[u], v1[u + w]);
                            }
                        t0 = h == 0 ? v0[0] : part_add(t0, v0[0]);
                        t1 = h == 0 ? v1[0] : part_add(t1, v1[0]);
                    }
                    acc0 = part_add(acc0, t0);
                    acc1 = part_add(acc1, t1);
                }
            }
            if (on0) acc0 = part_warp_sum(acc0);
            if (on1) acc1 = part_warp_sum(acc1);
            if (lane == 0) {
                fin[wid][e0] = acc0;
                if (e1 < NC * QT) fin[wid][e1] = acc1;
            }
        }
        __syncthreads();
        static_assert(kThreads / 32 == 8, "the warp tree below sums 8 warps");
        if (tid < NC * QT) {
            const PT* f = &fin[0][tid];
            constexpr int W = NC * QT;
            tot[tid] = part_value(part_add(part_add(part_add(f[0], f[W]), part_add(f[2 * W], f[3 * W])),
                                           part_add(part_add(f[4 * W], f[5 * W]), part_add(f[6 * W], f[7 * W]))));
        }
    }
    if (*last) {
        __syncthreads();
        if (tid < MVGD_NQ(P)) {
            RhsState T = S[tid];
            double cv[NC];
#pragma unroll
            for (int ch = 0; ch < NC; ch++) cv[ch] = tot[ch * QT + tid];
            advance<MIXED, AMG>(P, ph, T, cv, ctl, true);
            P.st[tid] = T;
        }
        // the grid barrier that ends this phase releases the new states and the
        // reset counter before any block reads them
        if (tid == 0) P.arrive[slot] = 0;
    }
    __syncthreads();
}

enum VStep : int { V_DOWN = 0, V_COARSE = 1, V_UP = 2 };

// The tile a block takes after tile c of a request of nrows rows, if this warp's
// slice of it holds rows (its slice in *slice2); else -1.  Such a tile is staged
// exactly like tile c, so its slice can be requested ahead.
__device__ __forceinline__ int next_tile(int c, int step, int nchunks, int64_t nrows, int wid, int64_t& slice2) {
    const int c2 = c + step;
    if (c2 < 0 || c2 >= nchunks) return -1;
    slice2 = (int64_t)c2 * (kCh / kSlice) + wid;
    return slice2 * kSlice < nrows ? c2 : -1;
}

template <bool MIXED, int QT, bool AMG, int SHARING>
__global__ void __launch_bounds__(kThreads, QT <= 2 ? 3 : 2)
    k_solve(ReqTable tab, Ctl ctl, int iter_budget, int kmax, int nbuf) {
    using VT = typename std::conditional<MIXED, float, double>::type;
    constexpr bool LOCAL = SHARING == S_LOCAL, listed = SHARING == S_LISTED;
    __shared__ RhsState S[QT];
    __shared__ __align__(16) Prob sP;
    __shared__ __align__(16) AmgHeader sH;
    static_assert(sizeof(Prob) % 8 == 0 && sizeof(AmgHeader) % 8 == 0, "descriptors are copied in 8-byte words");
    // per-warp partials of the block's pending tiles, summed into tile partials
    // (in warp order) only when kRedTiles are pending or the request changes:
    // the warps of a block do not wait for each other tile by tile
    constexpr int NC = chan_count(AMG);
    // about 5 KB of pending partials at most
    constexpr int kRedTiles = 80 / (NC * QT) > 16 ? 16 : (80 / (NC * QT) < 2 ? 2 : 80 / (NC * QT));
    __shared__ Part<MIXED> red[kRedTiles][kThreads / 32][NC * QT];
    __shared__ int red_lc[kRedTiles];
    __shared__ Part<MIXED> fin[kThreads / 32][NC * QT];
    __shared__ double tot[NC * QT];
    __shared__ int last;
    __shared__ float vagg[kThreads / kAmgAgg];  // a block's row residuals on a small level (agg_sum)
    __shared__ __align__(8) uint64_t stage_bar[kThreads / 32][2];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int bid = block_place(tab), nblk = block_count(tab);
    // this warp's nbuf slice buffers: kmax column slots, then kmax + 1 weight slots each
    Stager<VT> st;
    st.next_c = -1;
    st.have = -1;
    st.st = 0;
#define MVGD_STAGE_BAR stage_bar[threadIdx.x >> 5]
    if (lane == 0) {
        mbar_init(&stage_bar[wid][0], 1);
        mbar_init(&stage_bar[wid][1], 1);
        fence_mbar_init();
    }
    __syncthreads();

    extern __shared__ __align__(16) unsigned char stage_smem[];
    int* const act = reinterpret_cast<int*>(stage_smem + (size_t)nbuf * (kThreads / kWarp) * stage_bytes_per_warp<VT>(kmax));
    __shared__ int act_sum[kThreads / kWarp];
    int nact = 0;  // running requests in the list
    bool uneven = false;  // some right-hand side restarts in this iteration's A
    bool inner[QT], restart[QT];
    bool any_inner = false, any_restart = false, all_done = true;
    float c1[QT], c2[QT];
    // the request whose state S holds, while no phase has advanced it since
    int held = -1;
    unsigned bar_epoch = 0;  // grid barriers passed (the same count in every block)
    // The descriptor (and multigrid header) of the request the block works on,
    // copied into shared memory when the request changes.  Each grid barrier's
    // acquire leaves none of them in L1, so read from global memory every step
    // would start with a chain of dependent L2 round trips (table -> descriptor
    // -> header -> level arrays) before the first row is touched.  Neither is
    // written while the solver runs.
    int desc = -1;
    bool fit = true;  // that request fits the launch
    auto load_desc = [&](int ri) {
        if (ri == desc) return;
        __syncthreads();  // every thread is done with the previous one
        const unsigned long long* gp =
            reinterpret_cast<const unsigned long long*>(tab.prob[ri]);
        for (int w = tid; w < (int)(sizeof(Prob) / 8); w += kThreads)
            reinterpret_cast<unsigned long long*>(&sP)[w] = __ldcg(gp + w);
        __syncthreads();
        if (AMG && sP.amg != nullptr) {
            const unsigned long long* gh = reinterpret_cast<const unsigned long long*>(sP.amg);
            for (int w = tid; w < (int)(sizeof(AmgHeader) / 8); w += kThreads)
                reinterpret_cast<unsigned long long*>(&sH)[w] = __ldcg(gh + w);
            __syncthreads();
            if (tid == 0) sP.amg = &sH;
            __syncthreads();
        }
        if (tab.groups > 1) {  // this group's columns of every [n][Q] array, its states, partials and counters
            if (tid == 0) {
                const int g = (int)blockIdx.x % tab.groups, q0 = g * tab.gq;
                auto shift = [&](auto*& p) { if (p) p += q0; };
                auto shift_vt = [&](void*& p) { if (p) p = static_cast<VT*>(p) + q0; };
                shift(sP.f); shift(sP.u); shift(sP.r64); shift(sP.st);
                shift_vt(sP.x); shift_vt(sP.xb); shift_vt(sP.r); shift_vt(sP.rh);
                shift_vt(sP.p[0]); shift_vt(sP.p[1]); shift_vt(sP.v[0]); shift_vt(sP.v[1]);
                shift_vt(sP.s); shift_vt(sP.t); shift_vt(sP.ph); shift_vt(sP.sh);
                for (int l = 0; l < kAmgMaxLevels; l++) {
                    shift(sP.vy[l]); shift(sP.vr[l]); shift(sP.vb[l]); shift(sP.vx[l]);
                }
                sP.part = static_cast<Part<MIXED>*>(sP.part) + q0;
                sP.arrive += g * kRedSlots;
                sP.nq = tab.gq;
                sP.q0 = q0;
            }
            __syncthreads();
        }
        desc = ri;
        // a K above the one the staging buffers were sized for (a wrong K in the
        // request list) would overrun shared memory, right-hand sides other than the
        // list's would put a group's columns past the arrays or overrun the states,
        // and a hierarchy of another operator would be read out of bounds: do no work
        // and end the launch
        const Prob& P = sP;
        fit = P.k <= kmax && ((P.amg != nullptr) == AMG) &&
              (tab.groups > 1 ? P.Q == tab.groups * tab.gq : P.Q <= tab.gq);
        if (AMG && fit) fit = P.amg->n == P.n && P.amg->k == P.k;
        if (!fit && tid == 0) atomicCAS(ctl.err, 0, (int)MVGD_EINVAL);
    };
    // This step's masks from the states in S.
    auto masks = [&](int ph) {
        any_inner = any_restart = false;
        all_done = true;
#pragma unroll
        for (int q = 0; q < QT; q++) {
            const int md = S[q].mode;
            inner[q] = md == M_INNER;
            restart[q] = md == M_RESTART;
            any_inner |= inner[q];
            any_restart |= restart[q];
            all_done &= (md == M_DONE);
            c1[q] = (float)(ph == P_A ? S[q].beta : S[q].alpha);
            c2[q] = (float)S[q].omega;
        }
    };
    // Loads request ri's per-RHS state into S (block-wide) and its masks.
    auto enter = [&](int ri, int ph) {
        held = ri;
        load_desc(ri);
        __syncthreads();
        const Prob& P = sP;
        if (tid < QT) {
            if (tid < MVGD_NQ(P) && fit) {
                load_state(S[tid], P.st + tid);
            } else {  // a slot past the request's RHS count: no work of any kind
                S[tid].mode = M_DONE;
                S[tid].pending = 0;
            }
        }
        __syncthreads();
        masks(ph);
    };

    // Level-0 steps that stage the operator take the block's tiles forwards and
    // backwards in turn, so that the slice a warp holds from one step is the first of
    // the next: a block of 1M rows' nine tiles reads eight (an iteration 389 -> 382 us).
    int rev = 0;
    auto table = [&](int t) -> const ChunkTable& { return t == 0 ? tab.fine : (t == tab.ntab - 1 ? tab.coarse : tab.lvl[t]); };
    // The list of running requests and the prefixes of their units (block-wide).
    auto relist = [&]() {
        const int count = tab.nreq, pitch = count + 1;
        if (!tab.act) {
            nact = count;
            return;
        }
        __syncthreads();
        nact = 0;
        st.have = -1;  // tiles are renumbered
        for (int i0 = 0; i0 < count; i0 += kThreads) {
            const int i = i0 + tid;
            bool on = false;
            if (i < count) {
                const Prob* R = tab.prob[i];
                const RhsState* rs = R->st;
                for (int q = 0; q < R->Q; q++) on |= __ldcg(&rs[q].mode) != M_DONE;
            }
            const unsigned who = __ballot_sync(0xffffffffu, on);
            if (lane == 0) act_sum[wid] = __popc(who);
            __syncthreads();
            int at = nact, all = 0;
            for (int w = 0; w < kThreads / kWarp; w++) {
                if (w < wid) at += act_sum[w];
                all += act_sum[w];
            }
            if (on) act[at + __popc(who & ((1u << lane) - 1u))] = i;
            nact += all;
            __syncthreads();
        }
        for (int t = wid; t < tab.ntab; t += kThreads / kWarp) {
            const ChunkTable& T = table(t);
            int* pre = act + pitch * (1 + t);
            int run = 0;
            for (int j0 = 0; j0 < nact; j0 += 32) {
                const int j = j0 + lane;
                const int n = j < nact ? T.chunk_base[act[j] + 1] - T.chunk_base[act[j]] : 0;
                int x = n;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, x, o);
                    if (lane >= o) x += y;
                }
                if (j < nact) pre[j] = run + x - n;
                run += __shfl_sync(0xffffffffu, x, 31);
            }
            if (lane == 0) pre[nact] = run;
        }
        __syncthreads();
    };
    // This block's units of table t; unit i of them: its request, its place in the
    // request, and (returned) its number among the units in the list.
    // runs: a run of them (S_LISTED), else every nblk-th.
    auto units_of = [&](int t, bool runs) {
        Units U;
        U.cur = 0;
        if (listed) {
            U.pre = tab.act ? act + (tab.nreq + 1) * (1 + t) : table(t).chunk_base;
            const int n = U.pre[nact];
            if (runs) {
                U.lo = (int)(bid * (int64_t)n / nblk);
                U.cnt = (int)((bid + 1) * (int64_t)n / nblk) - U.lo;
                U.step = 1;
            } else {
                U.lo = bid;
                U.cnt = bid < n ? (n - 1 - bid) / nblk + 1 : 0;
                U.step = nblk;
            }
            int hi = nact;  // the last j with pre[j] <= lo
            while (hi - U.cur > 1) {
                const int mid = (U.cur + hi) >> 1;
                if (U.pre[mid] <= U.lo) U.cur = mid;
                else hi = mid;
            }
        } else {
            const int n = table(t).nchunks;
            U.pre = nullptr;
            U.lo = bid;
            U.step = nblk;
            U.cnt = bid < n ? (n - 1 - bid) / nblk + 1 : 0;
        }
        return U;
    };
    auto unit_at = [&](Units& U, int i, int& ri, int& place) -> int {
        if (listed) {
            const int a = U.lo + i * U.step;
            while (a >= U.pre[U.cur + 1]) U.cur++;
            while (a < U.pre[U.cur]) U.cur--;
            ri = tab.act ? act[U.cur] : U.cur;
            place = a - U.pre[U.cur];
            return a;
        }
        ri = 0;
        place = U.lo + i * nblk;
        return place;
    };

    // One request of few tiles (LOCAL): after a reducing step's barrier every block
    // sums the tile partials and advances its own copy of the states, the same
    // operations on the same values everywhere.  That takes the arrival counter, the
    // last block's sums before the barrier and the states' way through L2 off the
    // critical path.  Block 0 of a group keeps the launch's counts; they are read a step
    // later, after the next barrier, and the states go back to memory at the end.
    // Reducing steps with it: 7.4 -> 4.8 us at 2,562 rows in FP64, 8.2 and 9.9 -> 4.7 us
    // (A, B) at 20,000 rows.
    auto local_advance = [&](int ph) {
        const int nch = (AMG && ph == P_B) ? kChanAmg : kChan;
        sum_few_tiles<MIXED, QT, NC>(sP, red_slot(ph), nch, tot);
        __syncthreads();
        if (tid < MVGD_NQ(sP)) {
            RhsState T = S[tid];
            double cv[NC];
#pragma unroll
            for (int ch = 0; ch < NC; ch++) cv[ch] = tot[ch * QT + tid];
            advance<MIXED, AMG>(sP, ph, T, cv, ctl, bid == 0);
            S[tid] = T;
        }
        __syncthreads();
        masks(ph);
    };
    if constexpr (LOCAL) enter(0, P_PRE_A);
    int stop_word = 0;  // LOCAL: the stop word at the end of the last iteration

    // One Krylov phase over every request's level-0 tiles, then the grid barrier.
    // the step that ends an iteration: it restarts the Krylov vectors of the
    // right-hand sides in RESTART and its barrier precedes the exit test
    constexpr int ph_end = AMG ? P_B : P_C;
    auto fine_phase = [&](int ph) -> bool {
        const bool reduce = ph == P_A || ph == P_B || ph == P_C;
        const int nch = (AMG && ph == P_B) ? kChanAmg : kChan;  // the channels this step reduces
        const int slot = red_slot(ph);
        int cur = -1, tiles = 0, nred = 0;
        // tile partials of the pending tiles of request P: each the sum of its 8 warp partials (a pairwise tree)
        auto flush = [&](const Prob& P) {
            __syncthreads();
            for (int e = tid; e < nred * NC * QT; e += kThreads) {
                const int t = e / (NC * QT), j = e % (NC * QT);
                if (j / QT >= nch) continue;
                const Part<MIXED>* rw = &red[t][0][j];
                constexpr int W = NC * QT;  // stride between warps
                const Part<MIXED> v = part_add(part_add(part_add(rw[0], rw[W]), part_add(rw[2 * W], rw[3 * W])),
                                               part_add(part_add(rw[4 * W], rw[5 * W]), part_add(rw[6 * W], rw[7 * W])));
                const int ch = j / QT, q = j % QT;
                if (q < MVGD_NQ(P))
                    static_cast<Part<MIXED>*>(P.part)[(((int64_t)slot * NC + ch) * P.nchunk + red_lc[t]) * P.Q + q] = v;
            }
            __syncthreads();
            nred = 0;
        };
        Units U = units_of(0, !(ph == P_A && uneven));
        for (int i = 0;; i++) {
            int ri = -1, lc = 0, c = 0;
            if (i < U.cnt) c = unit_at(U, rev ? U.cnt - 1 - i : i, ri, lc);
            if (ri != cur || ri < 0) {  // (a block may have no level-0 tile at all)
                // leaving request `cur`: publish this block's tiles of it
                if (cur >= 0 && reduce && tiles > 0) {
                    flush(sP);  // still request cur's descriptor
                    if constexpr (!LOCAL)
                        arrive_and_finalize<MIXED, QT, AMG>(sP, ph, slot, tiles, S, fin, tot, &last, ctl);
                }
                if (ri < 0) break;
                cur = ri;
                tiles = 0;
                if constexpr (LOCAL) masks(ph);
                else enter(ri, ph);
            }
            if (all_done) continue;  // the whole request is finished: no work, no arrival
            const Prob& P = sP;
            const int64_t r = (int64_t)lc * kCh + tid;
            const int64_t slice = (int64_t)lc * (kCh / kSlice) + wid;
            F2 af[NC][QT];
            double ad[NC][QT];
#pragma unroll
            for (int ch = 0; ch < NC; ch++)
#pragma unroll
                for (int q = 0; q < QT; q++) { af[ch][q].hi = 0.0f; af[ch][q].lo = 0.0f; ad[ch][q] = 0.0; }
            // warp-uniform: lane 0 stages the whole slice and every lane waits for it
            const bool staged = (ph == P_A || ph == P_B) && any_inner && slice * kSlice < P.n && st.ok();
            if (staged) {
                int64_t slice2 = 0;
                const int cn = listed ? -1 : next_tile(c, rev ? -nblk : nblk, tab.fine.nchunks, P.n, wid, slice2);
                // FP32 multigrid flow: the hierarchy's level-0 weights (the operator's hi
                // values, copied at set-up), the array the V-cycle's level-0 steps read too
                const void* vsrc = (AMG && MIXED) ? static_cast<const void*>(P.amg->lv[0].val) : P.val;
                const int b = st.acquire(kmax, nbuf, MVGD_STAGE_BAR, c, slice, cn, slice2, P.col, vsrc, (int)sizeof(VT), P.k, ctl.err);
                const int* colS = st.col(kmax, nbuf, b);
                const VT* valS = static_cast<const VT*>(st.val(kmax, nbuf, b));
                auto landed = [&]() { return st.wait(MVGD_STAGE_BAR, b, ctl.err); };
                if constexpr (AMG) amg_spmv_row<MIXED, QT>(P, r, r < P.n, ph, S, inner, af, ad, colS, valS, landed);
                else spmv_row<MIXED, QT>(P, r, r < P.n, ph, S, inner, c1, c2, af, ad, colS, valS, landed);
            }
            if (r < P.n) {
                // a restart computes its residual in A and resets the Krylov vectors in
                // the iteration's last step, so that its first inner step starts at the
                // next iteration
                if (ph == P_A) {
                    if (any_restart) restart_row<MIXED, QT, NC>(P, r, ph, S, restart, ad);
                } else if (ph == ph_end) {
                    if constexpr (!AMG) {
                        if (any_inner) {
                            if (MIXED) elementwise_row<MIXED, QT>(P, r, ph, S, inner, restart, af);
                            else c_row_f64<QT>(P, r, S, inner, ad);
                        }
                    }
                    if (any_restart) restart_row<MIXED, QT, NC>(P, r, ph, S, restart, ad);
                } else if (ph != P_B) {
                    if constexpr (AMG) amg_pre_row<MIXED, QT>(P, r, ph, S, inner, restart);
                    else elementwise_row<MIXED, QT>(P, r, ph, S, inner, restart, af);
                }
            }
            if (!reduce) continue;
            // tile partials in a fixed order: FP32 partials within the warp in FP32,
            // then (at the next flush) the 8 warps in order
            {
                const bool with64 = any_restart || !MIXED;
                if constexpr (AMG) {
                    if (ph == P_B) tile_partials<MIXED, QT, NC, kChanAmg>(af, ad, with64, lane, red[nred][wid]);
                    else tile_partials<MIXED, QT, NC, kChan>(af, ad, with64, lane, red[nred][wid]);
                } else {
                    tile_partials<MIXED, QT, NC, kChan>(af, ad, with64, lane, red[nred][wid]);
                }
            }
            if (tid == 0) red_lc[nred] = lc;
            nred++;
            tiles++;
            if (nred == kRedTiles) flush(P);
        }
        // the stop word is written only before the last barrier of an iteration and
        // read only after it, so every block takes the same exit decision
        if (ph == ph_end && blockIdx.x == 0 && tid == 0 && ctl.cancel && *(const volatile int*)ctl.cancel != 0)
            *ctl.stop = 1;
        if (reduce && !LOCAL) held = -1;  // the states were advanced at the arrivals
        if (ph == P_A || ph == P_B) rev ^= 1;
        const bool ok = grid_sync(ctl.bar, bar_epoch, ctl.err, ctl.limit,
                                  !(ctl.withhold && blockIdx.x == 0 && bar_epoch == 0));
        trace_step(ctl, (unsigned)ph);
        if constexpr (LOCAL) {
            // (loaded with the partials: no round trip of its own)
            if (ph == ph_end) stop_word = *(const volatile int*)ctl.stop;
            if (reduce && ok) local_advance(ph);
        }
        return ok;
    };

    // PRE_A / PRE_B of the multigrid flow with one or two right-hand sides:
    // up to NT of the block's tiles of one request at a time (amg_pre_rows), so
    // their loads overlap; a request with a RESTART goes row by row (the fold of
    // x into u).  The rows and their arithmetic are those of fine_phase.
    auto pre_phase = [&](int ph) -> bool {
        constexpr int NT = MIXED ? (QT == 1 ? 4 : 2) : (QT == 1 ? 2 : 1);  // operands in registers
        const int step = listed ? 1 : nblk;  // from a unit's place to the block's next one's
        Units U = units_of(0, true);
        for (int i = 0; i < U.cnt;) {
            int ri, lc;
            unit_at(U, i, ri, lc);
            if (ri != held) enter(ri, ph);
            int n;
            if (listed) n = min(NT, min(U.cnt - i, U.pre[U.cur + 1] - U.lo - i));
            else n = min(NT, U.cnt - i);
            if (!all_done) {
                const Prob& P = sP;
                if (any_restart) {
                    for (int k = 0; k < n; k++) {
                        const int64_t r = (int64_t)(lc + k * step) * kCh + tid;
                        if (r < P.n) amg_pre_row<MIXED, QT>(P, r, ph, S, inner, restart);
                    }
                } else {
                    int64_t rows[NT];
                    bool ok[NT];
#pragma unroll
                    for (int k = 0; k < NT; k++) {
                        rows[k] = (int64_t)(lc + k * step) * kCh + tid;
                        ok[k] = k < n && rows[k] < P.n;
                    }
                    amg_pre_rows<MIXED, QT, NT>(P, rows, ok, ph, S, inner);
                }
            }
            i += n;
        }
        const bool ok = grid_sync(ctl.bar, bar_epoch, ctl.err, ctl.limit,
                                  !(ctl.withhold && blockIdx.x == 0 && bar_epoch == 0));
        trace_step(ctl, (unsigned)ph);
        return ok;
    };

    // One step of the V-cycle applied to p (side 0) or s (side 1) of every
    // INNER right-hand side, then the grid barrier.
    auto vstep = [&](int kind, int l, int side) -> bool {
        int cur = -1;
        Units U = kind == V_COARSE ? units_of(tab.ntab - 1, false) : units_of(l, true);
        for (int i = 0; i < U.cnt; i++) {
            int ri, lc;
            const int c = unit_at(U, rev && kind != V_COARSE && l == 0 ? U.cnt - 1 - i : i, ri, lc);
            if (ri != cur) {
                cur = ri;
                // V-cycle steps leave the states alone: the one loaded by the
                // preceding PRE phase (or step) stays valid
                if (ri != held) enter(ri, P_PRE_A);
            }
            const Prob& P = sP;
            const int m = P.amg_levels - 1;  // the request's coarsest level
            if (!any_inner || (kind != V_COARSE && l >= m)) continue;
            const AmgHeader& H = *P.amg;
            const int Q = P.Q;
            const VT* B0 = static_cast<const VT*>(side == 0 ? P.p[0] : P.s);
            VT* X0 = static_cast<VT*>(side == 0 ? P.ph : P.sh);
            if (kind == V_COARSE) {
                // a warp per row, every right-hand side at once
                const int64_t rho = (int64_t)lc * tab.coarse_rows + wid;
                if (wid >= tab.coarse_rows || rho >= H.nc) continue;
                auto store = [&](int q, float x) {
                    if (q >= MVGD_NQ(P) || S[q].mode != M_INNER) return;
                    if (m == 0) X0[rho * Q + q] = (VT)x;
                    else P.vx[m][rho * Q + q] = x;
                };
                if (m == 0) coarse_rows<QT>(H, rho, B0, Q, store);
                else coarse_rows<QT>(H, rho, P.vb[m], Q, store);
                continue;
            }
            const int64_t nl = H.lv[l].n;
            // level 0: a lane per row (staged slices); level >= 1: G lanes per row
            const int G = l == 0 ? 1 : amg_lanes(tab.G[l], nl, QT);
            const int64_t r = (int64_t)lc * (kThreads / G) + tid / G;
            const bool valid = r < nl;
            // whole warps past the level's end have nothing to do, except in a down
            // step whose aggregates span warps (G >= 8: block barriers in agg_sum)
            const bool warp_idle = (int64_t)lc * (kThreads / G) + (wid * kWarp) / G >= nl;
            if (warp_idle && (kind == V_UP || G < 8)) continue;
            // level 0 reads the operator's slice from a staged buffer, like A and B
            const int* colS = nullptr;
            const float* w0S = nullptr;
            int b = 0;
            if (l == 0) {
                if (!st.ok()) continue;
                const int64_t slice = (int64_t)lc * (kCh / kSlice) + wid;
                int64_t slice2 = 0;
                const int cn = listed ? -1 : next_tile(c, rev ? -nblk : nblk, tab.fine.nchunks, nl, wid, slice2);
                b = st.acquire(kmax, nbuf, MVGD_STAGE_BAR, c, slice, cn, slice2, P.col, H.lv[0].val, 4, P.k, ctl.err);
                colS = st.col(kmax, nbuf, b);
                w0S = static_cast<const float*>(st.val(kmax, nbuf, b));
            }
            const float sig = (float)P.sigma;
            const int k = P.k;
            auto a0 = [&](float xi, auto&& xv) {
                return l == 0 ? a0_row_staged(colS, w0S, lane, k, sig, xi, xv) : a0_row(H, r, xi, xv);
            };
            if (kind == V_DOWN) {
                float* Yn = (l + 1 < m) ? P.vy[l + 1] : nullptr;
                const float* Y = P.vy[l];
                float bi[QT], yi[QT];
#pragma unroll
                for (int q = 0; q < QT; q++) {  // the row's own values, loaded while the slice lands
                    bi[q] = (valid && inner[q]) ? (l == 0 ? (float)B0[r * Q + q] : P.vb[l][r * Q + q]) : 0.0f;
                    yi[q] = (valid && inner[q]) ? Y[r * Q + q] : 0.0f;
                }
                if (l == 0) {
                    // level 0: every right-hand side in one pass over the neighbours
                    if (!st.wait(MVGD_STAGE_BAR, b, ctl.err)) continue;
                    float ay[QT];
#pragma unroll
                    for (int q = 0; q < QT; q++) ay[q] = 0.0f;
                    if (valid)
                        a0_rows_staged<QT>(colS, w0S, lane, k, sig, yi, ay,
                                           [&](int64_t j, float (&x)[QT]) { load_row<QT>(Y, j, Q, x); });
#pragma unroll
                    for (int q = 0; q < QT; q++)
                        if (inner[q]) vdown_finish(H, 0, 1, r, valid, Q, q, bi[q] - ay[q], P.vr[0], P.vb[1], Yn, vagg);
                    continue;
                }
                // level >= 1: every right-hand side in one pass over the row's entries
                float ay[QT];
                al_rows<QT>(H.lv[l], r, valid, G, yi, [&](int64_t j, float (&x)[QT]) { load_row<QT>(Y, j, Q, x); },
                            ay);
#pragma unroll
                for (int q = 0; q < QT; q++) {
                    if (!inner[q]) continue;  // block-uniform
                    vdown_finish(H, l, G, r, valid, Q, q, bi[q] - ay[q], P.vr[l], P.vb[l + 1], Yn, vagg);
                }
            } else {
                const float* Xc = P.vx[l + 1];
                float yi[QT], rr[QT];
#pragma unroll
                for (int q = 0; q < QT; q++) {
                    yi[q] = (valid && inner[q]) ? P.vy[l][r * Q + q] : 0.0f;
                    rr[q] = (valid && inner[q]) ? P.vr[l][r * Q + q] : 0.0f;
                }
                if (l == 0) {
                    // level 0: x = y + x_c + d (r - A_0 P x_c), every right-hand side in one pass
                    if (!st.wait(MVGD_STAGE_BAR, b, ctl.err) || !valid) continue;
                    float xc[QT], apx[QT];
                    load_row<QT>(Xc, r / kAmgAgg, Q, xc);
                    a0_rows_staged<QT>(colS, w0S, lane, k, sig, xc, apx,
                                       [&](int64_t j, float (&x)[QT]) { load_row<QT>(Xc, j / kAmgAgg, Q, x); });
                    const float d0 = H.lv[0].dinv[r];
#pragma unroll
                    for (int q = 0; q < QT; q++)
                        if (inner[q]) X0[r * Q + q] = (VT)(yi[q] + xc[q] + d0 * (rr[q] - apx[q]));
                    continue;
                }
                if (!valid && G == 1) continue;
                // level >= 1: x = y + x_c + d (r - A_l P x_c), every right-hand side in one pass
                float xc[QT], apx[QT];
#pragma unroll
                for (int q = 0; q < QT; q++) xc[q] = 0.0f;
                if (valid) load_row<QT>(Xc, r / kAmgAgg, Q, xc);
                al_rows<QT>(H.lv[l], r, valid, G, xc,
                            [&](int64_t j, float (&x)[QT]) { load_row<QT>(Xc, j / kAmgAgg, Q, x); }, apx);
                if (!valid || (lane & (G - 1)) != 0) continue;
                const float dl = H.lv[l].dinv[r];
#pragma unroll
                for (int q = 0; q < QT; q++)
                    if (inner[q]) P.vx[l][r * Q + q] = yi[q] + xc[q] + dl * (rr[q] - apx[q]);
            }
        }
        if (kind != V_COARSE && l == 0) rev ^= 1;
        const bool ok = grid_sync(ctl.bar, bar_epoch, ctl.err, ctl.limit,
                                  !(ctl.withhold && blockIdx.x == 0 && bar_epoch == 0));
        trace_step(ctl, 0x1000u | ((unsigned)side << 8) | ((unsigned)kind << 4) | (unsigned)l);
        return ok;
    };
    auto vcycle = [&](int side) -> bool {
        for (int l = 0; l < tab.mlev; l++)
            if (!vstep(V_DOWN, l, side)) return false;
        if (!vstep(V_COARSE, 0, side)) return false;
        for (int l = tab.mlev - 1; l >= 0; l--)
            if (!vstep(V_UP, l, side)) return false;
        return true;
    };

    // the counts are stable between the barrier that follows their last change and the
    // next reducing step: identical in every block.  A launch that is told to stop leaves
    // at an iteration's end, before the next PRE_A: what PRE_A applies (a pending step, a
    // new p, the fold into u) the saved states still ask for, and a later launch of the
    // same request would apply it again.  LOCAL reads its count behind PRE_A, but leaves
    // there only with every right-hand side done, when PRE_A changes nothing.
    auto finished = [&]() { return *(volatile int*)ctl.active == 0; };
    auto stopped = [&]() { return LOCAL ? stop_word != 0 : *(volatile int*)ctl.stop != 0; };
    int running = -1;  // the launch's running right-hand sides when the list was formed
    for (int it = 0; it < iter_budget; ++it) {
        bool ok = true, leave = false;
        if (listed && *(volatile int*)ctl.active != running) {
            running = *(volatile int*)ctl.active;
            relist();
        }
        if (listed) uneven = *(volatile int*)ctl.nrestart > 0;
        if (AMG) {
            if constexpr (QT <= 2) {
                ok = pre_phase(P_PRE_A);
                leave = LOCAL && ok && finished();
                if (!leave)
                    ok = ok && vcycle(0) && fine_phase(P_A) && pre_phase(P_PRE_B) && vcycle(1) && fine_phase(P_B);
            } else {
                ok = fine_phase(P_PRE_A);
                leave = LOCAL && ok && finished();
                if (!leave)
                    ok = ok && vcycle(0) && fine_phase(P_A) && fine_phase(P_PRE_B) && vcycle(1) && fine_phase(P_B);
            }
        } else {
            // read after the last barrier of the previous iteration: identical in every block
            const bool pre_a = !MIXED || *(volatile int*)ctl.nrestart > 0;
            for (int ph = 0; ph < P_COUNT && ok && !leave; ++ph) {
                if (ph == P_PRE_A && !pre_a) continue;
                if (ph == P_PRE_B && MIXED) continue;
                ok = fine_phase(ph);
                if (LOCAL && ph == P_PRE_A) leave = ok && finished();
            }
        }
        if (!ok || leave) break;  // (an error exit: after the drain below)
        if (stopped() || (!LOCAL && finished())) break;
    }
    if (LOCAL && bid == 0 && fit && tid < MVGD_NQ(sP)) sP.st[tid] = S[tid];
    // copies still landing (a missed wait): bounded waits before the block's
    // shared memory is released
    st.drain(MVGD_STAGE_BAR);
}

// The dynamic shared memory that an instantiation's launches may ask for, set to the
// largest any of them does and not to the launch's own: a kernel's attribute is the
// process's, and another thread's smaller launch could lower it between this one's set
// and its launch.
constexpr size_t kStageMax = 112 << 10;  // two buffers a warp, at most
constexpr size_t kDynamicMax = kStageMax + kActBytes;
static_assert(stage_bytes_per_warp<double>(kMaxK) * (kThreads / kWarp) <= kStageMax, "one buffer a warp always fits");

// Slice buffers per warp.  One by default: a second buffer (the next tile's
// slice requested ahead) costs a resident block per SM, and on GB300 at 1M
// rows, K = 20, three single-buffered blocks ran the FP32 multigrid solve 8 %
// faster than two double-buffered ones (every step that is not a product
// loses the third block's latency hiding).  mvgd_set_launch_tuning selects two.
// With several requests it is one whatever is selected: their steps ask for
// nothing ahead, and a second buffer would only take its block (4 requests of
// 200,000 rows, FP32: 32.6 ms a batch with one, 38.5 with an idle second one,
// 37.9 with the request's next tile asked for ahead, whose code also cost the
// launches with one buffer 1 %).
template <typename VT, int SHARING>
int stage_buffers(int kmax) {
    if (SHARING != S_LISTED && tuned_stage_buffers() == 2 &&
        2 * stage_bytes_per_warp<VT>(kmax) * (kThreads / kWarp) <= kStageMax)
        return 2;
    return 1;
}

// Resident blocks of one instantiation (0: a CUDA error).
template <bool MIXED, int QT, bool AMG, int SHARING>
int solve_capacity(int kmax, size_t* smem_out = nullptr, size_t more = 0) {
    using VT = typename std::conditional<MIXED, float, double>::type;
    auto fn = k_solve<MIXED, QT, AMG, SHARING>;
    const size_t smem = stage_bytes_per_warp<VT>(kmax) * (kThreads / kWarp) * stage_buffers<VT, SHARING>(kmax) + more;
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDynamicMax) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kThreads, smem) != cudaSuccess)
        return 0;
    const int want = tuned_solver_blocks_per_sm();
    if (want > 0 && want < per_sm) per_sm = want;
    if (smem_out) *smem_out = smem;
    return sms * per_sm;
}

template <bool MIXED, int QT, bool AMG, int SHARING>
mvgd_status launch_solve_as(const ReqTable& tab, Ctl ctl, int budget, int kmax, cudaStream_t s) {
    using VT = typename std::conditional<MIXED, float, double>::type;
    size_t smem = 0;
    int grid = solve_capacity<MIXED, QT, AMG, SHARING>(
        kmax, &smem, tab.act ? act_bytes(tab.nreq, tab.ntab) : 0);
    if (grid < 1) return MVGD_ECUDA;
    // a block for every unit of the step that has most of them (a level whose rows
    // must take many lanes, or the coarsest one of a small system, can have more
    // units than level 0)
    int units = tab.fine.nchunks;
    if (AMG) {
        for (int l = 1; l < tab.mlev; l++) units = units > tab.lvl[l].nchunks ? units : tab.lvl[l].nchunks;
        units = units > tab.coarse.nchunks ? units : tab.coarse.nchunks;
    }
    units *= tab.groups;
    if (grid > units) grid = units;
    grid -= grid % tab.groups;  // units is a multiple of groups, and groups <= 8 blocks always fit
    int nbuf = stage_buffers<VT, SHARING>(kmax);
    ReqTable t = tab;
    void* args[] = {(void*)&t, (void*)&ctl, (void*)&budget, (void*)&kmax, (void*)&nbuf};
    MVGD_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)k_solve<MIXED, QT, AMG, SHARING>, dim3(grid), dim3(kThreads), args,
                                              smem, s));
    return MVGD_OK;
}

// The step kernel that skips nothing is the row-scaled FP64 or the multigrid one: the
// mixed row-scaled flow leaves PRE_A out on a count that every block must see at once.
template <bool MIXED, bool AMG>
constexpr bool has_local() { return AMG || !MIXED; }

template <bool MIXED, int QT, bool AMG>
mvgd_status launch_solve(const ReqTable& tab, Ctl ctl, int budget, int kmax, cudaStream_t s) {
    if constexpr (has_local<MIXED, AMG>()) {
        if (tab.sharing == S_LOCAL) return launch_solve_as<MIXED, QT, AMG, S_LOCAL>(tab, ctl, budget, kmax, s);
    }
    if (tab.sharing == S_LISTED) return launch_solve_as<MIXED, QT, AMG, S_LISTED>(tab, ctl, budget, kmax, s);
    return launch_solve_as<MIXED, QT, AMG, S_SINGLE>(tab, ctl, budget, kmax, s);
}

// The multigrid flows' widest instantiations, which take a third of their build, have
// translation units of their own (solve_*_amg_wide.cu).
extern template mvgd_status launch_solve<true, 8, true>(const ReqTable&, Ctl, int, int, cudaStream_t);
extern template mvgd_status launch_solve<false, 8, true>(const ReqTable&, Ctl, int, int, cudaStream_t);

template <bool MIXED, bool AMG>
mvgd_status dispatch_q(int Q, const ReqTable& tab, Ctl ctl, int budget, int kmax, cudaStream_t s) {
    if (Q <= 1) return launch_solve<MIXED, 1, AMG>(tab, ctl, budget, kmax, s);
    if (Q <= 2) return launch_solve<MIXED, 2, AMG>(tab, ctl, budget, kmax, s);
    if (Q <= 4) return launch_solve<MIXED, 4, AMG>(tab, ctl, budget, kmax, s);
    return launch_solve<MIXED, 8, AMG>(tab, ctl, budget, kmax, s);
}

// Right-hand sides a group of a one-request launch takes (Q: no split): the
// fewest (1, 2 or 4, dividing Q) whose level-0 units all fit the GPU at once.
// A small system with several right-hand sides leaves most SMs idle, and its
// steps last as long as one SM needs for all of them -- in FP64 above all,
// where an SM's pipe takes 2 FMAs a clock.  Once a second round of units would
// start, the operator read again for each group costs more than it gives.
// 16,000 rows x 8 right-hand sides in FP64: 257 us an iteration unsplit, 115 in
// groups of two; 7,001 rows x 4 in FP32: 124 and 64.
template <bool MIXED, bool AMG>
int rhs_group(int Q, int tiles, int kmax) {
    constexpr int kOneRequest = has_local<MIXED, AMG>() ? S_LOCAL : S_SINGLE;
    const int64_t t = tiles;
    if (t * Q <= solve_capacity<MIXED, 1, AMG, kOneRequest>(kmax)) return 1;
    if (Q > 2 && Q % 2 == 0 && t * (Q / 2) <= solve_capacity<MIXED, 2, AMG, kOneRequest>(kmax)) return 2;
    if (Q > 4 && Q % 4 == 0 && t * (Q / 4) <= solve_capacity<MIXED, 4, AMG, kOneRequest>(kmax)) return 4;
    return Q;
}


// One translation unit an instantiation: launch of a request table, and the
// right-hand sides a group of a one-request launch takes.
#define MVGD_SOLVE_FLOW(name)                                                                                   \
    mvgd_status launch_##name(int Q, const ReqTable& tab, Ctl ctl, int budget, int kmax, cudaStream_t s);        \
    int rhs_group_##name(int Q, int tiles, int kmax);
MVGD_SOLVE_FLOW(mixed_amg)
MVGD_SOLVE_FLOW(mixed_plain)
MVGD_SOLVE_FLOW(fp64_amg)
MVGD_SOLVE_FLOW(fp64_plain)
#undef MVGD_SOLVE_FLOW

}  // namespace solver
}  // namespace mvgd
