// Aggregation multigrid hierarchy of sigma I - L and its standalone V-cycle.
//
// The paper solves its MVGD systems with algebraic multigrid and reports its
// CPU time growing about linearly with N (Sec. 4.2, the timing table), without
// naming the variant.  This is plain aggregation (Braess 1995) on the
// stored row order, whose consecutive rows are spatial neighbours (the kNN
// step sorts points by cell along a Z-order curve):
//   * aggregate I of level l is rows kAmgAgg*I .. kAmgAgg*I + kAmgAgg-1;
//   * level l+1 is the Galerkin product P^T A_l P (entry (I, J) sums a_ij over
//     the rows of aggregate I and the columns of aggregate J), computed in
//     FP64 one warp per coarse row, with a fixed summation order;
//   * the first level with at most kAmgCoarsest rows is inverted by blocked
//     Gauss-Jordan elimination with partial pivoting (FP32, a cluster of CTAs),
//     refined by two Newton-Schulz steps to the FP64 level;
//   * smoothing is a Jacobi step x += d (b - A x) with d_i = omega / a_ii on
//     rows with a strong diagonal (a_ii > theta sum_j |a_ij|; omega = 0.9,
//     theta = 0.3) and the l1 scaling d_i = 1 / sum_j |a_ij| (Baker, Falgout,
//     Kolev, Yang 2011), positive whatever the sign pattern, on the others:
//     MVGD rows with few neighbours on irregular samples can have a small or
//     negative diagonal.  Against l1-Jacobi everywhere this took 15-30 % off
//     the preconditioned iteration counts (K 12 and 20, 7k-262k points).
// Everything the V-cycle reads is FP32; the FP64 Galerkin values stay
// available for inspection.
#include <cooperative_groups.h>
#include <limits.h>

#include <string.h>

#include <type_traits>

#include "vcycle.cuh"

namespace mvgd {
namespace {

struct AmgLayout {
    AmgHeader* hdr;
    AmgHeader h;  // host copy of the pointers and sizes
};

AmgLayout amg_layout(void* ws, int64_t n, int k) {
    AmgLayout A;
    memset(&A.h, 0, sizeof(A.h));
    Carver cv(ws);
    A.hdr = cv.take<AmgHeader>(1);
    int64_t sizes[kAmgMaxLevels];
    const int nlev = amg_levels(n, sizes);
    A.h.nlev = nlev;
    A.h.k = k;
    A.h.n = n;
    for (int l = 0; l < nlev; l++) {
        const int64_t nl = sizes[l], np = n_padded(nl);
        AmgLevel& L = A.h.lv[l];
        L.n = nl;
        if (l == 0) {
            L.val = cv.take<float>(np * (k + 1));
        } else {
            L.col = cv.take<int32_t>(np * kAmgStride);
            L.val = cv.take<float>(np * kAmgStride);
            L.val64 = cv.take<double>(np * kAmgStride);
            L.cnt = cv.take<int32_t>(np);
            L.sw = cv.take<int32_t>(np / kSlice);
            L.rs = cv.take<float>(np);
        }
        L.dinv = cv.take<float>(np);
    }
    const int64_t nc = nlev > 0 ? sizes[nlev - 1] : 0;
    A.h.nc = nc;
    A.h.cinv = cv.take<float>(nc * nc);
    A.h.dense64 = cv.take<double>(nc * nc);
    A.h.cinv64 = cv.take<double>(nc * nc);
    A.h.ns_x = cv.take<double>(nc * nc);
    A.h.ns_t = cv.take<double>(nc * nc);
    A.h.ns_s = cv.take<float>(2 * nc * nc);
    A.h.bytes = cv.used;
    return A;
}

// Where the set-up reads the operator's own weights (FP64, or hi + lo).
struct OpView {
    const int32_t* col;
    const void* val;
    const float* val_lo;
    int prec;
};

__device__ __forceinline__ double op_weight(const OpView& O, int64_t idx) {
    return O.prec == MVGD_FP64 ? static_cast<const double*>(O.val)[idx]
                               : (double)static_cast<const float*>(O.val)[idx] + (double)O.val_lo[idx];
}

// The header, and the slice widths that the coarse levels collect, zeroed.
__global__ void k_amg_header(AmgHeader h, AmgHeader* dst) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, threads = (int64_t)gridDim.x * blockDim.x;
    if (t == 0) *dst = h;
    for (int l = 1; l < h.nlev; l++)
        for (int64_t s = t; s < n_padded(h.lv[l].n) / kSlice; s += threads) h.lv[l].sw[s] = 0;
}

// Level 0: FP32 copy of the weights and the smoother's scaling of sigma I - L.
// Weights are loaded kLevel0Batch at a time before any is stored: stores to the
// copy could alias the operator for all the compiler knows, and a load a slot
// made the kernel a chain of K + 1 memory latencies.
constexpr int kLevel0Batch = 7;
__global__ void __launch_bounds__(256) k_amg_level0(const AmgHeader* __restrict__ Hp, OpView O) {
    const AmgHeader& H = *Hp;
    const int k = H.k, m = k + 1;
    const double sigma = H.sigma;
    float* const out = H.lv[0].val;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < H.n; r += (int64_t)gridDim.x * blockDim.x) {
        const int64_t vb = (r / kSlice) * (int64_t)(kSlice * m) + (r % kSlice);
        double l1 = 0.0, diag = 0.0;
        for (int s0 = 0; s0 < m; s0 += kLevel0Batch) {
            double w[kLevel0Batch];
            float hi[kLevel0Batch];
#pragma unroll
            for (int u = 0; u < kLevel0Batch; u++) {
                const int64_t idx = vb + (int64_t)(s0 + u < m ? s0 + u : s0) * kSlice;
                if (O.prec == MVGD_FP64) {
                    w[u] = static_cast<const double*>(O.val)[idx];
                    hi[u] = (float)w[u];
                } else {  // the mixed format's hi is already the weight's rounding
                    hi[u] = static_cast<const float*>(O.val)[idx];
                    w[u] = (double)hi[u] + (double)O.val_lo[idx];
                }
            }
#pragma unroll
            for (int u = 0; u < kLevel0Batch; u++) {
                if (s0 + u >= m) break;
                out[vb + (int64_t)(s0 + u) * kSlice] = hi[u];
                if (s0 + u == 0) diag = sigma - w[u];
                l1 += s0 + u == 0 ? fabs(sigma - w[u]) : fabs(w[u]);
            }
        }
        H.lv[0].dinv[r] = amg_smoother_scale(diag, l1);
    }
}

// Row I of level l+1 by one warp, from the `total` entries of its aggregate's
// rows: `fetch(e, key, v)` gives entry e < total (column aggregate and value),
// PL of them a lane (entry t * 32 + lane).  Distinct columns come out in
// increasing order, each with the FP64 sum of its entries: the lane's own in
// entry order, then a butterfly over the warp, the same order on every run.
//
// FP64 instructions are what the kernel is bound by (an SM's FP64 pipe takes
// one a warp in 16 clocks), then the search for the next column.  So each lane
// first sorts its entries by (column, entry) and adds up its equal columns
// once; columns are emitted kCoarsenGroup at a time, whose partial sums share
// one butterfly (16 additions for 16 columns, 80 in separate ones, bit for bit
// the same); and the row's l1 norm and sum gather in the lanes that end with
// the totals.  Entries a lane is a template parameter because the sorting
// network grows with its square: 15 exchanges for the 6 of K = 20 on level 0,
// 120 for the 16 that a level of 64-entry rows can need.  All levels of
// 1,048,576 rows, K = 20: 1.81 -> 0.82 ms, 0.71 ms of it level 1.
constexpr int kCoarsenGroup = 16;
template <int PL, typename Fetch>
__device__ __forceinline__ void coarsen_row(const AmgHeader* Hp, const AmgLevel& Cl, int64_t I, int total,
                                            Fetch&& fetch) {
    const int lane = (int)lane_id();
    int key[PL];
    double v[PL];
#pragma unroll
    for (int t = 0; t < PL; t++) {
        key[t] = INT_MAX;
        v[t] = 0.0;
        const int e = t * kWarp + lane;
        if (e < total) fetch(e, key[t], v[t]);
    }
    // sort the lane's entries by (column, entry): an odd-even transposition network
    int tt[PL];
#pragma unroll
    for (int t = 0; t < PL; t++) tt[t] = t;
#pragma unroll
    for (int ph = 0; ph < PL; ph++)
#pragma unroll
        for (int i = ph & 1; i + 1 < PL; i += 2) {
            const bool sw = key[i] > key[i + 1] || (key[i] == key[i + 1] && tt[i] > tt[i + 1]);
            const int ka = key[i], ta = tt[i];
            const double va = v[i];
            key[i] = sw ? key[i + 1] : ka;
            tt[i] = sw ? tt[i + 1] : ta;
            v[i] = sw ? v[i + 1] : va;
            key[i + 1] = sw ? ka : key[i + 1];
            tt[i + 1] = sw ? ta : tt[i + 1];
            v[i + 1] = sw ? va : v[i + 1];
        }
    // the lane's sum of each column, in entry order, left on its last entry
#pragma unroll
    for (int t = 1; t < PL; t++)
        if (key[t] != INT_MAX && key[t] == key[t - 1]) {
            v[t] = v[t - 1] + v[t];
            key[t - 1] = INT_MAX;
        }
    const int64_t ob = (I / kSlice) * (int64_t)(kSlice * kAmgStride) + (I % kSlice);
    int out = 0;
    double l1 = 0.0, rsum = 0.0, diag = 0.0;  // this lane's columns
    bool more = true;
    while (more) {
        double part[kCoarsenGroup];
        int cols = 0, mycol = INT_MAX;  // columns of this group; the one whose total this lane ends with
#pragma unroll
        for (int c = 0; c < kCoarsenGroup; c++) {
            part[c] = 0.0;
            if (!more) continue;  // warp-uniform
            int mine = INT_MAX;
#pragma unroll
            for (int t = 0; t < PL; t++) mine = min(mine, key[t]);
            const int m = __reduce_min_sync(0xffffffffu, mine);
            if (m == INT_MAX) {
                more = false;
                continue;
            }
            if (mine == m) {
#pragma unroll
                for (int t = 0; t < PL; t++)
                    if (key[t] == m) {  // at most one entry of the lane holds column m now
                        part[c] = v[t];
                        key[t] = INT_MAX;
                    }
            }
            if (lane / (kWarp / kCoarsenGroup) == c) mycol = m;
            cols++;
        }
        if (cols == 0) break;
        int chan;
        const double tot = warp_sum_multi<kCoarsenGroup>(part, lane, chan);
        // lanes 2c and 2c + 1 hold value c (the halves a lane keeps follow its bits from the top)
        if (chan < cols && (lane & 1) == 0) {
            const int pos = out + chan;
            if (pos < kAmgStride) {
                Cl.col[ob + (int64_t)pos * kSlice] = mycol;
                Cl.val64[ob + (int64_t)pos * kSlice] = tot;
                Cl.val[ob + (int64_t)pos * kSlice] = (float)tot;
            }
            l1 += fabs(tot);
            rsum += tot;
            if (mycol == (int)I) diag = tot;
        }
        out += cols;
    }
    l1 = warp_sum(l1);
    rsum = warp_sum(rsum);
    diag = warp_sum(diag);  // one lane's value, zeros elsewhere
    if (lane == 0) {
        if (out > kAmgStride) atomicCAS((int*)&Hp->status, 0, (int)MVGD_EDEGENERATE);
        if (out > *(volatile const int*)&Hp->width_max) atomicMax((int*)&Hp->width_max, out);
        const int c = min(out, kAmgStride);
        Cl.cnt[I] = c;
        atomicMax(&Cl.sw[I / kSlice], c);  // the slice's widest row (zeroed with the header)
        Cl.dinv[I] = amg_smoother_scale(diag, l1);
        Cl.rs[I] = (float)rsum;
    }
    // padding: (own row, 0) up to the full stride, so slice loops need no bounds
    for (int s = min(out, kAmgStride) + lane; s < kAmgStride; s += kWarp) {
        Cl.col[ob + (int64_t)s * kSlice] = (int32_t)I;
        Cl.val64[ob + (int64_t)s * kSlice] = 0.0;
        Cl.val[ob + (int64_t)s * kSlice] = 0.0f;
    }
}

// Level 1 from the operator: every row has its K + 1 weights, so PL >= 8 (K + 1) / 32.
template <int PL>
__global__ void __launch_bounds__(256) k_amg_coarsen0(const AmgHeader* Hp, OpView O) {
    const AmgHeader& H = *Hp;
    const AmgLevel& Cl = H.lv[1];
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x / kWarp);
    const int64_t n = H.lv[0].n;
    const int k = H.k, W = k + 1;
    for (int64_t I = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / kWarp; I < Cl.n; I += warps) {
        const int rows = (int)(n - I * kAmgAgg < kAmgAgg ? n - I * kAmgAgg : kAmgAgg);
        coarsen_row<PL>(Hp, Cl, I, rows * W, [&](int e, int& key, double& v) {
            const int f = e / W, s = e % W;
            const int64_t i = I * kAmgAgg + f;
            const double w = op_weight(O, (i / kSlice) * (int64_t)(kSlice * W) + (int64_t)s * kSlice + (i % kSlice));
            if (s == 0) {
                key = (int)I;
                v = H.sigma - w;
            } else {
                const int64_t j = O.col[(i / kSlice) * (int64_t)(kSlice * k) + (int64_t)(s - 1) * kSlice + (i % kSlice)];
                key = (int)(j / kAmgAgg);
                v = -w;
            }
        });
    }
}

// Level l+1 from level l >= 1: the rows' entries back to back, as many a lane
// as they need (rows hold 10 to 25 entries typically, 64 at most).
__global__ void __launch_bounds__(256) k_amg_coarsen(const AmgHeader* Hp, int l) {
    const AmgHeader& H = *Hp;
    const AmgLevel& F = H.lv[l];
    const AmgLevel& Cl = H.lv[l + 1];
    const int lane = (int)lane_id();
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x / kWarp);
    for (int64_t I = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / kWarp; I < Cl.n; I += warps) {
        const int64_t mine = I * kAmgAgg + lane;
        int end = lane < kAmgAgg && mine < F.n ? F.cnt[mine] : 0;  // inclusive prefix of the rows' counts
#pragma unroll
        for (int o = 1; o < kAmgAgg; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += t;
        }
        int ends[kAmgAgg];
#pragma unroll
        for (int f = 0; f < kAmgAgg; f++) ends[f] = __shfl_sync(0xffffffffu, end, f);
        const int total = ends[kAmgAgg - 1];
        auto fetch = [&](int e, int& key, double& v) {
            int f = 0, s = e;
#pragma unroll
            for (int g = 0; g + 1 < kAmgAgg; g++)
                if (e >= ends[g]) {
                    f = g + 1;
                    s = e - ends[g];
                }
            const int64_t i = I * kAmgAgg + f;
            const int64_t idx = (i / kSlice) * (int64_t)(kSlice * kAmgStride) + (int64_t)s * kSlice + (i % kSlice);
            key = F.col[idx] / kAmgAgg;
            v = F.val64[idx];
        };
        if (total <= 4 * kWarp) coarsen_row<4>(Hp, Cl, I, total, fetch);
        else if (total <= 8 * kWarp) coarsen_row<8>(Hp, Cl, I, total, fetch);
        else coarsen_row<kAmgAgg * kAmgStride / kWarp>(Hp, Cl, I, total, fetch);
    }
}

// x as hi + lo FP32 words (48 bits).
__device__ __forceinline__ float2 split_f2(double x) {
    const float hi = (float)x;
    return make_float2(hi, (float)(x - (double)hi));
}

// The coarsest level as a dense FP64 matrix and its hi + lo split (in ns_x), a warp a row.
__global__ void k_amg_dense(const AmgHeader* __restrict__ Hp, OpView O) {
    const AmgHeader& H = *Hp;
    const int m = H.nlev - 1, lane = (int)lane_id();
    const int64_t nc = H.nc, r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / kWarp;
    if (r >= nc) return;
    double* row = H.dense64 + r * nc;
    float2* row2 = reinterpret_cast<float2*>(H.ns_x) + r * nc;
    for (int64_t c = lane; c < nc; c += kWarp) {
        row[c] = 0.0;
        row2[c] = make_float2(0.0f, 0.0f);
    }
    __syncwarp();
    auto put = [&](int64_t c, double v) {
        row[c] = v;
        row2[c] = split_f2(v);
    };
    if (m == 0) {
        // a lane a slot.  A folded operator's row may name a column twice, or itself (a
        // point beside its ghost): such slots add up, in slot order, as in its products
        static_assert(kMaxK + 1 <= kWarp, "a lane a slot");
        const int k = H.k;
        const int64_t vb = (r / kSlice) * (int64_t)(kSlice * (k + 1)) + (r % kSlice);
        const int64_t cb = (r / kSlice) * (int64_t)(kSlice * k) + (r % kSlice);
        int c = -1 - lane;  // (no slot)
        double v = 0.0;
        if (lane == 0) {
            c = (int)r;
            v = H.sigma - op_weight(O, vb);
        } else if (lane <= k) {
            c = O.col[cb + (int64_t)(lane - 1) * kSlice];
            v = -op_weight(O, vb + (int64_t)lane * kSlice);
        }
        unsigned rest = __match_any_sync(0xffffffffu, c);
        const bool first = (rest & ((1u << lane) - 1u)) == 0;
        double t = v;
        rest &= rest - 1u;  // the slots that follow the column's first
        while (__any_sync(0xffffffffu, rest != 0u)) {
            const double x = __shfl_sync(0xffffffffu, v, rest ? __ffs(rest) - 1 : lane);
            if (rest) t += x;
            rest &= rest - 1u;
        }
        if (first && c >= 0) put(c, t);
    } else {
        const AmgLevel& L = H.lv[m];
        const int64_t b = (r / kSlice) * (int64_t)(kSlice * kAmgStride) + (r % kSlice);
        for (int s = lane; s < L.cnt[r]; s += kWarp) {
            const int64_t e = b + (int64_t)s * kSlice;
            put(L.col[e], L.val64[e]);
        }
    }
}

// ---------------------------------------------------------------------------
// Inverse of the coarsest level: Gauss-Jordan in place with partial pivoting
// in FP32, blocked.  Rows are not swapped: step k takes the largest |a_ik| of
// the rows not yet used as a pivot (the lowest row on ties), and the
// permutation p_k is undone on the way out, (A^-1)[k][p_j] = B[p_k][j].
//
// Steps go by panels of kInvPanel columns.  A panel's steps touch only its own
// columns; their effect on any other column is the product with the panel's
// result, a_new[i] = (i a pivot of the panel ? 0 : a[i]) + sum_t panel[i][t]
// a_old[p_t].  A cluster of up to 8 CTAs holds the matrix in shared memory, 64
// columns a CTA (139 KB at 512 rows).  Four warps of the CTA that owns the
// panel's columns do the steps without any other CTA: a thread holds the 32
// panel values of up to four rows in registers, one barrier of 128 threads a step.
// (With a row a thread, 16 warps each read the pivot row, 8 LDS.128 a step, and
// a step took 1,600 clocks.)  Then every CTA applies the panel to its columns in
// 8 x 8 register tiles.  So the cluster meets once a panel; a matrix cut by rows
// met four times a step, which made a step 4 us.  110 rows 0.44 -> 0.08 ms, 256
// rows 1.17 -> 0.26 ms, 512 rows about 2.5 -> 0.57 ms; the chain of a step (two
// warp reductions, the candidate row through shared memory, a reciprocal, one
// register update a row) still takes about 1 us.
// ---------------------------------------------------------------------------
constexpr int kInvCols = 64;                // columns a CTA
constexpr int kInvStride = kInvCols + 4;    // row stride: float4 accesses of consecutive rows hit all banks
constexpr int kInvPanel = 32;
constexpr int kInvThreads = 256;
constexpr int kInvStepThreads = 128;        // threads that do a panel's steps

// Rows of the panel's result, transposed [kInvPanel][pitch]; also the exchange
// area in global memory (set-up scratch), followed by the pivots and a flag.
__host__ __device__ constexpr int inv_pitch(int n) { return (n + 7) / 8 * 8; }
__host__ __device__ constexpr size_t inv_panel_floats(int n) { return (size_t)inv_pitch(n) * kInvPanel + 64; }
constexpr size_t inv_smem_floats(int n) {
    return (size_t)n * kInvStride + (size_t)inv_pitch(n) * kInvPanel + kInvPanel * kInvCols;
}

// kInvRows: rows a step thread holds, n <= kInvRows * kInvStepThreads.
template <int kInvRows>
__global__ void __launch_bounds__(kInvThreads) k_amg_invert(AmgHeader* Hp) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), ncta = (int)cl.num_blocks();
    const int n = (int)Hp->nc, pitch = inv_pitch(n);
    extern __shared__ __align__(16) float smf[];
    float* A = smf;                                    // [n][kInvStride] this CTA's columns
    float* Pn = A + (size_t)n * kInvStride;            // [kInvPanel][pitch] the panel's result
    float* U = Pn + (size_t)pitch * kInvPanel;         // [kInvPanel][kInvCols] the pivot rows before it
    constexpr int kStepWarps = kInvStepThreads / kWarp;
    __shared__ __align__(16) float cand[2][kStepWarps][kInvPanel];  // each warp's candidate row
    __shared__ unsigned cand_key[2][kStepWarps];
    __shared__ int cand_row[2][kStepWarps];
    __shared__ int piv[kAmgCoarsest];       // pivot row of step k
    __shared__ int panel_of[kAmgCoarsest];  // panel in which a row was the pivot
    __shared__ int failed;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int c0 = rank * kInvCols, ncols = min(kInvCols, n - c0);
    float* const xch = reinterpret_cast<float*>(Hp->ns_t);
    for (int e = tid; e < n * kInvCols; e += kInvThreads) {
        const int r = e / kInvCols, j = e % kInvCols;
        A[r * kInvStride + j] = j < ncols ? (float)Hp->dense64[(int64_t)r * n + c0 + j] : 0.0f;
    }
    for (int r = tid; r < n; r += kInvThreads) panel_of[r] = -1;
    if (tid == 0) failed = 0;
    __syncthreads();
    for (int p = 0; p * kInvPanel < n; p++) {
        const int k0 = p * kInvPanel, kb = min(kInvPanel, n - k0), owner = k0 / kInvCols, lk = k0 % kInvCols;
        float* const buf = xch + (p & 1) * inv_panel_floats(n);
        int* const bufi = reinterpret_cast<int*>(buf + (size_t)pitch * kInvPanel);
        if (rank == owner && tid < kInvStepThreads) {
            float v[kInvRows][kInvPanel];
            bool used[kInvRows];
#pragma unroll
            for (int q = 0; q < kInvRows; q++) {
                const int i = tid + q * kInvStepThreads;
                used[q] = i >= n || panel_of[i] >= 0;  // a row past the end is never a pivot
#pragma unroll
                for (int j = 0; j < kInvPanel; j += 4) {
                    const float4 t = i < n ? *reinterpret_cast<const float4*>(A + i * kInvStride + lk + j)
                                           : make_float4(0.f, 0.f, 0.f, 0.f);
                    v[q][j] = t.x; v[q][j + 1] = t.y; v[q][j + 2] = t.z; v[q][j + 3] = t.w;
                }
            }
            bool bad = false;
            // step t works on v[.][0] and turns the registers by one place: the loop is one body
#pragma unroll 1
            for (int t = 0; t < kInvPanel; t++) {
                if (t >= kb || bad) {  // uniform over the step threads: past the last column (zeros), only turn
#pragma unroll
                    for (int q = 0; q < kInvRows; q++) {
                        const float first = v[q][0];
#pragma unroll
                        for (int j = 0; j + 1 < kInvPanel; j++) v[q][j] = v[q][j + 1];
                        v[q][kInvPanel - 1] = first;
                    }
                    continue;
                }
                const int b = t & 1;
                unsigned key = 0u;
                int mq = -1;  // this thread's candidate: its largest unused |v[.][0]|, the lowest row on ties
#pragma unroll
                for (int q = 0; q < kInvRows; q++) {
                    const unsigned kq = __float_as_uint(fabsf(v[q][0]));
                    if (!used[q] && (mq < 0 || kq > key)) { key = kq; mq = q; }
                }
                const unsigned wm = __reduce_max_sync(0xffffffffu, key);
                const int row_of = mq >= 0 && key == wm ? tid + mq * kInvStepThreads : INT_MAX;
                const int wr = __reduce_min_sync(0xffffffffu, row_of);
                if (row_of == wr && wr != INT_MAX) {
#pragma unroll
                    for (int q = 0; q < kInvRows; q++)
                        if (q == mq) {
#pragma unroll
                            for (int j = 0; j < kInvPanel; j += 4)
                                *reinterpret_cast<float4*>(&cand[b][wid][j]) =
                                    make_float4(v[q][j], v[q][j + 1], v[q][j + 2], v[q][j + 3]);
                        }
                }
                if (lane == 0) {
                    cand_key[b][wid] = wr == INT_MAX ? 0u : wm;
                    cand_row[b][wid] = wr;
                }
                asm volatile("bar.sync 1, %0;" ::"n"(kInvStepThreads) : "memory");
                unsigned m = cand_key[b][0];
                int pr = cand_row[b][0], w = 0;
#pragma unroll
                for (int o = 1; o < kStepWarps; o++) {
                    const unsigned ko = cand_key[b][o];
                    const int ro = cand_row[b][o];
                    if (ko > m || (ko == m && ro < pr)) { m = ko; pr = ro; w = o; }
                }
                if (m == 0u || m >= 0x7f800000u) {  // no pivot, or one that is not finite
                    bad = true;
                    t--;  // turn the rest of the way
                    continue;
                }
                const float* row = cand[b][w];
                const float inv = 1.0f / row[0];
                float f[kInvRows];
#pragma unroll
                for (int q = 0; q < kInvRows; q++) f[q] = v[q][0] * inv;
                // every row but the pivot: v - f x
#pragma unroll
                for (int j = 0; j < kInvPanel; j += 4) {
                    const float4 x = *reinterpret_cast<const float4*>(row + j);
#pragma unroll
                    for (int q = 0; q < kInvRows; q++) {
                        if (j > 0) v[q][j - 1] = fmaf(-f[q], x.x, v[q][j]);
                        v[q][j] = fmaf(-f[q], x.y, v[q][j + 1]);
                        v[q][j + 1] = fmaf(-f[q], x.z, v[q][j + 2]);
                        v[q][j + 2] = fmaf(-f[q], x.w, v[q][j + 3]);
                    }
                }
#pragma unroll
                for (int q = 0; q < kInvRows; q++) v[q][kInvPanel - 1] = -f[q];
                if ((pr & (kInvStepThreads - 1)) == tid) {  // the pivot row: x inv
#pragma unroll
                    for (int q = 0; q < kInvRows; q++)
                        if (pr == tid + q * kInvStepThreads) {
                            used[q] = true;
#pragma unroll
                            for (int j = 0; j + 1 < kInvPanel; j++) v[q][j] = row[j + 1] * inv;
                            v[q][kInvPanel - 1] = inv;
                        }
                }
                if (tid == 0) piv[k0 + t] = pr;
            }
#pragma unroll
            for (int q = 0; q < kInvRows; q++) {
                const int i = tid + q * kInvStepThreads;
                if (i >= n) continue;
#pragma unroll
                for (int j = 0; j < kInvPanel; j++) {
                    Pn[j * pitch + i] = v[q][j];
                    if (ncta > 1) buf[j * pitch + i] = v[q][j];
                }
#pragma unroll
                for (int j = 0; j < kInvPanel; j += 4)
                    *reinterpret_cast<float4*>(A + i * kInvStride + lk + j) =
                        make_float4(v[q][j], v[q][j + 1], v[q][j + 2], v[q][j + 3]);
            }
            asm volatile("bar.sync 1, %0;" ::"n"(kInvStepThreads) : "memory");  // piv
            if (ncta > 1) {
                if (tid < kb) bufi[tid] = bad ? 0 : piv[k0 + tid];
                if (tid == 0) bufi[kInvPanel] = bad;
            }
            if (tid == 0) failed = bad;
        }
        if (ncta > 1) {
            cl.sync();  // the panel is in global memory (its buffer was last read two panels ago)
            if (rank != owner) {
                for (int e = tid; e < pitch * kInvPanel / 4; e += kInvThreads)
                    reinterpret_cast<float4*>(Pn)[e] = __ldcg(reinterpret_cast<const float4*>(buf) + e);
                if (tid < kb) piv[k0 + tid] = __ldcg(bufi + tid);
                if (tid == 0) failed = __ldcg(bufi + kInvPanel);
            }
        }
        __syncthreads();
        if (failed) break;  // the same decision in every CTA
        if (tid < kb) panel_of[piv[k0 + tid]] = p;
        for (int e = tid; e < kInvPanel * kInvCols; e += kInvThreads) {
            const int t = e / kInvCols, j = e % kInvCols;
            U[e] = t < kb ? A[piv[k0 + t] * kInvStride + j] : 0.0f;
        }
        __syncthreads();
        for (int tile = tid; tile < pitch / 8 * (kInvCols / 8); tile += kInvThreads) {
            const int rg = tile / (kInvCols / 8) * 8, cg8 = tile % (kInvCols / 8) * 8;
            if (cg8 >= ncols || (rank == owner && cg8 >= lk && cg8 < lk + kInvPanel)) continue;
            float acc[8][8];
#pragma unroll
            for (int r = 0; r < 8; r++) {
                const int i = rg + r;
                const bool old = i < n && panel_of[i] != p;
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const float4 t = old ? *reinterpret_cast<const float4*>(A + i * kInvStride + cg8 + 4 * h)
                                         : make_float4(0.f, 0.f, 0.f, 0.f);
                    acc[r][4 * h] = t.x; acc[r][4 * h + 1] = t.y; acc[r][4 * h + 2] = t.z; acc[r][4 * h + 3] = t.w;
                }
            }
#pragma unroll 2
            for (int t = 0; t < kInvPanel; t++) {
                const float4 u0 = *reinterpret_cast<const float4*>(U + t * kInvCols + cg8);
                const float4 u1 = *reinterpret_cast<const float4*>(U + t * kInvCols + cg8 + 4);
                const float4 x0 = *reinterpret_cast<const float4*>(Pn + t * pitch + rg);
                const float4 x1 = *reinterpret_cast<const float4*>(Pn + t * pitch + rg + 4);
                const float x[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
#pragma unroll
                for (int r = 0; r < 8; r++) {
                    acc[r][0] = fmaf(x[r], u0.x, acc[r][0]); acc[r][1] = fmaf(x[r], u0.y, acc[r][1]);
                    acc[r][2] = fmaf(x[r], u0.z, acc[r][2]); acc[r][3] = fmaf(x[r], u0.w, acc[r][3]);
                    acc[r][4] = fmaf(x[r], u1.x, acc[r][4]); acc[r][5] = fmaf(x[r], u1.y, acc[r][5]);
                    acc[r][6] = fmaf(x[r], u1.z, acc[r][6]); acc[r][7] = fmaf(x[r], u1.w, acc[r][7]);
                }
            }
#pragma unroll
            for (int r = 0; r < 8; r++) {
                if (rg + r >= n) continue;  // (the panel's columns past n hold whatever was there)
                float* d = A + (rg + r) * kInvStride + cg8;
                *reinterpret_cast<float4*>(d) = make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
                *reinterpret_cast<float4*>(d + 4) = make_float4(acc[r][4], acc[r][5], acc[r][6], acc[r][7]);
            }
        }
        __syncthreads();  // this CTA's columns are up to date
    }
    if (failed) {
        if (rank == 0 && tid == 0) atomicCAS((int*)&Hp->status, 0, (int)MVGD_EDEGENERATE);
        return;
    }
    // the pivots of every panel are in every CTA: the inverse in FP32, column-major
    for (int e = tid; e < n * kInvCols; e += kInvThreads) {
        const int j = e / n, k = e % n;
        if (j >= ncols) continue;
        Hp->cinv[(int64_t)piv[c0 + j] * n + k] = A[piv[k] * kInvStride + j];
    }
}

// ---------------------------------------------------------------------------
// Newton-Schulz X <- X + X (I - A X), twice, which squares the FP32 inverse's
// residual R = I - A X (~1e-5) each time, down to the FP64 level: four products
// of small n x n matrices.
//   kNsR0  R0 = I - A X0    A split into hi + lo FP32 words, X0 the FP32 inverse
//   kNsX1  X1 = X0 + X0 R0  (FP64, and split)
//   kNsR1  R1 = I - A X1    in FP64
//   kNsX2  X2 = X1 + X1 R1  both split; the inverse that the cycle uses
// The FP64 pipe takes 2 FMAs a clock an SM, so only the residual that decides
// the final accuracy runs there.  The other products sum hi hi in compensated
// FP32 arithmetic (f2_add_prod, about 2^-45 of sum |a||x|) with the cross terms
// beside it, 11 FP32 instructions a term.  X R is a correction of 1e-5 of X and
// less, so its error is below 2^-53 of X in the last step; in the first step the
// error of R0 enters X2 squared.
// A block of 4 warps takes a 16 x 16 tile (256 tiles at n = 256: more than SMs);
// each warp takes every fourth group of 8 of the sum, 8 outputs a lane, and the
// block adds the four partial sums.  All four: 317 -> 98 us at n = 256, of which
// R1 43 us (27 at the FP64 pipe's rate).  Against 80-bit arithmetic, with all four
// in FP64 before: the residual I - A X 0.07 to 0.16 of it, the error of X 0.68
// (300 rows of a one-level hierarchy) and 1.2 (Galerkin levels of 110 to 469 rows,
// from the order of R1's sums; the splits add nothing).
// ---------------------------------------------------------------------------
enum NsStep : int { kNsR0 = 0, kNsX1 = 1, kNsR1 = 2, kNsX2 = 3 };
constexpr int kNsTile = 16, kNsDeep = 32, kNsWarps = 4;

template <int STEP>
__global__ void __launch_bounds__(kNsWarps * kWarp) k_amg_ns(const AmgHeader* __restrict__ Hp) {
    constexpr bool kFast = STEP != kNsR1;
    using LT = typename std::conditional<STEP == kNsR1, double, typename std::conditional<STEP == kNsX1, float, float2>::type>::type;
    using RT = typename std::conditional<STEP == kNsR1, double, typename std::conditional<STEP == kNsR0, float, float2>::type>::type;
    using AT = typename std::conditional<kFast, F2, double>::type;
    __shared__ LT Ls[kNsTile][kNsDeep + 1];
    __shared__ RT Rs[kNsDeep][kNsTile + 1];
    __shared__ AT sum[kNsWarps][kNsTile * kNsTile];
    const AmgHeader& H = *Hp;
    const int n = (int)H.nc;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int row0 = blockIdx.y * kNsTile, col0 = blockIdx.x * kNsTile;
    const float* x0t = H.cinv;  // X0, column-major
    auto left = [&](int r, int c) -> LT {
        const int64_t e = (int64_t)r * n + c;
        if constexpr (STEP == kNsR0) return reinterpret_cast<const float2*>(H.ns_x)[e];       // A
        else if constexpr (STEP == kNsX1) return x0t[(int64_t)c * n + r];                     // X0
        else if constexpr (STEP == kNsR1) return H.dense64[e];                                // A
        else return reinterpret_cast<const float2*>(H.ns_s)[e];                               // X1
    };
    auto right = [&](int r, int c) -> RT {
        const int64_t e = (int64_t)r * n + c;
        if constexpr (STEP == kNsR0) return x0t[(int64_t)c * n + r];                          // X0
        else if constexpr (STEP == kNsR1) return H.ns_x[e];                                   // X1
        else return reinterpret_cast<const float2*>(H.ns_t)[e];                               // R0, R1
    };
    // lane: rows 2 (lane / 4) and the next, columns 4 (lane % 4) .. + 3
    const int lr = 2 * (lane >> 2), lc = 4 * (lane & 3);
    AT acc[2][4];
#pragma unroll
    for (int a = 0; a < 2; a++)
#pragma unroll
        for (int b = 0; b < 4; b++) acc[a][b] = AT{};
    for (int k0 = 0; k0 < n; k0 += kNsDeep) {
#pragma unroll
        for (int e = tid; e < kNsTile * kNsDeep; e += kNsWarps * kWarp) {
            // consecutive threads along the operand's contiguous index
            const int r = STEP == kNsX1 ? e % kNsTile : e / kNsDeep, c = STEP == kNsX1 ? e / kNsTile : e % kNsDeep;
            Ls[r][c] = row0 + r < n && k0 + c < n ? left(row0 + r, k0 + c) : LT{};
            const int r2 = STEP == kNsR0 ? e % kNsDeep : e / kNsTile, c2 = STEP == kNsR0 ? e / kNsDeep : e % kNsTile;
            Rs[r2][c2] = k0 + r2 < n && col0 + c2 < n ? right(k0 + r2, col0 + c2) : RT{};
        }
        __syncthreads();
#pragma unroll 2
        for (int kk = 0; kk < kNsDeep / kNsWarps; kk++) {
            const int k = wid * (kNsDeep / kNsWarps) + kk;
            LT x[2];
            RT y[4];
#pragma unroll
            for (int a = 0; a < 2; a++) x[a] = Ls[lr + a][k];
#pragma unroll
            for (int b = 0; b < 4; b++) y[b] = Rs[k][lc + b];
#pragma unroll
            for (int a = 0; a < 2; a++)
#pragma unroll
                for (int b = 0; b < 4; b++) {
                    if constexpr (STEP == kNsR1) {
                        acc[a][b] = fma(x[a], y[b], acc[a][b]);
                    } else if constexpr (STEP == kNsR0) {
                        f2_add_prod(acc[a][b], x[a].x, y[b]);
                        acc[a][b].lo = fmaf(x[a].y, y[b], acc[a][b].lo);
                    } else if constexpr (STEP == kNsX1) {
                        f2_add_prod(acc[a][b], x[a], y[b].x);
                        acc[a][b].lo = fmaf(x[a], y[b].y, acc[a][b].lo);
                    } else {
                        f2_add_prod(acc[a][b], x[a].x, y[b].x);
                        acc[a][b].lo = fmaf(x[a].x, y[b].y, fmaf(x[a].y, y[b].x, acc[a][b].lo));
                    }
                }
        }
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < 2; a++)
#pragma unroll
        for (int b = 0; b < 4; b++) sum[wid][(lr + a) * kNsTile + lc + b] = acc[a][b];
    __syncthreads();
    for (int e = tid; e < kNsTile * kNsTile; e += kNsWarps * kWarp) {
        const int r = row0 + e / kNsTile, c = col0 + e % kNsTile;
        if (r >= n || c >= n) continue;
        const AT t = part_add(part_add(sum[0][e], sum[1][e]), part_add(sum[2][e], sum[3][e]));
        double s;
        if constexpr (kFast) s = f2_to_double(t);
        else s = t;
        const int64_t o = (int64_t)r * n + c;
        if constexpr (STEP == kNsR0 || STEP == kNsR1) {
            reinterpret_cast<float2*>(H.ns_t)[o] = split_f2((r == c ? 1.0 : 0.0) - s);
        } else if constexpr (STEP == kNsX1) {
            const double x1 = (double)x0t[(int64_t)c * n + r] + s;
            H.ns_x[o] = x1;
            reinterpret_cast<float2*>(H.ns_s)[o] = split_f2(x1);
        } else {
            H.cinv64[o] = H.ns_x[o] + s;
        }
    }
}

int grid_for(int64_t threads) {
    int64_t g = (threads + 255) / 256;
    return (int)(g > 16384 ? 16384 : (g < 1 ? 1 : g));
}

// ---------------------------------------------------------------------------
// Standalone V-cycle (stored order): one kernel per step.
// ---------------------------------------------------------------------------
struct ApplyVecs {
    float* y[kAmgMaxLevels];
    float* r[kAmgMaxLevels];
    float* b[kAmgMaxLevels];  // b[0] unused: level 0 reads the FP64 input
    float* x[kAmgMaxLevels];  // x[0] unused: level 0 writes the FP64 output
    size_t bytes;
};

ApplyVecs apply_layout(void* ws, int64_t n, int Q) {
    ApplyVecs V;
    memset(&V, 0, sizeof(V));
    int64_t sizes[kAmgMaxLevels];
    const int nlev = amg_levels(n, sizes);
    Carver cv(ws);
    for (int l = 0; l < nlev; l++) {
        const int64_t m = n_padded(sizes[l]) * Q;
        V.y[l] = cv.take<float>(m);
        V.r[l] = cv.take<float>(m);
        if (l > 0) {
            V.b[l] = cv.take<float>(m);
            V.x[l] = cv.take<float>(m);
        }
    }
    V.bytes = cv.used;
    return V;
}

// Rows of a level in whole warps: rows past the end only join the shuffles.
__global__ void k_vpre(const AmgHeader* __restrict__ Hp, const double* __restrict__ b, int Q, float* y0) {
    const AmgHeader& H = *Hp;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < H.n * Q; e += (int64_t)gridDim.x * blockDim.x)
        y0[e] = H.lv[0].dinv[e / Q] * (float)b[e];
}

// Blocks of kApplyThreads threads take kApplyThreads / G consecutive rows at a
// time (G lanes a row, amg_group; level 0: G = 1), like the solver's steps.
constexpr int kApplyThreads = 256;

__global__ void __launch_bounds__(kApplyThreads) k_vdown(const AmgHeader* __restrict__ Hp, int l,
                                                         const double* __restrict__ b0, int Q, ApplyVecs V) {
    __shared__ float agg[kApplyThreads / kAmgAgg];
    const AmgHeader& H = *Hp;
    const int64_t nl = H.lv[l].n;
    const int G = l == 0 ? 1 : amg_group(nl);
    const int64_t rows = kApplyThreads / G;
    const float* Y = V.y[l];
    const bool last = (l + 1 == H.nlev - 1);
    // block-uniform loop: every thread reaches the barriers of agg_sum
    for (int64_t c = blockIdx.x; c * rows < nl; c += gridDim.x) {
        const int64_t r = c * rows + threadIdx.x / G;
        const bool valid = r < nl;
        for (int q = 0; q < Q; q++) {
            const float bi = valid ? (l == 0 ? (float)b0[r * Q + q] : V.b[l][r * Q + q]) : 0.0f;
            const float yi = valid ? Y[r * Q + q] : 0.0f;
            vdown_row(H, l, G, r, valid, Q, q, bi, yi, [&](int64_t j) { return Y[j * Q + q]; }, V.r[l], V.b[l + 1],
                      last ? nullptr : V.y[l + 1], [&](float xi, auto&& xv) { return a0_row(H, r, xi, xv); }, agg);
        }
    }
}

__global__ void k_vcoarse(const AmgHeader* __restrict__ Hp, const double* __restrict__ b0, double* x0, int Q,
                          ApplyVecs V) {
    const AmgHeader& H = *Hp;
    const int m = H.nlev - 1;
    const int64_t rho = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / kWarp;
    if (rho >= H.nc) return;  // warp-uniform
    auto store = [&](int q, float x) {
        if (m == 0) x0[rho * Q + q] = (double)x;
        else V.x[m][rho * Q + q] = x;
    };
    if (m == 0) coarse_rows<8>(H, rho, b0, Q, store);
    else coarse_rows<8>(H, rho, V.b[m], Q, store);
}

__global__ void __launch_bounds__(kApplyThreads) k_vup(const AmgHeader* __restrict__ Hp, int l, double* x0, int Q,
                                                       ApplyVecs V) {
    const AmgHeader& H = *Hp;
    const int64_t nl = H.lv[l].n;
    const int G = l == 0 ? 1 : amg_group(nl);
    const int64_t rows = kApplyThreads / G;
    const float* Xc = V.x[l + 1];
    for (int64_t c = blockIdx.x; c * rows < nl; c += gridDim.x) {
        const int64_t r = c * rows + threadIdx.x / G;
        const bool valid = r < nl;
        for (int q = 0; q < Q; q++) {
            const float x = vup_row(H, l, G, r, valid, valid ? V.y[l][r * Q + q] : 0.0f,
                                    valid ? V.r[l][r * Q + q] : 0.0f, [&](int64_t J) { return Xc[J * Q + q]; },
                                    [&](float xi, auto&& xv) { return a0_row(H, r, xi, xv); });
            if (!valid || (threadIdx.x & (G - 1)) != 0) continue;
            if (l == 0) x0[r * Q + q] = (double)x;
            else V.x[l][r * Q + q] = x;
        }
    }
}

}  // namespace
}  // namespace mvgd

using namespace mvgd;

MVGD_API size_t mvgd_amg_workspace_bytes(int64_t n, int32_t k) {
    if (n < 1 || k < kMinK || k > kMaxK || amg_levels(n, nullptr) == 0) return 0;
    return amg_layout(nullptr, n, k).h.bytes;
}

MVGD_API mvgd_status mvgd_amg_setup(const mvgd_ell* L, double sigma, void* amg_ws, size_t amg_bytes,
                                    mvgd_stream_t stream) {
    if (!L || !amg_ws || !L->col || !L->val || L->n < 2 || L->n >= (1ll << 31) || L->k < kMinK || L->k > kMaxK)
        return MVGD_EINVAL;
    if (L->prec != MVGD_FP64 && L->prec != MVGD_FP32_REFINE) return MVGD_EINVAL;
    if (L->prec == MVGD_FP32_REFINE && !L->val_lo) return MVGD_EINVAL;
    if (!aligned(amg_ws) || !aligned(L->col) || !aligned(L->val) || !aligned(L->val_lo)) return MVGD_EINVAL;
    if (!(sigma == sigma)) return MVGD_EINVAL;
    if (amg_levels(L->n, nullptr) == 0) return MVGD_EINVAL;
    AmgLayout A = amg_layout(amg_ws, L->n, L->k);
    if (amg_bytes < A.h.bytes) return MVGD_EWORKSPACE;
    A.h.sigma = sigma;
    A.h.col0 = L->col;
    A.h.val0 = L->val;
    A.h.val0_lo = L->val_lo;
    A.h.prec0 = L->prec;
    A.h.status = MVGD_OK;
    A.h.width_max = 0;
    cudaStream_t s = (cudaStream_t)stream;
    OpView O{L->col, L->val, L->val_lo, L->prec};
    k_amg_header<<<grid_for(n_padded(L->n) / kSlice / kAmgAgg + 1), 256, 0, s>>>(A.h, A.hdr);
    k_amg_level0<<<grid_for(L->n), 256, 0, s>>>(A.hdr, O);
    for (int l = 0; l + 1 < A.h.nlev; l++) {
        const int gb = grid_for(A.h.lv[l + 1].n * kWarp);
        if (l > 0) k_amg_coarsen<<<gb, 256, 0, s>>>(A.hdr, l);
        else if (L->k < 16) k_amg_coarsen0<4><<<gb, 256, 0, s>>>(A.hdr, O);
        else if (L->k < 24) k_amg_coarsen0<6><<<gb, 256, 0, s>>>(A.hdr, O);
        else k_amg_coarsen0<8><<<gb, 256, 0, s>>>(A.hdr, O);
    }
    const int64_t nc = A.h.nc;
    k_amg_dense<<<grid_for(nc * kWarp), 256, 0, s>>>(A.hdr, O);
    {
        const int ncta = (int)((nc + kInvCols - 1) / kInvCols);
        const size_t smem = sizeof(float) * inv_smem_floats((int)nc);
        const int rows = nc <= kInvStepThreads ? 1 : (nc <= 2 * kInvStepThreads ? 2 : 4);
        auto fn = rows == 1 ? k_amg_invert<1> : (rows == 2 ? k_amg_invert<2> : k_amg_invert<4>);
        // the instantiation's largest, whatever this level needs: the attribute is the
        // process's, and another thread may be setting up a smaller level
        const int most = (int)(sizeof(float) * inv_smem_floats(rows * kInvStepThreads));
        MVGD_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)ncta);
        cfg.blockDim = dim3(kInvThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)ncta;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        MVGD_CUDA_TRY(cudaLaunchKernelEx(&cfg, fn, A.hdr));
    }
    const dim3 gg((unsigned)((nc + kNsTile - 1) / kNsTile), (unsigned)((nc + kNsTile - 1) / kNsTile));
    k_amg_ns<kNsR0><<<gg, kNsWarps * kWarp, 0, s>>>(A.hdr);
    k_amg_ns<kNsX1><<<gg, kNsWarps * kWarp, 0, s>>>(A.hdr);
    k_amg_ns<kNsR1><<<gg, kNsWarps * kWarp, 0, s>>>(A.hdr);
    k_amg_ns<kNsX2><<<gg, kNsWarps * kWarp, 0, s>>>(A.hdr);
    return launch_status();
}

MVGD_API mvgd_status mvgd_amg_describe(const void* amg_ws, int32_t level, mvgd_amg_info* out) {
    if (!amg_ws || !out || !aligned(amg_ws)) return MVGD_EINVAL;
    AmgHeader h;
    MVGD_CUDA_TRY(cudaMemcpy(&h, amg_ws, sizeof(h), cudaMemcpyDeviceToHost));
    if (level < 0 || level >= h.nlev) return MVGD_EINVAL;
    const AmgLevel& L = h.lv[level];
    memset(out, 0, sizeof(*out));
    out->levels = h.nlev;
    out->status = h.status;
    out->width_max = h.width_max;
    out->n = L.n;
    out->stride = level == 0 ? h.k + 1 : kAmgStride;
    out->col = level == 0 ? h.col0 : L.col;
    out->val = L.val;
    out->val64 = L.val64;
    out->cnt = L.cnt;
    out->dinv = L.dinv;
    out->cinv = level == h.nlev - 1 ? h.cinv : nullptr;
    out->cinv64 = level == h.nlev - 1 ? h.cinv64 : nullptr;
    return MVGD_OK;
}

MVGD_API size_t mvgd_amg_apply_workspace_bytes(int64_t n, int32_t nrhs) {
    if (n < 1 || nrhs < 1 || nrhs > 8 || amg_levels(n, nullptr) == 0) return 0;
    return apply_layout(nullptr, n, nrhs).bytes;
}

MVGD_API mvgd_status mvgd_amg_apply(const void* amg_ws, int64_t n, int32_t nrhs, const double* b, double* x,
                                    void* ws, size_t ws_bytes, mvgd_stream_t stream) {
    if (!amg_ws || !b || !x || !ws || n < 1 || nrhs < 1 || nrhs > 8) return MVGD_EINVAL;
    if (!aligned(amg_ws) || !aligned(b) || !aligned(x) || !aligned(ws)) return MVGD_EINVAL;
    int64_t sizes[kAmgMaxLevels];
    const int nlev = amg_levels(n, sizes);
    if (nlev == 0) return MVGD_EINVAL;
    ApplyVecs V = apply_layout(ws, n, nrhs);
    if (ws_bytes < V.bytes) return MVGD_EWORKSPACE;
    const AmgHeader* H = static_cast<const AmgHeader*>(amg_ws);
    cudaStream_t s = (cudaStream_t)stream;
    const int m = nlev - 1;
    if (m > 0) k_vpre<<<grid_for(n * nrhs), 256, 0, s>>>(H, b, nrhs, V.y[0]);
    // a block for every kApplyThreads lanes of a level, kApplyThreads / G rows: by its rows
    // alone a level of 876 rows (32 lanes each) had 4 blocks for 110 blocks' work, and each
    // of its steps took microseconds a right-hand side
    auto blocks = [&](int l) { return grid_for(sizes[l] * (l == 0 ? 1 : amg_group(sizes[l]))); };
    for (int l = 0; l < m; l++) k_vdown<<<blocks(l), kApplyThreads, 0, s>>>(H, l, b, nrhs, V);
    k_vcoarse<<<grid_for(sizes[m] * kWarp), 256, 0, s>>>(H, b, x, nrhs, V);
    for (int l = m - 1; l >= 0; l--) k_vup<<<blocks(l), kApplyThreads, 0, s>>>(H, l, x, nrhs, V);
    return launch_status();
}
