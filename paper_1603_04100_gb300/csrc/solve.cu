// Device-resident Krylov solves of (sigma I - L) u = f (Sec. 4.2; the paper
// solves with AMG -- here BiCGSTAB, van der Vorst 1992, optionally left-scaled
// by the diagonal).
//
// Every system being solved is a "request" whose whole solver state (Krylov
// vectors, per-RHS scalars, reduction partials) lives in its own caller-owned
// workspace.  One persistent cooperative kernel advances any set of requests
// together; an iteration is a fixed sequence of phases separated by a bounded
// grid barrier:
//   PRE_A  FP64: p = r + beta (p - omega v)       | FP32: fold u += s x on restart
//   A      v = A p  (FP32: p formed on the fly at the neighbours)      -> (rh, v)
//   PRE_B  FP64: s = r - alpha v                   | FP32: skipped
//   B      t = A s  (FP32: s formed on the fly)                     -> (t, s), (t, t)
//   C      x += alpha p + omega s, r = s - omega t                  -> (rh, r), (r, r)
// FP64 materialises p and s because forming them at every neighbour would
// multiply the FP64 work by K on a part whose FP64 pipe is 1/56 of FP32; the
// FP32 path forms them on the fly and saves two barriers.  Rows are cut into
// fixed chunks of kCh rows; a chunk's partials are reduced in a fixed order
// and the block that finishes a request's last chunk of a phase sums that
// request's partials in chunk order and advances its per-RHS state (in a launch
// of one request of few chunks every block does both, for itself).  Results
// therefore depend neither on the grid size nor on the other requests.
// The kernel is in solve_kernel.cuh; this file has the host side and the small
// kernels around it.
//
// Per right-hand side:
//   RESTART  FP64 true residual r64 = f - A u (FP32 path: on hi + lo weights,
//            after folding the last inner correction into u); stop at rtol,
//            else restart the Krylov vectors from D^-1 r64 (FP32 path: scaled
//            by 1 / ||r64|| and rounded to FP32)
//   INNER    BiCGSTAB until the recursive residual meets the restart target;
//            a diverging FP32 inner solve is abandoned and its correction dropped
//   DONE
#include <stdlib.h>
#include <string.h>

#include "solve_kernel.cuh"

namespace mvgd {
namespace {

using namespace solver;

// ------------------------------------------------------------------------------
// Step trace: block 0 of the solver stamps the device clock after every grid
// barrier, with the step it closed, into a static device ring that the host
// reads with mvgd_trace_read.  Off unless mvgd_trace_enable(1).
// ------------------------------------------------------------------------------
static __device__ unsigned long long g_trace[kTraceMax];
static __device__ unsigned int g_trace_n;
int g_trace_on = 0;

// ------------------------------------------------------------------------------
// Request workspace layout, set-up and tear-down
// ------------------------------------------------------------------------------
struct ReqLayout {
    Prob* prob;
    RhsState* st;
    double* part;
    unsigned* arrive;
    mvgd_solve_info* info;
    double* fs;
    double* us;
    double* r64;
    void* invd;
    void* vec[12];  // x r rh p0 p1 v0 v1 s t x_best ph sh
    int nlev;       // multigrid levels (precond == 2), else 0
    float* vy[kAmgMaxLevels];
    float* vr[kAmgMaxLevels];
    float* vb[kAmgMaxLevels];
    float* vx[kAmgMaxLevels];
    size_t bytes;
};

ReqLayout req_layout(void* ws, int64_t n, int Q, int prec, int precond) {
    ReqLayout L;
    memset(&L, 0, sizeof(L));
    Carver cv(ws);
    const int64_t nchunk = (n + kCh - 1) / kCh;
    const size_t vt = prec == MVGD_FP64 ? sizeof(double) : sizeof(float);
    L.prob = cv.take<Prob>(1);
    L.st = cv.take<RhsState>(Q);
    L.part = cv.take<double>(kRedSlots * chan_count(precond == 2) * nchunk * Q);
    L.arrive = cv.take<unsigned>(kRedSlots * 8);  // a set for each right-hand-side group (256 bytes either way)
    L.info = cv.take<mvgd_solve_info>(Q);
    L.fs = cv.take<double>(n * Q);
    L.us = cv.take<double>(n * Q);
    L.r64 = cv.take<double>(n * Q);
    L.invd = cv.take<char>(vt * n);
    const int nvec = precond == 2 ? 12 : 10;
    for (int v = 0; v < nvec; v++) L.vec[v] = cv.take<char>(vt * n * Q);
    if (precond == 2) {
        int64_t sizes[kAmgMaxLevels];
        L.nlev = amg_levels(n, sizes);
        for (int l = 0; l < L.nlev; l++) {
            const int64_t m = n_padded(sizes[l]) * Q;
            L.vy[l] = cv.take<float>(m);
            L.vr[l] = cv.take<float>(m);
            if (l > 0) {
                L.vb[l] = cv.take<float>(m);
                L.vx[l] = cv.take<float>(m);
            }
        }
    }
    L.bytes = cv.used;
    return L;
}

// Chunk tables of one launch: level 0 (Krylov phases), levels 1 .. kAmgMaxLevels-1
// and the coarsest solves; each with its per-request first-unit array.
struct CtlLayout {
    unsigned* bar;
    int* words;     // err, active, nrestart, stop
    const Prob** prob;
    int* chunk_base[kAmgMaxLevels + 1];  // [0] fine, [l] level l, [kAmgMaxLevels] coarsest
    size_t bytes;
};

CtlLayout ctl_layout(void* ws, int max_req) {
    CtlLayout C;
    memset(&C, 0, sizeof(C));
    Carver cv(ws);
    C.bar = cv.take<unsigned>(2);
    C.words = cv.take<int>(4);
    C.prob = cv.take<const Prob*>(max_req);
    for (int t = 0; t <= kAmgMaxLevels; t++) C.chunk_base[t] = cv.take<int>(max_req + 1);
    C.bytes = cv.used;
    return C;
}

__global__ void k_request_init(Prob P, Prob* dst, int64_t n) {
    // Prob travels by value (kernel parameter), so set-up is capturable in a graph
    if (blockIdx.x == 0 && threadIdx.x == 0) *dst = P;
    if (blockIdx.x == 0 && threadIdx.x < P.Q) {
        RhsState T;
        T.rho = T.alpha = T.omega = 1.0;
        T.beta = 0.0;
        T.fnorm = -1.0;
        T.relres = 1.0;
        T.scale = 0.0;
        T.target = 0.0;
        T.rnorm = 0.0;
        T.rmin = 0.0;
        T.mode = M_RESTART;
        T.pp = 0;
        T.iters = T.inner_iters = T.outer = 0;
        T.status = MVGD_OK;
        T.discard = 0;
        T.stall = 0;
        T.best_flag = T.fold_best = T.since_best = T.pending = 0;
        P.st[threadIdx.x] = T;
    }
    if (blockIdx.x == 0 && threadIdx.x < kRedSlots * 8) P.arrive[threadIdx.x] = 0;
}

// Left scaling of the Krylov system: d_r = sigma + sum_s |w_rs| over the row's
// FP64 (or hi + lo) weights.  Always positive, unlike sigma - w_self: rows of an
// MVGD operator on irregular samples need not be diagonally dominant, and a
// self weight near sigma would make the Jacobi divisor vanish.
__global__ void k_prep_scaling(Prob P) {
    const int k = P.k, m = k + 1;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < P.n; r += (int64_t)gridDim.x * blockDim.x) {
        const int64_t vb = (r / kSlice) * (int64_t)(kSlice * m) + (r % kSlice);
        double d = fabs(P.sigma);
        for (int s = 0; s < m; s++) {
            const int64_t e = vb + (int64_t)s * kSlice;
            double w = P.prec == MVGD_FP64 ? static_cast<const double*>(P.val)[e]
                                           : (double)static_cast<const float*>(P.val)[e] + (double)P.val_lo[e];
            d += fabs(w);
        }
        const double inv = d > 0 ? 1.0 / d : 1.0;
        if (P.prec == MVGD_FP64) static_cast<double*>(P.invd)[r] = inv;
        else static_cast<float*>(P.invd)[r] = (float)inv;
    }
}

__global__ void k_gather_rows(const double* __restrict__ src, const int32_t* __restrict__ order, int64_t n, int Q,
                              double* __restrict__ dst, int zero) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * Q; e += (int64_t)gridDim.x * blockDim.x) {
        if (zero || src == nullptr) { dst[e] = 0.0; continue; }
        const int64_t r = e / Q, q = e % Q;
        const int64_t from = order ? (int64_t)order[r] : r;
        dst[e] = src[from * Q + q];
    }
}

__global__ void k_finish(const Prob* P, mvgd_solve_info* out) {
    const int q = threadIdx.x;
    if (q >= P->Q) return;
    RhsState T;
    load_state(T, P->st + q);
    mvgd_solve_info I;
    I.iters = T.iters;
    I.outer = T.outer;
    I.relres = T.relres;
    int s = T.status;
    if (T.mode != M_DONE && s == MVGD_OK) s = MVGD_ENOCONV;
    I.status = s;
    I.reserved = 0;
    out[q] = I;
}

__global__ void k_scatter_solution(const Prob* P, double* __restrict__ dst) {
    const int64_t n = P->n;
    const int Q = P->Q;
    const int32_t* order = P->order;
    const double* src = P->u;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * Q; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = e / Q, q = e % Q;
        const int64_t to = order ? (int64_t)order[r] : r;
        dst[to * Q + q] = src[e];
    }
}

constexpr int kTableMax = 256;
struct TableArgs {
    const Prob* prob[kTableMax];
    int nchunk[kTableMax];
    int count;
    int first_chunk;
};

// Request and chunk tables from by-value parameters (capturable in a graph);
// the first group also resets the barrier and the control words.
__global__ void k_build_table(TableArgs A, int base, const Prob** prob, int* chunk_base, unsigned* bar,
                              int* words, int first_group) {
    __shared__ int start[kTableMax + 1];
    if (threadIdx.x == 0) {
        start[0] = A.first_chunk;
        for (int i = 0; i < A.count; i++) start[i + 1] = start[i] + A.nchunk[i];
    }
    __syncthreads();
    for (int i = threadIdx.x; i <= A.count; i += blockDim.x) {
        if (prob && i < A.count) prob[base + i] = A.prob[i];
        chunk_base[base + i] = start[i];
    }
    if (first_group && threadIdx.x == 0) {
        bar[0] = 0;
        bar[1] = 0;
        words[0] = 0;  // err
        words[3] = 0;  // stop
    }
}

// The tables, control words and counts of a launch of one request: it needs no
// unit tables (its units are numbered from 0).
__global__ void k_start_one(const Prob* req, const Prob** prob, unsigned* bar, int* words) {
    if (threadIdx.x != 0) return;
    prob[0] = req;
    bar[0] = 0;
    bar[1] = 0;
    int act = 0, rst = 0;
    for (int q = 0; q < req->Q; q++) {
        const int md = __ldcg(&req->st[q].mode);
        act += md != M_DONE;
        rst += md == M_RESTART;
    }
    words[0] = 0;  // err
    words[1] = act;
    words[2] = rst;
    words[3] = 0;  // stop
}

// Counts running and restarting right-hand sides of the listed requests.
__global__ void k_count_active(const Prob** prob, int count, int* words) {
    __shared__ int act, rst;
    if (threadIdx.x == 0) { act = 0; rst = 0; }
    __syncthreads();
    for (int i = threadIdx.x; i < count; i += blockDim.x) {
        const Prob* P = prob[i];
        for (int q = 0; q < P->Q; q++) {
            const int md = __ldcg(&P->st[q].mode);
            if (md != M_DONE) atomicAdd(&act, 1);
            if (md == M_RESTART) atomicAdd(&rst, 1);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        words[1] = act;
        words[2] = rst;
    }
}

// After a launch that a cancel word or a barrier time-out ended, mark the
// right-hand sides that did not finish.
__global__ void k_mark_exit(const Prob** prob, int count, const int* words) {
    const int err = words[0], stop = words[3];
    if (!err && !stop) return;
    for (int i = threadIdx.x; i < count; i += blockDim.x) {
        const Prob* P = prob[i];
        for (int q = 0; q < P->Q; q++)
            if (P->st[q].mode != M_DONE) P->st[q].status = err ? err : MVGD_ECANCELLED;
    }
}

// done[i] = 1 when every right-hand side of request i has finished.
__global__ void k_poll(TableArgs A, int32_t* done) {
    for (int i = threadIdx.x; i < A.count; i += blockDim.x) {
        const Prob* P = A.prob[i];
        int all = 1;
        for (int q = 0; q < P->Q; q++) all &= (__ldcg(&P->st[q].mode) == M_DONE);
        done[i] = all;
    }
}

int rhs_group(bool mixed, bool amg, int Q, int tiles, int kmax) {
    if (mixed) return amg ? rhs_group_mixed_amg(Q, tiles, kmax) : rhs_group_mixed_plain(Q, tiles, kmax);
    return amg ? rhs_group_fp64_amg(Q, tiles, kmax) : rhs_group_fp64_plain(Q, tiles, kmax);
}

int gather_blocks(int64_t elems) {
    int64_t gb = (elems + 255) / 256;
    return (int)(gb > 8192 ? 8192 : (gb < 1 ? 1 : gb));
}

}  // namespace
}  // namespace mvgd

using namespace mvgd;

// ---------------------------------------------------------------------------------
// Requests
// ---------------------------------------------------------------------------------
MVGD_API size_t mvgd_request_workspace_bytes(int64_t n, int32_t k, int32_t nrhs, int32_t prec, int32_t precond) {
    (void)k;
    if (n <= 0 || nrhs < 1 || nrhs > 8 || precond < 0 || precond > 2) return 0;
    if (precond == 2 && amg_levels(n, nullptr) == 0) return 0;
    return req_layout(nullptr, n, nrhs, prec, precond).bytes;
}

MVGD_API mvgd_status mvgd_request_init(void* req_ws, size_t req_bytes, const mvgd_ell* L, int32_t nrhs, double sigma,
                                       const double* f, const double* u0, const mvgd_solve_opts* opts,
                                       mvgd_stream_t stream) {
    if (!req_ws || !L || !f || !opts || nrhs < 1 || nrhs > 8) return MVGD_EINVAL;
    if (L->n < 2 || L->n >= (1ll << 31) || L->k < kMinK || L->k > kMaxK || !L->col || !L->val) return MVGD_EINVAL;
    if (L->prec != MVGD_FP64 && L->prec != MVGD_FP32_REFINE) return MVGD_EINVAL;
    if (L->prec == MVGD_FP32_REFINE && !L->val_lo) return MVGD_EINVAL;
    if (!aligned(f) || !aligned(u0) || !aligned(req_ws) || !aligned(L->col) || !aligned(L->val) ||
        !aligned(L->val_lo) || !aligned(L->order))
        return MVGD_EINVAL;
    if (!(opts->rtol > 0) || opts->maxit < 1 || !(sigma == sigma)) return MVGD_EINVAL;
    if (opts->precond < 0 || opts->precond > 2) return MVGD_EINVAL;
    if (opts->precond == 2 && (!opts->amg || !aligned(opts->amg))) return MVGD_EINVAL;
    const bool mixed = L->prec == MVGD_FP32_REFINE;
    if (mixed && (opts->inner_maxit < 1 || !(opts->inner_rtol > 0) || opts->max_outer < 1)) return MVGD_EINVAL;
    const int64_t n = L->n;
    ReqLayout W = req_layout(req_ws, n, nrhs, L->prec, opts->precond);
    if (req_bytes < W.bytes) return MVGD_EWORKSPACE;
    cudaStream_t s = (cudaStream_t)stream;
    const int gb = gather_blocks(n * nrhs);
    k_gather_rows<<<gb, 256, 0, s>>>(f, L->order, n, nrhs, W.fs, 0);
    k_gather_rows<<<gb, 256, 0, s>>>(u0, L->order, n, nrhs, W.us, u0 == nullptr);
    Prob P;
    P.n = n;
    P.k = L->k;
    P.Q = nrhs;
    P.prec = L->prec;
    P.precond = opts->precond == 1 ? 1 : 0;
    P.sigma = sigma;
    P.col = L->col;
    P.val = L->val;
    P.val_lo = L->val_lo;
    P.order = L->order;
    P.f = W.fs;
    P.u = W.us;
    P.x = mixed ? W.vec[0] : (void*)W.us;
    P.xb = W.vec[9];
    P.r = W.vec[1];
    P.rh = W.vec[2];
    P.p[0] = W.vec[3];
    P.p[1] = W.vec[4];
    P.v[0] = W.vec[5];
    P.v[1] = W.vec[6];
    P.s = W.vec[7];
    P.t = W.vec[8];
    P.r64 = W.r64;
    P.invd = W.invd;
    P.st = W.st;
    P.part = W.part;
    P.arrive = W.arrive;
    P.nchunk = (int)((n + kCh - 1) / kCh);
    P.nq = nrhs;
    P.rtol = opts->rtol;
    P.inner_rtol = mixed ? opts->inner_rtol : 0.0;
    P.maxit = opts->maxit;
    P.inner_maxit = mixed ? opts->inner_maxit : opts->maxit;
    P.max_outer = mixed ? opts->max_outer : 1000;
    P.pad2 = 0;
    P.amg = opts->precond == 2 ? static_cast<const AmgHeader*>(opts->amg) : nullptr;
    P.amg_levels = W.nlev;
    P.q0 = 0;
    P.ph = W.vec[10];
    P.sh = W.vec[11];
    for (int l = 0; l < kAmgMaxLevels; l++) {
        P.vy[l] = W.vy[l];
        P.vr[l] = W.vr[l];
        P.vb[l] = W.vb[l];
        P.vx[l] = W.vx[l];
    }
    k_request_init<<<1, 32, 0, s>>>(P, W.prob, n);
    if (P.precond) k_prep_scaling<<<gather_blocks(n), 256, 0, s>>>(P);
    return launch_status();
}

MVGD_API size_t mvgd_iterate_workspace_bytes(int32_t max_requests, int64_t max_total_rows) {
    if (max_requests < 1 || max_total_rows < 1) return 0;
    return ctl_layout(nullptr, max_requests).bytes;
}

MVGD_API mvgd_status mvgd_iterate(const mvgd_request* reqs, int32_t count, int32_t prec, int32_t precond,
                                  int32_t max_iterations, const int32_t* cancel, void* ctl_ws, size_t ctl_bytes,
                                  mvgd_stream_t stream) {
    if (!reqs || count < 1 || count > kMaxReq || max_iterations < 0 || !ctl_ws) return MVGD_EINVAL;
    if (prec != MVGD_FP64 && prec != MVGD_FP32_REFINE) return MVGD_EINVAL;
    if (precond < 0 || precond > 2) return MVGD_EINVAL;
    const bool amg = precond == 2;
    int64_t total_rows = 0;
    int maxQ = 1, kmax = kMinK, mlev = 0;
    for (int i = 0; i < count; i++) {
        const mvgd_request& R = reqs[i];
        if (!R.workspace || !aligned(R.workspace) || R.n < 2 || R.n >= (1ll << 31) || R.nrhs < 1 || R.nrhs > 8 ||
            R.k < kMinK || R.k > kMaxK)
            return MVGD_EINVAL;
        total_rows += R.n;
        if (R.nrhs > maxQ) maxQ = R.nrhs;
        if (R.k > kmax) kmax = R.k;
        if (amg) {
            const int nl = amg_levels(R.n, nullptr);
            if (nl == 0) return MVGD_EINVAL;
            if (nl - 1 > mlev) mlev = nl - 1;
        }
    }
    if (!aligned(ctl_ws) || !aligned(cancel)) return MVGD_EINVAL;
    if (ctl_bytes < mvgd_iterate_workspace_bytes(count, total_rows)) return MVGD_EWORKSPACE;
    if (max_iterations == 0) return MVGD_OK;
    cudaStream_t s = (cudaStream_t)stream;
    CtlLayout C = ctl_layout(ctl_ws, count);
    ReqTable tab;
    memset(&tab, 0, sizeof(tab));
    tab.prob = C.prob;
    tab.mlev = mlev;
    tab.nreq = count;
    const bool mixed = prec == MVGD_FP32_REFINE;
    // one request: its right-hand sides in groups where they leave SMs idle
    const int gq = count == 1 && maxQ > 1
                       ? rhs_group(mixed, amg, maxQ, (int)((reqs[0].n + kCh - 1) / kCh), kmax) : maxQ;
    tab.groups = maxQ / gq;
    tab.gq = gq;
    const int qt = gq <= 1 ? 1 : (gq <= 2 ? 2 : (gq <= 4 ? 4 : 8));  // the solver's right-hand-side width
    // lanes of a coarse level's rows: what fills the blocks that level 0 brings
    // along, and no more.  A small system's levels could use more blocks, but every
    // grid barrier then waits for those too: 20,000 rows have 79 tiles; with 313
    // blocks (32 lanes a row on level 1) each of the 14 steps of an iteration took
    // 0.7 to 1 us longer than with 79 blocks and 8 lanes a row.
    int64_t threads = 0;
    for (int i = 0; i < count; i++) threads += ((reqs[i].n + kCh - 1) / kCh) * kThreads;
    threads *= tab.groups;
    for (int l = 0; l < kAmgMaxLevels; l++) {
        int64_t rows = 0;
        for (int i = 0; amg && l > 0 && i < count; i++) {
            int64_t sizes[kAmgMaxLevels];
            const int nl = amg_levels(reqs[i].n, sizes);
            if (l < nl - 1) rows += sizes[l] * tab.groups;
        }
        int g = l == 0 || rows == 0 ? 1 : amg_group(rows);
        while (g > 1 && rows * g > threads) g >>= 1;
        tab.G[l] = g;
    }
    tab.sharing = count > 1 ? S_LISTED
                            : ((reqs[0].n + kCh - 1) / kCh <= kFinWarpTiles && (amg || !mixed) ? S_LOCAL : S_SINGLE);
    tab.ntab = amg ? (mlev > 0 ? mlev + 1 : 2) : 1;
    tab.act = count > 1 && act_bytes(count, tab.ntab) <= kActBytes;
    // rows of the coarsest level a block takes: eight (a warp each), fewer while the
    // blocks of one request last -- the FP64 sums of eight warps queue for one SM's pipe
    tab.coarse_rows = kThreads / kWarp;
    if (count == 1 && amg) {
        int64_t sizes[kAmgMaxLevels];
        const int64_t nc = sizes[amg_levels(reqs[0].n, sizes) - 1];
        const int64_t blocks = threads / tab.groups / kThreads < kAmgLanesOnePass / kThreads / tab.groups
                                   ? threads / tab.groups / kThreads : kAmgLanesOnePass / kThreads / tab.groups;
        while (tab.coarse_rows > 1 && (nc + tab.coarse_rows / 2 - 1) / (tab.coarse_rows / 2) <= blocks)
            tab.coarse_rows /= 2;
    }
    // table t: 0 = level-0 tiles, 1 .. mlev-1 = level-t tiles, kAmgMaxLevels = coarsest rows
    for (int t = 0; t <= kAmgMaxLevels; t++) {
        const bool coarse = t == kAmgMaxLevels;
        if (t > 0 && (!amg || (!coarse && t >= mlev))) continue;
        int units = 0;
        for (int g = 0; g < count; g += kTableMax) {
            TableArgs A;
            A.count = count - g < kTableMax ? count - g : kTableMax;
            A.first_chunk = units;
            for (int i = 0; i < A.count; i++) {
                const mvgd_request& R = reqs[g + i];
                A.prob[i] = reinterpret_cast<const Prob*>(R.workspace);  // the Prob record opens every workspace
                int64_t sizes[kAmgMaxLevels];
                const int nl = amg ? amg_levels(R.n, sizes) : 1;
                if (t == 0) A.nchunk[i] = (int)((R.n + kCh - 1) / kCh);
                else if (coarse) A.nchunk[i] = (int)((sizes[nl - 1] + tab.coarse_rows - 1) / tab.coarse_rows);
                else if (t < nl - 1) {
                    const int64_t rows = kThreads / amg_lanes(tab.G[t], sizes[t], qt);  // rows per unit
                    A.nchunk[i] = (int)((sizes[t] + rows - 1) / rows);
                } else {
                    A.nchunk[i] = 0;
                }
                units += A.nchunk[i];
            }
            if (count > 1)
                k_build_table<<<1, 256, 0, s>>>(A, g, t == 0 ? C.prob : nullptr, C.chunk_base[t], C.bar, C.words,
                                                t == 0 && g == 0);
        }
        ChunkTable& T = coarse ? tab.coarse : (t == 0 ? tab.fine : tab.lvl[t]);
        T.chunk_base = C.chunk_base[t];
        T.nchunks = units;
    }
    if (count > 1) {
        k_count_active<<<1, 256, 0, s>>>(C.prob, count, C.words);
    } else {
        k_start_one<<<1, 32, 0, s>>>(reinterpret_cast<const Prob*>(reqs[0].workspace), C.prob, C.bar, C.words);
    }
    Ctl ctl;
    ctl.bar.count = C.bar;
    ctl.bar.gen = C.bar + 1;
    ctl.err = C.words;
    ctl.active = C.words + 1;
    ctl.nrestart = C.words + 2;
    ctl.stop = C.words + 3;
    ctl.cancel = cancel;
    ctl.limit = wait_limit_or(20000000ll);  // polls of >= 32 ns each: seconds, never reached by co-resident blocks
    ctl.trace = nullptr;
    ctl.trace_n = nullptr;
    if (g_trace_on) {
        void *buf = nullptr, *cnt = nullptr;
        MVGD_CUDA_TRY(cudaGetSymbolAddress(&buf, g_trace));
        MVGD_CUDA_TRY(cudaGetSymbolAddress(&cnt, g_trace_n));
        ctl.trace = static_cast<unsigned long long*>(buf);
        ctl.trace_n = static_cast<unsigned*>(cnt);
    }
    ctl.withhold = take_withhold() ? 1 : 0;
    mvgd_status st;
    if (mixed)
        st = amg ? launch_mixed_amg(gq, tab, ctl, max_iterations, kmax, s)
                 : launch_mixed_plain(gq, tab, ctl, max_iterations, kmax, s);
    else
        st = amg ? launch_fp64_amg(gq, tab, ctl, max_iterations, kmax, s)
                 : launch_fp64_plain(gq, tab, ctl, max_iterations, kmax, s);
    if (st != MVGD_OK) return st;
    k_mark_exit<<<1, 256, 0, s>>>(C.prob, count, C.words);
    return launch_status();
}

MVGD_API mvgd_status mvgd_request_poll(void* const* reqs, int32_t count, int32_t* done, mvgd_stream_t stream) {
    if (!reqs || count < 1 || !done || !aligned(done)) return MVGD_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    for (int g = 0; g < count; g += kTableMax) {
        TableArgs A;
        A.count = count - g < kTableMax ? count - g : kTableMax;
        A.first_chunk = 0;
        for (int i = 0; i < A.count; i++) {
            if (!reqs[g + i] || !aligned(reqs[g + i])) return MVGD_EINVAL;
            A.prob[i] = reinterpret_cast<const Prob*>(reqs[g + i]);
            A.nchunk[i] = 0;
        }
        k_poll<<<1, 256, 0, s>>>(A, done + g);
    }
    return launch_status();
}

MVGD_API mvgd_status mvgd_request_finish(void* req_ws, int64_t n, int32_t nrhs, double* u, mvgd_solve_info* info,
                                         mvgd_stream_t stream) {
    if (!req_ws || !u || !info || n < 1 || nrhs < 1 || nrhs > 8) return MVGD_EINVAL;
    if (!aligned(req_ws) || !aligned(u)) return MVGD_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const Prob* P = reinterpret_cast<const Prob*>(req_ws);
    k_scatter_solution<<<gather_blocks(n * nrhs), 256, 0, s>>>(P, u);
    k_finish<<<1, 32, 0, s>>>(P, info);
    return launch_status();
}

// ---------------------------------------------------------------------------------
// One system: init + iterate to the end + finish
// ---------------------------------------------------------------------------------
MVGD_API size_t mvgd_solve_workspace_bytes(int64_t n, int32_t k, int32_t nrhs, int32_t prec, int32_t precond) {
    if (n <= 0 || nrhs < 1 || nrhs > 8) return 0;
    const size_t req = mvgd_request_workspace_bytes(n, k, nrhs, prec, precond);
    if (req == 0) return 0;
    size_t amg = 0;
    if (precond == 2) {
        amg = mvgd_amg_workspace_bytes(n, k);
        if (amg == 0) return 0;
    }
    return req + mvgd_iterate_workspace_bytes(1, n) + align_up(sizeof(mvgd_solve_info) * 8) + align_up(amg);
}

MVGD_API mvgd_status mvgd_solve(const mvgd_ell* L, int32_t nrhs, double sigma, const double* f, double* u,
                                const mvgd_solve_opts* opts, mvgd_solve_info* info, const int32_t* cancel,
                                void* ws, size_t ws_bytes, mvgd_stream_t stream) {
    if (!L || !f || !u || !opts || !info || !ws || nrhs < 1 || nrhs > 8) return MVGD_EINVAL;
    if (L->n < 2 || L->n >= (1ll << 31) || L->k < kMinK || L->k > kMaxK || !L->col || !L->val) return MVGD_EINVAL;
    if (L->prec != MVGD_FP64 && L->prec != MVGD_FP32_REFINE) return MVGD_EINVAL;
    if (!(opts->rtol > 0) || opts->maxit < 1 || !(sigma == sigma)) return MVGD_EINVAL;
    if (L->prec == MVGD_FP32_REFINE &&
        (!L->val_lo || opts->inner_maxit < 1 || !(opts->inner_rtol > 0) || opts->max_outer < 1))
        return MVGD_EINVAL;
    if (opts->precond < 0 || opts->precond > 2 || (opts->amg && !aligned(opts->amg))) return MVGD_EINVAL;
    size_t need = mvgd_solve_workspace_bytes(L->n, L->k, nrhs, L->prec, opts->precond);
    if (need == 0) return MVGD_EINVAL;
    if (opts->precond == 2 && opts->amg) need -= align_up(mvgd_amg_workspace_bytes(L->n, L->k));  // not built here
    if (!aligned(ws) || !aligned(u) || !aligned(f)) return MVGD_EINVAL;
    if (ws_bytes < need) return MVGD_EWORKSPACE;
    cudaPointerAttributes pa;
    MVGD_CUDA_TRY(cudaPointerGetAttributes(&pa, info));
    const bool host_info = pa.type != cudaMemoryTypeDevice && pa.type != cudaMemoryTypeManaged;
    char* base = static_cast<char*>(ws);
    const size_t req_bytes = mvgd_request_workspace_bytes(L->n, L->k, nrhs, L->prec, opts->precond);
    const size_t ctl_bytes = mvgd_iterate_workspace_bytes(1, L->n);
    void* req = base;
    void* ctl = base + req_bytes;
    mvgd_solve_info* staged = reinterpret_cast<mvgd_solve_info*>(base + req_bytes + ctl_bytes);
    mvgd_solve_opts o = *opts;
    mvgd_status st;
    if (o.precond == 2 && !o.amg) {
        // no hierarchy given: build one after the info staging area
        void* amg = base + req_bytes + ctl_bytes + align_up(sizeof(mvgd_solve_info) * 8);
        st = mvgd_amg_setup(L, sigma, amg, mvgd_amg_workspace_bytes(L->n, L->k), stream);
        if (st != MVGD_OK) return st;
        o.amg = amg;
    }
    st = mvgd_request_init(req, req_bytes, L, nrhs, sigma, f, u, &o, stream);
    if (st != MVGD_OK) return st;
    // every inner iteration and every restart is one pass of the phases
    const bool mixed = L->prec == MVGD_FP32_REFINE;
    long long budget = (long long)opts->maxit + 2ll * ((mixed ? opts->max_outer : 1000) + 2) + 4;
    if (budget > (1ll << 30)) budget = 1ll << 30;
    mvgd_request one;
    one.workspace = req;
    one.n = L->n;
    one.nrhs = nrhs;
    one.k = L->k;
    st = mvgd_iterate(&one, 1, L->prec, o.precond, (int32_t)budget, cancel, ctl, ctl_bytes, stream);
    if (st != MVGD_OK) return st;
    st = mvgd_request_finish(req, L->n, nrhs, u, host_info ? staged : info, stream);
    if (st != MVGD_OK) return st;
    if (!host_info) return MVGD_OK;
    cudaStream_t s = (cudaStream_t)stream;
    MVGD_CUDA_TRY(cudaMemcpyAsync(info, staged, sizeof(mvgd_solve_info) * nrhs, cudaMemcpyDeviceToHost, s));
    MVGD_CUDA_TRY(cudaStreamSynchronize(s));
    int worst = MVGD_OK;
    for (int i = 0; i < nrhs; i++)
        if (info[i].status != MVGD_OK && worst == MVGD_OK) worst = info[i].status;
    return (mvgd_status)worst;
}

// ---------------------------------------------------------------------------------
// Step trace
// ---------------------------------------------------------------------------------
MVGD_API mvgd_status mvgd_trace_enable(int32_t on) {
    g_trace_on = on ? 1 : 0;
    if (on) {
        const unsigned zero = 0;
        MVGD_CUDA_TRY(cudaMemcpyToSymbol(g_trace_n, &zero, sizeof(zero)));
    }
    return MVGD_OK;
}

MVGD_API int32_t mvgd_trace_read(uint64_t* out, int32_t max) {
    if (!out || max < 1) return -1;
    unsigned n = 0;
    if (cudaMemcpyFromSymbol(&n, g_trace_n, sizeof(n)) != cudaSuccess) return -1;
    const int32_t count = (int32_t)(n < (unsigned)kTraceMax ? n : (unsigned)kTraceMax);
    const int32_t take = count < max ? count : max;
    if (take > 0 && cudaMemcpyFromSymbol(out, g_trace, sizeof(uint64_t) * take) != cudaSuccess) return -1;
    return take;
}
