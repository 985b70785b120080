// y = alpha (sigma x - L x) + beta y on the sliced ELL operator (the product a
// Krylov solve of (sigma I - L) u = f repeats; Sec. 3.1, Sec. 4.2).
//
// One thread per row: within a warp the 32 rows of one slice read every slot
// of col / val as one coalesced 128-byte (FP32) or 256-byte (FP64) line; x is
// gathered through L1/L2.  Three arithmetic forms:
//   F64       standard form  w_0 x_i + sum_s w_s x_{c_s}, FP64 weights;
//   F32       difference form sum_s w_s (x_{c_s} - x_i) with FP32 hi weights:
//             rows of L sum to zero, so the self weight is implied and the
//             products act on small differences of a smooth vector;
//   F64_HILO  standard form with w = hi + lo evaluated in FP64.
#include <type_traits>

#include "common.cuh"

namespace mvgd {
namespace {

// The operator's columns and weights are streamed once per product: loaded
// past L1 (read-only path, no L1 allocation), so that L1 keeps the lines of x
// the neighbour gathers reuse.  At 1M rows, K = 20 this took the FP32 product
// from 45 us to 35 us.  (Plain asm: the arrays do not change while a kernel runs.)
__device__ __forceinline__ int32_t ld_stream(const int32_t* p) {
    int32_t v;
    asm("ld.global.nc.L1::no_allocate.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float ld_stream(const float* p) {
    float v;
    asm("ld.global.nc.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ double ld_stream(const double* p) {
    double v;
    asm("ld.global.nc.L1::no_allocate.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}

// Row j of x (Q right-hand sides side by side), by the widest loads that Q allows: x is
// 256-byte aligned (checked at the entry), so a row of an even Q starts on two elements'
// boundary, one of Q = 4 or 8 on four's.  FP32, 1,048,576 rows, K = 20, eight vectors:
// 213 -> 90 us (a warp's gather of one element of 32 rows takes as many L1 passes as one of
// four); four of 100,003 rows, K = 16: 12.3 -> 10.3.
template <int Q>
__device__ __forceinline__ void load_x(const double* __restrict__ x, int64_t j, double (&v)[Q]) {
    const double* p = x + j * Q;
    if constexpr (Q % 2 == 0) {
#pragma unroll
        for (int q = 0; q < Q; q += 2) {
            const double2 t = *reinterpret_cast<const double2*>(p + q);
            v[q] = t.x;
            v[q + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int q = 0; q < Q; q++) v[q] = p[q];
    }
}
template <int Q>
__device__ __forceinline__ void load_x(const float* __restrict__ x, int64_t j, float (&v)[Q]) {
    const float* p = x + j * Q;
    if constexpr (Q % 4 == 0) {
#pragma unroll
        for (int q = 0; q < Q; q += 4) {
            const float4 t = *reinterpret_cast<const float4*>(p + q);
            v[q] = t.x;
            v[q + 1] = t.y;
            v[q + 2] = t.z;
            v[q + 3] = t.w;
        }
    } else if constexpr (Q % 2 == 0) {
#pragma unroll
        for (int q = 0; q < Q; q += 2) {
            const float2 t = *reinterpret_cast<const float2*>(p + q);
            v[q] = t.x;
            v[q + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int q = 0; q < Q; q++) v[q] = p[q];
    }
}

// Rows a block of the FP64 products.  With several right-hand sides they are bound by the
// FP64 pipe (2 FMAs a clock an SM), and blocks of 256 leave some SMs a third more rows than
// others (100,003 rows: 391 blocks on 152 SMs); one warp a block spreads them within 3 %
// and a small operator over every SM.  The hi + lo product has two FP64 conversions and an
// addition a weight more on that pipe and gains with a loop over K too (1,048,576 rows,
// K = 20: 177 -> 172 us; 524,288, K = 31: 141 -> 131).
constexpr int kF64Threads = 32;

// The row's k slots in order, `add(weight, row of x)` for each: GROUPS = k / 4 groups of
// four, known at compile time, and (REST) the k % 4 slots left over.  The columns, weights
// and rows of x of a batch of BATCH slots are all requested before its first product,
// whatever K is; a loop over a K known at run time keeps four slots' loads in flight.
template <int Q, int GROUPS, bool REST, int BATCH, typename T, typename Add>
__device__ __forceinline__ void walk_slots(int k, const int32_t* __restrict__ col, const T* __restrict__ val,
                                           const T* __restrict__ x, Add&& add) {
    auto batch = [&](auto width, int s0) {  // slots s0 .. s0 + width - 1
        constexpr int W = decltype(width)::value;
        int32_t c[W];
        T w[W], xj[W][Q];
#pragma unroll
        for (int u = 0; u < W; u++) c[u] = ld_stream(col + (int64_t)(s0 + u) * kSlice);
#pragma unroll
        for (int u = 0; u < W; u++) w[u] = ld_stream(val + (int64_t)(s0 + u + 1) * kSlice);
#pragma unroll
        for (int u = 0; u < W; u++) load_x<Q>(x, c[u], xj[u]);
#pragma unroll
        for (int u = 0; u < W; u++) add(w[u], xj[u]);
    };
    constexpr int F = 4 * GROUPS;
#pragma unroll
    for (int b = 0; b < F / BATCH; b++) batch(std::integral_constant<int, BATCH>{}, b * BATCH);
    if constexpr (F % BATCH != 0) batch(std::integral_constant<int, F % BATCH>{}, F / BATCH * BATCH);
    if constexpr (REST) {  // branches, not predicates: an FMA that is off still takes its turn on the pipe
        const int rest = k - F;
        if (rest == 1) batch(std::integral_constant<int, 1>{}, F);
        else if (rest == 2) batch(std::integral_constant<int, 2>{}, F);
        else if (rest == 3) batch(std::integral_constant<int, 3>{}, F);
    }
}

// `launch(groups)` with groups = k / 4 at compile time.
template <typename Launch>
void by_groups(int k, Launch&& launch) {
    static_assert(kMaxK / 4 == 7, "a case a group count");
    switch (k / 4) {
        case 0: launch(std::integral_constant<int, 0>{}); break;
        case 1: launch(std::integral_constant<int, 1>{}); break;
        case 2: launch(std::integral_constant<int, 2>{}); break;
        case 3: launch(std::integral_constant<int, 3>{}); break;
        case 4: launch(std::integral_constant<int, 4>{}); break;
        case 5: launch(std::integral_constant<int, 5>{}); break;
        case 6: launch(std::integral_constant<int, 6>{}); break;
        default: launch(std::integral_constant<int, 7>{}); break;
    }
}

// FP64, in us, against a loop over K of blocks of 256 rows with scalar loads of x: 20,001
// rows, K = 18, one vector 5.0 -> 3.1, K = 31 7.9 -> 3.5, K = 20, eight 25 -> 16; 524,288
// rows, K = 25, four vectors 108 -> 103, K = 24, eight 230 -> 197; 100,003 rows, K = 16,
// four 20.5 -> 19.2 (12 of them the FP64 pipe), but K = 28, seven 47 -> 52 (its registers
// leave a partial second wave there).
// REST: K is not 4 GROUPS (else it is known at compile time: 5 % at 100,003 rows, K = 16).
template <int Q, int GROUPS, bool REST>
__global__ void __launch_bounds__(kF64Threads) k_spmv_f64(int64_t n, int kr, const int32_t* __restrict__ col,
                                                   const double* __restrict__ val, double sigma, double alpha,
                                                   const double* __restrict__ x, double beta,
                                                   double* __restrict__ y) {
    const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int k = REST ? kr : 4 * GROUPS;
    const int m = k + 1;
    const int64_t vb = (r / kSlice) * (int64_t)(kSlice * m) + (r % kSlice);
    const int64_t cb = (r / kSlice) * (int64_t)(kSlice * k) + (r % kSlice);
    const double w0 = ld_stream(val + vb);
    double xi[Q], acc[Q];
    load_x<Q>(x, r, xi);
#pragma unroll
    for (int q = 0; q < Q; q++) {
        acc[q] = w0 * xi[q];
    }
    walk_slots<Q, GROUPS, REST, (Q <= 2 ? 8 : 4)>(k, col + cb, val + vb, x, [&](double w, const double (&xj)[Q]) {
#pragma unroll
        for (int q = 0; q < Q; q++) acc[q] = fma(w, xj[q], acc[q]);
    });
#pragma unroll
    for (int q = 0; q < Q; q++) {
        double out = alpha * (sigma * xi[q] - acc[q]);
        if (beta != 0.0) out = fma(beta, y[r * Q + q], out);
        y[r * Q + q] = out;
    }
}

// KK > 0: K fixed at compile time (the K of the workloads; every slot's loads can be issued
// at once).  KK < 0: -KK - 1 groups of four and the rest, with up to three vectors: 20,001
// rows, K = 25, one vector 5.2 -> 2.8 us, two 4.2 -> 3.2; 524,288 rows, K = 28, one 27 -> 20.
// KK == 0: a loop over K, with more (K = 28, four, 100,003 rows: 9 us, 14 by groups).
template <int Q, int KK>
__global__ void __launch_bounds__(256) k_spmv_f32(int64_t n, int kr, const int32_t* __restrict__ col,
                                                   const float* __restrict__ val, float sigma, float alpha,
                                                   const float* __restrict__ x, float beta,
                                                   float* __restrict__ y) {
    const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int k = KK > 0 ? KK : kr;
    const int m = k + 1;
    const int64_t vb = (r / kSlice) * (int64_t)(kSlice * m) + (r % kSlice);
    const int64_t cb = (r / kSlice) * (int64_t)(kSlice * k) + (r % kSlice);
    float xi[Q], acc[Q];
    load_x<Q>(x, r, xi);
#pragma unroll
    for (int q = 0; q < Q; q++) {
        acc[q] = 0.0f;
    }
    auto add = [&](float w, const float (&xj)[Q]) {
#pragma unroll
        for (int q = 0; q < Q; q++) acc[q] = fmaf(w, xj[q] - xi[q], acc[q]);
    };
    if constexpr (KK < 0) {
        walk_slots<Q, -KK - 1, true, 8>(k, col + cb, val + vb, x, add);
    } else {
#pragma unroll (KK > 0 ? KK : 4)
        for (int s = 0; s < k; s++) {
            const int64_t j = ld_stream(col + cb + (int64_t)s * kSlice);
            const float w = ld_stream(val + vb + (int64_t)(s + 1) * kSlice);
            float xj[Q];
            load_x<Q>(x, j, xj);
            add(w, xj);
        }
    }
#pragma unroll
    for (int q = 0; q < Q; q++) {
        float out = alpha * (sigma * xi[q] - acc[q]);
        if (beta != 0.0f) out = fmaf(beta, y[r * Q + q], out);
        y[r * Q + q] = out;
    }
}

template <int Q, int KK>
void launch_f32(const mvgd_ell* L, double sigma, double alpha, const void* x, double beta, void* y, cudaStream_t s) {
    k_spmv_f32<Q, KK><<<(unsigned)((L->n + 255) / 256), 256, 0, s>>>(
        L->n, L->k, L->col, static_cast<const float*>(L->val), (float)sigma, (float)alpha,
        static_cast<const float*>(x), (float)beta, static_cast<float*>(y));
}

template <int Q, int GROUPS>
void launch_f64(const mvgd_ell* L, double sigma, double alpha, const void* x, double beta, void* y, cudaStream_t s) {
    auto fn = L->k == 4 * GROUPS ? k_spmv_f64<Q, GROUPS, false> : k_spmv_f64<Q, GROUPS, true>;
    fn<<<(unsigned)((L->n + kF64Threads - 1) / kF64Threads), kF64Threads, 0, s>>>(
        L->n, L->k, L->col, static_cast<const double*>(L->val), sigma, alpha, static_cast<const double*>(x), beta,
        static_cast<double*>(y));
}

template <int Q>
mvgd_status launch_spmv(const mvgd_ell* L, int mode, double sigma, double alpha, const void* x, double beta,
                        void* y, cudaStream_t s) {
    if (mode == MVGD_SPMV_F32) {
        switch (L->k) {
            case 12: launch_f32<Q, 12>(L, sigma, alpha, x, beta, y, s); break;
            case 16: launch_f32<Q, 16>(L, sigma, alpha, x, beta, y, s); break;
            case 20: launch_f32<Q, 20>(L, sigma, alpha, x, beta, y, s); break;
            case 24: launch_f32<Q, 24>(L, sigma, alpha, x, beta, y, s); break;
            default:
                if constexpr (Q <= 3)
                    by_groups(L->k, [&](auto g) { launch_f32<Q, -decltype(g)::value - 1>(L, sigma, alpha, x, beta, y, s); });
                else
                    launch_f32<Q, 0>(L, sigma, alpha, x, beta, y, s);
        }
    } else if (mode == MVGD_SPMV_F64) {
        by_groups(L->k, [&](auto g) { launch_f64<Q, decltype(g)::value>(L, sigma, alpha, x, beta, y, s); });
    } else {
        // hi + lo: hi is stored as float in val; read it through a float view
        return MVGD_EINVAL;
    }
    return launch_status();
}

template <int Q>
__global__ void __launch_bounds__(kF64Threads) k_spmv_hilo(int64_t n, int k, const int32_t* __restrict__ col,
                                                    const float* __restrict__ hi, const float* __restrict__ lo,
                                                    double sigma, double alpha, const double* __restrict__ x,
                                                    double beta, double* __restrict__ y) {
    const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int m = k + 1;
    const int64_t vb = (r / kSlice) * (int64_t)(kSlice * m) + (r % kSlice);
    const int64_t cb = (r / kSlice) * (int64_t)(kSlice * k) + (r % kSlice);
    const double w0 = (double)ld_stream(hi + vb) + (double)ld_stream(lo + vb);
    double xi[Q], acc[Q];
    load_x<Q>(x, r, xi);
#pragma unroll
    for (int q = 0; q < Q; q++) {
        acc[q] = w0 * xi[q];
    }
    // the compiler's unrolling, with wide loads of x only for eight vectors (100,003 rows,
    // K = 30, four: 32.7 us without, 33.4 with)
#pragma unroll 4
    for (int s = 0; s < k; s++) {
        const int64_t j = ld_stream(col + cb + (int64_t)s * kSlice);
        const int64_t e = vb + (int64_t)(s + 1) * kSlice;
        const double w = (double)ld_stream(hi + e) + (double)ld_stream(lo + e);
        double xj[Q];
        if constexpr (Q == 8) {
            load_x<Q>(x, j, xj);
        } else {
#pragma unroll
            for (int q = 0; q < Q; q++) xj[q] = x[j * Q + q];
        }
#pragma unroll
        for (int q = 0; q < Q; q++) acc[q] = fma(w, xj[q], acc[q]);
    }
#pragma unroll
    for (int q = 0; q < Q; q++) {
        double out = alpha * (sigma * xi[q] - acc[q]);
        if (beta != 0.0) out = fma(beta, y[r * Q + q], out);
        y[r * Q + q] = out;
    }
}

template <int Q>
mvgd_status launch_hilo(const mvgd_ell* L, double sigma, double alpha, const void* x, double beta, void* y,
                        cudaStream_t s) {
    const unsigned blocks = (unsigned)((L->n + kF64Threads - 1) / kF64Threads);
    k_spmv_hilo<Q><<<blocks, kF64Threads, 0, s>>>(L->n, L->k, L->col, static_cast<const float*>(L->val), L->val_lo,
                                          sigma, alpha, static_cast<const double*>(x), beta,
                                          static_cast<double*>(y));
    return launch_status();
}

}  // namespace
}  // namespace mvgd

using namespace mvgd;

MVGD_API mvgd_status mvgd_spmv(const mvgd_ell* L, int32_t mode, int32_t nrhs, double sigma, double alpha,
                               const void* x, double beta, void* y, mvgd_stream_t stream) {
    if (!L || !x || !y || !L->col || !L->val || L->n < 1 || L->k < 1 || L->k > kMaxK) return MVGD_EINVAL;
    if (nrhs < 1 || nrhs > 8) return MVGD_EINVAL;
    if (!aligned(x) || !aligned(y) || !aligned(L->col) || !aligned(L->val) || !aligned(L->val_lo))
        return MVGD_EINVAL;
    if (mode == MVGD_SPMV_F64 && L->prec != MVGD_FP64) return MVGD_EINVAL;
    if ((mode == MVGD_SPMV_F32 || mode == MVGD_SPMV_F64_HILO) && L->prec != MVGD_FP32_REFINE) return MVGD_EINVAL;
    if (mode == MVGD_SPMV_F64_HILO && !L->val_lo) return MVGD_EINVAL;
    if (mode < 0 || mode > 2) return MVGD_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    if (mode == MVGD_SPMV_F64_HILO) {
        switch (nrhs) {
            case 1: return launch_hilo<1>(L, sigma, alpha, x, beta, y, s);
            case 2: return launch_hilo<2>(L, sigma, alpha, x, beta, y, s);
            case 3: return launch_hilo<3>(L, sigma, alpha, x, beta, y, s);
            case 4: return launch_hilo<4>(L, sigma, alpha, x, beta, y, s);
            case 5: return launch_hilo<5>(L, sigma, alpha, x, beta, y, s);
            case 6: return launch_hilo<6>(L, sigma, alpha, x, beta, y, s);
            case 7: return launch_hilo<7>(L, sigma, alpha, x, beta, y, s);
            default: return launch_hilo<8>(L, sigma, alpha, x, beta, y, s);
        }
    }
    switch (nrhs) {
        case 1: return launch_spmv<1>(L, mode, sigma, alpha, x, beta, y, s);
        case 2: return launch_spmv<2>(L, mode, sigma, alpha, x, beta, y, s);
        case 3: return launch_spmv<3>(L, mode, sigma, alpha, x, beta, y, s);
        case 4: return launch_spmv<4>(L, mode, sigma, alpha, x, beta, y, s);
        case 5: return launch_spmv<5>(L, mode, sigma, alpha, x, beta, y, s);
        case 6: return launch_spmv<6>(L, mode, sigma, alpha, x, beta, y, s);
        case 7: return launch_spmv<7>(L, mode, sigma, alpha, x, beta, y, s);
        default: return launch_spmv<8>(L, mode, sigma, alpha, x, beta, y, s);
    }
}
