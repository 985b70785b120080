// kNN on a periodic cell grid (Sec. 2: N(i) = the K nearest neighbours).
//
// Build: bounding box -> cell edge s (given, or estimated from the surface area
// covered by a 64^3 occupancy bitmap) -> every point gets integer cell
// coordinates c = floor((p - lo) / s) and a bucket, the row-major index of
// (c mod M) with power-of-two wrap sizes M per axis, so that at most ~2n
// buckets exist whatever the extent; a counting sort groups points by bucket.
// Any block of <= M consecutive cells per axis maps to distinct buckets, so a
// query scans each bucket at most once; points of far cells that share a
// bucket are merely extra candidates.  Row-major buckets make the three cells
// of a block's row one run of buckets (two where the wrap cuts it): the 27
// cells around a query are 9 ranges of points.
//
// Query (one warp per point, points visited in bucket order for locality):
//   1. the 9 rows of cells around the query are turned into point ranges;
//      lanes take candidates 32 at a time from the concatenated ranges;
//   2. screen: candidates beyond the nearest face of the block are dropped (a
//      K-th neighbour out there needs another ring anyway); the others get a
//      32-bit key, the FP32 squared distance with the low bits replaced by the
//      candidate's place in the warp's list, and the 32 smallest are sorted
//      across lanes.  A compare-exchange is a shuffle and a min or max (96-bit
//      (distance, index) keys took some fifteen instructions, for all of a
//      block's candidates, and the integer pipe bound the kernel); past 256
//      candidates the list is cut to the 32 smallest whenever it is full;
//   3. proof: the kept candidates' FP32 distances with a bound on their error
//      settle the order of the K nearest, and that no other point is nearer;
//   4. where only the order is unsettled (distances closer than the bound), the
//      32 kept ones are re-ranked by their exact FP64 keys
//      fl(fl(fl(dx dx) + fl(dy dy)) + fl(dz dz)) and index;
//   5. anything else goes to the general scan: rings that grow until the K-th
//      exact distance is inside the block, 96-bit keys, and exact FP64 keys
//      throughout where the screen cannot separate the 32nd candidate.
// All bounds are evaluated with directed rounding or a generous factor.
// 1,048,576 points, K = 20: the query 2.7 -> 0.97 ms (881 warp instructions a
// query before candidates beyond the guard were dropped), about a tenth of the
// queries re-ranked; the whole call with the row order 3.53 -> 1.27 ms.
#include <cfloat>
#include <mutex>

#include "common.cuh"

namespace mvgd {
namespace {

constexpr int kOccBits = 64;                 // occupancy bitmap edge
constexpr int kOccWords = kOccBits * kOccBits * kOccBits / 32;
constexpr int64_t kOccSample = 1 << 18;      // points it looks at, at most
constexpr int kBboxBlocks = 512;
constexpr int kScanTile = 2048;
constexpr int kQueryWarps = 8;
constexpr int kQueryPerWarp = 8;  // at most: consecutive queries of a block share their cells in L1

struct KnnParams {
    double lo[3];
    double ext[3];
    double s;
    float inv_s_f;  // cells are assigned in FP32 (the query's margin covers it)
    int D[3];       // cells per axis
    int Mb[3];      // log2 of the wrap per axis
    int nbuckets;
    int pad;
    float s_f;      // cell edge in FP32
    float ext_f;    // largest extent in FP32
    float eps_abs;  // bound on |d_fp32 - d_exact| from rounding the coordinates
    float margin;   // bound on the error of FP32 cell-boundary positions
};

struct Key {
    uint64_t a;  // distance bits (FP32 or FP64, non-negative so integer order = value order)
    uint32_t b;  // point index
};

__device__ __forceinline__ bool key_less(const Key& x, const Key& y) {
    return x.a < y.a || (x.a == y.a && x.b < y.b);
}
__device__ __forceinline__ Key key_shfl_xor(const Key& k, int m) {
    Key o;
    o.a = shfl_xor_u64(k.a, m);
    o.b = __shfl_xor_sync(0xffffffffu, k.b, m);
    return o;
}
__device__ __forceinline__ Key key_shfl(const Key& k, int src) {
    Key o;
    o.a = shfl_u64(k.a, src);
    o.b = __shfl_sync(0xffffffffu, k.b, src);
    return o;
}
__device__ __forceinline__ Key key_empty() { return Key{~0ull, 0xffffffffu}; }

// Ascending bitonic sort of one key per lane.
__device__ __forceinline__ void warp_sort(Key& k) {
    const unsigned lane = lane_id();
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            Key o = key_shfl_xor(k, stride);
            bool up = (lane & size) == 0 || size == 32;
            bool lower = (lane & stride) == 0;
            bool o_less = key_less(o, k);
            // lower element keeps the min when ascending
            if ((lower == up) ? o_less : !o_less) k = o;
        }
    }
}

// list (ascending) <- the 32 smallest of list and chunk (chunk sorted ascending).
__device__ __forceinline__ void warp_merge(Key& list, Key chunk) {
    const unsigned lane = lane_id();
    Key rev = key_shfl(chunk, 31 - lane);
    if (key_less(rev, list)) list = rev;
#pragma unroll
    for (int stride = 16; stride > 0; stride >>= 1) {
        Key o = key_shfl_xor(list, stride);
        bool lower = (lane & stride) == 0;
        bool o_less = key_less(o, list);
        if (lower ? o_less : !o_less) list = o;
    }
}

__device__ __forceinline__ uint32_t bucket_of(uint32_t x, uint32_t y, uint32_t z, const int* Mb) {
    return ((z & ((1u << Mb[2]) - 1)) << (Mb[0] + Mb[1])) | ((y & ((1u << Mb[1]) - 1)) << Mb[0]) |
           (x & ((1u << Mb[0]) - 1));
}

// Cell coordinate of x >= 0 (the point's offset from the box corner, FP32).
__device__ __forceinline__ int cell_of(float x, float inv_s, int D) {
    const float t = floorf(x * inv_s);
    if (!(t >= 0.0f)) return 0;
    return t > (float)(D - 1) ? D - 1 : (int)t;
}

// Cell coordinates -1 .. 2^20 - 1 as one word, 21 bits each.  An axis whose extent is
// not finite has no cells (D = 0) and its points the coordinate -1: such a query finds
// no range and no ring to grow, and its list is empty (-1).  Packed as it is, -1 would
// fill the word, and the ring sizes formed from it run into 10^8 rounds a query.
__device__ __forceinline__ uint64_t pack_cell(const int (&c)[3]) {
    return (uint64_t)(c[0] + 1) | (uint64_t)(c[1] + 1) << 21 | (uint64_t)(c[2] + 1) << 42;
}
__device__ __forceinline__ void unpack_cell(uint64_t w, int (&c)[3]) {
    c[0] = (int)(w & 0x1fffffu) - 1;
    c[1] = (int)((w >> 21) & 0x1fffffu) - 1;
    c[2] = (int)(w >> 42) - 1;
}

// True in the last block of the grid to arrive (every thread of the block
// returns it); everything the other blocks wrote before is visible to it.
__device__ __forceinline__ bool last_block(unsigned* ticket) {
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(ticket, 1u) + 1u == gridDim.x;
        if (last) __threadfence();
    }
    __syncthreads();
    return last;
}

// ---------------------------------------------------------------------------
// Build kernels
// ---------------------------------------------------------------------------
// Bounding box: a partial a block, the last block to finish combines them.
__global__ void __launch_bounds__(256) k_bbox(const double* __restrict__ pts, int64_t n, double* part,
                                              unsigned* ticket, KnnParams* P) {
    double mn[3] = {DBL_MAX, DBL_MAX, DBL_MAX}, mx[3] = {-DBL_MAX, -DBL_MAX, -DBL_MAX};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        for (int a = 0; a < 3; a++) {
            double v = pts[3 * i + a];
            mn[a] = fmin(mn[a], v);
            mx[a] = fmax(mx[a], v);
        }
    }
    __shared__ double sm[6][32];
    const int w = threadIdx.x / 32, nw = blockDim.x / 32;
    auto combine = [&]() {  // the block's minima and maxima, in sm[.][0]
        for (int a = 0; a < 3; a++) {
            for (int o = 16; o > 0; o >>= 1) {
                mn[a] = fmin(mn[a], __shfl_xor_sync(0xffffffffu, mn[a], o));
                mx[a] = fmax(mx[a], __shfl_xor_sync(0xffffffffu, mx[a], o));
            }
        }
        if (lane_id() == 0)
            for (int a = 0; a < 3; a++) { sm[a][w] = mn[a]; sm[3 + a][w] = mx[a]; }
        __syncthreads();
        if (threadIdx.x < 6) {
            double v = sm[threadIdx.x][0];
            for (int q = 1; q < nw; q++)
                v = threadIdx.x < 3 ? fmin(v, sm[threadIdx.x][q]) : fmax(v, sm[threadIdx.x][q]);
            sm[threadIdx.x][0] = v;
        }
        __syncthreads();
    };
    combine();
    if (threadIdx.x < 6) part[blockIdx.x * 6 + threadIdx.x] = sm[threadIdx.x][0];
    if (!last_block(ticket)) return;
    for (int a = 0; a < 3; a++) { mn[a] = DBL_MAX; mx[a] = -DBL_MAX; }
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x)
        for (int a = 0; a < 3; a++) {
            mn[a] = fmin(mn[a], __ldcg(part + b * 6 + a));
            mx[a] = fmax(mx[a], __ldcg(part + b * 6 + 3 + a));
        }
    combine();
    if (threadIdx.x < 3) {
        P->lo[threadIdx.x] = sm[threadIdx.x][0];
        P->ext[threadIdx.x] = sm[3 + threadIdx.x][0] - sm[threadIdx.x][0];
    }
}

// Cell edge, grid dimensions and wrap sizes.
__device__ void set_params(const unsigned* bits, int64_t n, int k, double cell_size, int nbuckets_max, KnnParams* P) {
    // occupied cells of the 64^3, 32^3, 16^3 and 8^3 grids (a word holds 32 cells of a
    // row: pairs of bits, words 2 apart in y and z merge into the next coarser grid)
    __shared__ int occ[4];
    __shared__ unsigned half[32 * 32 * 2];  // the 32^3 grid: 16 bits a word
    const int tid = threadIdx.x;
    if (tid < 4) occ[tid] = 0;
    __syncthreads();
    if (cell_size <= 0) {
        int c = 0;
        const uint4* b4 = reinterpret_cast<const uint4*>(bits);
        uint4 v[kOccWords / 4 / 256];
#pragma unroll
        for (int u = 0; u < kOccWords / 4 / 256; u++) v[u] = __ldcg(b4 + tid + 256 * u);
#pragma unroll
        for (int u = 0; u < kOccWords / 4 / 256; u++)
            c += __popc(v[u].x) + __popc(v[u].y) + __popc(v[u].z) + __popc(v[u].w);
        atomicAdd(&occ[0], c);
        auto pairs = [](unsigned w) {  // bit b: either of bits 2b, 2b + 1
            w = (w | (w >> 1)) & 0x55555555u;
            w = (w | (w >> 1)) & 0x33333333u;
            w = (w | (w >> 2)) & 0x0f0f0f0fu;
            w = (w | (w >> 4)) & 0x00ff00ffu;
            return (w | (w >> 8)) & 0xffffu;
        };
        c = 0;
        for (int e = tid; e < 32 * 32 * 2; e += 256) {
            const int x = e & 1, y = (e >> 1) & 31, z = e >> 6;
            unsigned w = 0;
            for (int q = 0; q < 4; q++) w |= __ldcg(bits + ((2 * z + (q >> 1)) * 64 + 2 * y + (q & 1)) * 2 + x);
            half[e] = pairs(w);
            c += __popc(half[e]);
        }
        atomicAdd(&occ[1], c);
        __syncthreads();
        if (tid < 256) {  // 16^3: row (y, z) of 16 bits, both words of the finer grid's rows
            const int y = tid & 15, z = tid >> 4;
            unsigned w = 0;
            for (int q = 0; q < 4; q++) {
                const unsigned* h = half + ((2 * z + (q >> 1)) * 32 + 2 * y + (q & 1)) * 2;
                w |= h[0] | (h[1] << 16);
            }
            w = pairs(w);
            atomicAdd(&occ[2], __popc(w));
            __syncthreads();
            half[tid] = w;
        }
        __syncthreads();
        if (tid < 64) {
            const int y = tid & 7, z = tid >> 3;
            unsigned w = 0;
            for (int q = 0; q < 4; q++) w |= half[(2 * z + (q >> 1)) * 16 + 2 * y + (q & 1)];
            atomicAdd(&occ[3], __popc(pairs(w)));
        }
    }
    __syncthreads();
    if (tid != 0) return;
    double e = fmax(P->ext[0], fmax(P->ext[1], P->ext[2]));
    double s = cell_size;
    if (s <= 0) {
        // surface-area estimate: occupied cells x cell area / mean |n|_1 of a surface, on the
        // finest grid that has three points a cell on average: on a finer one most cells of
        // the surface are empty, the estimate is small and every query scans several rings
        // (2,562 points on the 64^3 grid: cells 2.7 times too small)
        int lv = 0;
        while (lv < 3 && (int64_t)occ[lv] * 3 > n) lv++;
        double s0 = e / (kOccBits >> lv);
        double area = (double)occ[lv] * s0 * s0 / 1.5;
        double rk = sqrt((double)k * area / (3.141592653589793 * (double)n));
        s = 1.25 * rk * (cell_size < 0 ? -cell_size : 1.0);  // a negative cell_size scales the estimate
    }
    if (!(s > 0) || !isfinite(s)) s = e > 0 ? e : 1.0;
    if (e > 0 && s < e * 1e-6) s = e * 1e-6;   // keep cell coordinates below 2^20
    double inv_s = 1.0 / s;
    int Mb[3];
    for (int a = 0; a < 3; a++) {
        double d = floor(P->ext[a] * inv_s) + 1.0;
        if (d > 1048576.0) d = 1048576.0;
        P->D[a] = d >= 0.0 ? (int)d : 0;  // (no finite extent: an infinite coordinate, or none that is a number)
        int b = 0;
        while ((1 << b) < P->D[a] && b < 20) b++;
        Mb[a] = b < 2 ? 2 : b;  // wrap >= 4 so a 3-cell block never aliases
    }
    while (Mb[0] + Mb[1] + Mb[2] > 2 && (1ll << (Mb[0] + Mb[1] + Mb[2])) > nbuckets_max) {
        int a = (Mb[0] >= Mb[1] && Mb[0] >= Mb[2]) ? 0 : (Mb[1] >= Mb[2] ? 1 : 2);
        if (Mb[a] <= 2) break;
        Mb[a]--;
    }
    for (int a = 0; a < 3; a++) P->Mb[a] = Mb[a];
    P->nbuckets = 1 << (Mb[0] + Mb[1] + Mb[2]);
    P->s = s;
    P->inv_s_f = (float)inv_s;
    P->s_f = (float)s;
    P->ext_f = (float)e;
    // |fl32(x - lo) - (x - lo)| <= 2^-24 e per coordinate, for both points: the
    // distance moves by at most 2 sqrt(3) 2^-24 e; rounded up generously.
    P->eps_abs = (float)(4.0 * e * 5.9604644775390625e-08) + 1e-30f;
    // cell boundaries in FP32: the coordinate, its product with 1 / s and the boundary's
    // own position round by at most 2^-24 e each; rounded up generously
    P->margin = (float)(16.0 * e * 5.9604644775390625e-08 + 4.0 * s * 5.9604644775390625e-08) + 1e-30f;
}

// Occupied cells of a 64^3 grid; the last block to finish sets the parameters.
__global__ void __launch_bounds__(256) k_occupancy(const double* __restrict__ pts, int64_t n, unsigned* bits, int k,
                                                   double cell_size, int nbuckets_max, unsigned* ticket,
                                                   KnnParams* P) {
    const double e = fmax(P->ext[0], fmax(P->ext[1], P->ext[2]));
    const float inv = e > 0 ? (float)((double)kOccBits / e) : 0.0f;
    if (cell_size <= 0) {
        const double lo[3] = {P->lo[0], P->lo[1], P->lo[2]};
        // at most kOccSample points, evenly spaced: an estimate needs no more
        const int64_t step = n > kOccSample ? n / kOccSample : 1;
        for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * step; i < n;
             i += (int64_t)gridDim.x * blockDim.x * step) {
            int c[3];
            for (int a = 0; a < 3; a++) {
                const int t = (int)((float)(pts[3 * i + a] - lo[a]) * inv);
                c[a] = t < 0 ? 0 : (t >= kOccBits ? kOccBits - 1 : t);
            }
            const unsigned cell = (c[2] * kOccBits + c[1]) * kOccBits + c[0];
            const unsigned bit = 1u << (cell & 31);
            if (!(__ldcg(&bits[cell >> 5]) & bit)) atomicOr(&bits[cell >> 5], bit);
        }
    }
    if (last_block(ticket)) set_params(bits, n, k, cell_size, nbuckets_max, P);
}

// Exclusive scan of a[0 .. len) in two passes: tile sums (the last block scans
// those), then each tile again with its offset; a[len] = total.
template <int WARPS>
__device__ __forceinline__ int block_scan(int v, int* sh) {  // exclusive; sh: WARPS + 1 ints, the total in the last
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += t;
    }
    if (lane == 31) sh[wid] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        int acc = 0;
#pragma unroll
        for (int q = 0; q < WARPS; q++) {
            const int t = sh[q];
            sh[q] = acc;
            acc += t;
        }
        sh[WARPS] = acc;
    }
    __syncthreads();
    return x - v + sh[wid];
}

constexpr int kScanPer = kScanTile / 256;
__device__ __forceinline__ void scan_load(const int* a, int base, int len, int (&v)[kScanPer]) {
    const int at = base + (int)threadIdx.x * kScanPer;
#pragma unroll
    for (int u = 0; u < kScanPer; u += 4) {
        const int4 t = at + u + 4 <= len ? *reinterpret_cast<const int4*>(a + at + u)
                                         : make_int4(at + u < len ? a[at + u] : 0, at + u + 1 < len ? a[at + u + 1] : 0,
                                                     at + u + 2 < len ? a[at + u + 2] : 0, 0);
        v[u] = t.x; v[u + 1] = t.y; v[u + 2] = t.z; v[u + 3] = t.w;
    }
}

__global__ void __launch_bounds__(256) k_scan_sums(const int* __restrict__ a, int len, int* sums, unsigned* ticket) {
    __shared__ int sh[9];
    int v[kScanPer], t = 0;
    scan_load(a, blockIdx.x * kScanTile, len, v);
#pragma unroll
    for (int u = 0; u < kScanPer; u++) t += v[u];
    block_scan<8>(t, sh);
    if (threadIdx.x == 0) sums[blockIdx.x] = sh[8];
    if (!last_block(ticket)) return;
    int carry = 0;
    for (int b0 = 0; b0 < (int)gridDim.x; b0 += 256) {
        const int b = b0 + (int)threadIdx.x;
        const int x = b < (int)gridDim.x ? __ldcg(sums + b) : 0;
        __syncthreads();  // sh of the previous round is consumed
        const int ex = block_scan<8>(x, sh);
        if (b < (int)gridDim.x) sums[b] = carry + ex;
        carry += sh[8];
    }
}

__global__ void __launch_bounds__(256) k_scan_apply(int* __restrict__ a, int len, const int* __restrict__ sums,
                                                    int64_t total) {
    __shared__ int sh[9];
    const int base = blockIdx.x * kScanTile, at = base + (int)threadIdx.x * kScanPer;
    int v[kScanPer], t = 0;
    scan_load(a, base, len, v);
#pragma unroll
    for (int u = 0; u < kScanPer; u++) t += v[u];
    int acc = sums[blockIdx.x] + block_scan<8>(t, sh);
#pragma unroll
    for (int u = 0; u < kScanPer; u++) {
        if (at + u < len) a[at + u] = acc;
        acc += v[u];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) a[len] = (int)total;
}

__device__ __forceinline__ uint64_t spread3_21(uint32_t v) {
    uint64_t x = v & 0x1fffffu;
    x = (x | x << 32) & 0x1f00000000ffffull;
    x = (x | x << 16) & 0x1f0000ff0000ffull;
    x = (x | x << 8) & 0x100f00f00f00f00full;
    x = (x | x << 4) & 0x10c30c30c30c30c3ull;
    x = (x | x << 2) & 0x1249249249249249ull;
    return x;
}

// The exported order's key: 21-bit Z-order of the point's offset x from the box
// corner, in FP64.  The conversion saturates (and takes a NaN to 0).
__device__ __forceinline__ uint64_t zorder_key(const double (&x)[3], double scale) {
    uint64_t k = 0;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const uint32_t t = __double2uint_rz(x[a] * scale);
        k |= spread3_21(t > 2097151u ? 2097151u : t) << a;
    }
    return k;
}
__device__ __forceinline__ double zorder_scale(const KnnParams& p) {
    const double e = fmax(p.ext[0], fmax(p.ext[1], p.ext[2]));
    return e > 0.0 ? 2097152.0 / e : 0.0;
}

// Each point's cell and place in its bucket and, where the exported order goes by
// radix passes (key not null), its Z-order key.
__global__ void __launch_bounds__(256) k_count(const double* __restrict__ pts, int64_t n,
                                               const KnnParams* __restrict__ P, int* __restrict__ counts,
                                               int* __restrict__ pbucket, int* __restrict__ prank,
                                               uint64_t* __restrict__ pcell, uint64_t* __restrict__ key,
                                               int* __restrict__ val) {
    const KnnParams p = *P;
    const double scale = zorder_scale(p);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double x[3] = {pts[3 * i] - p.lo[0], pts[3 * i + 1] - p.lo[1], pts[3 * i + 2] - p.lo[2]};
        int c[3];
        for (int a = 0; a < 3; a++) c[a] = cell_of((float)x[a], p.inv_s_f, p.D[a]);
        const uint32_t b = bucket_of(c[0], c[1], c[2], p.Mb);
        pbucket[i] = (int)b;
        prank[i] = atomicAdd(&counts[b], 1);
        pcell[i] = pack_cell(c);
        if (key) {
            key[i] = zorder_key(x, scale);
            val[i] = (int)i;
        }
    }
}

// Points and their cells in bucket order (within a bucket in arrival order,
// which no result depends on: the query ranks by exact distance and index).
__global__ void k_scatter(const double* __restrict__ pts, int64_t n, const KnnParams* __restrict__ P,
                          const int* __restrict__ start, const int* __restrict__ pbucket,
                          const int* __restrict__ prank, const uint64_t* __restrict__ pcell,
                          float4* __restrict__ sorted, uint64_t* __restrict__ scell) {
    const KnnParams p = *P;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int pos = start[pbucket[i]] + prank[i];
        float4 v;
        v.x = (float)(pts[3 * i + 0] - p.lo[0]);
        v.y = (float)(pts[3 * i + 1] - p.lo[1]);
        v.z = (float)(pts[3 * i + 2] - p.lo[2]);
        v.w = __int_as_float((int)i);
        sorted[pos] = v;
        scell[pos] = pcell[i];
    }
}

// ---------------------------------------------------------------------------
// The row order exported to callers: every point along one Z-order curve of
// the bounding cube (21 bits per axis), ties by index.  Consecutive points of
// this order are spatial neighbours at every scale down to a few points --
// which the kNN's hashed cell buckets are not where the hash wraps around the
// grid -- and aggregation multigrid, which groups consecutive rows, relies on
// it.
// ---------------------------------------------------------------------------
// Up to kZSmall points one block sorts them in shared memory; above, a stable LSD
// radix sort of (key, index) pairs, 8 bits a pass, two launches a pass.
constexpr int kZSmall = 8192;
constexpr int kZThreads = 512;
constexpr int kRadixThreads = 256;
constexpr int kRadixTile = 4096;  // elements per block: 512 consecutive ones a warp
constexpr int kRadixSmem = kRadixTile * (int)(sizeof(uint64_t) + sizeof(int));
constexpr int kRadixWarps = kRadixThreads / 32;
constexpr int kRadixRounds = kRadixTile / kRadixThreads;

// Ranks of a warp's elements by digit, in element order: rank[r] counts the
// elements of the same digit before element r * 32 + lane of the warp's run,
// and wcnt[d] becomes the run's count of digit d (zero on entry).
template <int ROUNDS>
__device__ __forceinline__ void radix_ranks(const uint64_t (&k)[ROUNDS], const bool (&valid)[ROUNDS], int rounds,
                                            int shift, int* wcnt, int (&rank)[ROUNDS]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int r = 0; r < ROUNDS; r++) {
        if (r >= rounds) break;  // uniform
        const unsigned d = valid[r] ? (unsigned)((k[r] >> shift) & 255u) : 256u + lane;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const int ahead = __popc(peers & ((1u << lane) - 1u));
        const int seen = valid[r] ? wcnt[d] : 0;
        __syncwarp();
        if (valid[r] && ahead == 0) wcnt[d] = seen + __popc(peers);
        __syncwarp();
        rank[r] = seen + ahead;
    }
}

// The whole sort of a small cloud by one block: the same eight stable radix
// passes on (key, index) pairs in shared memory, warp w holding a run of the
// elements in registers.  Separate launches a pass took over 100 us for a few
// thousand points, nearly all of it launch latency; a bitonic sort of 4,096 in
// this block 69 us (78 barriers).
__global__ void __launch_bounds__(kZThreads) k_zorder_small(const double* __restrict__ pts, int n,
                                                            const KnnParams* __restrict__ P, int* __restrict__ order) {
    constexpr int kWarps = kZThreads / 32, kRounds = kZSmall / kZThreads;
    extern __shared__ uint64_t zkey[];  // [n] keys, then [n] indices
    uint16_t* zidx = reinterpret_cast<uint16_t*>(zkey + n);
    __shared__ int wcnt[kWarps][256];
    __shared__ int sh[kWarps + 1];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const KnnParams p = *P;
    const double scale = zorder_scale(p);
    const int rounds = (n + kZThreads - 1) / kZThreads;
    uint64_t k[kRounds];
    int v[kRounds], rank[kRounds];
    bool valid[kRounds];
#pragma unroll
    for (int r = 0; r < kRounds; r++) {
        const int i = (wid * rounds + r) * 32 + lane;
        valid[r] = r < rounds && i < n;
        k[r] = 0;
        v[r] = i;
        if (valid[r]) {
            const double x[3] = {pts[3 * i] - p.lo[0], pts[3 * i + 1] - p.lo[1], pts[3 * i + 2] - p.lo[2]};
            k[r] = zorder_key(x, scale);
        }
    }
    // the upper 32 bits first: where no two points share them they are the order
    __shared__ int tied;
    if (tid == 0) tied = 0;
    for (int pass = 4; pass < 8 + 8; pass++) {
        const int shift = 8 * (pass & 7);
        for (int e = tid; e < kWarps * 256; e += kZThreads) (&wcnt[0][0])[e] = 0;
        __syncthreads();
        radix_ranks<kRounds>(k, valid, rounds, shift, wcnt[wid], rank);
        __syncthreads();
        int total = 0;
        if (tid < 256) {
#pragma unroll
            for (int w = 0; w < kWarps; w++) total += wcnt[w][tid];
        }
        int acc = block_scan<kWarps>(tid < 256 ? total : 0, sh);
        if (tid < 256) {
#pragma unroll
            for (int w = 0; w < kWarps; w++) {
                const int c = wcnt[w][tid];
                wcnt[w][tid] = acc;
                acc += c;
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kRounds; r++)
            if (valid[r]) {
                const int pos = wcnt[wid][(k[r] >> shift) & 255u] + rank[r];
                zkey[pos] = k[r];
                zidx[pos] = (uint16_t)v[r];
            }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kRounds; r++)
            if (valid[r]) {
                const int i = (wid * rounds + r) * 32 + lane;
                k[r] = zkey[i];
                v[r] = zidx[i];
                if (pass == 7 && i > 0 && (zkey[i - 1] >> 32) == (k[r] >> 32)) tied = 1;
            }
        __syncthreads();
        if (pass == 7) {
            if (!tied) break;
            // ties: all eight passes, from the points' own order
#pragma unroll
            for (int r = 0; r < kRounds; r++)
                if (valid[r]) order[v[r]] = (wid * rounds + r) * 32 + lane;  // where each point is now
            __syncthreads();
#pragma unroll
            for (int r = 0; r < kRounds; r++)
                if (valid[r]) {
                    const int i = (wid * rounds + r) * 32 + lane;
                    k[r] = zkey[order[i]];
                    v[r] = i;
                }
            __syncthreads();
        }
    }
#pragma unroll
    for (int r = 0; r < kRounds; r++)
        if (valid[r]) order[(wid * rounds + r) * 32 + lane] = v[r];
}

// One radix pass is two launches.  The first counts each tile's digits,
// counts[tile][256], and adds them up over groups of `group` tiles,
// super[tile / group][256] (zeroed before).  In the second each tile forms its
// own offsets from at most (groups + group) rows of 256 counts -- about
// 2 sqrt(tiles) of them, 32 at 1M points -- so no scan launches lie between.
struct RadixPass {
    int* counts;
    int* super;
    int group, groups;
};

__global__ void __launch_bounds__(kRadixThreads) k_radix_count(const uint64_t* __restrict__ key, int64_t n, int shift,
                                                               RadixPass R) {
    __shared__ int h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kRadixTile;
    const int64_t end = base + kRadixTile < n ? base + kRadixTile : n;
    for (int64_t i = base + threadIdx.x; i < end; i += kRadixThreads) atomicAdd(&h[(key[i] >> shift) & 255u], 1);
    __syncthreads();
    const int c = h[threadIdx.x];
    R.counts[(int64_t)blockIdx.x * 256 + threadIdx.x] = c;
    if (c) atomicAdd(&R.super[(int64_t)(blockIdx.x / R.group) * 256 + threadIdx.x], c);
}

// Stable scatter of a tile: warp w takes elements 512 w .. 512 w + 511 of it in
// order, and each element goes after every earlier element of its digit.  The
// tile is put in digit order in shared memory first, so that what leaves it is
// runs of about 16 consecutive places (written from where they were read, single
// 8- and 4-byte stores made a pass of 1M points 26 us).
__global__ void __launch_bounds__(kRadixThreads) k_radix_scatter(const uint64_t* __restrict__ kin,
                                                                 const int* __restrict__ vin, int64_t n, int shift,
                                                                 RadixPass R, uint64_t* __restrict__ kout,
                                                                 int* __restrict__ vout) {
    __shared__ int wcnt[kRadixWarps][256];
    __shared__ int sh[9];
    __shared__ int gofs[256];  // a digit's first place in the output less its first place in the tile
    extern __shared__ uint64_t zkey[];
    uint64_t* tkey = zkey;  // [kRadixTile] keys, then indices
    int* tval = reinterpret_cast<int*>(tkey + kRadixTile);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int w = 0; w < kRadixWarps; w++) wcnt[w][tid] = 0;
    __syncthreads();
    const int64_t tile0 = (int64_t)blockIdx.x * kRadixTile;
    const int64_t base = tile0 + wid * (kRadixTile / kRadixWarps);
    uint64_t k[kRadixRounds];
    int v[kRadixRounds], rank[kRadixRounds];
    bool valid[kRadixRounds];
#pragma unroll
    for (int r = 0; r < kRadixRounds; r++) {
        const int64_t i = base + r * 32 + lane;
        valid[r] = i < n;
        k[r] = valid[r] ? kin[i] : 0;
        v[r] = valid[r] ? vin[i] : 0;
    }
    // this tile's first place of digit tid: the digits below it, then the tiles before this one
    const int sg = blockIdx.x / R.group;
    int total = 0, before = 0;
#pragma unroll 4
    for (int g = 0; g < R.groups; g++) {
        const int c = __ldg(R.super + (int64_t)g * 256 + tid);
        total += c;
        if (g < sg) before += c;
    }
#pragma unroll 4
    for (int t = sg * R.group; t < (int)blockIdx.x; t++) before += __ldg(R.counts + (int64_t)t * 256 + tid);
    radix_ranks<kRadixRounds>(k, valid, kRadixRounds, shift, wcnt[wid], rank);
    const int digit0 = block_scan<8>(total, sh);  // (its barriers also close the ranking)
    int mine = 0;
    for (int w = 0; w < kRadixWarps; w++) mine += wcnt[w][tid];
    __syncthreads();  // sh is consumed
    const int local0 = block_scan<8>(mine, sh);
    gofs[tid] = digit0 + before - local0;
    int acc = local0;
    for (int w = 0; w < kRadixWarps; w++) {
        const int c = wcnt[w][tid];
        wcnt[w][tid] = acc;
        acc += c;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRadixRounds; r++) {
        if (!valid[r]) continue;
        const int pos = wcnt[wid][(k[r] >> shift) & 255u] + rank[r];
        tkey[pos] = k[r];
        tval[pos] = v[r];
    }
    __syncthreads();
    const int here = (int)(n - tile0 < kRadixTile ? n - tile0 : kRadixTile);
    for (int e = tid; e < here; e += kRadixThreads) {
        const uint64_t x = tkey[e];
        const int64_t to = (int64_t)gofs[(x >> shift) & 255u] + e;
        if (kout) kout[to] = x;
        vout[to] = tval[e];
    }
}

// ---------------------------------------------------------------------------
// Query
// ---------------------------------------------------------------------------
struct AxisRange {
    int first, len;  // first cell (or residue 0) and count
    bool full;       // all residues visited
};

__device__ __forceinline__ double exact_d2(const double* __restrict__ pts, int i, int j) {
    double dx = __dsub_rn(pts[3 * (int64_t)j + 0], pts[3 * (int64_t)i + 0]);
    double dy = __dsub_rn(pts[3 * (int64_t)j + 1], pts[3 * (int64_t)i + 1]);
    double dz = __dsub_rn(pts[3 * (int64_t)j + 2], pts[3 * (int64_t)i + 2]);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// FP32 squares and their sums round by at most half of 2^-149 where they are subnormal
// (clouds of an extent near 1e-20), which no relative bound covers: an absolute error
// bound of a squared distance, several times the three roundings.  Lost in the rounding
// of any normal number above 2^-122.
constexpr float kTinySq = 0x1p-146f;

// Scan the block of ring R around cell c; returns the running list.
template <bool EXACT>
__device__ Key scan_block(const double* __restrict__ pts, const float4* __restrict__ sorted,
                          const int* __restrict__ start, const KnnParams& p, const AxisRange* ax,
                          int i, float qx, float qy, float qz) {
    const unsigned lane = lane_id();
    Key list = key_empty();
    const int ncell = ax[0].len * ax[1].len * ax[2].len;
    for (int cb = 0; cb < ncell; cb += 32) {
        int cid = cb + (int)lane;
        int beg = 0, cnt = 0;
        if (cid < ncell) {
            int tx = cid % ax[0].len;
            int ty = (cid / ax[0].len) % ax[1].len;
            int tz = cid / (ax[0].len * ax[1].len);
            const uint32_t b = bucket_of(ax[0].first + tx, ax[1].first + ty, ax[2].first + tz, p.Mb);
            beg = start[b];
            cnt = start[b + 1] - beg;
        }
        // inclusive prefix of counts across lanes
        int off = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int v = __shfl_up_sync(0xffffffffu, off, o);
            if ((int)lane >= o) off += v;
        }
        const int total = __shfl_sync(0xffffffffu, off, 31);
        for (int t = 0; t < total; t += 32) {
            int c = t + (int)lane;
            Key key = key_empty();
            // owning lane: smallest l with off[l] > c (all lanes take part in the shuffles)
            int l = 0;
#pragma unroll
            for (int step = 16; step > 0; step >>= 1) {
                int probe = __shfl_sync(0xffffffffu, off, l + step - 1);
                if (probe <= c) l += step;
            }
            int lb = __shfl_sync(0xffffffffu, beg, l & 31);
            int lo = __shfl_sync(0xffffffffu, off, l & 31) - __shfl_sync(0xffffffffu, cnt, l & 31);
            if (c < total) {
                int pos = lb + (c - lo);
                float4 v = __ldg(&sorted[pos]);
                int j = __float_as_int(v.w);
                if (j != i) {
                    if (EXACT) {
                        key.a = (uint64_t)__double_as_longlong(exact_d2(pts, i, j));
                    } else {
                        float dx = v.x - qx, dy = v.y - qy, dz = v.z - qz;
                        float d2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
                        key.a = (uint32_t)__float_as_int(d2);
                    }
                    key.b = (uint32_t)j;
                }
            }
            // merge only if some candidate beats the current 32nd entry
            Key worst = key_shfl(list, 31);
            if (__any_sync(0xffffffffu, key_less(key, worst))) {
                warp_sort(key);
                warp_merge(list, key);
            }
        }
    }
    return list;
}

// The general query: rings double until the k-th distance is inside the block;
// a block of more than M cells per axis visits each residue once, so every
// scan is bounded by the bucket count and the loop by log2 of the grid size.  The
// first ring and whether FP32 keys are worth trying are what the screen has found.
__device__ __noinline__ Key query_general(const double* __restrict__ pts, const float4* __restrict__ sorted,
                                          const int* __restrict__ start, const KnnParams& p, int k, int i, float4 me,
                                          uint64_t cell, int ring, bool exact_mode) {
    const float qv[3] = {me.x, me.y, me.z};
    int c[3];
    unpack_cell(cell, c);
    for (int R = ring;;) {
        AxisRange ax[3];
        bool all_full = true;
        float guard = FLT_MAX;
        for (int a = 0; a < 3; a++) {
            int a0 = c[a] - R, a1 = c[a] + R;
            bool lo_open = a0 > 0, hi_open = a1 < p.D[a] - 1;
            if (a0 < 0) a0 = 0;
            if (a1 > p.D[a] - 1) a1 = p.D[a] - 1;
            int len = a1 - a0 + 1, M = 1 << p.Mb[a];
            ax[a].full = len > M;
            ax[a].first = ax[a].full ? 0 : a0;
            ax[a].len = ax[a].full ? M : len;
            if (lo_open || hi_open) all_full = false;
            // distance from the query to the faces of the block (FP32, rounded down)
            if (lo_open) guard = fminf(guard, __fsub_rd(qv[a], __fmul_ru((float)a0, p.s_f)));
            if (hi_open) guard = fminf(guard, __fsub_rd(__fmul_rd((float)(a1 + 1), p.s_f), qv[a]));
        }
        guard = __fsub_rd(guard, p.margin);
        Key list = exact_mode ? scan_block<true>(pts, sorted, start, p, ax, i, me.x, me.y, me.z)
                              : scan_block<false>(pts, sorted, start, p, ax, i, me.x, me.y, me.z);
        Key ex = list;
        if (!exact_mode && list.b != 0xffffffffu)
            ex.a = (uint64_t)__double_as_longlong(exact_d2(pts, i, (int)list.b));
        if (!exact_mode) warp_sort(ex);
        Key kth = key_shfl(ex, k - 1);
        bool have_k = kth.b != 0xffffffffu;
        double dk2 = have_k ? __longlong_as_double((long long)kth.a) : 0.0;
        float ub = __fsqrt_ru(__double2float_ru(dk2));
        bool cov_ok = have_k && (all_full || ub < guard);
        bool ex_ok = true;
        if (!exact_mode) {
            Key last = key_shfl(list, 31);
            if (last.b != 0xffffffffu) {
                float d = __fsqrt_rd(fmaxf(__fsub_rd(__uint_as_float((uint32_t)last.a), kTinySq), 0.0f));
                float lb = __fsub_rd(__fmul_rd(d, 1.0f - 8.0f * 5.9604645e-08f), p.eps_abs);
                ex_ok = lb > ub;
            }
        }
        if (cov_ok && ex_ok) return ex;
        if (!ex_ok && !exact_mode) {
            exact_mode = true;  // redo this ring with exact keys
            continue;
        }
        if (all_full) return ex;  // fewer than k points: impossible after host checks
        R *= 2;
    }
}

// Ascending bitonic sort of one word a lane, every comparison "lower lane keeps
// the smaller" (the first step of a merge pairs mirror images), so a step is a
// shuffle and a min or max by one bit of the lane.
__device__ __forceinline__ uint32_t word_step(uint32_t v, int mask, bool lower) {
    const uint32_t o = __shfl_xor_sync(0xffffffffu, v, mask);
    return lower ? min(v, o) : max(v, o);
}
__device__ __forceinline__ uint32_t warp_sort_words(uint32_t v, unsigned lane) {
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
        v = word_step(v, size - 1, (lane & (size >> 1)) == 0);
#pragma unroll
        for (int stride = size >> 2; stride > 0; stride >>= 1) v = word_step(v, stride, (lane & stride) == 0);
    }
    return v;
}
// The 32 smallest of two ascending lists, ascending.
__device__ __forceinline__ uint32_t warp_merge_words(uint32_t list, uint32_t chunk, unsigned lane) {
    uint32_t v = min(list, __shfl_sync(0xffffffffu, chunk, 31 - lane));
#pragma unroll
    for (int stride = 16; stride > 0; stride >>= 1) v = word_step(v, stride, (lane & stride) == 0);
    return v;
}

constexpr int kKept = 256;  // candidates inside the guard a warp can hold
constexpr uint32_t kKeptMask = kKept - 1;

// The 32 smallest of a warp's `kept` keys, ascending.
__device__ __forceinline__ uint32_t smallest_kept(const uint32_t* qkey, int kept, unsigned lane) {
    uint32_t list = (int)lane < kept ? qkey[lane] : 0xffffffffu;
    list = warp_sort_words(list, lane);
    for (int t0 = 32; t0 < kept; t0 += 32) {
        const uint32_t key = t0 + (int)lane < kept ? qkey[t0 + lane] : 0xffffffffu;
        if (__any_sync(0xffffffffu, key < __shfl_sync(0xffffffffu, list, 31)))
            list = warp_merge_words(list, warp_sort_words(key, lane), lane);
    }
    return list;
}

// The screen of a query with more candidates in its cells than a warp holds: points
// denser than the cells were sized for (a graded or clustered cloud).  A full list is cut
// down to its 32 smallest, and candidates at or above the last of those are dropped from
// there on.  `off` and `shift`: the lanes' ranges; `cut`: the guard's square, as the
// unsigned word whose order is that of non-negative floats.  Returns the candidates held.
// A function of its own, so that ordinary queries keep their registers.  In ms a call,
// 300,000 points most of which lie near two poles, K = 20 and 31: 2.6 and 5.2 (handed
// to the general scan and its 96-bit keys: 5.1 and 8.2; by the general scan alone, before
// there was a screen: 3.7 and 4.9).
__device__ __noinline__ int screen_dense(const float4* __restrict__ sorted, float4 me, int off, int shift,
                                         uint32_t cut, uint32_t* qkey, int* qpos) {
    const unsigned lane = lane_id();
    const int total = __shfl_sync(0xffffffffu, off, 31);
    int kept = 0;
    for (int t0 = 0; t0 < total; t0 += 32) {
        const int t = t0 + (int)lane;
        int l = 0;
#pragma unroll
        for (int step = 16; step > 0; step >>= 1)
            if (__shfl_sync(0xffffffffu, off, l + step - 1) <= t) l += step;
        const int pos = t + __shfl_sync(0xffffffffu, shift, l & 31);
        uint32_t d2 = 0xffffffffu;
        if (t < total) {
            const float4 v = __ldg(&sorted[pos]);
            const float dx = v.x - me.x, dy = v.y - me.y, dz = v.z - me.z;
            if (__float_as_int(v.w) != __float_as_int(me.w))
                d2 = __float_as_uint(fmaf(dz, dz, fmaf(dy, dy, dx * dx)));
        }
        unsigned who = __ballot_sync(0xffffffffu, d2 < cut);
        if (kept + __popc(who) > kKept) {
            __syncwarp();
            const uint32_t list = smallest_kept(qkey, kept, lane);
            const int at = qpos[list & kKeptMask];
            __syncwarp();
            qkey[lane] = (list & ~kKeptMask) | lane;
            qpos[lane] = at;
            __syncwarp();
            cut = min(cut, __shfl_sync(0xffffffffu, list, 31) & ~kKeptMask);
            kept = 32;
            who = __ballot_sync(0xffffffffu, d2 < cut);
        }
        if (d2 < cut) {
            const int at = kept + __popc(who & ((1u << lane) - 1u));
            qkey[at] = (d2 & ~kKeptMask) | (uint32_t)at;
            qpos[at] = pos;
        }
        kept += __popc(who);
    }
    return kept;
}

// (four blocks an SM: with the 80 registers that three leave the call took 1.52 ms instead
// of 1.31 at 1,048,576 points)
__global__ void __launch_bounds__(kQueryWarps * 32, 4)
k_query(const double* __restrict__ pts, int64_t n, int k, const KnnParams* __restrict__ P,
        const float4* __restrict__ sorted, const int* __restrict__ start, const uint64_t* __restrict__ scell,
        int32_t* __restrict__ nbr, int per_warp) {
    __shared__ uint32_t kept_key[kQueryWarps][kKept];
    __shared__ int kept_pos[kQueryWarps][kKept];
    const KnnParams& p = *P;
    const unsigned lane = lane_id();
    const float eps = p.eps_abs;
    uint32_t* const qkey = kept_key[threadIdx.x / 32];
    int* const qpos = kept_pos[threadIdx.x / 32];
    // this lane's row of cells (lanes 0 .. 17: row lane / 2, the part before or after the wrap)
    const int dy = (int)(lane / 2) % 3 - 1, dz = (int)(lane / 6) - 1;
    const int64_t q0 = blockIdx.x * (int64_t)(kQueryWarps * per_warp) + threadIdx.x / 32;
    for (int it = 0; it < per_warp; it++) {
        const int64_t q = q0 + it * kQueryWarps;
        if (q >= n) return;
        const float4 me = __ldg(&sorted[q]);
        const int i = __float_as_int(me.w);
        int c[3];
        unpack_cell(__ldg(&scell[q]), c);
        // the lane's point range
        int beg = 0, cnt = 0;
        {
            const int y = c[1] + dy, z = c[2] + dz;
            if (lane < 18 && y >= 0 && y < p.D[1] && z >= 0 && z < p.D[2]) {
                const int x0 = max(c[0] - 1, 0), len = min(c[0] + 1, p.D[0] - 1) - x0 + 1;
                const int M = 1 << p.Mb[0], xm = x0 & (M - 1), head = min(len, M - xm);
                const int first = (lane & 1) ? 0 : xm, run = (lane & 1) ? len - head : head;
                const uint32_t b = bucket_of(first, y, z, p.Mb);
                if (run > 0) {
                    beg = __ldg(start + b);
                    cnt = __ldg(start + b + run) - beg;
                }
            }
        }
        int off = cnt;  // inclusive prefix
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, off, o);
            if ((int)lane >= o) off += v;
        }
        int total = __shfl_sync(0xffffffffu, off, 31);
        total = total > kKept ? 0 : total;  // (more: screen_dense)
        const int shift = beg - (off - cnt);  // a candidate of this lane's range: its place + shift
        // the guard: the query's distance to the faces of the block, rounded down.  A K-th
        // neighbour beyond it needs more rings anyway, so candidates beyond it are dropped
        // as they come: about 40 of the 110 of K = 20 stay to be sorted
        float guard = FLT_MAX;
        const float qv[3] = {me.x, me.y, me.z};
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const int a0 = c[a] - 1, a1 = c[a] + 1;
            if (a0 > 0) guard = fminf(guard, __fsub_rd(qv[a], __fmul_ru((float)a0, p.s_f)));
            if (a1 < p.D[a] - 1) guard = fminf(guard, __fsub_rd(__fmul_rd((float)(a1 + 1), p.s_f), qv[a]));
        }
        const bool open = guard < FLT_MAX;  // (false: the block is the whole grid)
        guard = __fsub_rd(guard, p.margin);
        const float guard2 = open ? (guard > 0.0f ? guard * guard : 0.0f) : FLT_MAX;
        int kept = 0;
        for (int t0 = 0; t0 < total; t0 += 32) {
            const int t = t0 + (int)lane;
            int l = 0;  // the range holding place t: the smallest l with off[l] > t
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
                if (__shfl_sync(0xffffffffu, off, l + step - 1) <= t) l += step;
            const int pos = t + __shfl_sync(0xffffffffu, shift, l & 31);
            float d2 = 0.0f;
            bool keep = false;
            if (t < total) {
                const float4 v = __ldg(&sorted[pos]);
                const float dx = v.x - me.x, dyy = v.y - me.y, dzz = v.z - me.z;
                d2 = fmaf(dzz, dzz, fmaf(dyy, dyy, dx * dx));
                keep = __float_as_int(v.w) != i && !(d2 >= guard2);
            }
            const unsigned who = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                const int at = kept + __popc(who & ((1u << lane) - 1u));
                qkey[at] = (__float_as_uint(d2) & ~kKeptMask) | (uint32_t)at;
                qpos[at] = pos;
            }
            kept += __popc(who);
        }
        if (__shfl_sync(0xffffffffu, off, 31) > kKept)
            kept = screen_dense(sorted, me, off, shift, __float_as_uint(guard2), qkey, qpos);
        __syncwarp();
        int32_t nb = 0;
        bool done = false;
        // the general scan's first ring (fewer than K inside the guard: the next one), and
        // whether FP32 distances have already failed to tell the 32nd candidate from the K-th
        int ring = open && kept < k ? 2 : 1;
        bool tight = false;
        if (kept >= k) {
            const uint32_t list = smallest_kept(qkey, kept, lane);
            // the 32 smallest's FP32 squared distances with the bound on their error:
            // |d_fp32 - d| <= eps from the coordinates, 4 roundings in the square (and, where
            // they are subnormal, kTinySq)
            const bool have = list != 0xffffffffu;
            const float4 v = __ldg(&sorted[have ? qpos[list & kKeptMask] : (int)q]);
            const float dx = v.x - me.x, dyy = v.y - me.y, dzz = v.z - me.z;
            const float d2 = fmaf(dzz, dzz, fmaf(dyy, dyy, dx * dx));
            auto bound = [&](float x) {
                const float d = sqrtf(x + kTinySq) * 1.000001f;
                return (fmaf(2.0f, d, eps) * eps + x * (8.0f * 5.9604645e-08f)) * 1.001f + 2.0f * kTinySq;
            };
            const float err = bound(d2);
            const float lo = __fsub_rd(d2, err), hi = __fadd_ru(d2, err);
            const float kth_hi = __shfl_sync(0xffffffffu, hi, k - 1);
            // no candidate outside the list reaches a distance: those dropped are beyond the
            // guard, those screened out have keys above the last one kept
            const float out2 = __fmul_rd(fmaxf(__fsub_rd(__fmul_rd(guard, 1.0f - 8.0f * 5.9604645e-08f), eps), 0.0f),
                                         1.0f - 8.0f * 5.9604645e-08f);
            float out_lo = open ? __fsub_rd(__fmul_rd(out2, out2), 2.0f * kTinySq) : FLT_MAX;
            if (kept >= 32) {  // (32: a dense query's list may have been cut)
                const float x = __uint_as_float(__shfl_sync(0xffffffffu, list, 31) & ~kKeptMask);
                const float x_lo = __fsub_rd(x, bound(x));
                out_lo = fminf(out_lo, x_lo);
                tight = !(x_lo > kth_hi);
            }
            const float prev = __shfl_up_sync(0xffffffffu, hi, 1);
            const bool settled = lane == 0 || !have || ((int)lane < k ? lo > prev : lo > kth_hi);
            const bool covered = out_lo > kth_hi;
            if (covered && __all_sync(0xffffffffu, settled)) {
                nb = __float_as_int(v.w);
                done = true;
            } else if (covered) {  // only the order is open: the kept ones by their exact keys
                Key ex = key_empty();
                if (have) {
                    ex.b = (uint32_t)__float_as_int(v.w);
                    ex.a = (uint64_t)__double_as_longlong(exact_d2(pts, i, (int)ex.b));
                }
                warp_sort(ex);
                const Key kth = key_shfl(ex, k - 1);
                if (out_lo > __double2float_ru(__longlong_as_double((long long)kth.a))) {
                    nb = (int32_t)ex.b;
                    done = true;
                }
            }
        }
        if (!done) nb = (int32_t)query_general(pts, sorted, start, p, k, i, me, scell[q], ring, tight).b;
        if ((int)lane < k) nbr[(int64_t)i * k + lane] = nb;
        __syncwarp();  // the kept lists are read; the next query may write them
    }
}

struct KnnLayout {
    KnnParams* params;
    double* bbox;
    char* zeroed;       // tickets, occ and start lie together: one memset
    unsigned* tickets;  // of k_bbox, k_occupancy, k_scan_sums
    unsigned* occ;
    int* start;         // nbuckets_max + 1
    size_t zeroed_bytes;
    int* sums;
    int* pbucket;
    int* prank;
    uint64_t* pcell;    // packed cell coordinates, point order
    float4* sorted;     // points in bucket order (coordinates, index)
    uint64_t* scell;    // their cells
    uint64_t* zkey[2];  // radix-sort buffers of the exported order (clouds above kZSmall)
    int* zval[2];
    int* zcount;        // [radix tiles][256]
    int* zsuper;        // [8 passes][groups][256]
    int zgroup, zgroups;  // tiles a group, groups
    size_t bytes;
    int nbuckets_max;
};

int bucket_budget(int64_t n) {
    int64_t b = 1024;
    while (b < 2 * n && b < (1ll << 26)) b <<= 1;
    return (int)b;
}

KnnLayout knn_layout(void* ws, int64_t n) {
    KnnLayout L;
    Carver cv(ws);
    L.nbuckets_max = bucket_budget(n);
    int ntiles = (L.nbuckets_max + kScanTile - 1) / kScanTile;
    L.params = cv.take<KnnParams>(1);
    L.bbox = cv.take<double>(kBboxBlocks * 6);
    const size_t z0 = cv.used;
    L.tickets = cv.take<unsigned>(4);
    L.zeroed = reinterpret_cast<char*>(L.tickets);
    L.occ = cv.take<unsigned>(kOccWords);
    L.start = cv.take<int>(L.nbuckets_max + 1);
    L.zeroed_bytes = cv.used - z0;
    L.sums = cv.take<int>(ntiles);
    L.pbucket = cv.take<int>(n);
    L.prank = cv.take<int>(n);
    L.pcell = cv.take<uint64_t>(n);
    L.sorted = cv.take<float4>(n);
    L.scell = cv.take<uint64_t>(n);
    const bool radix = n > kZSmall;
    const int64_t rblocks = radix ? (n + kRadixTile - 1) / kRadixTile : 0;
    L.zgroup = 1;
    while ((int64_t)L.zgroup * L.zgroup < rblocks) L.zgroup *= 2;
    L.zgroups = (int)((rblocks + L.zgroup - 1) / L.zgroup);
    for (int b = 0; b < 2; b++) {
        L.zkey[b] = cv.take<uint64_t>(radix ? n : 0);
        L.zval[b] = cv.take<int>(radix ? n : 0);
    }
    L.zcount = cv.take<int>(256 * rblocks);
    L.zsuper = cv.take<int>((size_t)8 * 256 * L.zgroups);
    L.bytes = cv.used;
    return L;
}

}  // namespace
}  // namespace mvgd

using namespace mvgd;

MVGD_API size_t mvgd_knn_workspace_bytes(int64_t n, int32_t k) {
    (void)k;
    if (n <= 0) return 0;
    return knn_layout(nullptr, n).bytes;
}

MVGD_API mvgd_status mvgd_knn(const double* pts, int64_t n, int32_t k, int32_t* nbr, int32_t* order,
                              double cell_size, void* ws, size_t ws_bytes, mvgd_stream_t stream) {
    if (!pts || !nbr || !ws || n < 2 || n >= (1ll << 31) || k < 1 || k > kMaxK || k >= n)
        return MVGD_EINVAL;
    if (!aligned(pts) || !aligned(nbr) || !aligned(order) || !aligned(ws)) return MVGD_EINVAL;
    if (!(cell_size == cell_size)) return MVGD_EINVAL;
    KnnLayout L = knn_layout(ws, n);
    if (ws_bytes < L.bytes) return MVGD_EWORKSPACE;
    cudaStream_t s = (cudaStream_t)stream;
    int dev = 0, sms = 0;
    MVGD_CUDA_TRY(cudaGetDevice(&dev));
    MVGD_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int tb = 256;
    int gb = (int)((n + tb - 1) / tb);
    if (gb > sms * 8) gb = sms * 8;
    int nb_box = gb < kBboxBlocks ? gb : kBboxBlocks;

    MVGD_CUDA_TRY(cudaMemsetAsync(L.zeroed, 0, L.zeroed_bytes, s));
    k_bbox<<<nb_box, tb, 0, s>>>(pts, n, L.bbox, L.tickets, L.params);
    k_occupancy<<<cell_size <= 0 ? gb : 1, tb, 0, s>>>(pts, n, L.occ, k, cell_size, L.nbuckets_max, L.tickets + 1,
                                                       L.params);
    const bool radix = order && n > kZSmall;
    k_count<<<gb, tb, 0, s>>>(pts, n, L.params, L.start, L.pbucket, L.prank, L.pcell, radix ? L.zkey[0] : nullptr,
                              L.zval[0]);
    // scan over the whole budget; buckets past params->nbuckets stay empty
    const int len = L.nbuckets_max;
    const int ntiles = (len + kScanTile - 1) / kScanTile;
    k_scan_sums<<<ntiles, 256, 0, s>>>(L.start, len, L.sums, L.tickets + 2);
    k_scan_apply<<<ntiles, 256, 0, s>>>(L.start, len, L.sums, n);
    k_scatter<<<gb, tb, 0, s>>>(pts, n, L.params, L.start, L.pbucket, L.prank, L.pcell, L.sorted, L.scell);
    // queries a warp: one after the other only where the GPU is full without
    int64_t per_warp = n / ((int64_t)sms * 64);
    per_warp = per_warp < 1 ? 1 : (per_warp > kQueryPerWarp ? kQueryPerWarp : per_warp);
    const int64_t per_block = kQueryWarps * per_warp;
    k_query<<<(unsigned)((n + per_block - 1) / per_block), kQueryWarps * 32, 0, s>>>(
        pts, n, k, L.params, L.sorted, L.start, L.scell, nbr, (int)per_warp);
    if (order && n <= kZSmall) {
        const int smem = (int)n * (int)(sizeof(uint64_t) + sizeof(uint16_t));
        MVGD_CUDA_TRY(cudaFuncSetAttribute(k_zorder_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           kZSmall * (int)(sizeof(uint64_t) + sizeof(uint16_t))));
        k_zorder_small<<<1, kZThreads, smem, s>>>(pts, (int)n, L.params, order);
    } else if (order) {
        const int rblocks = (int)((n + kRadixTile - 1) / kRadixTile);
        MVGD_CUDA_TRY(cudaFuncSetAttribute(k_radix_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, kRadixSmem));
        MVGD_CUDA_TRY(cudaMemsetAsync(L.zsuper, 0, sizeof(int) * 8 * 256 * L.zgroups, s));
        for (int pass = 0; pass < 8; pass++) {
            const int a = pass & 1;
            const RadixPass R{L.zcount, L.zsuper + (int64_t)pass * 256 * L.zgroups, L.zgroup, L.zgroups};
            k_radix_count<<<rblocks, kRadixThreads, 0, s>>>(L.zkey[a], n, 8 * pass, R);
            k_radix_scatter<<<rblocks, kRadixThreads, kRadixSmem, s>>>(L.zkey[a], L.zval[a], n, 8 * pass, R,
                                                              pass < 7 ? L.zkey[a ^ 1] : nullptr,
                                                              pass < 7 ? L.zval[a ^ 1] : order);
        }
    }
    return launch_status();
}

// ---------------------------------------------------------------------------
// kNN for callers that cannot allocate device memory.
//
// Some callers of this library may not call cudaMalloc at all: code that is
// being recorded into a CUDA graph (an allocation would break the capture),
// latency-bound loops that must never wait on the allocator, and host
// applications or plug-in frameworks that own every device buffer and hand
// the library only its inputs and outputs.  For them the scratch that
// mvgd_knn takes from a caller workspace lives instead in one file-scope
// device array, reserved when the library's code is loaded on a GPU and held
// by every GPU that loads it until the process exits.  The array is sized for
// MVGD_KNN_NOALLOC_MAX_POINTS points; larger clouds are refused.
//
// In host code the array's name is only a host-side stand-in, never a device
// address, so its address is fetched with cudaGetSymbolAddress once per
// device, with that device current, on the first call made on that device;
// that first call should therefore come before any stream capture.  Every
// call on a device shares the one array: calls whose work overlaps on the GPU
// (different streams, no ordering between them) race on it and must be
// serialised by the caller.  The array keeps the last call's contents; the
// kNN zeroes what it needs zeroed (bucket counts, occupancy bits) itself.
// ---------------------------------------------------------------------------
namespace mvgd {
namespace {

constexpr size_t kNoAllocScratchBytes = size_t(8) << 20;  // >= knn workspace of 65,536 points
static __device__ __align__(256) unsigned char g_knn_scratch[kNoAllocScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mutex;
void* g_scratch_ptr[kMaxDevices] = {nullptr};

mvgd_status scratch_for_current_device(void** out) {
    int dev = 0;
    MVGD_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return MVGD_ECUDA;
    std::lock_guard<std::mutex> lock(g_scratch_mutex);
    if (!g_scratch_ptr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_knn_scratch) != cudaSuccess || p == nullptr) return MVGD_ECUDA;
        g_scratch_ptr[dev] = p;
    }
    *out = g_scratch_ptr[dev];
    return MVGD_OK;
}

}  // namespace
}  // namespace mvgd

MVGD_API mvgd_status mvgd_knn_noalloc(const double* pts, int64_t n, int32_t k, int32_t* nbr, int32_t* order,
                                      double cell_size, mvgd_stream_t stream) {
    if (n > MVGD_KNN_NOALLOC_MAX_POINTS || knn_layout(nullptr, n).bytes > kNoAllocScratchBytes) return MVGD_EINVAL;
    if (!pts || !nbr || n < 2 || k < 1 || k > kMaxK || k >= n) return MVGD_EINVAL;
    void* scratch = nullptr;
    mvgd_status st = scratch_for_current_device(&scratch);
    if (st != MVGD_OK) return st;
    return mvgd_knn(pts, n, k, nbr, order, cell_size, scratch, kNoAllocScratchBytes, stream);
}
