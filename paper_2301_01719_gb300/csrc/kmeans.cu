// kmeans.cu -- the encoder of palette textures: Lloyd's k-means over the
// buckets of a dense texture, each bucket a vector of n^2 x 4 values.
//
// Centroids are stored like a K x 1 texture in PLANES order: centroid k,
// texel (s, t) at float4 index (t n + s) K + k.
//
// Assignment is a distance matrix contraction (w h buckets x K centroids over
// n^2 x 4 values) with an argmin epilogue, in FP32 on the CUDA cores: a block
// holds 128 buckets and sweeps the centroids 64 at a time, 4 texels of each per
// shared-memory stage; each thread accumulates 8 x 4 dot products and keeps
// the running (distance, index) minimum of its 8 rows, ties to the lower
// index.  |x - c|^2 is ranked as |c|^2 - 2 x.c (|x|^2 is added for the
// reported distance only).
//
// Update: per-centroid counts, their prefix sums and a scatter of the buckets
// group every cluster's members; blocks then sum the members' texels (FP64, or
// exact integers) and write the mean rounded to FP32.  Empty clusters keep
// their centroid.
#include "rt_device.cuh"
#include "rt_encode.cuh"
#include "rt_internal.h"

namespace rt {

constexpr int kAM = 128;  // buckets per block
constexpr int kAN = 64;   // centroids per sweep step
constexpr int kAP = 4;    // texels per shared-memory stage
constexpr int kAThreads = 256;

// Texel p = t n + s of bucket (i, j) of a dense texture (ATLAS, PLANES or QUADS).
template <int FMT, int LAYOUT>
__device__ __forceinline__ float4 bucket_texel(const TexDesc& d, int i, int j, int p, float sc) {
    if (LAYOUT == RT_LAYOUT_ATLAS)
        return load_texel<FMT>(d.base, texel_index<RT_LAYOUT_ATLAS>(d, i, j, p % d.n, p / d.n), sc);
    return load_texel<FMT>(d.base, checked_texel(d, (int64_t)p * d.plane + bucket_slot<LAYOUT>(d, i, j)), sc);
}

// The E4M3 scale of bucket (i, j) (1 for the other formats).
template <int FMT, int LAYOUT>
__device__ __forceinline__ float bucket_scale_of(const TexDesc& d, int i, int j) {
    return FMT == RT_E4M3_BUCKET_SCALE ? __ldg(d.scale + bucket_slot<LAYOUT>(d, i, j)) : 1.0f;
}

__device__ __forceinline__ float dot4f(float4 a, float4 b) {
    return fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, a.w * b.w)));
}

template <int FMT, int LAYOUT>
__global__ void __launch_bounds__(kAThreads, 2) kmeans_assign_kernel(TexDesc d, int K, const float4* __restrict__ C,
                                                                  uint32_t* __restrict__ index,
                                                                  float* __restrict__ dist) {
    __shared__ float4 Xs[kAP][kAM];
    __shared__ float4 Cs[kAP][kAN];
    __shared__ float cnp[kAP][kAN];
    __shared__ float cn[kAN];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int64_t B = (int64_t)d.W * d.H;
    const int64_t b0 = (int64_t)blockIdx.x * kAM;
    const int planes = d.n * d.n;
    // loader role for X: bucket b0 + lb, stages q = tid / 128 and q + 2
    const int lb = tid & (kAM - 1);
    const int64_t bb = b0 + lb;
    const bool bvalid = bb < B;
    int bi = 0, bj = 0;
    float sc = 1.0f;
    if (bvalid) {
        bj = (int)(bb / d.W);
        bi = (int)(bb - (int64_t)bj * d.W);
        sc = bucket_scale_of<FMT, LAYOUT>(d, bi, bj);
    }
    // loader role for C: stage cq, centroid ck of the sweep step
    const int cq = tid >> 6, ck = tid & (kAN - 1);

    float best[8], xn[8];
    int bestk[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        best[r] = INFINITY;
        bestk[r] = 0;
        xn[r] = 0.0f;
    }
    for (int k0 = 0; k0 < K; k0 += kAN) {
        float acc[8][4];
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[r][c] = 0.0f;
        float cnorm = 0.0f;  // |c|^2 partial of centroid k0 + ck over stages cq
        for (int p0 = 0; p0 < planes; p0 += kAP) {
            __syncthreads();
            for (int q = tid >> 7; q < kAP; q += 2) {
                const int p = p0 + q;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (bvalid && p < planes) v = bucket_texel<FMT, LAYOUT>(d, bi, bj, p, sc);
                Xs[q][lb] = v;
            }
            {
                const int p = p0 + cq, k = k0 + ck;
                float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
                if (p < planes && k < K) c = __ldg(C + (int64_t)p * K + k);
                Cs[cq][ck] = c;
                cnorm += dot4f(c, c);
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < kAP; ++q) {
                float4 c[4];
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) c[cc] = Cs[q][tx + 16 * cc];
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const float4 x = Xs[q][ty * 8 + r];
#pragma unroll
                    for (int cc = 0; cc < 4; ++cc) acc[r][cc] += dot4f(x, c[cc]);
                    if (k0 == 0 && tx == 0) xn[r] += dot4f(x, x);
                }
            }
        }
        __syncthreads();
        cnp[cq][ck] = cnorm;
        __syncthreads();
        if (tid < kAN) cn[tid] = (cnp[0][tid] + cnp[1][tid]) + (cnp[2][tid] + cnp[3][tid]);
        __syncthreads();
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
            const int k = k0 + tx + 16 * cc;
            if (k >= K) continue;
            const float c2 = cn[tx + 16 * cc];
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const float dd = fmaf(-2.0f, acc[r][cc], c2);
                if (dd < best[r]) {  // k grows within a thread: equal distances keep the lower index
                    best[r] = dd;
                    bestk[r] = k;
                }
            }
        }
    }
    // reduce over the 16 threads (tx) of each row group; they share a half-warp
#pragma unroll
    for (int r = 0; r < 8; ++r) {
#pragma unroll
        for (int off = 8; off >= 1; off >>= 1) {
            const float ob = __shfl_xor_sync(0xffffffffu, best[r], off);
            const int ok = __shfl_xor_sync(0xffffffffu, bestk[r], off);
            if (ob < best[r] || (ob == best[r] && ok < bestk[r])) {
                best[r] = ob;
                bestk[r] = ok;
            }
        }
    }
    if (tx == 0) {
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int64_t b = b0 + ty * 8 + r;
            if (b >= B) continue;
            index[b] = (uint32_t)bestk[r];
            if (dist) dist[b] = fmaxf(best[r] + xn[r], 0.0f);
        }
    }
}

template <int FMT, int LAYOUT>
__global__ void kmeans_init_kernel(TexDesc d, int K, const int32_t* __restrict__ buckets, float4* __restrict__ C,
                                   unsigned* status) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int planes = d.n * d.n;
    if (e >= (int64_t)K * planes) return;
    const int p = (int)(e / K), k = (int)(e - (int64_t)p * K);
    const int64_t B = (int64_t)d.W * d.H;
    int64_t b = buckets[k];
    if (b < 0 || b >= B) {
        atomicOr(status, ST_BAD_ARG);
        b = b < 0 ? 0 : B - 1;
    }
    const int j = (int)(b / d.W), i = (int)(b - (int64_t)j * d.W);
    C[(int64_t)p * K + k] = bucket_texel<FMT, LAYOUT>(d, i, j, p, bucket_scale_of<FMT, LAYOUT>(d, i, j));
}

// Counting the members and grouping them.  Clusters are uneven, and atomics on
// one large cluster's counter serialise: a block counts its buckets in shared
// memory first and touches each counter once (K <= kLocalK; beyond it the
// counters outgrow shared memory and are many enough).  512^2 buckets, K = 1024:
// 24 us for each of the two kernels with global atomics alone, 5 and 8 us so.
constexpr int kLocalK = 4096, kGroupThreads = 512, kGroupItems = 4;

template <bool LOCAL>
__global__ void __launch_bounds__(kGroupThreads) kmeans_count_kernel(const uint32_t* __restrict__ index, int64_t B,
                                                                     int K, uint32_t* counts, unsigned* status) {
    extern __shared__ uint32_t local[];
    if (LOCAL) {
        for (int k = threadIdx.x; k < K; k += kGroupThreads) local[k] = 0;
        __syncthreads();
    }
    const int64_t b0 = (int64_t)blockIdx.x * (kGroupThreads * kGroupItems) + threadIdx.x;
#pragma unroll
    for (int u = 0; u < kGroupItems; ++u) {
        const int64_t b = b0 + u * kGroupThreads;
        if (b >= B) break;
        const uint32_t k = index[b];
        if (k >= (uint32_t)K)
            atomicOr(status, ST_BAD_ARG);
        else
            atomicAdd((LOCAL ? local : counts) + k, 1u);
    }
    if (LOCAL) {
        __syncthreads();
        for (int k = threadIdx.x; k < K; k += kGroupThreads)
            if (local[k]) atomicAdd(counts + k, local[k]);
    }
}

// Exclusive prefix sum of counts[0..K) into offsets[0..K] (one block).
__global__ void __launch_bounds__(1024) kmeans_scan_kernel(const uint32_t* __restrict__ counts, int K,
                                                           uint32_t* __restrict__ offsets) {
    __shared__ uint32_t part[1024];
    const int t = threadIdx.x;
    const int per = (K + 1023) / 1024;
    const int lo = t * per, hi = min(K, lo + per);
    uint32_t s = 0;
    for (int k = lo; k < hi; ++k) s += counts[k];
    part[t] = s;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {  // inclusive scan of the partial sums
        const uint32_t v = t >= off ? part[t - off] : 0u;
        __syncthreads();
        part[t] += v;
        __syncthreads();
    }
    uint32_t run = t ? part[t - 1] : 0u;
    for (int k = lo; k < hi; ++k) {
        offsets[k] = run;
        run += counts[k];
    }
    if (t == 1023) offsets[K] = part[1023];
}

// Groups the buckets by centroid: members holds each bucket's number (ATLAS) or
// its slot in a direction plane (PLANES, QUADS), found here once per bucket.
template <bool LOCAL>
__global__ void __launch_bounds__(kGroupThreads) kmeans_scatter_kernel(const uint32_t* __restrict__ index, int64_t B,
                                                                       int K, int W, int layout,
                                                                       const uint32_t* __restrict__ offsets,
                                                                       uint32_t* cursor,
                                                                       uint32_t* __restrict__ members) {
    extern __shared__ uint32_t local[];
    if (LOCAL) {
        for (int k = threadIdx.x; k < K; k += kGroupThreads) local[k] = 0;
        __syncthreads();
    }
    const int64_t b0 = (int64_t)blockIdx.x * (kGroupThreads * kGroupItems) + threadIdx.x;
    uint32_t cluster[kGroupItems], rank[kGroupItems];
#pragma unroll
    for (int u = 0; u < kGroupItems; ++u) {
        const int64_t b = b0 + u * kGroupThreads;
        cluster[u] = b < B ? index[b] : (uint32_t)K;
        if (cluster[u] < (uint32_t)K) rank[u] = atomicAdd((LOCAL ? local : cursor) + cluster[u], 1u);
    }
    if (LOCAL) {  // the block's places in each of its clusters
        __syncthreads();
        for (int k = threadIdx.x; k < K; k += kGroupThreads)
            if (local[k]) local[k] = atomicAdd(cursor + k, local[k]);
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < kGroupItems; ++u) {
        if (cluster[u] >= (uint32_t)K) continue;
        const int64_t b = b0 + u * kGroupThreads;
        const int j = (int)(b / W), i = (int)(b - (int64_t)j * W);
        const uint32_t at = layout == RT_LAYOUT_ATLAS ? (uint32_t)b : (uint32_t)slot_in(layout, W, i, j);
        members[offsets[cluster[u]] + (LOCAL ? local[cluster[u]] : 0u) + rank[u]] = at;
    }
}

// Centroid means.  A block is 16 rows of 16 threads over 16 planes: a row takes
// one member at a time, eight loads in flight, and R rows share a centroid and
// add their sums in shared memory (R = 1, 4 or 16 for small to large clusters).
// All centroids of one group of planes run together (blockIdx.x), so their
// scattered 8-byte reads find the planes in L2.
//
// The sums are FP64, but FP64 runs at a few additions and conversions per cycle
// and SM: FP16 texels, multiples of 2^-24, are summed in 64-bit integers
// instead, exactly, whenever all of the block's lie below 64 in magnitude
// (infinities and NaN do not; w h <= 2^30 members leave room), and the other
// formats' values are widened by moving their bits.  One thread per plane and
// centroid, walking the members one by one, took 1.65 ms on 512^2 x 16^2 FP16
// lobes with K = 1024 (and 66 ms where one cluster held 30 % of the buckets, now
// 1.6 ms); this takes 0.27 ms, bound by L1, which looks up each of a warp's 32
// lines by itself.
constexpr int kMeanPlanes = 16, kMeanRows = 16, kMeanThreads = kMeanPlanes * kMeanRows, kMeanUnroll = 8;
// The rows that share a centroid, by the average cluster.  512^2 x 16^2 FP16 and
// (128^2 x 5^2 FP16), random clusters, whole update in us for R = 1, 4, 16:
// average 8: 605, 993, 2709 (28, 30, 40); 32: 345, 440, 805 (31, 25, 27);
// 256: 556, 299, 344 (77, 37, 26); 1024: 759, 440, 297 (227, 72, 39).  Where one
// cluster holds 30 % of the buckets, R = 16 is four times faster than R = 4, so
// the lines lie a little early.
constexpr int64_t kMeanShare16 = 128, kMeanShare4 = 16;

template <int FMT, int LAYOUT>
__device__ __forceinline__ float4 member_texel(const TexDesc& d, uint32_t at, int p) {
    if (LAYOUT == RT_LAYOUT_ATLAS) {
        const int j = (int)(at / (uint32_t)d.W), i = (int)(at - (uint32_t)j * d.W);
        return load_texel<FMT>(d.base, texel_index<RT_LAYOUT_ATLAS>(d, i, j, p % d.n, p / d.n), 1.0f);
    }
#ifdef RADTEX_CHECKED
    at = (uint32_t)checked_slot(d, at, d.plane);
#endif
    const float sc = FMT == RT_E4M3_BUCKET_SCALE ? __ldg(d.scale + at) : 1.0f;
    return load_texel<FMT>(d.base, checked_texel(d, (int64_t)p * d.plane + at), sc);
}

// Calls f(texel) for members m, m + R, ... < m1 on plane p.
template <int FMT, int LAYOUT, int R, typename F>
__device__ __forceinline__ void for_members(const TexDesc& d, const uint32_t* members, uint32_t m, uint32_t m1, int p,
                                            F f) {
    for (; m < m1; m += kMeanUnroll * R) {
        float4 v[kMeanUnroll];
#pragma unroll
        for (int u = 0; u < kMeanUnroll; ++u)
            if (m + u * R < m1) v[u] = member_texel<FMT, LAYOUT>(d, __ldg(members + m + u * R), p);
#pragma unroll
        for (int u = 0; u < kMeanUnroll; ++u)
            if (m + u * R < m1) f(v[u]);
    }
}

// A call, so that the compiler does not compute it beside the other form.
__device__ __noinline__ double widen_any(float v) { return (double)v; }

// (double)v by moving its bits, but for zeros (0), denormals, infinities and NaN.
__device__ __forceinline__ double widen(float v) {
    const uint32_t b = __float_as_uint(v), a = b & 0x7fffffffu;
    if (a - 0x00800000u < 0x7f000000u)
        return __hiloint2double((int)((b & 0x80000000u) | ((a >> 3) + 0x38000000u)), (int)(b << 29));
    return a == 0 ? 0.0 : widen_any(v);
}

// The sums over R rows: in acc[c] of row c < 4 of each R, for R > 1.
template <int R, typename T>
__device__ __forceinline__ void sum_rows(T (&acc)[4], T (*part)[4][kMeanPlanes + 1]) {
    if (R == 1) return;
    const int row = threadIdx.x / kMeanPlanes, pl = threadIdx.x & (kMeanPlanes - 1), c = row & (R - 1);
#pragma unroll
    for (int k = 0; k < 4; ++k) part[row][k][pl] = acc[k];
    __syncthreads();
    if (c < 4) {
        T s = part[row - c][c][pl];
        for (int r = 1; r < R; ++r) s += part[row - c + r][c][pl];
        acc[0] = s;
    }
}

template <int FMT, int LAYOUT, int R>
__global__ void __launch_bounds__(kMeanThreads, 4) kmeans_mean_kernel(TexDesc d, int K,
                                                                   const uint32_t* __restrict__ offsets,
                                                                   const uint32_t* __restrict__ members,
                                                                   float* __restrict__ C) {
    __shared__ union {
        long long i[kMeanRows][4][kMeanPlanes + 1];
        double f[kMeanRows][4][kMeanPlanes + 1];
    } part;
    const int row = threadIdx.x / kMeanPlanes, c = row & (R - 1);
    const int64_t k = (int64_t)blockIdx.x * (kMeanRows / R) + row / R;
    const int p = blockIdx.y * kMeanPlanes + (threadIdx.x & (kMeanPlanes - 1));
    uint32_t m0 = 0, m1 = 0;
    if (k < K) {
        m0 = offsets[k];
        m1 = offsets[k + 1];
    }
    const uint32_t count = m1 - m0;  // empty: keep the centroid
    if (p >= d.n * d.n) m1 = m0;
    double sum[4];
    bool done = false;
    if (FMT == RT_F16) {
        long long acc[4] = {0, 0, 0, 0};
        bool wide = false;  // a texel of 64 or more, infinite or NaN
        for_members<FMT, LAYOUT, R>(d, members, m0 + c, m1, p, [&](float4 v) {
            wide |= !(fabsf(v.x) < 64.0f && fabsf(v.y) < 64.0f && fabsf(v.z) < 64.0f && fabsf(v.w) < 64.0f);
            acc[0] += __float2int_rn(v.x * 16777216.0f);
            acc[1] += __float2int_rn(v.y * 16777216.0f);
            acc[2] += __float2int_rn(v.z * 16777216.0f);
            acc[3] += __float2int_rn(v.w * 16777216.0f);
        });
        if (!__syncthreads_or(wide)) {
            sum_rows<R>(acc, part.i);
            for (int q = 0; q < (R > 1 ? 1 : 4); ++q) sum[q] = (double)acc[q] * (1.0 / 16777216.0);
            done = true;
        }
    }
    if (!done) {
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
        for_members<FMT, LAYOUT, R>(d, members, m0 + c, m1, p, [&](float4 v) {
            acc[0] += widen(v.x);
            acc[1] += widen(v.y);
            acc[2] += widen(v.z);
            acc[3] += widen(v.w);
        });
        sum_rows<R>(acc, part.f);
        for (int q = 0; q < (R > 1 ? 1 : 4); ++q) sum[q] = acc[q];
    }
    if (count == 0 || m1 == m0) return;
    const double inv = 1.0 / (double)count;
    const int64_t e = (int64_t)p * K + k;
    if (R == 1)
        reinterpret_cast<float4*>(C)[e] = make_float4((float)(sum[0] * inv), (float)(sum[1] * inv),
                                                      (float)(sum[2] * inv), (float)(sum[3] * inv));
    else if (c < 4)
        C[4 * e + c] = (float)(sum[0] * inv);
}

static unsigned blocks(int64_t items, int threads) { return (unsigned)((items + threads - 1) / threads); }

template <template <int, int> class Launch, int LAYOUT, typename... Args>
static cudaError_t dispatch_format(const TexDesc& d, Args... args) {
    switch (d.fmt) {
        case RT_F16:
            return Launch<RT_F16, LAYOUT>::run(d, args...);
        case RT_BF16:
            return Launch<RT_BF16, LAYOUT>::run(d, args...);
        case RT_E4M3_BUCKET_SCALE:
            return Launch<RT_E4M3_BUCKET_SCALE, LAYOUT>::run(d, args...);
        default:
            return Launch<RT_F32, LAYOUT>::run(d, args...);
    }
}

// Calls Launch<FMT, LAYOUT>::run(args...) for the texture's format and layout (dense textures only).
template <template <int, int> class Launch, typename... Args>
static cudaError_t dispatch_dense(const TexDesc& d, Args... args) {
    if (d.layout == RT_LAYOUT_ATLAS) return Launch<RT_F32, RT_LAYOUT_ATLAS>::run(d, args...);
    if (d.layout == RT_LAYOUT_QUADS) return dispatch_format<Launch, RT_LAYOUT_QUADS>(d, args...);
    if (d.layout != RT_LAYOUT_PLANES) return cudaErrorInvalidValue;
    return dispatch_format<Launch, RT_LAYOUT_PLANES>(d, args...);
}

template <int FMT, int LAYOUT>
struct InitLaunch {
    static cudaError_t run(const TexDesc& d, int K, const int32_t* buckets, float* C, unsigned* status,
                           cudaStream_t stream) {
        const int64_t items = (int64_t)K * d.n * d.n;
        kmeans_init_kernel<FMT, LAYOUT><<<blocks(items, 256), 256, 0, stream>>>(d, K, buckets,
                                                                              reinterpret_cast<float4*>(C), status);
        return cudaGetLastError();
    }
};

template <int FMT, int LAYOUT>
struct AssignLaunch {
    static cudaError_t run(const TexDesc& d, int K, const float* C, uint32_t* index, float* dist,
                           cudaStream_t stream) {
        const int64_t B = (int64_t)d.W * d.H;
        kmeans_assign_kernel<FMT, LAYOUT><<<blocks(B, kAM), kAThreads, 0, stream>>>(
            d, K, reinterpret_cast<const float4*>(C), index, dist);
        return cudaGetLastError();
    }
};

template <int FMT, int LAYOUT>
struct MeanLaunch {
    static cudaError_t run(const TexDesc& d, int K, const uint32_t* offsets, const uint32_t* members, float* C,
                           cudaStream_t stream) {
        const int64_t average = (int64_t)d.W * d.H / K;
        if (average >= kMeanShare16) return launch<16>(d, K, offsets, members, C, stream);
        if (average >= kMeanShare4) return launch<4>(d, K, offsets, members, C, stream);
        return launch<1>(d, K, offsets, members, C, stream);
    }
    template <int R>
    static cudaError_t launch(const TexDesc& d, int K, const uint32_t* offsets, const uint32_t* members, float* C,
                              cudaStream_t stream) {
        constexpr int per = kMeanRows / R;
        const dim3 grid((unsigned)((K + per - 1) / per), (unsigned)((d.n * d.n + kMeanPlanes - 1) / kMeanPlanes));
        kmeans_mean_kernel<FMT, LAYOUT, R><<<grid, kMeanThreads, 0, stream>>>(d, K, offsets, members, C);
        return cudaGetLastError();
    }
};

cudaError_t launch_kmeans_init(const TexDesc& d, int K, const int32_t* buckets, float* C, unsigned* status,
                               cudaStream_t stream) {
    return dispatch_dense<InitLaunch>(d, K, buckets, C, status, stream);
}

cudaError_t launch_kmeans_assign(const TexDesc& d, int K, const float* C, uint32_t* index, float* dist,
                                 cudaStream_t stream) {
    return dispatch_dense<AssignLaunch>(d, K, C, index, dist, stream);
}

cudaError_t launch_kmeans_update(const TexDesc& d, int K, const uint32_t* index, float* C, uint32_t* scratch,
                                 unsigned* status, cudaStream_t stream) {
    const int64_t B = (int64_t)d.W * d.H;
    uint32_t* counts = scratch;
    uint32_t* cursor = scratch + K;
    uint32_t* offsets = scratch + 2 * (int64_t)K;  // K + 1 entries
    uint32_t* members = scratch + 3 * (int64_t)K + 1;
    cudaError_t e = cudaMemsetAsync(scratch, 0, sizeof(uint32_t) * 2 * (size_t)K, stream);
    if (e != cudaSuccess) return e;
    const unsigned grid = blocks(B, kGroupThreads * kGroupItems);
    const size_t local = sizeof(uint32_t) * (size_t)K;
    if (K <= kLocalK)
        kmeans_count_kernel<true><<<grid, kGroupThreads, local, stream>>>(index, B, K, counts, status);
    else
        kmeans_count_kernel<false><<<grid, kGroupThreads, 0, stream>>>(index, B, K, counts, status);
    kmeans_scan_kernel<<<1, 1024, 0, stream>>>(counts, K, offsets);
    if (K <= kLocalK)
        kmeans_scatter_kernel<true><<<grid, kGroupThreads, local, stream>>>(index, B, K, d.W, d.layout, offsets,
                                                                            cursor, members);
    else
        kmeans_scatter_kernel<false><<<grid, kGroupThreads, 0, stream>>>(index, B, K, d.W, d.layout, offsets, cursor,
                                                                         members);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return dispatch_dense<MeanLaunch>(d, K, (const uint32_t*)offsets, (const uint32_t*)members, C, stream);
}

}  // namespace rt
