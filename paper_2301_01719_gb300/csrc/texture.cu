// texture.cu -- texture set-up kernels: encoding, read-back, lobe fill, layout
// conversion, and the footprint counter used to compute algorithmic bytes.
#include "launch.h"
#include "rt_device.cuh"
#include "rt_filter.cuh"
#include "rt_encode.cuh"
#include "rt_internal.h"

namespace rt {

constexpr int kThreads = 256;

static inline unsigned blocks_for(int64_t items) { return (unsigned)((items + kThreads - 1) / kThreads); }

// ---------------------------------------------------------------------------
// Copies between layouts: encoding a source, reading codes back, converting an
// FP32 buffer.  S is the source's texel type, D the destination's, and Op
// converts one texel.  Both kernels leave the padding of a QUADS destination
// unwritten.
// ---------------------------------------------------------------------------
struct CopyTexel {
    template <typename T>
    __device__ __forceinline__ T operator()(T v) const {
        return v;
    }
};
struct EncodeF16 {
    __device__ __forceinline__ uint2 operator()(float4 v) const { return pack_f16(v); }
};
struct EncodeBF16 {
    __device__ __forceinline__ uint2 operator()(float4 v) const { return pack_bf16(v); }
};

// A block moves tiles of 32 x 2 buckets at one in-bucket row t and up to 16
// in-bucket columns s through shared memory, reading in the order of the source
// and writing in the order of the destination: a tile is runs of 32 buckets
// (PLANES), of 16 quads (QUADS) or of 32 sc texels (ATLAS) on either side, so
// both sides move whole cache lines.  Bound: HBM.  One thread per texel in
// plane order instead stores every texel of an ATLAS destination n texels from
// the next thread's (8 of each 32-byte sector).  1024^2 x 16^2 codes from QUADS
// to ATLAS: FP16 4.76 -> 0.79 ms (5.4 TB/s read + written), E4M3 0.72 ms (the
// index arithmetic starts to show), FP32 1.21 ms (7.1 TB/s).
constexpr int kTileI = 32, kTileS = 16;
constexpr int kTileRow = 40;               // shared-memory pitch of the second bucket row
constexpr int kTilePitch = 2 * kTileRow - 7;  // and of the next s: 73, odd

struct RelayoutShape {
    int W, H, n, sc;             // sc: in-bucket columns per tile, the last chunk may hold fewer
    int ti, tj, chunks;          // tiles along i and j, chunks of s
    FastDiv div_sc;
    int step_b, step_s;          // kThreads = step_b sc + step_s
};

static RelayoutShape relayout_shape(int W, int H, int n) {
    RelayoutShape r;
    r.W = W;
    r.H = H;
    r.n = n;
    r.chunks = (n + kTileS - 1) / kTileS;
    r.sc = (n + r.chunks - 1) / r.chunks;
    r.ti = (W + kTileI - 1) / kTileI;
    r.tj = (H + 1) / 2;
    r.div_sc = make_fastdiv((uint32_t)r.sc);
    r.step_b = kThreads / r.sc;
    r.step_s = kThreads % r.sc;
    return r;
}

// Calls f(offset of the texel in the buffer, its place in the tile) for this
// thread's texels of the tile, in the buffer's order: texels threadIdx.x,
// threadIdx.x + kThreads, ... of 64 sc, stepped without divisions.
template <typename F>
__device__ __forceinline__ void for_tile_texels(int layout, const RelayoutShape& r, int i0, int j0, int t, int s0,
                                                F f) {
    constexpr int kSteps = 2 * kTileI * kTileS / kThreads;
    const int sc = min(r.sc, r.n - s0);
    if (layout == RT_LAYOUT_ATLAS) {
        const int64_t row = (int64_t)r.W * r.n;
        const int64_t base = ((int64_t)j0 * r.n + t) * row + (int64_t)i0 * r.n + s0;
        const int64_t next = row * r.n;  // from bucket row j0 to j0 + 1
        int b = (int)r.div_sc.div(threadIdx.x), s = (int)threadIdx.x - b * r.sc;
#pragma unroll
        for (int k = 0; k < kSteps; ++k) {
            const int ii = b & (kTileI - 1), jj = b / kTileI;
            if (jj < 2 && s < sc && i0 + ii < r.W && j0 + jj < r.H)
                f(base + (jj ? next : 0) + ii * r.n + s, s * kTilePitch + jj * kTileRow + ii);
            b += r.step_b;
            s += r.step_s;
            if (s >= r.sc) {
                s -= r.sc;
                ++b;
            }
        }
    } else {
        // kThreads is a multiple of 64: a thread keeps its bucket and takes every fourth s
        const bool quads = layout == RT_LAYOUT_QUADS;
        const int64_t plane = plane_buckets(layout, r.W, r.H);
        const int q = threadIdx.x & (2 * kTileI - 1), s1 = threadIdx.x / (2 * kTileI);
        const int jj = quads ? (q >> 1) & 1 : q / kTileI;
        const int ii = quads ? ((q >> 2) << 1) + (q & 1) : q & (kTileI - 1);
        if (i0 + ii >= r.W || j0 + jj >= r.H) return;
        int64_t o = ((int64_t)t * r.n + s0 + s1) * plane + slot_in(layout, r.W, i0 + ii, j0 + jj);
        int p = s1 * kTilePitch + jj * kTileRow + ii;
#pragma unroll
        for (int k = 0; k < kSteps; ++k) {
            if (s1 + k * (kThreads / (2 * kTileI)) < sc) f(o, p);
            o += (kThreads / (2 * kTileI)) * plane;
            p += (kThreads / (2 * kTileI)) * kTilePitch;
        }
    }
}

template <typename S, typename D, typename Op>
__global__ void __launch_bounds__(kThreads, 6) relayout_tiles(const S* __restrict__ src, int src_layout,
                                                           D* __restrict__ dst, int dst_layout, RelayoutShape r) {
    __shared__ D tile[kTileS * kTilePitch];
    const Op op;
    const int tj = (int)(blockIdx.x / (unsigned)r.ti), t = (int)(blockIdx.y / (unsigned)r.chunks);
    const int i0 = (int)(blockIdx.x - (unsigned)tj * r.ti) * kTileI, j0 = 2 * tj;
    const int s0 = (int)(blockIdx.y - (unsigned)t * r.chunks) * r.sc;
    for_tile_texels(src_layout, r, i0, j0, t, s0, [&](int64_t o, int p) { tile[p] = op(src[o]); });
    __syncthreads();
    for_tile_texels(dst_layout, r, i0, j0, t, s0, [&](int64_t o, int p) { dst[o] = tile[p]; });
}

// One thread per texel in plane order, for copies that leave most of a tile empty.
template <typename S, typename D, typename Op>
__global__ void relayout_texels(const S* __restrict__ src, int src_layout, D* __restrict__ dst, int dst_layout, int W,
                                int H, int n, int64_t total) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    int i, j, s, t;
    planes_coords(idx, W, H, n, i, j, s, t);
    dst[index_in(dst_layout, W, H, n, i, j, s, t)] = Op()(src[index_in(src_layout, W, H, n, i, j, s, t)]);
}

// Tiles, or a thread per texel.  A block's costs are those of a whole tile (64
// buckets x 16 columns), so it must hold enough of them: bucket rows of 24 and
// more, and 8 columns where the tile has two bucket rows, 16 where the matrix has
// one (a palette).  Tiles / texels in us, all pairs of layouts, on 2^20 to 2^23
// texels of FP32, 2-byte and E4M3 channels:
//   width (FP32, 2^17 buckets x 16^2), QUADS to ATLAS and PLANES to QUADS: 8 wide
//     545 / 492 and 473 / 195, 16 wide 311 / 476 and 258 / 195, 24 wide 164 / 472 and 159 / 195;
//   columns n: n = 1, 2, 4 are 4-6, 2-3 and 1.2-1.7 times as slow in tiles (1000 x 2097 x 2^2 FP32
//     PLANES to QUADS 149 / 72), n = 8 0.5-1.2 times, n = 16 0.4-1.0 (copies within one layout
//     0.5-0.9);
//   one bucket row: n = 8 1.0-1.4 times as slow, n = 12 0.7-1.1, n = 16 0.7-1.0, n = 17 (chunks of
//     9) 1.0-1.4.
// FP32 texels into an ATLAS, which a thread per texel stores one by one past L2,
// are faster in tiles from 5 columns on where the copy outgrows L2: 256 x 1310 x
// 5^2 from QUADS 68 / 100, 64 x 1820 x 6^2 33 / 33, 256 x 910 x 6^2 60 / 87.
constexpr int kTileMinWidth = 24, kTileMinColumns = 8;

static bool tiles_pay(const RelayoutShape& r, bool fp32_to_atlas) {
    // a texture's n is at most 64, but an FP32 buffer to convert may have more in-bucket rows and
    // chunks of columns than a grid has in y (n = 1024 and on)
    if (r.W < kTileMinWidth || (int64_t)r.n * r.chunks > 65535) return false;
    if (r.H == 1) return r.sc == kTileS;
    if (r.sc >= kTileMinColumns) return true;
    const int64_t texels = (int64_t)r.W * r.H * r.n * r.n;
    return fp32_to_atlas && r.sc >= 5 && texels >= (r.sc == 5 ? (int64_t)1 << 23 : (int64_t)1 << 22);
}

template <typename S, typename D, typename Op = CopyTexel>
static cudaError_t launch_relayout(const void* src, int src_layout, void* dst, int dst_layout, int W, int H, int n,
                                   cudaStream_t stream) {
    const S* s = static_cast<const S*>(src);
    D* d = static_cast<D*>(dst);
    const RelayoutShape r = relayout_shape(W, H, n);
    if (tiles_pay(r, sizeof(D) == 16 && dst_layout == RT_LAYOUT_ATLAS)) {
        // w h <= 2^30 (or a K x 1 palette, K <= 2^30) for a texture: at most 2^25 blocks in x
        const dim3 grid((unsigned)r.ti * (unsigned)r.tj, (unsigned)(n * r.chunks));
        relayout_tiles<S, D, Op><<<grid, kThreads, 0, stream>>>(s, src_layout, d, dst_layout, r);
    } else {
        const int64_t total = (int64_t)W * H * n * n;
        relayout_texels<S, D, Op><<<blocks_for(total), kThreads, 0, stream>>>(s, src_layout, d, dst_layout, W, H, n,
                                                                              total);
    }
    return cudaGetLastError();
}

// FP32 source -> E4M3 + per-bucket scale (stored at the bucket's slot of
// dst_layout), one thread per bucket (amax pass, then encode pass).
__global__ void encode_e4m3_buckets(const float4* __restrict__ src, int src_layout, unsigned* __restrict__ dst,
                                    float* __restrict__ scale, int dst_layout, int W, int H, int n) {
    int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= (int64_t)W * H) return;
    int j = (int)(b / W), i = (int)(b - (int64_t)j * W);
    float amax = 0.0f;
    for (int t = 0; t < n; ++t)
        for (int s = 0; s < n; ++s) amax = fmaxf(amax, amax4(src[index_in(src_layout, W, H, n, i, j, s, t)]));
    float sc = bucket_scale(amax);
    scale[slot_in(dst_layout, W, i, j)] = sc;
    for (int t = 0; t < n; ++t)
        for (int s = 0; s < n; ++s)
            dst[index_in(dst_layout, W, H, n, i, j, s, t)] = pack_e4m3(src[index_in(src_layout, W, H, n, i, j, s, t)], sc);
}

// FP32 source -> 1-bit storage: bit = (channel 0 >= 1/2); one thread per 32-bit word.
__global__ void encode_bits(const float4* __restrict__ src, int src_layout, unsigned* __restrict__ dst, int W, int H,
                            int n, int64_t total) {
    const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (w * 32 >= total) return;
    unsigned word = 0;
    for (int k = 0; k < 32; ++k) {
        const int64_t idx = w * 32 + k;
        if (idx >= total) break;
        int i, j, s, t;
        planes_coords(idx, W, H, n, i, j, s, t);
        if (src[index_in(src_layout, W, H, n, i, j, s, t)].x >= 0.5f) word |= 1u << k;
    }
    dst[w] = word;
}

cudaError_t launch_encode(const float* src, int src_layout, void* dst, float* scale, int W, int H, int n, int fmt,
                          int dst_layout, cudaStream_t stream) {
    if (fmt == RT_BIT1) {
        const int64_t total = (int64_t)W * H * n * n;
        encode_bits<<<blocks_for((total + 31) / 32), kThreads, 0, stream>>>(
            reinterpret_cast<const float4*>(src), src_layout, reinterpret_cast<unsigned*>(dst), W, H, n, total);
    } else if (fmt == RT_E4M3_BUCKET_SCALE) {
        int64_t buckets = (int64_t)W * H;
        encode_e4m3_buckets<<<blocks_for(buckets), kThreads, 0, stream>>>(
            reinterpret_cast<const float4*>(src), src_layout, reinterpret_cast<unsigned*>(dst), scale, dst_layout, W,
            H, n);
    } else if (fmt == RT_F32) {
        return launch_relayout<float4, float4>(src, src_layout, dst, dst_layout, W, H, n, stream);
    } else if (fmt == RT_F16) {
        return launch_relayout<float4, uint2, EncodeF16>(src, src_layout, dst, dst_layout, W, H, n, stream);
    } else {
        return launch_relayout<float4, uint2, EncodeBF16>(src, src_layout, dst, dst_layout, W, H, n, stream);
    }
    return cudaGetLastError();
}

// Per-bucket scales stored at their slots of src_layout -> row-major h x w.
__global__ void read_scales(const float* __restrict__ src, int src_layout, float* __restrict__ dst, int W, int H) {
    int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= (int64_t)W * H) return;
    const int j = (int)(b / W), i = (int)(b - (int64_t)j * W);
    dst[b] = src[slot_in(src_layout, W, i, j)];
}

// 1-bit storage -> one byte (0 or 1) per texel in dst_layout.
__global__ void read_bits(const unsigned* __restrict__ src, uint8_t* __restrict__ dst, int W, int H, int n,
                          int dst_layout, int64_t total) {
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    int i, j, s, t;
    planes_coords(idx, W, H, n, i, j, s, t);
    int64_t o = index_in(dst_layout, W, H, n, i, j, s, t);
    dst[o] = (uint8_t)((src[idx >> 5] >> (unsigned)(idx & 31)) & 1u);
}

// Stored codes (src_layout: PLANES or QUADS) -> codes in dst_layout.
cudaError_t launch_read(const void* src, int src_layout, const float* scale, int fmt, int W, int H, int n,
                        int dst_layout, void* dst, float* scale_dst, cudaStream_t stream) {
    cudaError_t e;
    if (fmt == RT_BIT1) {  // bit textures are always PLANES
        const int64_t total = (int64_t)W * H * n * n;
        read_bits<<<blocks_for(total), kThreads, 0, stream>>>(reinterpret_cast<const unsigned*>(src),
                                                              reinterpret_cast<uint8_t*>(dst), W, H, n, dst_layout,
                                                              total);
        e = cudaGetLastError();
    } else if (fmt == RT_F32) {
        e = launch_relayout<float4, float4>(src, src_layout, dst, dst_layout, W, H, n, stream);
    } else if (fmt == RT_E4M3_BUCKET_SCALE) {
        e = launch_relayout<unsigned, unsigned>(src, src_layout, dst, dst_layout, W, H, n, stream);
    } else {
        e = launch_relayout<uint2, uint2>(src, src_layout, dst, dst_layout, W, H, n, stream);
    }
    if (e != cudaSuccess) return e;
    if (scale && scale_dst)
        read_scales<<<blocks_for((int64_t)W * H), kThreads, 0, stream>>>(scale, src_layout, scale_dst, W, H);
    return cudaGetLastError();
}

__device__ __forceinline__ float4 lobe_value(const float* P, float3 I) {
    float c = I.x * P[3] + I.y * P[4] + I.z * P[5];
    float l = c > 0.f ? powf(c, P[6]) : 0.f;
    return make_float4(P[0] * l, P[1] * l, P[2] * l, l);
}

__global__ void fill_lobes_kernel(const float* __restrict__ params, void* __restrict__ dst, float* __restrict__ scale,
                                  int layout, int W, int H, int n, int fmt) {
    int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= (int64_t)W * H) return;
    int j = (int)(b / W), i = (int)(b - (int64_t)j * W);
    float P[8];
    const float4* p4 = reinterpret_cast<const float4*>(params) + 2 * b;
    float4 a = p4[0], c = p4[1];
    P[0] = a.x; P[1] = a.y; P[2] = a.z; P[3] = a.w;
    P[4] = c.x; P[5] = c.y; P[6] = c.z; P[7] = c.w;
    float sc = 1.0f;
    if (fmt == RT_E4M3_BUCKET_SCALE) {
        float amax = 0.f;
        for (int t = 0; t < n; ++t)
            for (int s = 0; s < n; ++s) amax = fmaxf(amax, amax4(lobe_value(P, texel_centre_direction(s, t, n))));
        sc = bucket_scale(amax);
        scale[slot_in(layout, W, i, j)] = sc;
    }
    for (int t = 0; t < n; ++t)
        for (int s = 0; s < n; ++s) {
            float4 v = lobe_value(P, texel_centre_direction(s, t, n));
            int64_t idx = index_in(layout, W, H, n, i, j, s, t);
            if (fmt == RT_F32)
                reinterpret_cast<float4*>(dst)[idx] = v;
            else if (fmt == RT_F16)
                reinterpret_cast<uint2*>(dst)[idx] = pack_f16(v);
            else if (fmt == RT_BF16)
                reinterpret_cast<uint2*>(dst)[idx] = pack_bf16(v);
            else
                reinterpret_cast<unsigned*>(dst)[idx] = pack_e4m3(v, sc);
        }
}

cudaError_t launch_fill_lobes(const float* params, void* dst, float* scale, int layout, int W, int H, int n, int fmt,
                              cudaStream_t stream) {
    int64_t buckets = (int64_t)W * H;
    fill_lobes_kernel<<<blocks_for(buckets), kThreads, 0, stream>>>(params, dst, scale, layout, W, H, n, fmt);
    return cudaGetLastError();
}

__global__ void check_index_kernel(const uint32_t* __restrict__ index, int64_t count, uint32_t K, unsigned* bad) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < count && index[k] >= K) atomicOr(bad, 1u);
}

cudaError_t launch_check_index(const uint32_t* index, int64_t count, uint32_t K, unsigned* bad, cudaStream_t stream) {
    if (count == 0) return cudaSuccess;
    check_index_kernel<<<blocks_for(count), kThreads, 0, stream>>>(index, count, K, bad);
    return cudaGetLastError();
}

cudaError_t launch_convert(const float* src, int src_layout, float* dst, int dst_layout, int W, int H, int n,
                           cudaStream_t stream) {
    return launch_relayout<float4, float4>(src, src_layout, dst, dst_layout, W, H, n, stream);
}

// Footprint: one bit per texel of every object (PLANES numbering), set for
// every tap the forward kernel reads.
template <int FILTER>
__global__ void __launch_bounds__(kThreads) footprint_kernel(const TexDesc* __restrict__ table, int n_obj,
                                                            const float* __restrict__ uv,
                                                            const float* __restrict__ dir,
                                                            const int32_t* __restrict__ obj, int64_t F,
                                                            uint32_t* __restrict__ bitmap,
                                                            const int64_t* __restrict__ word_offset,
                                                            unsigned* status) {
    __shared__ WarpStage<false> stages[kThreads / 32];
    const Tiling flat = flat_tiling();
    for_each_fragment<kThreads / 32, false, false, 2>(uv, dir, obj, nullptr, F, flat, stages,
                                                   [&](int64_t, const Frag& q, float4) {
        TexDesc d;
        if (!fragment_valid(table, n_obj, q.o, q.u, q.v, q.x, q.y, q.z, status, d)) return;
        Lookup<FILTER> L = locate<FILTER>(d, q.u, q.v, q.x, q.y, q.z);
        const int64_t base = word_offset[q.o] * 32;
        const int nu = FILTER == RT_QUADRILINEAR ? 2 : 1;
        const int ns = FILTER == RT_NEAREST ? 1 : 2;
        for (int b = 0; b < nu; ++b)
            for (int a = 0; a < nu; ++a)
                for (int t = 0; t < ns; ++t)
                    for (int p = 0; p < ns; ++p) {
                        const int i = a ? L.u.k1 : L.u.k0, j = b ? L.v.k1 : L.v.k0;
                        const int s = p ? L.s.k1 : L.s.k0, tt = t ? L.t.k1 : L.t.k0;
                        int64_t bit = base + (d.layout == kLayoutPalette
                                                  ? texel_index<kLayoutPalette>(d, i, j, s, tt)
                                                  : texel_index<RT_LAYOUT_PLANES>(d, i, j, s, tt));
                        atomicOr(bitmap + (bit >> 5), 1u << (bit & 31));
                    }
    });
}

template <int FILTER>
static cudaError_t launch_footprint_t(const TexDesc* table, int n_obj, const float* uv, const float* dir,
                                      const int32_t* obj, int64_t F, uint32_t* bitmap, const int64_t* word_offset,
                                      unsigned* status, cudaStream_t stream) {
    const unsigned grid = persistent_grid<footprint_kernel<FILTER>>(kThreads, (F + kChunk - 1) / kChunk);
    footprint_kernel<FILTER><<<grid, kThreads, 0, stream>>>(table, n_obj, uv, dir, obj, F, bitmap, word_offset,
                                                            status);
    return cudaGetLastError();
}

cudaError_t launch_footprint_mark(const TexDesc* table, int n_obj, const float* uv, const float* dir,
                                  const int32_t* obj, int64_t F, int filter, uint32_t* bitmap,
                                  const int64_t* word_offset, unsigned* status, cudaStream_t stream) {
    if (filter == RT_NEAREST)
        return launch_footprint_t<RT_NEAREST>(table, n_obj, uv, dir, obj, F, bitmap, word_offset, status, stream);
    if (filter == RT_ANGULAR_BILINEAR)
        return launch_footprint_t<RT_ANGULAR_BILINEAR>(table, n_obj, uv, dir, obj, F, bitmap, word_offset, status,
                                                       stream);
    return launch_footprint_t<RT_QUADRILINEAR>(table, n_obj, uv, dir, obj, F, bitmap, word_offset, status, stream);
}

__global__ void popcount_kernel(const uint32_t* __restrict__ bitmap, int64_t words, unsigned long long* count) {
    unsigned long long local = 0;
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < words; w += (int64_t)gridDim.x * blockDim.x)
        local += __popc(bitmap[w]);
    for (int o = 16; o > 0; o >>= 1) local += __shfl_down_sync(0xFFFFFFFFu, local, o);
    if ((threadIdx.x & 31) == 0 && local) atomicAdd(count, local);
}

cudaError_t launch_popcount(const uint32_t* bitmap, int64_t words, unsigned long long* count, cudaStream_t stream) {
    if (words <= 0) return cudaSuccess;
    int64_t b = (words + kThreads - 1) / kThreads;
    unsigned grid = (unsigned)(b < 4096 ? b : 4096);
    popcount_kernel<<<grid, kThreads, 0, stream>>>(bitmap, words, count);
    return cudaGetLastError();
}

}  // namespace rt
