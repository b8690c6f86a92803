// shade.cu -- forward synthesis and lookup-coordinate kernels.
//
// Persistent kernels: every warp walks 32-fragment chunks (a run of the flat
// stream, or a screen tile of a batch of frames) with the G-buffer of its next
// chunk prefetched into shared memory (rt_filter.cuh), one fragment per lane,
// and writes its colour with one 16-byte store.  Texels are gathered through
// the read-only path; fragments that are close on screen fall in neighbouring
// buckets, and in the PLANES layout neighbouring buckets at one in-bucket texel
// are neighbours in memory, so a warp's taps share cache lines.
#include "launch.h"
#include "rt_device.cuh"
#include "rt_filter.cuh"
#include "rt_internal.h"

namespace rt {

constexpr int kShadeThreads = 128;
constexpr int kShadeWarps = kShadeThreads / 32;

// The screen-tiled and the single-format forward keep three G-buffer chunks per
// warp (two in flight) and are held to 64 registers, 8 blocks (32 warps) per SM:
// measured 4% faster than two chunks at 72 registers.  The dispatching kernel of
// the flat stream keeps two chunks (it would spill at 64 registers).
template <bool TILED, int SPEC>
constexpr int shade_stages() { return TILED || SPEC >= 0 ? 3 : 2; }

template <int FILTER, bool TILED, int SPEC>
__global__ void __launch_bounds__(kShadeThreads, TILED || SPEC >= 0 ? 8 : 1) shade_kernel(const TexDesc* __restrict__ table, int n_obj,
                                                              const float* __restrict__ uv,
                                                              const float* __restrict__ dir,
                                                              const int32_t* __restrict__ obj, int64_t F,
                                                              Tiling tiling, float* __restrict__ out,
                                                              unsigned* status) {
    __shared__ WarpStage<false, shade_stages<TILED, SPEC>()> stages[kShadeWarps];
    for_each_fragment<kShadeWarps, false, TILED, shade_stages<TILED, SPEC>()>(uv, dir, obj, nullptr, F, tiling, stages,
                                                               [&](int64_t f, const Frag& q, float4) {
        float4 res = make_float4(0.f, 0.f, 0.f, 0.f);
        TexDesc d;
        if (fragment_valid(table, n_obj, q.o, q.u, q.v, q.x, q.y, q.z, status, d)) {
            Lookup<FILTER> L = locate<FILTER, (SPEC < 0)>(d, q.u, q.v, q.x, q.y, q.z);
            res = filter_spec<FILTER, SPEC>(d, L);
        }
        if (f >= 0) __stcs(reinterpret_cast<float4*>(out) + f, res);
    });
}

template <int FILTER, bool TILED>
__global__ void __launch_bounds__(kShadeThreads) locate_kernel(const TexDesc* __restrict__ table, int n_obj,
                                                               const float* __restrict__ uv,
                                                               const float* __restrict__ dir,
                                                               const int32_t* __restrict__ obj, int64_t F,
                                                               Tiling tiling, int32_t* __restrict__ idx,
                                                               float* __restrict__ coord, unsigned* status) {
    __shared__ WarpStage<false> stages[kShadeWarps];
    for_each_fragment<kShadeWarps, false, TILED, 2>(uv, dir, obj, nullptr, F, tiling, stages,
                                                    [&](int64_t f, const Frag& q, float4) {
        int4 I = make_int4(0, 0, 0, 0);
        float4 C = make_float4(0.f, 0.f, 0.f, 0.f);
        TexDesc d;
        if (fragment_valid(table, n_obj, q.o, q.u, q.v, q.x, q.y, q.z, status, d)) {
            Lookup<FILTER> L = locate<FILTER>(d, q.u, q.v, q.x, q.y, q.z);
            I = make_int4(L.u.fl, L.v.fl, L.s.fl, L.t.fl);
            C = make_float4(L.u.c, L.v.c, L.s.c, L.t.c);
        }
        if (f >= 0) {
            reinterpret_cast<int4*>(idx)[f] = I;
            reinterpret_cast<float4*>(coord)[f] = C;
        }
    });
}

// World-space forward and lookup (Eq. 1a with a per-fragment normal): the
// streamer of the tangent-space kernels with a fourth staged stream, the
// normal, over the flat fragment stream or, TILED, over screen tiles of a batch
// of frames.  Held to 64 registers and 8 blocks per SM, but for the dispatching
// quadrilinear kernels, which would spill (110 registers, 4 blocks): left to itself
// the compiler took 66 and 71 for the dispatching nearest and angular-bilinear ones,
// 7 blocks, and 4 frames of 1080p on FP16 took 84 and 92 us in the flat call instead of
// 73 and 80 (9 or 10 blocks: no better).
template <int FILTER, bool TILED, int SPEC>
__global__ void __launch_bounds__(kShadeThreads, SPEC >= 0 || FILTER != RT_QUADRILINEAR ? 8 : 1) world_shade_kernel(const TexDesc* __restrict__ table, int n_obj,
                                                                    const float* __restrict__ uv,
                                                                    const float* __restrict__ dir,
                                                                    const float* __restrict__ nrm,
                                                                    const int32_t* __restrict__ obj, int64_t F,
                                                                    Tiling tiling, float* __restrict__ out,
                                                                    int32_t* __restrict__ idx,
                                                                    float* __restrict__ coord, unsigned* status) {
    __shared__ WarpStage<false, 2, true> stages[kShadeWarps];
    for_each_fragment<kShadeWarps, false, TILED, 2, true>(uv, dir, obj, nullptr, F, tiling, stages,
                                                          [&](int64_t f, const Frag& q, float4) {
        float4 res = make_float4(0.f, 0.f, 0.f, 0.f);
        int4 Ix = make_int4(0, 0, 0, 0);
        float4 C = make_float4(0.f, 0.f, 0.f, 0.f);
        TexDesc d;
        const float3 N = make_float3(q.nx, q.ny, q.nz);
        if (fragment_valid(table, n_obj, q.o, q.u, q.v, q.x, q.y, q.z, status, d) && normal_valid(N, status)) {
            const Lookup<FILTER> L = locate_world<FILTER, (SPEC < 0)>(d, q.u, q.v, make_float3(q.x, q.y, q.z), N);
            if (out) res = filter_spec<FILTER, SPEC>(d, L);
            Ix = make_int4(L.u.fl, L.v.fl, L.s.fl, L.t.fl);
            C = make_float4(L.u.c, L.v.c, L.s.c, L.t.c);
        }
        if (f < 0) return;
        if (out) __stcs(reinterpret_cast<float4*>(out) + f, res);
        if (idx) {
            reinterpret_cast<int4*>(idx)[f] = Ix;
            reinterpret_cast<float4*>(coord)[f] = C;
        }
    }, nrm);
}

template <int FILTER, bool TILED, int SPEC>
static cudaError_t launch_world_shade_t(const TexDesc* table, int n_obj, const float* uv, const float* dir,
                                        const float* nrm, const int32_t* obj, int64_t F, const Tiling& T, float* out,
                                        int32_t* idx, float* coord, unsigned* status, cudaStream_t stream) {
    const unsigned grid = persistent_grid<world_shade_kernel<FILTER, TILED, SPEC>>(kShadeThreads,
                                          chunk_count_host(T, F, kShadeWarps));
    world_shade_kernel<FILTER, TILED, SPEC><<<grid, kShadeThreads, 0, stream>>>(table, n_obj, uv, dir, nrm, obj, F, T,
                                                                          out, idx, coord, status);
    return cudaGetLastError();
}

template <bool TILED, int SPEC>
static cudaError_t launch_world_shade_f(const TexDesc* table, int n_obj, const float* uv, const float* dir,
                                        const float* nrm, const int32_t* obj, int64_t F, int filter, const Tiling& T,
                                        float* out, int32_t* idx, float* coord, unsigned* status,
                                        cudaStream_t stream) {
    switch (filter) {
        case RT_NEAREST:
            return launch_world_shade_t<RT_NEAREST, TILED, SPEC>(table, n_obj, uv, dir, nrm, obj, F, T, out, idx, coord,
                                                           status, stream);
        case RT_ANGULAR_BILINEAR:
            return launch_world_shade_t<RT_ANGULAR_BILINEAR, TILED, SPEC>(table, n_obj, uv, dir, nrm, obj, F, T, out, idx,
                                                                    coord, status, stream);
        default:
            return launch_world_shade_t<RT_QUADRILINEAR, TILED, SPEC>(table, n_obj, uv, dir, nrm, obj, F, T, out, idx,
                                                                coord, status, stream);
    }
}

// Single-format instantiations of the screen-tiled path as for the tangent-space
// lookup: 64 registers and 8 blocks per SM instead of 112 and 4.  Forward and
// coordinate gradients of 12 poses of 1080p, FP16: 0.918 ms dispatching, 0.824 ms
// with these and the backward's (80 registers, 6 blocks, instead of 136 and 3).
cudaError_t launch_world_shade(const TexDesc* table, int n_obj, const float* uv, const float* dir, const float* nrm,
                               const int32_t* obj, int64_t F, int filter, const Tiling& T, int spec, float* out,
                               int32_t* idx, float* coord, unsigned* status, cudaStream_t stream) {
#define RT_WSHADE(TILED, SPEC)                                                                                    \
    launch_world_shade_f<TILED, SPEC>(table, n_obj, uv, dir, nrm, obj, F, filter, T, out, idx, coord, status, stream)
    if (T.W <= 0) return RT_WSHADE(false, -1);
    switch (spec) {
        case RT_F16:
            return RT_WSHADE(true, RT_F16);
        case RT_BF16:
            return RT_WSHADE(true, RT_BF16);
        case RT_F32:
            return RT_WSHADE(true, RT_F32);
        case RT_E4M3_BUCKET_SCALE:
            return RT_WSHADE(true, RT_E4M3_BUCKET_SCALE);
        default:
            return RT_WSHADE(true, -1);
    }
#undef RT_WSHADE
}

// S lookups per fragment, averaged (area lights over a shadow texture, Section
// 5: "more than one sample per bucket"): dirs holds S directions per fragment.
// General S: one fragment per thread, the samples in a loop.
template <int FILTER>
__global__ void __launch_bounds__(kShadeThreads) multi_shade_kernel(const TexDesc* __restrict__ table, int n_obj,
                                                                    const float* __restrict__ uv,
                                                                    const float* __restrict__ dirs, int S,
                                                                    const int32_t* __restrict__ obj, int64_t F,
                                                                    float* __restrict__ out, unsigned* status) {
    for (int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; f < F; f += (int64_t)gridDim.x * blockDim.x) {
        const float2 q = reinterpret_cast<const float2*>(uv)[f];
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        bool ok = true;
        for (int k = 0; k < S && ok; ++k) {
            const float* I = dirs + 3 * (f * S + k);
            TexDesc d;
            ok = fragment_valid(table, n_obj, obj[f], q.x, q.y, I[0], I[1], I[2], status, d);
            if (!ok) break;
            const float4 c = filter_any<FILTER>(d, locate<FILTER>(d, q.x, q.y, I[0], I[1], I[2]));
            acc.x += c.x;
            acc.y += c.y;
            acc.z += c.z;
            acc.w += c.w;
        }
        const float inv = 1.0f / (float)S;
        const float4 res = ok ? make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv)
                              : make_float4(0.f, 0.f, 0.f, 0.f);
        __stcs(reinterpret_cast<float4*>(out) + f, res);
    }
}

// S a power of two <= 32: one lookup per lane, lanes f S .. f S + S - 1 of a
// warp share fragment f (coalesced direction loads, 32 lookups in flight per
// warp) and sum by butterfly shuffles.  Each lane loads the inputs of its next
// lookup before filtering the current one, so their DRAM latency overlaps the
// gathers (which hit L1 and L2: a bit texture is small).
template <int FILTER>
__global__ void __launch_bounds__(kShadeThreads) multi_shade_lanes_kernel(const TexDesc* __restrict__ table,
                                                                          int n_obj, const float* __restrict__ uv,
                                                                          const float* __restrict__ dirs, int S,
                                                                          const int32_t* __restrict__ obj, int64_t F,
                                                                          float* __restrict__ out, unsigned* status) {
    const int lane = threadIdx.x & 31;
    const int lg = __ffs(S) - 1;  // S = 2^lg
    const int64_t total = F * S;
    const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t stride = (((int64_t)gridDim.x * blockDim.x) >> 5) * 32;
    float2 q = make_float2(0.f, 0.f);
    float ix = 0.f, iy = 0.f, iz = 0.f;
    int32_t o = -1;
    auto fetch = [&](int64_t e) {
        if (e < total) {
            const int64_t f = e >> lg;
            q = reinterpret_cast<const float2*>(uv)[f];
            o = obj[f];
            ix = dirs[3 * e];
            iy = dirs[3 * e + 1];
            iz = dirs[3 * e + 2];
        }
    };
    fetch(warp0 * 32 + lane);
    for (int64_t base = warp0 * 32; base < total; base += stride) {
        const int64_t e = base + lane;
        const float2 cq = q;
        const float cx = ix, cy = iy, cz = iz;
        const int32_t co = o;
        fetch(e + stride);
        float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
        int bad = 0;
        if (e < total) {
            TexDesc d;
            if (fragment_valid(table, n_obj, co, cq.x, cq.y, cx, cy, cz, status, d))
                c = filter_any<FILTER>(d, locate<FILTER>(d, cq.x, cq.y, cx, cy, cz));
            else
                bad = co >= 0;  // an invalid sample zeroes its fragment
        }
        for (int off = 1; off < S; off <<= 1) {
            c.x += __shfl_xor_sync(0xffffffffu, c.x, off);
            c.y += __shfl_xor_sync(0xffffffffu, c.y, off);
            c.z += __shfl_xor_sync(0xffffffffu, c.z, off);
            c.w += __shfl_xor_sync(0xffffffffu, c.w, off);
            bad |= __shfl_xor_sync(0xffffffffu, bad, off);
        }
        if (e < total && (lane & (S - 1)) == 0) {
            const float inv = 1.0f / (float)S;
            const float4 r = bad ? make_float4(0.f, 0.f, 0.f, 0.f)
                                 : make_float4(c.x * inv, c.y * inv, c.z * inv, c.w * inv);
            __stcs(reinterpret_cast<float4*>(out) + (e >> lg), r);
        }
    }
}

// The same when every object is a bit texture in clamp mode: one number per
// lookup instead of four equal channels, a row's two bits from one word, and a
// fragment per thread, its samples one after another with the next direction
// loaded ahead (the validity test, the spatial axes and the bucket offsets are
// then a fragment's, not a lookup's).  A power of two up to 32 samples is summed
// as the tree of multi_shade_lanes_kernel, others in their order.  Bound: issue
// (two thirds of the cycles) and the gathers' latency (L1 data pipe 62 %).
// 10 poses of 1080p, S = 4, quadrilinear on 2 x 1024^2 x 16^2 bits: 1.12 ms with the
// general kernel, 0.77 with a lane per lookup, 0.645 here (to 0.80 by input); 2 views of 1366 x 768
// (lane per lookup -> here): S = 3, angular 56 -> 36 us, S = 16, quadrilinear 351 -> 265.
template <int FILTER, int KIND>
__global__ void __launch_bounds__(kShadeThreads, 8) multi_bits_kernel(const TexDesc* __restrict__ table, int n_obj,
                                                                      const float* __restrict__ uv,
                                                                      const float* __restrict__ dirs, int S,
                                                                      const int32_t* __restrict__ obj, int64_t F,
                                                                      float* __restrict__ out, unsigned* status) {
    const float inv = 1.0f / (float)S;
    const bool tree = S <= 32 && (S & (S - 1)) == 0;
    for (int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; f < F; f += (int64_t)gridDim.x * blockDim.x) {
        const float2 q = reinterpret_cast<const float2*>(uv)[f];
        const int32_t o = obj[f];
        const float* I = dirs + 3 * (f * S);
        float x = I[0], y = I[1], z = I[2];
        float sum = 0.f, level[5];  // level[l]: the sum of the last whole left half of 2^l samples
        bool ok = true;
        for (int k = 0; k < S && ok; ++k) {
            const float cx = x, cy = y, cz = z;
            if (k + 1 < S) {
                I += 3;
                x = I[0];
                y = I[1];
                z = I[2];
            }
            TexDesc d;
            ok = fragment_valid(table, n_obj, o, q.x, q.y, cx, cy, cz, status, d);
            if (!ok) break;
            const float c = filter_bits<FILTER, KIND>(d, locate<FILTER, false>(d, q.x, q.y, cx, cy, cz));
            if (tree) {
                sum = c;
#pragma unroll
                for (int l = 0; l < 5; ++l) {
                    if (!((k >> l) & 1)) {
                        level[l] = sum;
                        break;
                    }
                    sum = level[l] + sum;
                }
            } else {
                sum += c;
            }
        }
        const float v = ok ? sum * inv : 0.f;
        __stcs(reinterpret_cast<float4*>(out) + f, make_float4(v, v, v, v));
    }
}

template <int FILTER, int KIND>
static void launch_multi_bits(const TexDesc* table, int n_obj, const float* uv, const float* dirs, int S,
                              const int32_t* obj, int64_t F, float* out, unsigned* status, cudaStream_t stream) {
    const unsigned grid = persistent_grid<multi_bits_kernel<FILTER, KIND>>(kShadeThreads, (F + 31) / 32);
    multi_bits_kernel<FILTER, KIND><<<grid, kShadeThreads, 0, stream>>>(table, n_obj, uv, dirs, S, obj, F, out, status);
}

// Below this many fragments a lane per lookup is faster where S divides a warp: a
// thread per fragment leaves the chip (155 648 threads at 8 blocks per SM) or its
// last round partly idle for as long as the samples of a fragment take, and the
// cheaper filters gain less from sharing the fragment's work.  Thread / lane, 1024 x
// 512 x 16^2 bits, every fragment with an object, S = 4, 8, 16, 32:
//   quadrilinear: 60 000 fragments 1.00, 0.86, 0.93, 1.00, 98 304 0.75, 0.73, 0.81, 0.91, 1.5 M 0.59,
//     0.54, 0.58, 0.67;
//   angular-bilinear: 60 000 1.00, 1.07, 1.14, 1.46, 98 304 0.75, 0.83, 1.00, 1.31, 200 000 0.83, 0.85, 1.05,
//     1.27, 250 000 0.72, 0.77, 0.97, 1.16, 480 000 0.67, 0.67, 0.85, 1.07, 1.5 M 0.60, 0.58, 0.78, 1.00
//     (with the background of a frame among them 0.91);
//   nearest: 98 304 1.00, 0.93, 1.00, 1.41, 200 000 0.84, 0.88, 1.08, 1.37, 250 000 0.83, 0.73, 1.00, 1.25, 1.5 M
//     0.63, 0.62, 0.86, 1.13.
template <int FILTER>
static int64_t few_fragments(int S) {
    if (FILTER == RT_QUADRILINEAR || S < 16) return 98304;
    if (S == 16) return 262144;
    return FILTER == RT_NEAREST ? INT64_MAX : 524288;
}

template <int FILTER>
static void launch_multi_t(const TexDesc* table, int n_obj, const float* uv, const float* dirs, int S,
                           const int32_t* obj, int64_t F, int bits, float* out, unsigned* status,
                           cudaStream_t stream) {
    const bool lanes = S <= 32 && (S & (S - 1)) == 0;
    if (lanes && F < few_fragments<FILTER>(S)) bits = kBitsNone;
    if (bits == kBitsWords) {
        launch_multi_bits<FILTER, kBitsWords>(table, n_obj, uv, dirs, S, obj, F, out, status, stream);
    } else if (bits == kBitsSmall) {
        launch_multi_bits<FILTER, kBitsSmall>(table, n_obj, uv, dirs, S, obj, F, out, status, stream);
    } else if (bits == kBitsLarge) {
        launch_multi_bits<FILTER, kBitsLarge>(table, n_obj, uv, dirs, S, obj, F, out, status, stream);
    } else if (lanes) {
        const unsigned grid = persistent_grid<multi_shade_lanes_kernel<FILTER>>(kShadeThreads, (F * S + 31) / 32);
        multi_shade_lanes_kernel<FILTER><<<grid, kShadeThreads, 0, stream>>>(table, n_obj, uv, dirs, S, obj, F, out,
                                                                              status);
    } else {
        const unsigned grid = persistent_grid<multi_shade_kernel<FILTER>>(kShadeThreads,
                                              (F + kShadeThreads - 1) / kShadeThreads);
        multi_shade_kernel<FILTER><<<grid, kShadeThreads, 0, stream>>>(table, n_obj, uv, dirs, S, obj, F, out,
                                                                        status);
    }
}

cudaError_t launch_multi_shade(const TexDesc* table, int n_obj, const float* uv, const float* dirs, int S,
                               const int32_t* obj, int64_t F, int filter, int bits, float* out, unsigned* status,
                               cudaStream_t stream) {
    switch (filter) {
        case RT_NEAREST:
            launch_multi_t<RT_NEAREST>(table, n_obj, uv, dirs, S, obj, F, bits, out, status, stream);
            break;
        case RT_ANGULAR_BILINEAR:
            launch_multi_t<RT_ANGULAR_BILINEAR>(table, n_obj, uv, dirs, S, obj, F, bits, out, status, stream);
            break;
        default:
            launch_multi_t<RT_QUADRILINEAR>(table, n_obj, uv, dirs, S, obj, F, bits, out, status, stream);
    }
    return cudaGetLastError();
}

template <int FILTER, bool TILED, int SPEC>
static cudaError_t launch_shade_t(const TexDesc* table, int n_obj, const float* uv, const float* dir,
                                  const int32_t* obj, int64_t F, const Tiling& T, float* out, unsigned* status,
                                  cudaStream_t stream) {
    const unsigned grid = persistent_grid<shade_kernel<FILTER, TILED, SPEC>>(kShadeThreads,
                                          chunk_count_host(T, F, kShadeWarps));
    shade_kernel<FILTER, TILED, SPEC><<<grid, kShadeThreads, 0, stream>>>(table, n_obj, uv, dir, obj, F, T, out,
                                                                          status);
    return cudaGetLastError();
}

template <bool TILED, int SPEC>
static cudaError_t launch_shade_f(const TexDesc* table, int n_obj, const float* uv, const float* dir,
                                  const int32_t* obj, int64_t F, int filter, const Tiling& T, float* out,
                                  unsigned* status, cudaStream_t stream) {
    switch (filter) {
        case RT_NEAREST:
            return launch_shade_t<RT_NEAREST, TILED, SPEC>(table, n_obj, uv, dir, obj, F, T, out, status, stream);
        case RT_ANGULAR_BILINEAR:
            return launch_shade_t<RT_ANGULAR_BILINEAR, TILED, SPEC>(table, n_obj, uv, dir, obj, F, T, out, status,
                                                                    stream);
        default:
            return launch_shade_t<RT_QUADRILINEAR, TILED, SPEC>(table, n_obj, uv, dir, obj, F, T, out, status,
                                                                stream);
    }
}

// A single-format instantiation per storage format, dense and palette (spec);
// contexts of several formats, with repeating or with borrowed objects of another
// layout run the dispatching kernels.  20 poses of 1080p, E4M3 palettes of 1024
// buckets: 0.591 ms dispatching (64 registers, spilling), 0.547 ms here (56).
template <bool TILED>
static cudaError_t launch_shade_s(const TexDesc* table, int n_obj, const float* uv, const float* dir,
                                  const int32_t* obj, int64_t F, int filter, const Tiling& T, int spec, float* out,
                                  unsigned* status, cudaStream_t stream) {
#define RT_SHADE(SPEC)  \
    case SPEC:          \
        return launch_shade_f<TILED, SPEC>(table, n_obj, uv, dir, obj, F, filter, T, out, status, stream)
    switch (spec) {
        RT_SHADE(RT_F16);
        RT_SHADE(RT_BF16);
        RT_SHADE(RT_F32);
        RT_SHADE(RT_E4M3_BUCKET_SCALE);
        RT_SHADE(RT_F16 + kSpecPalette);
        RT_SHADE(RT_BF16 + kSpecPalette);
        RT_SHADE(RT_F32 + kSpecPalette);
        RT_SHADE(RT_E4M3_BUCKET_SCALE + kSpecPalette);
        default:
            return launch_shade_f<TILED, -1>(table, n_obj, uv, dir, obj, F, filter, T, out, status, stream);
    }
#undef RT_SHADE
}

cudaError_t launch_shade(const TexDesc* table, int n_obj, const float* uv, const float* dir, const int32_t* obj,
                         int64_t F, int filter, const Tiling& T, int spec, float* out, unsigned* status,
                         cudaStream_t stream) {
    if (T.W > 0) return launch_shade_s<true>(table, n_obj, uv, dir, obj, F, filter, T, spec, out, status, stream);
    return launch_shade_s<false>(table, n_obj, uv, dir, obj, F, filter, T, spec, out, status, stream);
}

template <int FILTER, bool TILED>
static cudaError_t launch_locate_t(const TexDesc* table, int n_obj, const float* uv, const float* dir,
                                   const int32_t* obj, int64_t F, const Tiling& T, int32_t* idx, float* coord,
                                   unsigned* status, cudaStream_t stream) {
    const unsigned grid = persistent_grid<locate_kernel<FILTER, TILED>>(kShadeThreads,
                                          chunk_count_host(T, F, kShadeWarps));
    locate_kernel<FILTER, TILED><<<grid, kShadeThreads, 0, stream>>>(table, n_obj, uv, dir, obj, F, T, idx, coord,
                                                                     status);
    return cudaGetLastError();
}

cudaError_t launch_locate(const TexDesc* table, int n_obj, const float* uv, const float* dir, const int32_t* obj,
                          int64_t F, int filter, int32_t* idx, float* coord, unsigned* status, cudaStream_t stream) {
    const Tiling T = flat_tiling();
    switch (filter) {
        case RT_NEAREST:
            return launch_locate_t<RT_NEAREST, false>(table, n_obj, uv, dir, obj, F, T, idx, coord, status, stream);
        case RT_ANGULAR_BILINEAR:
            return launch_locate_t<RT_ANGULAR_BILINEAR, false>(table, n_obj, uv, dir, obj, F, T, idx, coord, status,
                                                               stream);
        default:
            return launch_locate_t<RT_QUADRILINEAR, false>(table, n_obj, uv, dir, obj, F, T, idx, coord, status,
                                                           stream);
    }
}

}  // namespace rt
