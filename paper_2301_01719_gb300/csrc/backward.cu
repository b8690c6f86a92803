// backward.cu -- gradients of the lookup: texels, UV and direction.
//
// The filter weights are recomputed exactly as the forward pass computes them
// (nothing is stored between the passes).  Texel gradients w_tap * dL/dout are
// summed into FP32 buffers with 16-byte vector reductions (red.global.add.v4.f32),
// one per tap of non-zero weight.  UV and direction gradients follow the chain
// rule through the nested lerps, the Note's clamp (zero derivative where a
// coordinate is clamped), Eq. 3 and Eq. 1b.
#include <cmath>

#include "launch.h"
#include "rt_backward.cuh"
#include "rt_internal.h"

namespace rt {

// The single-format tiled kernels are held to 80 registers (6 blocks, 24 warps
// per SM): measured 3 % faster than 95 registers at 5 blocks.
template <int FILTER, bool TILED, bool DET, int SPEC>
__global__ void __launch_bounds__(kBackThreads, DET ? 4 : (TILED && SPEC >= 0) ? 6 : 1) backward_kernel(
    const TexDesc* __restrict__ table, int n_obj, const float* __restrict__ uv, const float* __restrict__ dir,
    const int32_t* __restrict__ obj, int64_t F, Tiling tiling, const float* __restrict__ dL_dout,
    const __grid_constant__ GradTable grads, bool any_grad, float* __restrict__ dL_duv, float* __restrict__ dL_ddir,
    bool accumulate, unsigned* status) {
    __shared__ WarpStage<true> stages[kBackWarps];
    const bool coord_grads = (dL_duv != nullptr) || (dL_ddir != nullptr);
    for_each_fragment<kBackWarps, true, TILED, 2>(uv, dir, obj, dL_dout, F, tiling, stages,
                                               [&](int64_t f, const Frag& q, float4 go) {
        float2 guv = make_float2(0.f, 0.f);
        float3 gdir = make_float3(0.f, 0.f, 0.f);
        TexDesc d;
        Lookup<FILTER> L;
        void* grad = nullptr;
        const bool valid = fragment_valid(table, n_obj, q.o, q.u, q.v, q.x, q.y, q.z, status, d);
        if (valid) {
            L = locate<FILTER, (SPEC < 0)>(d, q.u, q.v, q.x, q.y, q.z);
            if (any_grad) grad = grads.p[q.o];
        }
        if (DET) {
            reduce_fixed_warp<FILTER, SPEC>(valid && grad && d.fmt != RT_BIT1, d, L, go, grad, status);
            grad = nullptr;
        }
        if (valid && (!DET || coord_grads)) {
            CoordGrad cg = backward_spec<FILTER, SPEC>(d, L, go, grad, coord_grads);
            coord_grads_of<FILTER>(d, L, q, cg, dL_ddir != nullptr, guv, gdir);
        }
        if (f < 0) return;
        store_coord_grads(f, guv, gdir, dL_duv, dL_ddir, accumulate);
    });
}

template <int FILTER, bool TILED, bool DET, int SPEC>
static cudaError_t launch_backward_t(const TexDesc* table, int n_obj, const float* uv, const float* dir,
                                     const int32_t* obj, int64_t F, const Tiling& T, const float* dL_dout,
                                     const GradTable& grads, bool any_grad, float* dL_duv, float* dL_ddir,
                                     bool accumulate, unsigned* status, cudaStream_t stream) {
    const unsigned grid = persistent_grid<backward_kernel<FILTER, TILED, DET, SPEC>>(kBackThreads,
                                          chunk_count_host(T, F, kBackWarps));
    backward_kernel<FILTER, TILED, DET, SPEC><<<grid, kBackThreads, 0, stream>>>(
        table, n_obj, uv, dir, obj, F, T, dL_dout, grads, any_grad, dL_duv, dL_ddir, accumulate, status);
    return cudaGetLastError();
}

template <bool TILED, bool DET, int SPEC>
static cudaError_t launch_backward_f(const TexDesc* table, int n_obj, const float* uv, const float* dir,
                                     const int32_t* obj, int64_t F, int filter, const Tiling& T,
                                     const float* dL_dout, const GradTable& grads, bool any_grad, float* dL_duv,
                                     float* dL_ddir, bool accumulate, unsigned* status, cudaStream_t stream) {
    switch (filter) {
        case RT_NEAREST:
            return launch_backward_t<RT_NEAREST, TILED, DET, SPEC>(table, n_obj, uv, dir, obj, F, T, dL_dout, grads,
                                                                   any_grad, dL_duv, dL_ddir, accumulate, status,
                                                                   stream);
        case RT_ANGULAR_BILINEAR:
            return launch_backward_t<RT_ANGULAR_BILINEAR, TILED, DET, SPEC>(table, n_obj, uv, dir, obj, F, T,
                                                                            dL_dout, grads, any_grad, dL_duv,
                                                                            dL_ddir, accumulate, status, stream);
        default:
            return launch_backward_t<RT_QUADRILINEAR, TILED, DET, SPEC>(table, n_obj, uv, dir, obj, F, T, dL_dout,
                                                                        grads, any_grad, dL_duv, dL_ddir,
                                                                        accumulate, status, stream);
    }
}

// The screen-tiled, non-deterministic path has a single-format instantiation
// per storage format (spec); the others run the dispatching kernels.
cudaError_t launch_backward(const TexDesc* table, int n_obj, const float* uv, const float* dir, const int32_t* obj,
                            int64_t F, int filter, const Tiling& T, int spec, const float* dL_dout,
                            const GradTable& grads, bool any_grad, float* dL_duv, float* dL_ddir, bool accumulate,
                            bool deterministic, unsigned* status, cudaStream_t stream) {
#define RT_BWD(TILED, DET, SPEC)                                                                                 \
    launch_backward_f<TILED, DET, SPEC>(table, n_obj, uv, dir, obj, F, filter, T, dL_dout, grads, any_grad, dL_duv, \
                                        dL_ddir, accumulate, status, stream)
    if (T.W > 0) {
        if (deterministic) return RT_BWD(true, true, -1);
        switch (spec) {
            case RT_F16:
                return RT_BWD(true, false, RT_F16);
            case RT_BF16:
                return RT_BWD(true, false, RT_BF16);
            case RT_F32:
                return RT_BWD(true, false, RT_F32);
            case RT_E4M3_BUCKET_SCALE:
                return RT_BWD(true, false, RT_E4M3_BUCKET_SCALE);
            default:
                return RT_BWD(true, false, -1);
        }
    }
    if (deterministic) return RT_BWD(false, true, -1);
    return RT_BWD(false, false, -1);
#undef RT_BWD
}

// World-space backward (Eq. 1a with a per-fragment normal): the streamer of
// the tangent-space backward with the normal as a fourth staged stream, over
// the flat fragment stream or, TILED, over screen tiles of a batch of frames.
// dL/dI = dL/dN, since A depends on h = I + N only.
// The dispatching kernels' blocks per SM: left to itself the compiler takes 136
// (tiled) and 128 registers for the quadrilinear ones, 85 for the angular-bilinear
// ones.  4 frames of 1080p, FP16 and FP32 objects, coordinate gradients / texel
// gradients as well, us (136, 128, 85 -> here): quadrilinear in tiles 223 -> 189 / 572 -> 542
// (5 blocks: 188 / 551), flat 217 -> 173 / 562 -> 517 (4 blocks: 182 / 518); angular-bilinear in
// tiles 146 -> 127, flat 144 -> 125 (6 blocks: 133, 134).  The deterministic ones: 4 blocks,
// quadrilinear in tiles 1869 -> 1844.
template <int FILTER, bool DET, bool TILED, int SPEC>
constexpr int world_backward_blocks() {
    if (SPEC >= 0) return 6;
    if (DET) return 4;
    return FILTER == RT_QUADRILINEAR ? (TILED ? 4 : 5) : FILTER == RT_ANGULAR_BILINEAR ? 7 : 1;
}

template <int FILTER, bool DET, bool TILED, int SPEC>
__global__ void __launch_bounds__(kBackThreads, world_backward_blocks<FILTER, DET, TILED, SPEC>()) world_backward_kernel(
    const TexDesc* __restrict__ table, int n_obj, const float* __restrict__ uv, const float* __restrict__ dir,
    const float* __restrict__ nrm, const int32_t* __restrict__ obj, int64_t F, Tiling tiling,
    const float* __restrict__ dL_dout,
    const __grid_constant__ GradTable grads, bool any_grad, float* __restrict__ dL_duv, float* __restrict__ dL_ddir,
    float* __restrict__ dL_dnrm, bool accumulate, unsigned* status) {
    __shared__ WarpStage<true, 2, true> stages[kBackWarps];
    const bool coord_grads = dL_duv || dL_ddir || dL_dnrm;
    for_each_fragment<kBackWarps, true, TILED, 2, true>(uv, dir, obj, dL_dout, F, tiling, stages,
                                                        [&](int64_t f, const Frag& q, float4 go) {
        float2 guv = make_float2(0.f, 0.f);
        float3 gh = make_float3(0.f, 0.f, 0.f);
        TexDesc d;
        const float3 I = make_float3(q.x, q.y, q.z), N = make_float3(q.nx, q.ny, q.nz);
        Lookup<FILTER> L;
        void* grad = nullptr;
        const bool valid = fragment_valid(table, n_obj, q.o, q.u, q.v, I.x, I.y, I.z, status, d) &&
                           normal_valid(N, status);
        if (valid) {
            L = locate_world<FILTER, (SPEC < 0)>(d, q.u, q.v, I, N);
            if (any_grad) grad = grads.p[q.o];
        }
        if (DET) {
            reduce_fixed_warp<FILTER, SPEC>(valid && grad && d.fmt != RT_BIT1, d, L, go, grad, status);
            grad = nullptr;
        }
        if (valid && (!DET || coord_grads)) {
            const CoordGrad cg = backward_spec<FILTER, SPEC>(d, L, go, grad, coord_grads);
            if (FILTER == RT_QUADRILINEAR) guv = uv_grad(d, q.u, q.v, cg.gu, cg.gv);
            if (FILTER != RT_NEAREST && (dL_ddir || dL_dnrm)) {
                const float gBx = (L.B.x > -d.hi && L.B.x < d.hi) ? cg.gs * d.half_n : 0.f;
                const float gBy = (L.B.y > -d.hi && L.B.y < d.hi) ? cg.gt * d.half_n : 0.f;
                gh = half_grad(I.x + N.x, I.y + N.y, I.z + N.z, gBx, gBy);
            }
        }
        if (f < 0) return;
        if (dL_duv) {
            float2* p = reinterpret_cast<float2*>(dL_duv) + f;
            if (accumulate) {
                const float2 o = *p;
                guv.x += o.x;
                guv.y += o.y;
            }
            *p = guv;
        }
        float* outs[2] = {dL_ddir, dL_dnrm};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            float* p = outs[k];
            if (!p) continue;
            p += 3 * f;
            p[0] = accumulate ? p[0] + gh.x : gh.x;
            p[1] = accumulate ? p[1] + gh.y : gh.y;
            p[2] = accumulate ? p[2] + gh.z : gh.z;
        }
    }, nrm);
}

template <int FILTER, bool DET, bool TILED, int SPEC>
static cudaError_t launch_world_backward_t(const TexDesc* table, int n_obj, const float* uv, const float* dir,
                                           const float* nrm, const int32_t* obj, int64_t F, const Tiling& T,
                                           const float* dL_dout, const GradTable& grads, bool any_grad, float* dL_duv,
                                           float* dL_ddir, float* dL_dnrm, bool accumulate, unsigned* status,
                                           cudaStream_t stream) {
    // with texel gradients more warps only queue at the reductions: angular-bilinear, 7 blocks 426 us in
    // tiles and 417 flat, 6 415 and 401, 5 413 and 393, 4 419 and 404
    const int most = FILTER == RT_ANGULAR_BILINEAR && SPEC < 0 && any_grad ? 5 : 0;
    const unsigned grid = persistent_grid<world_backward_kernel<FILTER, DET, TILED, SPEC>>(
        kBackThreads, chunk_count_host(T, F, kBackWarps), most);
    world_backward_kernel<FILTER, DET, TILED, SPEC><<<grid, kBackThreads, 0, stream>>>(
        table, n_obj, uv, dir, nrm, obj, F, T, dL_dout, grads, any_grad, dL_duv, dL_ddir, dL_dnrm, accumulate,
        status);
    return cudaGetLastError();
}

template <bool DET, bool TILED, int SPEC>
static cudaError_t launch_world_backward_d(const TexDesc* table, int n_obj, const float* uv, const float* dir,
                                           const float* nrm, const int32_t* obj, int64_t F, int filter,
                                           const Tiling& T, const float* dL_dout, const GradTable& grads,
                                           bool any_grad, float* dL_duv, float* dL_ddir, float* dL_dnrm,
                                           bool accumulate, unsigned* status, cudaStream_t stream) {
#define RT_WBWD(FILT)                                                                                              \
    launch_world_backward_t<FILT, DET, TILED, SPEC>(table, n_obj, uv, dir, nrm, obj, F, T, dL_dout, grads, any_grad,      \
                                              dL_duv, dL_ddir, dL_dnrm, accumulate, status, stream)
    switch (filter) {
        case RT_NEAREST:
            return RT_WBWD(RT_NEAREST);
        case RT_ANGULAR_BILINEAR:
            return RT_WBWD(RT_ANGULAR_BILINEAR);
        default:
            return RT_WBWD(RT_QUADRILINEAR);
    }
#undef RT_WBWD
}

cudaError_t launch_world_backward(const TexDesc* table, int n_obj, const float* uv, const float* dir,
                                  const float* nrm, const int32_t* obj, int64_t F, int filter, const Tiling& T,
                                  int spec, const float* dL_dout, const GradTable& grads, bool any_grad,
                                  float* dL_duv, float* dL_ddir, float* dL_dnrm, bool accumulate, bool deterministic,
                                  unsigned* status, cudaStream_t stream) {
#define RT_WBWD_D(DET, TILED, SPEC)                                                                               \
    launch_world_backward_d<DET, TILED, SPEC>(table, n_obj, uv, dir, nrm, obj, F, filter, T, dL_dout, grads,       \
                                              any_grad, dL_duv, dL_ddir, dL_dnrm, accumulate, status, stream)
    if (T.W <= 0) return deterministic ? RT_WBWD_D(true, false, -1) : RT_WBWD_D(false, false, -1);
    if (deterministic) return RT_WBWD_D(true, true, -1);
    switch (spec) {
        case RT_F16:
            return RT_WBWD_D(false, true, RT_F16);
        case RT_BF16:
            return RT_WBWD_D(false, true, RT_BF16);
        case RT_F32:
            return RT_WBWD_D(false, true, RT_F32);
        case RT_E4M3_BUCKET_SCALE:
            return RT_WBWD_D(false, true, RT_E4M3_BUCKET_SCALE);
        default:
            return RT_WBWD_D(false, true, -1);
    }
#undef RT_WBWD_D
}

// Fixed-point sums (deterministic mode) -> FP32 gradients: the sum times
// f = scale 2^-32, the product rounded to FP64 and then to FP32, added to or
// overwriting dst.  The FP64 pipe takes a few operations per cycle and SM, and
// converting to double, multiplying and converting back would bound the pass at
// three times its memory time.  So a magnitude below 2^52 becomes the mantissa
// of 2^52 + |a|, one FMA takes (2^52 + |a|) |f| - 2^52 |f| = |a| |f| with the
// one rounding a product has, and FP32 is rounded from its bits in integers.
struct FixedScale {
    double f, mag, minus;  // f, |f| and -2^52 |f|
    uint32_t sign;         // f's sign, in bit 31
};

static FixedScale fixed_scale(double scale) {
    FixedScale s;
    s.f = scale * (1.0 / 4294967296.0);
    s.mag = std::fabs(s.f);
    s.minus = -4503599627370496.0 * s.mag;  // infinite for a huge scale: no product of it passes the test below
    s.sign = std::signbit(s.f) ? 0x80000000u : 0u;
    return s;
}

// A call, so that the compiler does not compute it beside the other form.
__device__ __noinline__ float fixed_to_float_any(long long a, double f) { return (float)((double)a * f); }

__device__ __forceinline__ float fixed_to_float(long long a, const FixedScale& s) {
    const uint32_t sign = (a < 0 ? 0x80000000u : 0u) ^ s.sign;
    const uint64_t m = a < 0 ? 0ull - (uint64_t)a : (uint64_t)a;
    if (m == 0) return __uint_as_float(sign);
    const double d = __fma_rn(__longlong_as_double((long long)(m | 0x4330000000000000ull)), s.mag, s.minus);
    const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
    const uint32_t e = hi >> 20;  // d >= 0; an FP32 in its normal range for e in [897, 1150)
    if (m < (1ull << 52) && e - 897u < 253u) {
        const uint32_t y = __funnelshift_l(lo, hi, 3) - 0xC0000000u;  // the bits above the lowest 29, rebiased
        const uint32_t up = ((lo & 0x1fffffffu) + 0x0fffffffu + (y & 1u)) >> 29;
        return __uint_as_float(sign | (y + up));
    }
    return fixed_to_float_any(a, s.f);
}

// Two values per thread and load, so that a warp's loads (512 bytes) and stores
// (256) are whole lines, four loads in flight (acc and dst 16-byte aligned);
// an odd last value by itself.  Bound: HBM.  151 M values (1.8 GB): 0.83 ms with
// one value per thread and three FP64 operations each, 0.25-0.27 ms here.
constexpr int kFixedUnroll = 4;

__global__ void __launch_bounds__(256) fixed_to_float_kernel(const long long* __restrict__ acc,
                                                             float* __restrict__ dst, int64_t count, FixedScale f,
                                                             bool accumulate) {
    const longlong2* in = reinterpret_cast<const longlong2*>(acc);
    float2* out = reinterpret_cast<float2*>(dst);
    const int64_t pairs = count / 2, first = (int64_t)blockIdx.x * (blockDim.x * kFixedUnroll) + threadIdx.x;
    longlong2 a[kFixedUnroll];
#pragma unroll
    for (int u = 0; u < kFixedUnroll; ++u) {
        const int64_t k = first + u * 256;
        a[u] = k < pairs ? __ldcs(in + k) : make_longlong2(0, 0);
    }
#pragma unroll
    for (int u = 0; u < kFixedUnroll; ++u) {
        const int64_t k = first + u * 256;
        if (k >= pairs) break;
        float2 v = make_float2(fixed_to_float(a[u].x, f), fixed_to_float(a[u].y, f));
        if (accumulate) {
            const float2 o = out[k];
            v = make_float2(o.x + v.x, o.y + v.y);
        }
        out[k] = v;
    }
    if (first == 0 && (count & 1)) {
        const float v = fixed_to_float(acc[count - 1], f);
        dst[count - 1] = accumulate ? dst[count - 1] + v : v;
    }
}

cudaError_t launch_fixed_to_float(const long long* acc, float* dst, int64_t count, bool accumulate,
                                  cudaStream_t stream, double scale) {
    if (count <= 0) return cudaSuccess;
    const int64_t blocks = (count / 2 + 256 * kFixedUnroll - 1) / (256 * kFixedUnroll);
    if (blocks > 0x7fffffff) return cudaErrorInvalidValue;
    fixed_to_float_kernel<<<(unsigned)(blocks > 0 ? blocks : 1), 256, 0, stream>>>(acc, dst, count,
                                                                                 fixed_scale(scale), accumulate);
    return cudaGetLastError();
}

}  // namespace rt
