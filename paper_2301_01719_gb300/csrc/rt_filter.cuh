// rt_filter.cuh -- gathering and filtering the taps of one fragment (FP32).
//
// QUADRILINEAR: 2 x 2 buckets (u, v) x 2 x 2 texels (s, t) = 16 taps, all four
// buckets at the same in-bucket coordinate (one tangent-space direction per
// fragment).  ANGULAR_BILINEAR: the nearest bucket, 2 x 2 texels inside it
// ("single sample per bucket", Section 2).  NEAREST: one texel.
// Weights are applied as nested lerps a + w (b - a) in the order s, t, u, v, so
// a constant texture returns its constant exactly.
#pragma once

#include <type_traits>

#include "rt_device.cuh"

namespace rt {

// The four texels (s0,t0) (s1,t0) (s0,t1) (s1,t1) of bucket (i, j).
template <int FMT, int LAYOUT>
__device__ __forceinline__ void load_quadP(const TexDesc& d, int i, int j, const Axis& s, const Axis& t, P4& t00,
                                           P4& t10, P4& t01, P4& t11) {
    float sc = 1.0f;
    if (FMT == RT_E4M3_BUCKET_SCALE) sc = __ldg(d.scale + bucket_slot<LAYOUT>(d, i, j));
    t00 = load_texelP<FMT>(d.base, texel_index<LAYOUT>(d, i, j, s.k0, t.k0), sc);
    t10 = load_texelP<FMT>(d.base, texel_index<LAYOUT>(d, i, j, s.k1, t.k0), sc);
    t01 = load_texelP<FMT>(d.base, texel_index<LAYOUT>(d, i, j, s.k0, t.k1), sc);
    t11 = load_texelP<FMT>(d.base, texel_index<LAYOUT>(d, i, j, s.k1, t.k1), sc);
}

// Addresses of the taps.  PLANES / QUADS: the four in-bucket texels (s0|s1,
// t0|t1) select four planes (64-bit base indices), the (up to) four buckets
// select spatial offsets inside a plane (32-bit, w h < 2^31).
// The planes (64-bit bases, k = (s0,t0) (s1,t0) (s0,t1) (s1,t1)) and the spatial
// offsets (b = (u0,v0) (u1,v0) (u0,v1) (u1,v1)) of a quadrilinear lookup's 16 taps
// on a PLANES / QUADS / palette texture: tap (b, k) is texel pl[k] + o[b].
template <int LAYOUT>
__device__ __forceinline__ void quad_tap_addresses(const TexDesc& d, const Axis& U, const Axis& V, const Axis& S,
                                                   const Axis& T, int64_t (&pl)[4], int (&o)[4]) {
    const int64_t P = d.plane;
    const int64_t p00 = (int64_t)(T.k0 * d.n + S.k0) * P;
    const int64_t ds = (int64_t)(S.k1 - S.k0) * P, dt = (int64_t)(T.k1 - T.k0) * d.n * P;
    pl[0] = p00;
    pl[1] = p00 + ds;
    pl[2] = p00 + dt;
    pl[3] = p00 + dt + ds;
    bucket_slots4<LAYOUT>(d, U.k0, U.k1, V.k0, V.k1, o);
}

// The colour of 16 taps q[bucket][texel]: lerps in s, t, then u, v.
__device__ __forceinline__ P4 quadrilinear_combine(const P4 (&q)[4][4], const Axis& U, const Axis& V, const Axis& S,
                                                   const Axis& T) {
    const f32x2 ws = pack2(S.w, S.w), wt = pack2(T.w, T.w), wu = pack2(U.w, U.w), wv = pack2(V.w, V.w);
    P4 c[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) c[b] = lerpP(lerpP(q[b][0], q[b][1], ws), lerpP(q[b][2], q[b][3], ws), wt);
    return lerpP(lerpP(c[0], c[1], wu), lerpP(c[2], c[3], wu), wv);
}

// The same from FP16 / BF16 codes, bit for bit.
template <int FMT>
__device__ __forceinline__ P4 quadrilinear_combine_codes(const uint2 (&q)[4][4], const Axis& U, const Axis& V,
                                                         const Axis& S, const Axis& T) {
    const f32x2 ws = pack2(S.w, S.w), wt = pack2(T.w, T.w), wu = pack2(U.w, U.w), wv = pack2(V.w, V.w);
    P4 c[4];
#pragma unroll
    for (int b = 0; b < 4; ++b)
        c[b] = lerpP(lerp8<FMT>(q[b][0], q[b][1], ws), lerp8<FMT>(q[b][2], q[b][3], ws), wt);
    return lerpP(lerpP(c[0], c[1], wu), lerpP(c[2], c[3], wu), wv);
}

template <int FMT, int LAYOUT>
__device__ __forceinline__ P4 quadrilinear_planes(const TexDesc& d, const Axis& U, const Axis& V, const Axis& S,
                                                  const Axis& T) {
    int64_t pl[4];
    int o[4];
    quad_tap_addresses<LAYOUT>(d, U, V, S, T, pl, o);
    if constexpr (FMT == RT_F16 || FMT == RT_BF16) {
        uint2 code[4][4];
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int k = 0; k < 4; ++k)
                code[b][k] = __ldg(reinterpret_cast<const uint2*>(d.base) + checked_texel(d, pl[k] + o[b]));
        return quadrilinear_combine_codes<FMT>(code, U, V, S, T);
    }
    float sc[4] = {1.f, 1.f, 1.f, 1.f};
    if (FMT == RT_E4M3_BUCKET_SCALE) {
#pragma unroll
        for (int k = 0; k < 4; ++k) sc[k] = __ldg(d.scale + o[k]);
    }
    P4 q[4][4];  // [bucket][texel]
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int k = 0; k < 4; ++k) q[b][k] = load_texelP<FMT>(d.base, checked_texel(d, pl[k] + o[b]), sc[b]);
    return quadrilinear_combine(q, U, V, S, T);
}

template <int FILTER, int FMT, int LAYOUT>
__device__ __forceinline__ float4 filter_taps(const TexDesc& d, const Lookup<FILTER>& L) {
    if (FILTER == RT_NEAREST) {
        float sc = 1.0f;
        if (FMT == RT_E4M3_BUCKET_SCALE) sc = __ldg(d.scale + bucket_slot<LAYOUT>(d, L.u.k0, L.v.k0));
        return toF4(load_texelP<FMT>(d.base, texel_index<LAYOUT>(d, L.u.k0, L.v.k0, L.s.k0, L.t.k0), sc));
    } else if (FILTER == RT_ANGULAR_BILINEAR) {
        P4 a, b, c, e;
        load_quadP<FMT, LAYOUT>(d, L.u.k0, L.v.k0, L.s, L.t, a, b, c, e);
        const f32x2 ws = pack2(L.s.w, L.s.w), wt = pack2(L.t.w, L.t.w);
        return toF4(lerpP(lerpP(a, b, ws), lerpP(c, e, ws), wt));
    } else if (LAYOUT != RT_LAYOUT_ATLAS) {
        return toF4(quadrilinear_planes<FMT, LAYOUT>(d, L.u, L.v, L.s, L.t));
    } else {
        P4 q[2][2][4];
#pragma unroll
        for (int bv = 0; bv < 2; ++bv)
#pragma unroll
            for (int au = 0; au < 2; ++au)
                load_quadP<FMT, LAYOUT>(d, au ? L.u.k1 : L.u.k0, bv ? L.v.k1 : L.v.k0, L.s, L.t, q[bv][au][0],
                                        q[bv][au][1], q[bv][au][2], q[bv][au][3]);
        const f32x2 ws = pack2(L.s.w, L.s.w), wt = pack2(L.t.w, L.t.w), wu = pack2(L.u.w, L.u.w),
                    wv = pack2(L.v.w, L.v.w);
        P4 y[2];
#pragma unroll
        for (int bv = 0; bv < 2; ++bv) {
            P4 c[2];
#pragma unroll
            for (int au = 0; au < 2; ++au)
                c[au] = lerpP(lerpP(q[bv][au][0], q[bv][au][1], ws), lerpP(q[bv][au][2], q[bv][au][3], ws), wt);
            y[bv] = lerpP(c[0], c[1], wu);
        }
        return toF4(lerpP(y[0], y[1], wv));
    }
}

// How the bit textures of a context are indexed: planes of whole words and fewer
// than 2^32 texels, any planes with fewer than 2^32 texels, or any.
enum { kBitsNone = 0, kBitsWords = 1, kBitsSmall = 2, kBitsLarge = 3 };

// The value of a lookup in a bit texture (PLANES, clamp), equal in its four
// channels: the nested lerps of filter_taps on one number.  The two buckets of a
// row at one in-bucket texel are neighbouring bits, nearly always of one word;
// the pair is filtered as a packed pair.  With planes of whole words a row lies
// at the same bit of its word in all four planes.
template <int FILTER, int KIND>
__device__ __forceinline__ float filter_bits(const TexDesc& d, const Lookup<FILTER>& L) {
    using Idx = typename std::conditional<KIND == kBitsLarge, int64_t, uint32_t>::type;
    const unsigned* words = reinterpret_cast<const unsigned*>(d.base);
    auto value = [](unsigned bits) { return __uint_as_float((bits & 1u) * 0x3f800000u); };  // 0.0f or 1.0f
    auto lerpf = [](float a, float b, float w) { return fmaf(w, b - a, a); };
    const Idx P = (Idx)d.plane, p00 = (Idx)(L.t.k0 * d.n + L.s.k0) * P;
    const Idx o0 = (Idx)bucket_slot<RT_LAYOUT_PLANES>(d, L.u.k0, L.v.k0);
    auto texel = [&](Idx o) {
        const Idx e = (Idx)checked_texel(d, (int64_t)o);
        return value(__ldg(words + (e >> 5)) >> ((unsigned)e & 31u));
    };
    if constexpr (FILTER == RT_NEAREST) return texel(p00 + o0);
    const Idx ds = (Idx)(L.s.k1 - L.s.k0) * P, dt = (Idx)((L.t.k1 - L.t.k0) * d.n) * P;
    const Idx pl[4] = {p00, p00 + ds, p00 + dt, p00 + dt + ds};
    if constexpr (FILTER == RT_ANGULAR_BILINEAR) {
        return lerpf(lerpf(texel(pl[0] + o0), texel(pl[1] + o0), L.s.w),
                     lerpf(texel(pl[2] + o0), texel(pl[3] + o0), L.s.w), L.t.w);
    } else {
        const Idx o1 = (Idx)bucket_slot<RT_LAYOUT_PLANES>(d, L.u.k0, L.v.k1);
        const unsigned u1 = (unsigned)(L.u.k1 - L.u.k0);  // 0 (clamped) or 1
        const f32x2 ws = pack2(L.s.w, L.s.w), wt = pack2(L.t.w, L.t.w);
        float row[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const Idx o = r ? o1 : o0;
            f32x2 q[4];
#ifdef RADTEX_CHECKED
            // every tap by itself: a checked index decides which bit is read
#pragma unroll
            for (int k = 0; k < 4; ++k) q[k] = pack2(texel(pl[k] + o), texel(pl[k] + o + u1));
#else
            unsigned lo[4], hi[4], sh[4];  // the word of the first bucket's bit, the next one's, the bit
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const Idx a = pl[k] + o;
                if (KIND == kBitsWords) {
                    lo[k] = __ldg(words + ((pl[k] >> 5) + (o >> 5)));
                    sh[k] = (unsigned)o & 31u;
                } else {
                    lo[k] = __ldg(words + (a >> 5));
                    sh[k] = (unsigned)a & 31u;
                }
                hi[k] = lo[k];
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (u1 == 1u && sh[k] == 31u) hi[k] = __ldg(words + ((pl[k] + o + 1) >> 5));
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const unsigned x = __funnelshift_r(lo[k], hi[k], sh[k]);  // the two bits, lowest first
                q[k] = pack2(value(x), value(x >> u1));
            }
#endif
            const float2 c = unpack2(lerp2(lerp2(q[0], q[1], ws), lerp2(q[2], q[3], ws), wt));
            row[r] = lerpf(c.x, c.y, L.u.w);
        }
        return lerpf(row[0], row[1], L.v.w);
    }
}

// Dispatch on the object's storage format and layout: owned textures are
// QUADS (bit textures PLANES) or palettes; only a borrowed buffer, always
// FP32, may also be ATLAS or PLANES.
template <int FILTER, int FMT>
__device__ __forceinline__ float4 filter_dense(const TexDesc& d, const Lookup<FILTER>& L) {
    if (d.layout == kLayoutPalette) return filter_taps<FILTER, FMT, kLayoutPalette>(d, L);
    if (FMT == RT_BIT1) return filter_taps<FILTER, FMT, RT_LAYOUT_PLANES>(d, L);
    if (FMT != RT_F32 || d.layout == RT_LAYOUT_QUADS) return filter_taps<FILTER, FMT, RT_LAYOUT_QUADS>(d, L);
    return filter_taps<FILTER, FMT, RT_LAYOUT_PLANES>(d, L);
}

template <int FILTER>
__device__ __forceinline__ float4 filter_any(const TexDesc& d, const Lookup<FILTER>& L) {
    switch (d.fmt) {
        case RT_F16:
            return filter_dense<FILTER, RT_F16>(d, L);
        case RT_BF16:
            return filter_dense<FILTER, RT_BF16>(d, L);
        case RT_E4M3_BUCKET_SCALE:
            return filter_dense<FILTER, RT_E4M3_BUCKET_SCALE>(d, L);
        case RT_BIT1:
            return filter_dense<FILTER, RT_BIT1>(d, L);
        default:
            if (d.layout == RT_LAYOUT_ATLAS) return filter_taps<FILTER, RT_F32, RT_LAYOUT_ATLAS>(d, L);
            return filter_dense<FILTER, RT_F32>(d, L);
    }
}

// SPEC: -1 = any objects (format, layout, palette and repeat mode dispatched
// per fragment); a format = every object of the table is a dense QUADS
// texture of that format in clamp mode, a format + kSpecPalette = a palette of
// that format in clamp mode, so the fragment code is one path (the host picks
// the instantiation from the table).
constexpr int kSpecPalette = 16;

template <int FILTER, int SPEC>
__device__ __forceinline__ float4 filter_spec(const TexDesc& d, const Lookup<FILTER>& L) {
    if constexpr (SPEC < 0)
        return filter_any<FILTER>(d, L);
    else
        return filter_taps<FILTER, SPEC % kSpecPalette, SPEC < kSpecPalette ? RT_LAYOUT_QUADS : kLayoutPalette>(d, L);
}

// G-buffer staging.  Kernels that walk fragments are persistent: each warp
// takes 32-fragment chunks c, c + (warps in the grid), ...  and double-buffers
// them in its own slice of shared memory.  While the warp filters chunk c, the
// G-buffer of its next chunk is already in flight with 16-byte cp.async copies
// that bypass L1 -- so the DRAM latency of the G-buffer overlaps the texel
// gather, and no block-wide barrier is needed.
// Only __syncwarp orders the warp's own copies and reads.
//
// A chunk is either 32 consecutive fragments of the flat stream (rt_shade), or
// a tw x th screen tile of a batch of frames (rt_shade_batched): fragment
// (view, y, x) of views x H x W frames.  A block's warps take the tw x th
// sub-tiles of one bx x by block tile, so the warps that share an SM's L1 work
// on one compact screen region: vertically adjacent fragments read the same
// bucket rows.  Block tiles are visited in raster order, frame after frame.
constexpr int kChunk = 32;

// Division of a non-negative 31-bit integer by a fixed divisor d >= 1 with a
// multiply and a shift (the divisor's "magic" reciprocal is prepared on the
// host): q = umulhi(n, mul) >> shift, with shift = ceil(log2 d) and
// mul = ceil(2^(32 + shift) / d) - 2^32 handled as below for d = 1.
struct FastDiv {
    uint32_t d, mul, shift;
    __host__ __device__ __forceinline__ uint32_t div(uint32_t n) const {
        // q = (umulhi(n, mul) + n) >> shift, with the 33-bit sum taken in 64 bits
#ifdef __CUDA_ARCH__
        const uint32_t hi = __umulhi(n, mul);
#else
        const uint32_t hi = (uint32_t)(((uint64_t)n * mul) >> 32);
#endif
        return (uint32_t)(((uint64_t)hi + n) >> shift);
    }
};

// Prepares a FastDiv for divisor d >= 1 (exact for every n < 2^31).
__host__ __device__ inline FastDiv make_fastdiv(uint32_t d) {
    FastDiv f;
    f.d = d;
    uint32_t s = 0;
    while (s < 32 && (1ull << s) < d) ++s;
    f.shift = s;
    // mul = floor(2^32 (2^s - d) / d) + 1
    f.mul = (uint32_t)((((1ull << s) - d) << 32) / d + 1);
    return f;
}

struct Tiling {
    int32_t W, H, views;  // frame size and count; W = H = 0 selects the flat stream
    int32_t tw, th;       // warp tile, tw * th = 32, tw a multiple of 4
    int32_t bx, by;       // block tile in warp tiles, bx * by = warps per block
    int32_t btx, bty;     // block tiles per frame row / column
    int32_t tw_log2, bx_log2;
    FastDiv div_btx, div_frame;  // by btx, by btx * bty
    int64_t frame;        // W * H
};

// A warp's G-buffer buffers: the chunk being processed plus STAGES - 1
// prefetched ones.  A chunk is 24 pieces of 16 bytes of dir, 16 of uv and 8 of
// obj, in fragment order, then optionally a 16-byte-per-fragment extra stream
// such as dL/dout and (NRM) a second three-float stream, the normal of the
// world-space lookup.
template <bool EXTRA, int STAGES = 2, bool NRM = false>
struct __align__(16) WarpStage {
    static constexpr int kDir = 0, kUv = 12 * kChunk, kObj = 20 * kChunk, kExtra = 24 * kChunk;
    static constexpr int kNrm = kExtra + (EXTRA ? 16 * kChunk : 0);
    static constexpr int kBytes = kNrm + (NRM ? 12 * kChunk : 0);
    char b[STAGES][kBytes];
};

struct Frag {
    float u, v, x, y, z;
    int o;
    float nx, ny, nz;  // NRM streams only
};

// Asynchronous copies of BYTES (4 or 8 through L1, 16 past it) to shared address s.
template <int BYTES>
__device__ __forceinline__ void cp_async(unsigned s, const void* gmem) {
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(s), "l"(gmem), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// One chunk: the first fragment of its first row, whether all of it can be
// copied in aligned 16-byte pieces, and this lane's fragment (-1 = none).
struct Chunk {
    int64_t row0;
    int64_t f;
    bool fast;
};

// The chunks of one warp, in order.  Tiled: block tiles blockIdx.x,
// blockIdx.x + gridDim.x, ... in raster order, frame after frame, this warp's
// tile of each; the step is taken in tile coordinates, so that a chunk costs a
// few additions and no division.  Flat: 32-fragment runs.
template <int WARPS, bool TILED>
struct ChunkWalk {
    int tx, ty, view, dx, dy, dv;  // block tile and step (tiled)
    int wx, wy, lx, ly;            // this warp's tile in the block tile, this lane in the tile
    int64_t c, dc;                 // chunk and step (flat)
    int64_t count;                 // chunks left to hand out

    __device__ __forceinline__ ChunkWalk(const Tiling& T, int64_t F, int lane, int w) {
        if constexpr (TILED) {
            const uint32_t bt = blockIdx.x, step = gridDim.x;
            tiles(T, bt, tx, ty, view);
            tiles(T, step, dx, dy, dv);
            const int64_t total = (int64_t)T.btx * T.bty * T.views;
            count = bt < total ? (int64_t)((uint32_t)(total - 1 - bt) / step + 1) : 0;
            wx = (w & (T.bx - 1)) << T.tw_log2;
            wy = (w >> T.bx_log2) * T.th;
            lx = lane & (T.tw - 1);
            ly = lane >> T.tw_log2;
        } else {
            c = (int64_t)blockIdx.x * WARPS + w;
            dc = (int64_t)gridDim.x * WARPS;
            const int64_t total = (F + kChunk - 1) / kChunk;
            count = c < total ? (total - 1 - c) / dc + 1 : 0;
        }
    }

    __device__ __forceinline__ static void tiles(const Tiling& T, uint32_t n, int& x, int& y, int& v) {
        const uint32_t q = T.div_frame.div(n), r = n - q * T.div_frame.d, ry = T.div_btx.div(r);
        v = (int)q;
        y = (int)ry;
        x = (int)(r - ry * T.div_btx.d);
    }

    // The next chunk (any values once count is used up).
    __device__ __forceinline__ Chunk next(const Tiling& T, int64_t F, int lane) {
        Chunk g;
        if constexpr (TILED) {
            const int x0 = (tx * T.bx << T.tw_log2) + wx, y0 = ty * (T.by * T.th) + wy;
            g.row0 = (int64_t)view * T.frame + ((int64_t)y0 * T.W + x0);
            const bool whole = x0 + T.tw <= T.W && y0 + T.th <= T.H;
            g.fast = whole && (T.W & 3) == 0;
            g.f = whole || (x0 + lx < T.W && y0 + ly < T.H) ? g.row0 + (ly * T.W + lx) : -1;
            tx += dx;
            ty += dy;
            view += dv;
            if (tx >= T.btx) {
                tx -= T.btx;
                ++ty;
            }
            if (ty >= T.bty) {
                ty -= T.bty;
                ++view;
            }
        } else {
            g.row0 = c * kChunk;
            g.fast = g.row0 + kChunk <= F;
            g.f = g.row0 + lane < F ? g.row0 + lane : -1;
            c += dc;
        }
        return g;
    }
};

// This lane's share of a chunk's copies.  Piece q of a chunk (0-23 dir, 24-39
// uv, 40-47 obj) is 16 bytes of one stream, all in one tile row; lanes take
// pieces lane and lane + 32.  A piece starts at p + m row0 bytes: m is the
// stream's bytes per fragment, and p holds the rest, fixed for the launch.
struct LaneCopy {
    const char* p;
    uint32_t m;

    __device__ __forceinline__ LaneCopy(const float* dir, const float* uv, const int32_t* obj, int q, int tw_log2,
                                        int64_t pitch) {
        const int k = q < 24 ? 3 : q < 40 ? 2 : 1;             // values per fragment
        const int e = 4 * (q - (q < 24 ? 0 : q < 40 ? 24 : 40));  // first value of the piece
        const int row = (e / k) >> tw_log2;
        const char* base = reinterpret_cast<const char*>(q < 24 ? (const void*)dir : q < 40 ? (const void*)uv : obj);
        p = base + 4 * (k * ((int64_t)row * pitch) + (e - k * (row << tw_log2)));
        m = 4 * k;
    }
    __device__ __forceinline__ const void* at(int64_t row0) const { return p + row0 * (int64_t)m; }
};

// Issues the copies of one chunk into the buffer at shared address s.  A chunk
// that crosses the frame's edge or has unaligned rows is copied fragment by
// fragment, each lane its own; lanes without a fragment become background.
template <bool EXTRA, int STAGES, bool NRM>
__device__ __forceinline__ void stage_chunk(const float* __restrict__ uv, const float* __restrict__ dir,
                                            const int32_t* __restrict__ obj, const float* __restrict__ extra,
                                            const float* __restrict__ nrm, const Chunk& g, const LaneCopy& c0,
                                            const LaneCopy& c1, unsigned s, int lane) {
    using S = WarpStage<EXTRA, STAGES, NRM>;
    if (g.fast) {
        cp_async<16>(s + 16 * lane, c0.at(g.row0));
        if (lane < 16) cp_async<16>(s + 512 + 16 * lane, c1.at(g.row0));
        if (NRM && lane < 24)  // the pieces of nrm lie as those of dir
            cp_async<16>(s + S::kNrm + 16 * lane, reinterpret_cast<const char*>(c0.at(g.row0)) +
                                                      (reinterpret_cast<const char*>(nrm) -
                                                       reinterpret_cast<const char*>(dir)));
        if (EXTRA) cp_async<16>(s + S::kExtra + 16 * lane, extra + 4 * g.f);
    } else if (g.f >= 0) {
        const int64_t f = g.f;
        cp_async<8>(s + S::kUv + 8 * lane, uv + 2 * f);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            cp_async<4>(s + S::kDir + 12 * lane + 4 * k, dir + 3 * f + k);
            if (NRM) cp_async<4>(s + S::kNrm + 12 * lane + 4 * k, nrm + 3 * f + k);
        }
        cp_async<4>(s + S::kObj + 4 * lane, obj + f);
        if (EXTRA) cp_async<16>(s + S::kExtra + 16 * lane, extra + 4 * f);
    } else {
        asm volatile("st.shared.b32 [%0], %1;" ::"r"(s + S::kObj + 4 * lane), "r"(-1) : "memory");
    }
}

template <bool EXTRA, int STAGES, bool NRM>
__device__ __forceinline__ Frag read_frag(const char* S, int lane) {
    using St = WarpStage<EXTRA, STAGES, NRM>;
    Frag r;
    const float2 q = reinterpret_cast<const float2*>(S + St::kUv)[lane];
    const float* d = reinterpret_cast<const float*>(S + St::kDir) + 3 * lane;
    r.u = q.x;
    r.v = q.y;
    r.x = d[0];
    r.y = d[1];
    r.z = d[2];
    r.o = reinterpret_cast<const int*>(S + St::kObj)[lane];
    r.nx = r.ny = r.nz = 0.f;
    if (NRM) {
        const float* n = reinterpret_cast<const float*>(S + St::kNrm) + 3 * lane;
        r.nx = n[0];
        r.ny = n[1];
        r.nz = n[2];
    }
    return r;
}

// Runs body(f, frag, extra) with all 32 lanes of the warp, one fragment per
// lane, persistent over the grid, with the G-buffer of the next STAGES - 1
// chunks prefetched.  Lanes without a fragment get a background fragment
// (object id -1, other inputs arbitrary) and f = -1: the body must not store
// for them.  WARPS = warps per block; the block's shared memory holds WARPS
// stages.  Bound of the shading kernels: issue and latency, so what a chunk costs
// beside its lookups counts: with the tile found by division and each stream's
// addresses formed per chunk the 1080p FP16 quadrilinear forward took 360
// instructions per chunk, with the walk and the lane's pointers 316 (20 poses:
// 0.586 -> 0.498 ms).
template <int WARPS, bool EXTRA, bool TILED, int STAGES, bool NRM = false, typename Body>
__device__ __forceinline__ void for_each_fragment(const float* __restrict__ uv, const float* __restrict__ dir,
                                                  const int32_t* __restrict__ obj, const float* __restrict__ extra,
                                                  int64_t F, const Tiling& T, WarpStage<EXTRA, STAGES, NRM>* stages,
                                                  Body body, const float* __restrict__ nrm = nullptr) {
    using St = WarpStage<EXTRA, STAGES, NRM>;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const char* S = stages[w].b[0];
    const unsigned s0 = (unsigned)__cvta_generic_to_shared(S);
    ChunkWalk<WARPS, TILED> walk(T, F, lane, w);
    const int lg = TILED ? T.tw_log2 : 5;
    const LaneCopy c0(dir, uv, obj, lane, lg, TILED ? T.W : 0), c1(dir, uv, obj, lane + 32, lg, TILED ? T.W : 0);
    // fk[k]: this lane's fragment of the k-th chunk from the current one, staged in buffer (b + k) % STAGES
    int64_t fk[STAGES];
#pragma unroll
    for (int k = 0; k < STAGES - 1; ++k) {
        const Chunk g = walk.next(T, F, lane);
        if (k < walk.count) stage_chunk<EXTRA, STAGES, NRM>(uv, dir, obj, extra, nrm, g, c0, c1, s0 + k * St::kBytes, lane);
        cp_async_commit();
        fk[k] = g.f;
    }
    int b = 0;
    for (int64_t left = walk.count; left > 0; --left) {
        const Chunk g = walk.next(T, F, lane);
        const int bl = b + STAGES - 1 >= STAGES ? b - 1 : b + STAGES - 1;  // (b + STAGES - 1) % STAGES
        if (left > STAGES - 1)
            stage_chunk<EXTRA, STAGES, NRM>(uv, dir, obj, extra, nrm, g, c0, c1, s0 + bl * St::kBytes, lane);
        cp_async_commit();
        fk[STAGES - 1] = g.f;
        cp_async_wait<STAGES - 1>();  // the current chunk has landed (newer groups may still be in flight)
        __syncwarp();
        const Frag q = read_frag<EXTRA, STAGES, NRM>(S + b * St::kBytes, lane);
        float4 e = make_float4(0.f, 0.f, 0.f, 0.f);
        if (EXTRA) e = reinterpret_cast<const float4*>(S + b * St::kBytes + St::kExtra)[lane];
        __syncwarp();  // every lane has read buffer b before it is refilled
        body(fk[0], q, e);
#pragma unroll
        for (int k = 0; k < STAGES - 1; ++k) fk[k] = fk[k + 1];
        b = b + 1 == STAGES ? 0 : b + 1;
    }
    cp_async_wait<0>();
}

// Validity of one fragment: 1 = shade it, 0 = background or invalid (status
// bits raised for invalid ones).
__device__ __forceinline__ bool fragment_valid(const TexDesc* __restrict__ table, int n_obj, int o, float u, float v,
                                               float x, float y, float z, unsigned* status, TexDesc& d) {
    if (o < 0) return false;
    if (o >= n_obj) {
        atomicOr(status, ST_BAD_OBJ);
        return false;
    }
    d = load_desc(table, o);
    if (!d.live) {
        atomicOr(status, ST_BAD_OBJ);
        return false;
    }
    // 0 * t is 0 for finite t and NaN for an infinity or a NaN: one test covers all five inputs
    const float probe = fmaf(z, 0.f, fmaf(y, 0.f, fmaf(x, 0.f, fmaf(v, 0.f, u * 0.f))));
    if (probe != 0.f) {
        atomicOr(status, ST_NONFINITE);
        return false;
    }
    return true;
}

// A world-space fragment's normal must be finite (status bit otherwise).
__device__ __forceinline__ bool normal_valid(float3 N, unsigned* status) {
    const float probe = fmaf(N.z, 0.f, fmaf(N.y, 0.f, N.x * 0.f));
    if (probe != 0.f) {
        atomicOr(status, ST_NONFINITE);
        return false;
    }
    return true;
}

}  // namespace rt
