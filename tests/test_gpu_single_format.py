"""GPU: contexts of one storage format, dense or palettes, which run single-format
kernels, against contexts that hold an object of another format besides, whose
kernels dispatch per fragment.

The per-fragment arithmetic is the same, so colours and the UV, direction and
normal gradients are bit-identical; texel gradients differ by the order of FP32
atomic additions: within 1e-4 of the sum of w |g|."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_2301_01719_gb300 import api
from parity_util import FILTERS, to_dev

pytestmark = pytest.mark.gpu

FORMATS = [api.RT_F32, api.RT_F16, api.RT_BF16, api.RT_E4M3_BUCKET_SCALE]
SHAPES = [(2, 50, 60), (1, 33, 201), (1, 7, 3)]  # rows of whole 16-byte pieces, ragged rows, less than one tile


def make(ctx, fmt, k, palette, flags=0):
    """An object of 37 x 23 buckets (odd sides: padded quads), from 9 palette buckets if `palette`."""
    W, H, n, K = 37, 23, 8, 9
    if not palette:
        src = to_dev(oracle.fill_field(W, H, n, synth.field_lobes(900 + k)))
        return api.rt_create_texture(ctx, W, H, n, fmt, api.RT_LAYOUT_ATLAS, src, flags)
    src = to_dev(oracle.fill_field(K, 1, n, synth.field_lobes(900 + k)))
    index = np.random.default_rng(k).integers(0, K, (H, W)).astype(np.int32)
    return api.rt_create_palette_texture(ctx, W, H, n, K, fmt, api.RT_LAYOUT_ATLAS, src, to_dev(index), flags)


def frames(shape, oids):
    V, H, W = shape
    g = synth.sphere_plane_scene(1002, views=V, width=W, height=H)
    obj = np.where(g.obj >= 0, np.array(oids, np.int32)[np.maximum(g.obj, 0)], -1).astype(np.int32)
    rng = np.random.default_rng(3)
    N = np.concatenate([rng.normal(scale=0.3, size=(V * H * W, 2)), np.ones((V * H * W, 1))], 1)
    N = (N / np.linalg.norm(N, axis=1, keepdims=True)).astype(np.float32)
    uv = (1.1 * g.uv - 0.05).astype(np.float32)  # past both edges
    return (to_dev(uv).reshape(V, H, W, 2), to_dev(g.dir).reshape(V, H, W, 3), to_dev(N).reshape(V, H, W, 3),
            to_dev(obj).reshape(V, H, W))


@pytest.fixture
def pair():
    """A context of the case's objects alone, and one that gets an object of another format as well."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2301_01719_gb300 import build

    build.build()
    c = [api.Context(0), api.Context(0)]
    yield c
    for x in c:
        x.close()


def objects(pair, fmt, palettes, flags=(0, 0)):
    for c in pair:
        oids = [make(c, fmt, k, palettes[k], flags[k]) for k in range(2)]
    make(pair[1], api.RT_F32 if fmt != api.RT_F32 else api.RT_F16, 2, False)
    return oids


@pytest.mark.parametrize("palettes,flags", [((False, False), (0, 0)), ((True, True), (0, 0)), ((True, False), (0, 0)),
                                            ((True, True), (api.RT_WRAP_U, 0))])
@pytest.mark.parametrize("fmt", FORMATS)
def test_forward(pair, fmt, palettes, flags):
    """(Dense beside palette and a repeating palette take the dispatching kernel in both contexts.)"""
    oids = objects(pair, fmt, palettes, flags)
    for shape in SHAPES:
        uv, d, N, o = frames(shape, oids)
        flat = uv.reshape(-1, 2), d.reshape(-1, 3), N.reshape(-1, 3), o.reshape(-1)
        for filt in FILTERS:
            got, ref = ([api.rt_shade(c, flat[0], flat[1], flat[3], filt),
                         api.rt_shade_batched(c, uv, d, o, filt).reshape(-1, 4),
                         api.rt_shade_world(c, *flat, filt),
                         api.rt_shade_world_batched(c, uv, d, N, o, filt).reshape(-1, 4)] for c in pair)
            for x, y in zip(got, ref):
                assert torch.equal(x, y)
            assert torch.equal(got[0], got[1]) and torch.equal(got[2], got[3])
    assert api.rt_get_error(pair[0]) == api.RT_OK


@pytest.mark.parametrize("fmt", FORMATS)
@pytest.mark.parametrize("palette", [False, True])
def test_world_backward(pair, fmt, palette):
    oids = objects(pair, fmt, (palette, palette))
    for shape in SHAPES:
        uv, d, N, o = frames(shape, oids)
        gout = to_dev(np.random.default_rng(2).normal(size=(*shape, 4)).astype(np.float32))
        for filt in FILTERS:

            def run(c, g):
                duv, ddir, dnrm = torch.empty_like(uv), torch.empty_like(d), torch.empty_like(d)
                dt = {k: torch.empty(api.storage_numel(c, k), device=uv.device) for k in oids}
                api.rt_shade_world_batched_backward(c, uv, d, N, o, filt, g, dt, duv, ddir, dnrm)
                return (duv, ddir, dnrm), dt

            (a, at), (b, bt), (_, weight) = run(pair[0], gout), run(pair[1], gout), run(pair[1], gout.abs())
            for x, y in zip(a, b):
                assert torch.equal(x, y)
            for k in oids:
                assert bool(((at[k] - bt[k]).abs() <= 1e-4 * weight[k]).all())
    assert api.rt_get_error(pair[0]) == api.RT_OK


@pytest.mark.parametrize("fmt,dtype", [(api.RT_F16, torch.float16), (api.RT_BF16, torch.bfloat16)])
def test_16_bit_codes_shade_as_their_values(pair, fmt, dtype):
    """An FP16 / BF16 texture shades, bit for bit, as an FP32 one of the same values: widening is
    exact.  Random codes: every magnitude, subnormals, infinities (no NaN)."""
    W, H, n = 37, 23, 8
    rng = np.random.default_rng(11)
    codes = torch.from_numpy(rng.integers(-32768, 32768, (n, n, H, W, 4)).astype(np.int16)).view(dtype)
    values = torch.where(codes.isnan(), torch.zeros_like(codes), codes).float().to("cuda")
    for c, f in ((pair[0], fmt), (pair[1], api.RT_F32)):
        api.rt_create_texture(c, W, H, n, f, api.RT_LAYOUT_PLANES, values)
        api.rt_create_texture(c, W, H, n, f, api.RT_LAYOUT_PLANES, values.flip(2))
    for shape in SHAPES:
        uv, d, N, o = frames(shape, [0, 1])
        for filt in FILTERS:
            a, b = (torch.stack([api.rt_shade_batched(c, uv, d, o, filt),
                                 api.rt_shade_world_batched(c, uv, d, N, o, filt)]) for c in pair)
            assert torch.allclose(a, b, rtol=0.0, atol=0.0, equal_nan=True)
