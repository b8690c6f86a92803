"""rt_shade_multi on contexts of bit textures alone against the dispatching kernels, which run as
soon as the context holds an object of another format: the same colours bit for bit, for every
filter, sample counts that do and do not divide a warp, odd sizes and invalid samples."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_2301_01719_gb300 import api
from parity_util import COLOUR_TOL, floor_mismatch

pytestmark = pytest.mark.gpu

FILTERS = [api.RT_NEAREST, api.RT_ANGULAR_BILINEAR, api.RT_QUADRILINEAR]


def _inputs(F, S, seed, objects):
    rng = np.random.default_rng(seed)
    uv = rng.uniform(-0.1, 1.1, (F, 2)).astype(np.float32)  # beyond both edges
    d = rng.standard_normal((F, S, 3)).astype(np.float32)
    d[..., 2] = np.abs(d[..., 2])
    d /= np.linalg.norm(d, axis=-1, keepdims=True)
    obj = rng.integers(-1, objects, F).astype(np.int32)
    return uv, d, obj


def _both(sizes, seed, uv, d, obj, filt, fill=None):
    """The call on a context of bit textures, then with an FP32 object added: colours and statuses."""
    got = []
    with_other = (False, True)
    for other in with_other:
        ctx = api.Context(0)
        for k, (w, h, n) in enumerate(sizes):
            if fill is None:
                src = torch.rand(api.layout_shape(api.RT_LAYOUT_PLANES, w, h, n),
                                 generator=torch.Generator("cuda").manual_seed(seed + k), device="cuda")
                api.rt_create_texture(ctx, w, h, n, api.RT_BIT1, api.RT_LAYOUT_PLANES, src)
            else:
                fill(ctx, api.rt_create_texture(ctx, w, h, n, api.RT_BIT1))
        if other:
            api.rt_create_texture(ctx, 1, 1, 1, api.RT_F32)
        out = api.rt_shade_multi(ctx, torch.from_numpy(uv).cuda(), torch.from_numpy(d).cuda(),
                                 torch.from_numpy(obj).cuda(), filt)
        got.append((out.cpu().numpy(), api.rt_get_error(ctx)))
        ctx.close()
    return got


@pytest.mark.parametrize("filt", FILTERS)
@pytest.mark.parametrize("S", [1, 2, 3, 4, 5, 7, 8, 11, 16, 31, 32, 33])
@pytest.mark.parametrize("sizes", [[(37, 23, 5), (64, 32, 8), (1, 1, 1)],  # planes of whole words or not,
                                   [(64, 32, 8), (37, 32, 3), (1, 32, 2)]])  # and all of whole words
def test_bit_contexts_match_the_dispatching_kernels(filt, S, sizes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    uv, d, obj = _inputs(1003, S, S, 3)
    (a, ea), (b, eb) = _both(sizes, 5, uv, d, obj, filt)
    np.testing.assert_array_equal(a.view(np.int32), b.view(np.int32))
    assert ea == eb == api.RT_OK and a.any() and not a[obj < 0].any()


@pytest.mark.parametrize("S", [3, 4])
def test_invalid_samples_zero_their_fragment(S):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    for where, status in (("direction", api.RT_ERR_NONFINITE), ("uv", api.RT_ERR_NONFINITE),
                          ("object", api.RT_ERR_BAD_OBJ_ID)):
        uv, d, obj = _inputs(257, S, 9, 1)
        obj[:] = 0
        if where == "direction":
            d[100, S - 1, 1] = np.nan
        elif where == "uv":
            uv[100, 0] = np.inf
        else:
            obj[100] = 900
        (a, ea), (b, eb) = _both([(16, 16, 4)], 6, uv, d, obj, api.RT_QUADRILINEAR)
        np.testing.assert_array_equal(a.view(np.int32), b.view(np.int32))
        assert ea == eb == status and not a[100].any()


def test_textures_of_2_to_the_32_texels_take_64_bit_indices():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    uv, d, obj = _inputs(40001, 4, 3, 1)
    obj[:] = 0
    scene = synth.bake_scene(11)

    def fill(ctx, oid):
        api.rt_bake_shadow(ctx, oid, api.RT_SURFACE_PLANE, scene)

    (a, ea), (b, eb) = _both([(65536, 16384, 2)], 0, uv, d, obj, api.RT_QUADRILINEAR, fill)
    np.testing.assert_array_equal(a.view(np.int32), b.view(np.int32))
    assert ea == eb == api.RT_OK and 0.0 < a.mean() < 1.0


@pytest.mark.parametrize("filt", FILTERS)
@pytest.mark.parametrize("S", [1, 2, 4, 8, 16, 32])
def test_many_fragments_sum_powers_of_two_as_the_lanes_do(filt, S):
    """Enough fragments for a thread each: the samples' tree of sums is that of the lanes, bit for bit."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    uv, d, obj = _inputs(100003, S, S, 2)
    (a, ea), (b, eb) = _both([(37, 23, 5), (64, 32, 8)], 5, uv, d, obj, filt)
    np.testing.assert_array_equal(a.view(np.int32), b.view(np.int32))
    assert ea == eb == api.RT_OK and a.any()


@pytest.mark.parametrize("filt", FILTERS)
def test_64_bit_indices_a_thread_per_fragment(filt):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    uv, d, obj = _inputs(10007, 3, 4, 1)
    obj[:] = 0
    scene = synth.bake_scene(11)

    def fill(ctx, oid):
        api.rt_bake_shadow(ctx, oid, api.RT_SURFACE_PLANE, scene)

    (a, ea), (b, eb) = _both([(65536, 16384, 2)], 0, uv, d, obj, filt, fill)
    np.testing.assert_array_equal(a.view(np.int32), b.view(np.int32))
    assert ea == eb == api.RT_OK and 0.0 < a.mean() < 1.0


WORDS = [(64, 32, 8), (37, 32, 3), (1, 32, 2)]  # planes of whole words
ANY = [(37, 23, 5), (64, 32, 8), (1, 1, 1)]


@pytest.mark.parametrize("sizes", [WORDS, ANY])
@pytest.mark.parametrize("S,filt,F", [
    (4, api.RT_QUADRILINEAR, 98303), (4, api.RT_QUADRILINEAR, 98304), (8, api.RT_NEAREST, 98304),
    (16, api.RT_QUADRILINEAR, 98304), (16, api.RT_NEAREST, 262143), (16, api.RT_NEAREST, 262144),
    (16, api.RT_ANGULAR_BILINEAR, 262144), (32, api.RT_ANGULAR_BILINEAR, 524287),
    (32, api.RT_ANGULAR_BILINEAR, 524288), (32, api.RT_NEAREST, 524288)])
def test_both_sides_of_the_few_fragments_rule(sizes, S, filt, F):
    """Where a lane per lookup gives way to a thread per fragment, by sample count and filter."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    uv, d, obj = _inputs(F, S, S, 3)
    (a, ea), (b, eb) = _both(sizes, 5, uv, d, obj, filt)
    np.testing.assert_array_equal(a.view(np.int32), b.view(np.int32))
    assert ea == eb == api.RT_OK and a.any() and not a[obj < 0].any()


@pytest.mark.parametrize("bad", ["first", "middle", "last", "uv", "object"])
@pytest.mark.parametrize("S", [4, 8])
@pytest.mark.parametrize("sizes", [WORDS, ANY])
def test_invalid_samples_with_a_thread_per_fragment(sizes, S, bad):
    """An invalid sample anywhere in a power of two of them zeroes its fragment and no other."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    uv, d, obj = _inputs(100003, S, 9, 3)
    at = np.arange(500, 100003, 5000)
    obj[at] = 1
    status = api.RT_ERR_BAD_OBJ_ID if bad == "object" else api.RT_ERR_NONFINITE
    if bad == "object":
        obj[at] = 900
    elif bad == "uv":
        uv[at, 1] = np.nan
    else:
        d[at, {"first": 0, "middle": S // 2, "last": S - 1}[bad], 2] = np.inf
    (a, ea), (b, eb) = _both(sizes, 6, uv, d, obj, api.RT_QUADRILINEAR)
    np.testing.assert_array_equal(a.view(np.int32), b.view(np.int32))
    assert ea == eb == status and not a[at].any() and a[at + 1].any()


@pytest.mark.parametrize("filt", FILTERS)
@pytest.mark.parametrize("S", [2, 4])
def test_64_bit_indices_with_a_tree_of_sums(S, filt):
    """2^32 texels, enough fragments for a thread each: power-of-two sample counts."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    uv, d, obj = _inputs(100003, S, 4, 1)
    obj[:] = 0
    scene = synth.bake_scene(11)

    def fill(ctx, oid):
        api.rt_bake_shadow(ctx, oid, api.RT_SURFACE_PLANE, scene)

    (a, ea), (b, eb) = _both([(65536, 16384, 2)], 0, uv, d, obj, filt, fill)
    np.testing.assert_array_equal(a.view(np.int32), b.view(np.int32))
    assert ea == eb == api.RT_OK and 0.0 < a.mean() < 1.0


@pytest.mark.parametrize("filt", FILTERS)
@pytest.mark.parametrize("W,H,S", [(64, 32, 4), (37, 23, 4), (64, 32, 16), (64, 32, 5)])
def test_thread_per_fragment_against_the_oracle(W, H, S, filt):
    """The mean of the oracle's single lookups, whole-word planes and others, tree and sequential sums;
    the last 2000 fragments of a call large enough for a thread each (S = 16: of 262 144).  Tolerance: a
    lookup of random bits changes by at most the sum of its coordinates' errors: 2^-19 and 2^-20 spatial
    (64 and 32 buckets, one rounding), 2e-6 in either in-bucket one (3 times some 8 roundings of B), 5e-7 for
    the lerps; a mean of lookups has no larger error than the worst, and its sum adds S 2^-24: below
    COLOUR_TOL in all."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n, F, T = 6, 262144 if S == 16 else 98304, 2000
    uv, d, obj = _inputs(F, S, W + S, 1)
    bits = np.random.default_rng(S).integers(0, 2, (H * n, W * n), dtype=np.uint8)
    ctx = api.Context(0)
    src = torch.from_numpy(np.repeat(bits[..., None], 4, axis=2).astype(np.float32)).cuda()
    oid = api.rt_create_texture(ctx, W, H, n, api.RT_BIT1, api.RT_LAYOUT_ATLAS, src)
    obj[obj >= 0] = oid
    out = api.rt_shade_multi(ctx, torch.from_numpy(uv).cuda(), torch.from_numpy(d).cuda(),
                             torch.from_numpy(obj).cuda(), filt)[-T:].cpu().numpy()
    table = [None] * oid + [oracle.bit_texture(bits, W, H, n)]
    uvS, dS, objS = np.repeat(uv[-T:], S, axis=0), d[-T:].reshape(-1, 3), np.repeat(obj[-T:], S)
    ref, flags = oracle.shade(table, uvS, dS, objS, filt)
    assert flags == 0
    mism = np.zeros(T, bool)  # the linear filters are continuous where floors differ
    if filt == api.RT_NEAREST:
        g = synth.GBuffer(uv=uvS, dir=dS, obj=objS, width=0, height=0, views=1)
        mism = floor_mismatch(ctx, g, objS, filt, table).reshape(T, S).any(axis=1)
        assert (~mism).mean() > 0.95
    assert np.abs(out - ref.reshape(T, S, 4).mean(axis=1))[~mism].max() <= COLOUR_TOL
    assert api.rt_get_error(ctx) == api.RT_OK and (out[:, 0] == out[:, 3]).all()
    ctx.close()
