"""The deterministic mode's arithmetic against exact integers: a contribution v becomes
round(v 2^32) to nearest even, and a sum a becomes the FP32 value
of the FP64 product a (2^-32 scale)."""
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_2301_01719_gb300 import api
from parity_util import storage_index

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = api.Context(0)
    yield c
    c.close()


def _half_even(x: Fraction) -> int:
    return round(x)  # Python rounds a Fraction to the nearest integer, ties to even


def test_contributions_round_to_nearest_even(ctx):
    """One fragment per texel under the nearest filter (weight 1): the sums are the rounded gradients."""
    rng = np.random.default_rng(7)
    w = h = 32
    g = rng.standard_normal((h * w, 4)) * 10.0 ** rng.uniform(-12, 9, (h * w, 4))
    g = g.astype(np.float32)
    edge = [0.0, 4096.0, np.nextafter(np.float32(4096), np.float32(5000)), -4096.0, 4095.9998, 2.0 ** 30, -(2.0 ** 30),
            1.5 * 2.0 ** -32, 2.5 * 2.0 ** -32, -0.5 * 2.0 ** -32, 0.5 * 2.0 ** -32, 2.0 ** -33 * 1.0000001, 2.0 ** -11,
            2.0 ** -10, 1.5 * 2.0 ** -10, 2.5 * 2.0 ** -10, 2.0 ** -11 + 2.0 ** -33, 2.0 ** -20 + 2.0 ** -33, 1e-30, -1.0]
    g.reshape(-1)[:len(edge)] = np.asarray(edge, np.float32)
    oid = api.rt_create_texture(ctx, w, h, 1, api.RT_F32)
    jj, ii = np.meshgrid(np.arange(h), np.arange(w), indexing="ij")
    uv = torch.from_numpy(np.stack([(ii.ravel() + 0.5) / w, (jj.ravel() + 0.5) / h], 1).astype(np.float32)).cuda()
    dirs = torch.tensor([[0.0, 0.0, 1.0]], device="cuda").repeat(h * w, 1)
    obj = torch.full((h * w,), oid, dtype=torch.int32, device="cuda")
    acc = torch.zeros(api.layout_shape(api.RT_LAYOUT_PLANES, w, h, 1), dtype=torch.int64, device="cuda")
    quads = torch.zeros(api.layout_shape(api.RT_LAYOUT_QUADS, w, h, 1), dtype=torch.int64, device="cuda")
    api.rt_shade_backward(ctx, uv, dirs, obj, api.RT_NEAREST, torch.from_numpy(g).cuda(), {oid: quads}, None, None,
                          api.RT_FIXED_POINT_GRADS)
    acc = quads.view(h // 2, w // 2, 2, 2, 4).permute(0, 2, 1, 3, 4).reshape(h * w, 4).cpu().numpy()
    want = [_half_even(Fraction(float(v)) * (1 << 32)) for v in g.reshape(-1)]
    assert [int(a) for a in acc.reshape(-1)] == want
    api.rt_destroy_texture(ctx, oid)


@pytest.mark.parametrize("scale", [1.0, -1.0, 1.0 / (4.0 * 15728640.0), 0.3, 1e-12, 7.25e10, 1e-36, 1e30, 1e300, 0.0])
@pytest.mark.parametrize("count", [1, 3, 4, 5, 1023, 4099])
def test_sums_convert_as_the_fp64_product(scale, count):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(count)
    a = (rng.uniform(-1.0, 1.0, count) * 2.0 ** rng.uniform(0, 62, count)).astype(np.int64)
    edge = [0, 1, -1, (1 << 24) + 1, (1 << 25) + 2, (1 << 25) + 6, -(1 << 53) - 1, (1 << 62) + (1 << 38), 1 << 40,
            (1 << 52) - 1, 1 << 52, -(1 << 52), -(1 << 52) + 1, -(1 << 63), (1 << 63) - 1]
    a[:len(edge)] = edge[:count]
    got = api.rt_fixed_to_float(torch.from_numpy(a).cuda(), scale=scale).cpu().numpy()
    with np.errstate(over="ignore"):
        want = (a.astype(np.float64) * (scale * 2.0 ** -32)).astype(np.float32)
    np.testing.assert_array_equal(got.view(np.int32), want.view(np.int32))
    base = torch.ones(count, device="cuda")
    api.rt_fixed_to_float(torch.from_numpy(a).cuda(), base, api.RT_ACCUMULATE, scale=scale)
    np.testing.assert_array_equal(base.cpu().numpy(), np.float32(1.0) + want)


@pytest.mark.parametrize("layout", [api.RT_LAYOUT_QUADS, api.RT_LAYOUT_PLANES, api.RT_LAYOUT_ATLAS])
@pytest.mark.parametrize("filt", [api.RT_NEAREST, api.RT_ANGULAR_BILINEAR, api.RT_QUADRILINEAR])
def test_sums_of_every_layout_are_the_rounded_products(ctx, layout, filt):
    """The sums of the flat, batched and fused calls, recomputed from the lookup's coordinates: a tap's
    weight is the FP32 product ((wu wv) ws) wt, in the ATLAS layout (wu wv) (ws wt), and its
    contribution round(weight g 2^32)."""
    w, h, n, V, H, W = 13, 9, 6, 1, 48, 64
    rng = np.random.default_rng(21 + filt)
    F = V * H * W
    shape = api.layout_shape(layout, w, h, n)
    numel = api.layout_numel(layout, w, h, n)
    tex = torch.from_numpy(rng.random(shape, dtype=np.float32)).cuda()
    oid = api.rt_create_texture(ctx, w, h, n, api.RT_F32, layout, tex, api.RT_BORROW)
    uv = torch.from_numpy(rng.uniform(-0.1, 1.1, (F, 2)).astype(np.float32)).cuda()
    d = rng.standard_normal((F, 3)).astype(np.float32)
    d[:, 2] = np.abs(d[:, 2])
    d = torch.from_numpy(d / np.linalg.norm(d, axis=1, keepdims=True)).cuda()
    obj = torch.full((F,), oid, dtype=torch.int32, device="cuda")
    obj[::7] = -1
    g = (rng.standard_normal((F, 4)) * 10.0 ** rng.uniform(-8, 5, (F, 4))).astype(np.float32)
    idx, coord = (x.cpu().numpy() for x in api.rt_locate(ctx, uv, d, obj, filt))
    frac = np.float32(coord - idx.astype(np.float32))
    one = np.float32(1.0)
    want = [0] * numel
    live = np.flatnonzero(obj.cpu().numpy() >= 0)

    def axis(k, linear, size):
        a = idx[live, k]
        if not linear:
            return [(np.clip(a, 0, size - 1), None)]
        f = frac[live, k]
        return [(np.clip(a, 0, size - 1), one - f), (np.clip(a + 1, 0, size - 1), f)]

    spatial, angular = filt == api.RT_QUADRILINEAR, filt != api.RT_NEAREST
    for j, wv in axis(1, spatial, h):
        for i, wu in axis(0, spatial, w):
            for t, wt in axis(3, angular, n):
                for s, ws in axis(2, angular, n):
                    wb = wu * wv if spatial else np.full(len(live), one)
                    if not angular:
                        weight = wb
                    elif layout == api.RT_LAYOUT_ATLAS:
                        weight = wb * (ws * wt)
                    else:
                        weight = wb * ws * wt
                    if layout == api.RT_LAYOUT_ATLAS:
                        at = (j.astype(np.int64) * n + t) * (w * n) + i * n + s
                    else:
                        at = storage_index(layout, w, h, n, i, j, s, t)
                    c = weight[:, None] * g[live]
                    assert c.dtype == np.float32
                    for f in range(len(live)):
                        for ch in range(4):
                            want[4 * int(at[f]) + ch] += _half_even(Fraction(float(c[f, ch])) * (1 << 32))
    want = np.array(want, dtype=np.int64)
    gd = torch.from_numpy(g).cuda()
    for call in ("flat", "batched", "fused"):
        acc = torch.empty(shape, dtype=torch.int64, device="cuda")
        if call == "flat":
            api.rt_shade_backward(ctx, uv, d, obj, filt, gd, {oid: acc}, None, None, api.RT_FIXED_POINT_GRADS)
        elif call == "batched":
            api.rt_shade_batched_backward(ctx, uv.view(V, H, W, 2), d.view(V, H, W, 3), obj.view(V, H, W), filt,
                                          gd.view(V, H, W, 4), {oid: acc}, None, None, api.RT_FIXED_POINT_GRADS)
        else:  # dL/dout = scale (out - target) with a zero texture: -target
            tex.zero_()
            api.rt_shade_batched_l2_step(ctx, uv.view(V, H, W, 2), d.view(V, H, W, 3), obj.view(V, H, W), filt,
                                         -gd.view(V, H, W, 4), 1.0, None, None, {oid: acc}, None, None,
                                         api.RT_FIXED_POINT_GRADS)
        np.testing.assert_array_equal(acc.cpu().numpy().reshape(-1), want)
    assert api.rt_get_error(ctx) == api.RT_OK
    api.rt_destroy_texture(ctx, oid)
