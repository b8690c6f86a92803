"""Copies between texture layouts at the edges of their tiles (32 x 2 buckets, up to 16 in-bucket
columns): every texel must land at its layout's index, bit for bit, and the padding of a quads
destination must stay as it was.  The reference is numpy's permutation of the atlas."""
import numpy as np
import pytest
import torch

from paper_2301_01719_gb300 import api
from parity_util import atlas_to_quads

pytestmark = pytest.mark.gpu

SIZES = [(1, 1, 1), (7, 3, 5), (8, 2, 16), (31, 1, 17), (32, 4, 16), (33, 5, 33), (64, 3, 64), (130, 2, 3), (9, 70, 15)]
LAYOUTS = [api.RT_LAYOUT_ATLAS, api.RT_LAYOUT_PLANES, api.RT_LAYOUT_QUADS]


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = api.Context(0)
    yield c
    c.close()


def _in_layout(atlas, layout, w, h, n, pad=0):
    """The (h n, w n, ...) atlas as an array of the layout's shape."""
    tail = atlas.shape[2:]
    planes = atlas.reshape(h, n, w, n, *tail).swapaxes(1, 2).transpose(2, 3, 0, 1, *range(4, 4 + len(tail)))
    if layout == api.RT_LAYOUT_ATLAS:
        return atlas
    if layout == api.RT_LAYOUT_PLANES:
        return np.ascontiguousarray(planes)
    full = np.full((n, n, h + h % 2, w + w % 2, *tail), pad, dtype=atlas.dtype)
    full[:, :, :h, :w] = planes
    full = full.reshape(n, n, (h + 1) // 2, 2, (w + 1) // 2, 2, *tail)
    return np.ascontiguousarray(full.swapaxes(3, 4))


@pytest.mark.parametrize("w,h,n", SIZES)
def test_convert_layout_moves_every_texel(ctx, w, h, n):
    atlas = np.random.default_rng(w * 1000 + h * 10 + n).standard_normal((h * n, w * n, 4)).astype(np.float32)
    np.testing.assert_array_equal(_in_layout(atlas, api.RT_LAYOUT_QUADS, w, h, n), atlas_to_quads(atlas, w, h, n))
    for src in LAYOUTS:
        a = torch.from_numpy(_in_layout(atlas, src, w, h, n, pad=7.0)).cuda()
        for dst in LAYOUTS:
            to = torch.full(api.layout_shape(dst, w, h, n), -3.0, device="cuda")
            got = api.rt_convert_layout(a, src, dst, w, h, n, to)
            np.testing.assert_array_equal(got.cpu().numpy(), _in_layout(atlas, dst, w, h, n, pad=-3.0))


@pytest.mark.parametrize("w,h,n", SIZES)
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16", "e4m3"])
def test_stored_codes_read_back_in_every_layout(ctx, w, h, n, storage):
    atlas = np.random.default_rng(w + h + n).uniform(-2.0, 2.0, (h * n, w * n, 4)).astype(np.float32)
    want = None
    for src in LAYOUTS:
        t = torch.from_numpy(_in_layout(atlas, src, w, h, n)).cuda()
        oid = api.rt_create_texture(ctx, w, h, n, api.FORMAT_NAMES[storage], src, t)
        codes = api.rt_read_texture(ctx, oid, api.RT_LAYOUT_ATLAS)[0].cpu().numpy()
        if storage in ("f32", "f16", "bf16"):
            kind = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}[storage]
            enc = torch.from_numpy(atlas).to(kind)
            want = enc.numpy() if storage == "f32" else enc.view(torch.int16).numpy()
        want = codes if want is None else want  # E4M3: the same codes whatever the source's layout
        np.testing.assert_array_equal(codes, want)
        for dst in LAYOUTS[1:]:
            got = api.rt_read_texture(ctx, oid, dst)[0].cpu().numpy()
            np.testing.assert_array_equal(got, _in_layout(want, dst, w, h, n))
        api.rt_destroy_texture(ctx, oid)


@pytest.mark.parametrize("w,n", [(24, 1023), (24, 1024), (23, 1024)])
def test_convert_layout_of_many_in_bucket_texels(w, n):
    """rt_convert_layout has no limit on n; a grid has one on its second dimension (reached at n = 1024)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    a = torch.arange(n * n * w * 4, dtype=torch.int32, device="cuda").view(n, n, 1, w, 4)
    planes = a.view(torch.float32)  # distinct bit patterns
    got = api.rt_convert_layout(planes, api.RT_LAYOUT_PLANES, api.RT_LAYOUT_ATLAS, w, 1, n)
    assert torch.equal(got.view(torch.int32), a[:, :, 0].permute(0, 2, 1, 3).reshape(n, w * n, 4))
    back = api.rt_convert_layout(got, api.RT_LAYOUT_ATLAS, api.RT_LAYOUT_PLANES, w, 1, n)
    assert torch.equal(back.view(torch.int32), a)


@pytest.mark.parametrize("w,h,n", [(40, 3, 7), (40, 3, 8), (24, 2, 8), (23, 2, 8), (40, 1, 15), (40, 1, 16), (40, 1, 17),
                                   (40, 1, 31), (40, 1, 32), (40, 2, 5), (64, 1820, 6), (64, 1821, 6), (100, 3355, 5),
                                   (100, 3356, 5)])
def test_copies_on_both_sides_of_the_tiles_rule(ctx, w, h, n):
    """Every pair of layouts where tiles begin and end (widths, in-bucket columns, one bucket row, large
    FP32 copies into an atlas), and the FP16 codes of the same sizes."""
    planes = torch.arange(n * n * w * h * 4, dtype=torch.int32, device="cuda").view(n, n, h, w, 4)
    atlas = planes.permute(2, 0, 3, 1, 4).reshape(h * n, w * n, 4)
    full = torch.full((n, n, h + h % 2, w + w % 2, 4), -7, dtype=torch.int32, device="cuda")
    full[:, :, :h, :w] = planes
    quads = full.view(n, n, full.shape[2] // 2, 2, full.shape[3] // 2, 2, 4).transpose(3, 4).contiguous()
    held = {api.RT_LAYOUT_ATLAS: atlas.contiguous(), api.RT_LAYOUT_PLANES: planes, api.RT_LAYOUT_QUADS: quads}
    for src in LAYOUTS:
        for dst in LAYOUTS:
            to = torch.full(held[dst].shape, -7, dtype=torch.int32, device="cuda").view(torch.float32)
            api.rt_convert_layout(held[src].view(torch.float32), src, dst, w, h, n, to)
            assert torch.equal(to.view(torch.int32), held[dst])
    values = (atlas % 2039).float()  # exact in FP16
    oid = api.rt_create_texture(ctx, w, h, n, api.RT_F16, api.RT_LAYOUT_ATLAS, values)
    for dst, want in ((api.RT_LAYOUT_ATLAS, values), (api.RT_LAYOUT_PLANES, (planes % 2039).float())):
        assert torch.equal(api.rt_read_texture(ctx, oid, dst)[0].view(torch.float16).float(), want)
    api.rt_destroy_texture(ctx, oid)
