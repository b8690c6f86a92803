"""The palette encoder at the edges of its tiles: bucket matrices that no tile divides, planes that
no group divides, every format and layout, clusters of very different sizes, texels that the exact
integer sums leave to FP64 (large, infinite, NaN), and assignments on converted operands."""
import numpy as np
import pytest
import torch

import synth
from paper_2301_01719_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = api.Context(0)
    yield c
    c.close()


def _texture(ctx, values, storage, layout=api.RT_LAYOUT_PLANES, flags=0):
    """values (n, n, h, w, 4) FP32 planes; the object and the (h w, n n 4) FP64 vectors it holds."""
    n, _, h, w, _ = values.shape
    t = torch.from_numpy(values).cuda()
    if layout != api.RT_LAYOUT_PLANES:
        t = api.rt_convert_layout(t, api.RT_LAYOUT_PLANES, layout, w, h, n)
    oid = api.rt_create_texture(ctx, w, h, n, storage, layout, t, flags)
    if storage == api.RT_F32:
        held = values.astype(np.float64)
    else:
        codes, scales = api.rt_read_texture(ctx, oid, api.RT_LAYOUT_PLANES)
        kind = {api.RT_F16: torch.float16, api.RT_BF16: torch.bfloat16, api.RT_E4M3_BUCKET_SCALE: torch.float8_e4m3fn}
        held = codes.view(kind[storage]).float().cpu().numpy()
        if scales is not None:  # decoded values are FP32 products
            held = held * scales.cpu().numpy()[None, None, :, :, None]
        held = held.astype(np.float64)
    return oid, t, held.reshape(n * n, h * w, 4).transpose(1, 0, 2).reshape(h * w, n * n * 4)


def _update(ctx, oid, K, index, C):
    return api.rt_kmeans_update(ctx, oid, K, torch.from_numpy(index.astype(np.int32)).cuda(), C)


SHAPES = [(1, 1, 1, 1), (3, 5, 2, 4), (17, 9, 3, 7), (33, 16, 4, 300), (64, 31, 5, 33), (129, 2, 9, 20),
          (300, 40, 1, 4096), (300, 40, 1, 4097), (64, 40, 5, 20),
          (64, 40, 5, 21), (64, 40, 5, 160), (64, 40, 5, 161)]
KINDS = [(api.RT_F16, api.RT_LAYOUT_PLANES, 0), (api.RT_BF16, api.RT_LAYOUT_PLANES, 0),
         (api.RT_F32, api.RT_LAYOUT_PLANES, 0), (api.RT_E4M3_BUCKET_SCALE, api.RT_LAYOUT_PLANES, 0),
         (api.RT_F32, api.RT_LAYOUT_ATLAS, api.RT_BORROW), (api.RT_F32, api.RT_LAYOUT_PLANES, api.RT_BORROW)]


@pytest.mark.parametrize("w,h,n,K", SHAPES)
@pytest.mark.parametrize("storage,layout,flags", KINDS)
def test_update_is_the_mean_of_the_members(ctx, w, h, n, K, storage, layout, flags):
    """Skewed clusters (one holds half of the buckets, some none).  The mean of FP64 sums, in any
    order, rounds to FP32 within one unit of the exact mean's rounding."""
    rng = np.random.default_rng(w + 7 * h + n)
    oid, keep, X = _texture(ctx, rng.uniform(-1.0, 1.0, (n, n, h, w, 4)).astype(np.float32), storage, layout, flags)
    index = np.where(rng.random(w * h) < 0.5, 0, rng.integers(0, K, w * h))
    old = torch.full((n, n, K, 4), 0.125, device="cuda")
    C = _update(ctx, oid, K, index, old.clone()).cpu().numpy().reshape(n * n, K, 4).transpose(1, 0, 2).reshape(K, -1)
    for k in range(K):
        at = index == k
        want = X[at].mean(axis=0) if at.any() else np.full(n * n * 4, 0.125)
        np.testing.assert_allclose(C[k], want, rtol=2.0 ** -23, atol=1e-15)
    assert api.rt_get_error(ctx) == api.RT_OK
    api.rt_destroy_texture(ctx, oid)
    del keep


@pytest.mark.parametrize("value", [63.96875, 64.0, 65504.0, np.inf, -np.inf, np.nan, 5.9604645e-08, -0.0])
def test_update_of_extreme_fp16_texels(ctx, value):
    w, h, n, K = 24, 6, 3, 5
    rng = np.random.default_rng(3)
    v = rng.uniform(-1.0, 1.0, (n, n, h, w, 4)).astype(np.float16).astype(np.float32)
    v[1, 1, 2, 5, 2] = value
    oid, _, X = _texture(ctx, v, api.RT_F16)
    index = rng.integers(0, K, w * h)
    C = _update(ctx, oid, K, index, torch.zeros((n, n, K, 4), device="cuda")).cpu().numpy()
    C = C.reshape(n * n, K, 4).transpose(1, 0, 2).reshape(K, -1)
    for k in range(K):
        # sums of up to 144 multiples of 2^-24 below 2^17 are exact in FP64, so the rounding is too
        want = (X[index == k].sum(axis=0) * (1.0 / (index == k).sum())).astype(np.float32)
        np.testing.assert_array_equal(C[k], want)
    api.rt_destroy_texture(ctx, oid)


@pytest.mark.parametrize("w,h,n,K", [(1, 1, 1, 1), (16, 2, 4, 3), (17, 3, 4, 5), (15, 33, 8, 40), (130, 7, 5, 257)])
@pytest.mark.parametrize("storage,layout,flags", KINDS)
def test_tensor_core_assignment_and_reassignment(ctx, w, h, n, K, storage, layout, flags):
    """The chosen centroid is a nearest one up to 2^-10 (|x|^2 + |c|^2), the documented bound, and
    assigning again on the converted operands gives the same as converting again."""
    rng = np.random.default_rng(n + K)
    oid, keep, X = _texture(ctx, rng.uniform(-1.0, 1.0, (n, n, h, w, 4)).astype(np.float32), storage, layout, flags)
    first = torch.from_numpy(rng.uniform(-1.0, 1.0, (n, n, K, 4)).astype(np.float32)).cuda()
    then = torch.from_numpy(rng.uniform(-1.0, 1.0, (n, n, K, 4)).astype(np.float32)).cuda()
    scratch = api.TcScratch(api.rt_kmeans_tc_scratch_bytes(w, h, n, K), first.device)
    api.rt_kmeans_assign_tc(ctx, oid, K, first, scratch=scratch)
    index = torch.empty((h, w), dtype=torch.int32, device="cuda")
    dist = torch.empty((h, w), device="cuda")
    api.rt_kmeans_reassign_tc(ctx, oid, K, then, index, dist, scratch)
    i2, d2 = api.rt_kmeans_assign_tc(ctx, oid, K, then, want_dist=True)
    assert torch.equal(index, i2) and torch.equal(dist, d2)
    C = then.cpu().numpy().astype(np.float64).reshape(n * n, K, 4).transpose(1, 0, 2).reshape(K, -1)
    D = (X ** 2).sum(1)[:, None] + (C ** 2).sum(1)[None] - 2.0 * X @ C.T
    got = index.cpu().numpy().reshape(-1)
    bound = 2.0 ** -10 * ((X ** 2).sum(1) + (C ** 2).sum(1).max())
    rows = np.arange(w * h)
    assert (D[rows, got] <= D.min(1) + bound).all()
    assert (np.abs(dist.cpu().numpy().reshape(-1) - D[rows, got]) <= bound).all()
    assert api.rt_get_error(ctx) == api.RT_OK
    api.rt_destroy_texture(ctx, oid)
    del keep


@pytest.mark.parametrize("w,h,n,K", [(8, 8, 16, 5), (9, 5, 17, 3), (16, 16, 15, 4), (5, 3, 33, 2), (16, 16, 64, 16),
                                     (160, 59, 16, 7),
                                     (160, 61, 16, 7)])
@pytest.mark.parametrize("storage,layout,flags", KINDS)
def test_tensor_core_distances_of_few_buckets_with_many_planes(ctx, w, h, n, K, storage, layout, flags):
    """The conversion of few buckets (160 x 61 are the first with enough) splits their planes among blocks,
    from 4 groups of 64 planes on, groups that the split does not divide among them: indices and distances within the documented bound."""
    rng = np.random.default_rng(w + h + n)
    oid, keep, X = _texture(ctx, rng.uniform(-1.0, 1.0, (n, n, h, w, 4)).astype(np.float32), storage, layout, flags)
    C = rng.uniform(-1.0, 1.0, (n, n, K, 4)).astype(np.float32)
    index, dist = api.rt_kmeans_assign_tc(ctx, oid, K, torch.from_numpy(C).cuda(), want_dist=True)
    C = C.astype(np.float64).reshape(n * n, K, 4).transpose(1, 0, 2).reshape(K, -1)
    D = (X ** 2).sum(1)[:, None] + (C ** 2).sum(1)[None] - 2.0 * X @ C.T
    bound = 2.0 ** -10 * ((X ** 2).sum(1) + (C ** 2).sum(1).max())
    got = D[np.arange(w * h), index.cpu().numpy().reshape(-1)]
    assert (got <= D.min(1) + bound).all()
    assert (np.abs(dist.cpu().numpy().reshape(-1) - got) <= bound).all()
    assert api.rt_get_error(ctx) == api.RT_OK
    api.rt_destroy_texture(ctx, oid)
    del keep


def _reassign_setup(ctx, w=24, h=10, n=4, K=6):
    oid, _, _ = _texture(ctx, np.random.default_rng(1).random((n, n, h, w, 4), dtype=np.float32), api.RT_F16)
    C = torch.rand((n, n, K, 4), device="cuda")
    scratch = api.TcScratch(api.rt_kmeans_tc_scratch_bytes(w, h, n, K + 300), C.device)  # for another K too
    index = torch.empty((h, w), dtype=torch.int32, device="cuda")
    return oid, C, scratch, index


@pytest.mark.parametrize("change", ["none", "never converted", "other object", "other K", "baked", "filled",
                                    "created anew"])
def test_reassignment_reports_a_scratch_of_other_texels(ctx, change):
    """The scratch carries what it was converted from; a reassignment on another one is an error."""
    w, h, n, K = 24, 10, 4, 6
    oid, C, scratch, index = _reassign_setup(ctx)
    ids = [oid]
    scratch.buf.zero_()
    if change != "never converted":
        api.rt_kmeans_assign_tc(ctx, oid, K, C, index, scratch=scratch)
    if change == "other object":
        ids.append(api.rt_create_texture(ctx, w, h, n, api.RT_F16))
    elif change == "other K":
        K = 300
        C = torch.rand((n, n, K, 4), device="cuda")
    elif change == "baked":
        api.rt_bake(ctx, oid, api.RT_SURFACE_SPHERE, synth.bake_scene(3))
    elif change == "filled":
        api.rt_fill_bucket_lobes(ctx, oid, torch.rand((h, w, 8), device="cuda"))
    elif change == "created anew":
        api.rt_destroy_texture(ctx, oid)
        assert api.rt_create_texture(ctx, w, h, n, api.RT_F16) == oid
    assert api.rt_get_error(ctx) == api.RT_OK
    api.rt_kmeans_reassign_tc(ctx, ids[-1], K, C, index, None, scratch)
    assert api.rt_get_error(ctx) == (api.RT_OK if change == "none" else api.RT_ERR_INVALID_ARG)
    api.rt_kmeans_assign_tc(ctx, ids[-1], K, C, index, scratch=scratch)  # converts: the scratch is good again
    api.rt_kmeans_reassign_tc(ctx, ids[-1], K, C, index, None, scratch)
    assert api.rt_get_error(ctx) == api.RT_OK
    for o in ids:
        api.rt_destroy_texture(ctx, o)


def test_reassignment_checks_its_tensors(ctx):
    oid, C, scratch, index = _reassign_setup(ctx)
    api.rt_kmeans_assign_tc(ctx, oid, 6, C, index, scratch=scratch)
    dist = torch.empty((10, 24), device="cuda")
    for bad_index, bad_dist, error in ((None, None, TypeError), (index.cpu(), None, TypeError),
                                       (index.long(), None, TypeError), (index[:, ::2], None, ValueError),
                                       (index[:5].clone(), None, ValueError), (index, dist.double(), TypeError),
                                       (index, dist[:9].clone(), ValueError), (index, dist.cpu(), TypeError)):
        with pytest.raises(error):
            api.rt_kmeans_reassign_tc(ctx, oid, 6, C, bad_index, bad_dist, scratch)
    api.rt_kmeans_reassign_tc(ctx, oid, 6, C, index.view(torch.uint32), dist, scratch)
    assert api.rt_get_error(ctx) == api.RT_OK
    api.rt_destroy_texture(ctx, oid)
