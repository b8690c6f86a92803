"""palette_encode called in other ways than with a positive number of steps on the current stream."""
import numpy as np
import pytest
import torch

from paper_2301_01719_gb300 import api

pytestmark = pytest.mark.gpu

W, H, N, K = 64, 48, 8, 37


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = api.Context(0)
    yield c
    c.close()


@pytest.fixture(scope="module")
def oid(ctx):
    """FP16: its means are exact sums, so an encoding repeats bit for bit."""
    values = np.random.default_rng(4).random((N, N, H, W, 4), dtype=np.float32)
    return api.rt_create_texture(ctx, W, H, N, api.RT_F16, api.RT_LAYOUT_PLANES, torch.from_numpy(values).cuda())


def same(a, b):
    return torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and a[2] == b[2]


@pytest.mark.parametrize("tensor_cores", [True, False])
def test_a_negative_number_of_steps_is_none(ctx, oid, tensor_cores):
    """The first assignment converts the buckets whichever step it is."""
    none = api.palette_encode(ctx, oid, K, 0, tensor_cores=tensor_cores)
    assert len(none[2]) == 1 and none[2][0] > 0.0
    for steps in (-1, -5):
        torch.full((1 << 22,), float("nan"), device="cuda")  # what the scratch may be given next
        assert same(api.palette_encode(ctx, oid, K, steps, tensor_cores=tensor_cores), none)


@pytest.mark.parametrize("tensor_cores", [True, False])
@pytest.mark.parametrize("busy", ["given", "current"])
@pytest.mark.parametrize("kind", ["torch", "handle"])
def test_a_given_stream_runs_the_whole_encoding(ctx, oid, tensor_cores, busy, kind):
    """With work queued on either stream (some 20 ms of fills), an encoding on a side stream equals the
    one on the current stream: its sums are taken after each assignment and before the next."""
    want = api.palette_encode(ctx, oid, K, 3, seed=2, tensor_cores=tensor_cores)
    side = torch.cuda.Stream()
    filler = torch.empty(1 << 28, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(side if busy == "given" else torch.cuda.current_stream()):
        for k in range(100):
            filler.fill_(float(k))
    got = api.palette_encode(ctx, oid, K, 3, seed=2, stream=side if kind == "torch" else side.cuda_stream,
                             tensor_cores=tensor_cores)
    assert same(got, want)
    torch.cuda.synchronize()


def test_the_default_streams_handle_is_a_stream_too(ctx, oid):
    want = api.palette_encode(ctx, oid, K, 1)
    assert same(api.palette_encode(ctx, oid, K, 1, stream=0), want)
    with torch.cuda.stream(torch.cuda.Stream()):
        assert same(api.palette_encode(ctx, oid, K, 1, stream=torch.cuda.default_stream()), want)
