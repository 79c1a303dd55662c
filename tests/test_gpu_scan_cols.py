"""Whole-column form of psr_scan (32 units x the whole sequence) at its edges:
sequences shorter than, equal to and just over a 32-site stage and over the
ring's four stages, more columns than resident warps, and in place.

Tolerance: one fused multiply-add a site, so h_t carries at most one rounding
(2^-24) of every partial value, 1e-5 of the recurrence on |a|, |b|, |h0| being
far above it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2605_13807_gb300 import api, binding as B, inputs  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    yield


def _scan64(a, b, h0):
    h = np.zeros(b[:, 0].shape) if h0 is None else h0.astype(np.float64)
    out = np.empty(a.shape)
    for t in range(a.shape[1]):
        h = a[:, t].astype(np.float64) * h + b[:, t]
        out[:, t] = h
    return out


@pytest.mark.parametrize("n,N,H,with_h0,in_place", [
    (1, 1, 32, True, None), (3, 31, 64, False, None), (2, 32, 96, True, "a"), (5, 33, 32, True, "b"),
    (2, 127, 128, False, None), (2, 129, 64, True, "b"), (1300, 65, 32, True, None), (700, 40, 64, False, "a")])
def test_whole_columns(n, N, H, with_h0, in_place):
    a, b, h0 = inputs.scan_inputs(21, n, N, H)
    h0 = h0 if with_h0 else None
    ref = _scan64(a, b, h0)
    mag = _scan64(np.abs(a), np.abs(b), None if h0 is None else np.abs(h0))
    ta, tb = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    th0 = None if h0 is None else torch.from_numpy(h0).cuda()
    out = {"a": ta, "b": tb, None: None}[in_place]
    h = api.scan(ta, tb, th0, tile=(32, N), out=out)
    api.sync()
    assert np.all(np.abs(h.cpu().numpy() - ref) <= 1e-5 * mag)


def test_default_takes_whole_columns():
    ctx = B.context()
    assert B.psr_scan_tile_for(ctx, 200, 2704, 128) == ((32, 2704), False)
    assert B.psr_scan_tile_for(ctx, 64, 700, 64) == ((32, 700), False)
    assert B.psr_scan_tile_for(ctx, 16384, 100, 128) == ((128, 100), False)
    (units, chunk), _ = B.psr_scan_tile_for(ctx, 8, 2704, 32)
    assert chunk < 2704  # few long columns: look-back chunks
    (units, _), _ = B.psr_scan_tile_for(ctx, 100, 100, 36)
    assert units == 4
