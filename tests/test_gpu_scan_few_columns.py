"""psr_scan of one to four columns of 32 units around the lengths where the
default tile changes from whole columns to look-back chunks, also in place.

Tolerance: one rounding (2^-24) of every partial value a site, composed maps
the same; 1e-5 of the recurrence on |a|, |b|, |h0| is far above it."""
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


@pytest.mark.parametrize("n,H,N,whole", [(1, 32, 896, True), (1, 32, 897, False), (1, 64, 1000, False), (3, 32, 1024, False),
                                         (1, 128, 1024, True), (4, 32, 1024, True), (1, 128, 1025, False)])
def test_few_columns(n, H, N, whole):
    (units, chunk), tuned = B.psr_scan_tile_for(B.context(), n, N, H)
    assert not tuned and ((units, chunk) == (32, N)) == whole and (whole or chunk < N)
    a, b, h0 = inputs.scan_inputs(31, n, N, H)
    ref, mag = h0.astype(np.float64), np.abs(h0).astype(np.float64)
    refs, mags = [], []
    for t in range(N):
        ref = a[:, t].astype(np.float64) * ref + b[:, t]
        mag = np.abs(a[:, t]).astype(np.float64) * mag + np.abs(b[:, t])
        refs.append(ref)
        mags.append(mag)
    refs, mags = np.stack(refs, 1), np.stack(mags, 1)
    for alias in (None, "a", "b"):
        ta, tb = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
        h = api.scan(ta, tb, torch.from_numpy(h0).cuda(), out={"a": ta, "b": tb, None: None}[alias])
        api.sync()
        assert np.all(np.abs(h.cpu().numpy() - refs) <= 1e-5 * mags)
