"""FP32 gradient of the chain minGRU, layer by layer, at the edges of its tiles:
site counts around the 128-site tile and the 256 / 512-site ranges, one to four
layers, every width, a parameter vector that does not start on 16 bytes.

Tolerance: a weight gradient is a sum of FP32 products whose rounding errors
(2^-24 each, independent) grow like the square root of the terms; with the few
hundred roundings along a site's path the relative error of the whole vector
stays near 1e-6.  The bound is 2e-5 of the norm (50 times below the stated
1e-3)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2605_13807_gb300 import api, inputs  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    yield


def _close(got, ref):
    got = got.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - ref) <= 2e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("nL,H,n,N,u1", [
    (1, 32, 1, 1, False), (1, 64, 3, 7, False), (2, 32, 2, 64, True), (3, 64, 3, 43, False), (3, 128, 1, 129, False),
    (4, 32, 5, 103, False), (3, 128, 4, 128, True), (2, 128, 3, 171, False), (3, 32, 9, 57, False)])
def test_rows_and_weighted_sum_match_the_oracle(oracle_mod, nL, H, n, N, u1):
    theta = inputs.random_params(nL, H, seed=nL * 100 + H)
    spins = inputs.zero_magnetisation_spins(5, n, N) if u1 else inputs.random_spins(5, n, N)
    w = np.linspace(-1.0, 1.5, n).astype(np.float32)
    cfg = api.ModelConfig(nL, H, u1, "fp32")
    _, ref = oracle_mod.grad(theta, nL, H, spins, u1=u1)
    buf = torch.empty(theta.size + 1, dtype=torch.float32, device="cuda")
    buf[1:] = torch.from_numpy(theta).cuda()
    for th in (torch.from_numpy(theta).cuda(), buf[1:]):  # the second starts 4 bytes off
        s = torch.from_numpy(spins).cuda()
        rows = api.grad(th, s, cfg)
        tot = api.grad(th, s, cfg, dout=torch.from_numpy(w).cuda())
        api.sync()
        for i in range(n):
            _close(rows[i], ref[i])
        _close(tot, w.astype(np.float64) @ ref)
