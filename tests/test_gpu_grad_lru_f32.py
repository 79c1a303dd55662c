"""FP32 gradient of the LRU, layer by layer, at the edges of its tiles (site
counts around 128 and 256, one to four layers, every width, a parameter vector
off 16 bytes): rows against central differences of the oracle's FP64 log psi
along random directions, and the weighted sum against the rows.

Tolerances: the differences (unit directions, eps 1e-4, FP64) are good to about
1e-8; the FP32 rows carry some hundred roundings of 2^-24, about 1e-6 of their
norm; 2e-5 of the norm is asserted.  The sum equals the weighted rows to
2e-5 of the sum of their norms."""
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


@pytest.mark.parametrize("nL,H,n,N,u1", [
    (1, 32, 1, 1, False), (1, 64, 3, 7, False), (2, 32, 2, 64, True), (3, 64, 3, 43, False), (3, 128, 1, 129, False),
    (4, 32, 5, 52, False), (3, 128, 4, 32, True), (2, 64, 2, 257, False)])
def test_rows_and_weighted_sum(oracle_mod, nL, H, n, N, u1):
    theta = inputs.lru_params(nL, H, seed=nL * 100 + H)
    spins = inputs.zero_magnetisation_spins(5, n, N) if u1 else inputs.random_spins(5, n, N)
    w = np.linspace(-1.0, 1.5, n).astype(np.float32)
    cfg = api.ModelConfig(nL, H, u1, "fp32")
    rng = np.random.default_rng(nL)
    dirs = rng.standard_normal((3, theta.size))
    dirs /= np.linalg.norm(dirs, axis=1)[:, None]
    eps, t64 = 1e-4, theta.astype(np.float64)
    fd = [(oracle_mod.logpsi_lru(t64 + eps * d, nL, H, spins, u1=u1) -
           oracle_mod.logpsi_lru(t64 - eps * d, nL, H, spins, u1=u1)) / (2 * eps) for d in dirs]
    buf = torch.empty(theta.size + 1, dtype=torch.float32, device="cuda")
    buf[1:] = torch.from_numpy(theta).cuda()
    for th in (torch.from_numpy(theta).cuda(), buf[1:]):  # the second starts 4 bytes off
        s = torch.from_numpy(spins).cuda()
        rows = api.grad_lru(th, s, cfg)
        tot = api.grad_lru(th, s, cfg, dout=torch.from_numpy(w).cuda())
        api.sync()
        r = rows.cpu().numpy().astype(np.float64)
        for d, f in zip(dirs, fd):
            assert np.all(np.abs(r @ d - f) <= 2e-5 * np.linalg.norm(r, axis=1) + 1e-7)
        err = np.linalg.norm(tot.cpu().numpy() - w.astype(np.float64) @ r)
        assert err <= 2e-5 * np.sum(np.abs(w) * np.linalg.norm(r, axis=1)) + 1e-12
