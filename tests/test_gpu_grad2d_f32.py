"""FP32 gradient of the 2D patched minGRU, layer by layer, at the edges of its
tiles and rows: one patch row or column, rows of 32 patches, odd row counts,
one to four layers, widths 32 to 256, a parameter vector off 16 bytes: rows
against central differences of the oracle's FP64 log psi along random
directions, and the weighted sum against the rows.

Tolerances: the differences (unit directions, eps 1e-4, FP64) are good to about
1e-8; the FP32 rows carry some hundred roundings of 2^-24, about 1e-6 of their
norm; 2e-5 of the norm is asserted, and 2e-5 of the sum of the norms for the
weighted sum."""
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


@pytest.mark.parametrize("nL,H,n,Lx,Ly,u1", [
    (1, 32, 1, 2, 2, False), (2, 32, 3, 64, 2, False), (3, 64, 5, 2, 6, True), (3, 128, 3, 6, 6, True),
    (4, 64, 2, 18, 4, False), (3, 256, 5, 4, 10, False), (2, 256, 2, 34, 2, True)])
def test_rows_and_weighted_sum(oracle_mod, nL, H, n, Lx, Ly, u1):
    rng = np.random.default_rng(nL)
    theta = inputs.glorot_params2d(nL, H, seed=nL * 100 + H)
    theta = (theta + 0.05 * rng.standard_normal(theta.size)).astype(np.float32)
    spins = inputs.zero_magnetisation_spins(5, n, Lx * Ly) if u1 else inputs.random_spins(5, n, Lx * Ly)
    w = np.linspace(-1.0, 1.5, n).astype(np.float32)
    cfg = api.ModelConfig(nL, H, u1, "fp32")
    dirs = rng.standard_normal((3, theta.size))
    dirs /= np.linalg.norm(dirs, axis=1)[:, None]
    eps, t64 = 1e-4, theta.astype(np.float64)
    fd = [(oracle_mod.logpsi2d(t64 + eps * d, nL, H, Lx, Ly, spins, u1=u1) -
           oracle_mod.logpsi2d(t64 - eps * d, nL, H, Lx, Ly, spins, u1=u1)) / (2 * eps) for d in dirs]
    buf = torch.empty(theta.size + 1, dtype=torch.float32, device="cuda")
    buf[1:] = torch.from_numpy(theta).cuda()
    for th in (torch.from_numpy(theta).cuda(), buf[1:]):  # the second starts 4 bytes off
        s = torch.from_numpy(spins).cuda()
        rows = api.grad2d(th, s, cfg, Lx, Ly)
        tot = api.grad2d(th, s, cfg, Lx, Ly, dout=torch.from_numpy(w).cuda())
        api.sync()
        r = rows.cpu().numpy().astype(np.float64)
        for d, f in zip(dirs, fd):
            assert np.all(np.abs(r @ d - f) <= 2e-5 * np.linalg.norm(r, axis=1) + 1e-7)
        err = np.linalg.norm(tot.cpu().numpy() - w.astype(np.float64) @ r)
        assert err <= 2e-5 * np.sum(np.abs(w) * np.linalg.norm(r, axis=1)) + 1e-12
