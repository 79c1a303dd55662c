"""2D patched minGRU on the tensor cores at the edges of its 8-column epilogue
chunks (patch rows of 7, 8, 9, 15, 17 and 25), with fewer jobs than slots, and
the c4v images' configurations in one launch.

Tolerances: the stated log psi bound of the 16-bit path against the FP64 oracle,
|d| <= 2e-2 + 2e-5 |log psi|; E_loc 1e-3 (|diag| + |E_loc - diag|), the FP16 path's
stated bound.  A sample's value does not depend on its slot or its neighbours:
bitwise."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle import vmc  # noqa: E402
from paper_2605_13807_gb300 import api, binding as B, inputs  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    yield


@pytest.mark.parametrize("Lx,Ly,H", [(14, 4, 128), (16, 6, 256), (18, 6, 128), (30, 4, 256), (34, 4, 128),
                                     (50, 4, 128)])
def test_chunk_edges(oracle_mod, Lx, Ly, H):
    nL = 3
    theta = inputs.glorot_params2d(nL, H, seed=Lx)
    s = inputs.zero_magnetisation_spins(Lx + 1, 21, Lx * Ly)
    ref = oracle_mod.logpsi2d(theta.astype(np.float64), nL, H, Lx, Ly, s, u1=True)
    th, sd = torch.from_numpy(theta).cuda(), torch.from_numpy(s).cuda()
    cfg = api.ModelConfig(nL, H, True, "fp16")
    got = api.logpsi2d(th, sd, cfg, Lx, Ly)
    one = torch.cat([api.logpsi2d(th, sd[i:i + 1].contiguous(), cfg, Lx, Ly) for i in (0, 20)])
    api.sync()
    assert torch.equal(one, got[[0, 20]])
    assert np.all(np.abs(got.cpu().numpy() - ref) <= 2e-2 + 2e-5 * np.abs(ref))


@pytest.mark.parametrize("L,n", [(4, 1), (6, 40)])
def test_images_in_one_launch(oracle_mod, L, n):
    nL, H = 3, 128
    theta = inputs.glorot_params2d(nL, H, seed=L)
    s = inputs.neel_like_spins(9, n, L, L)
    th64 = theta.astype(np.float64)
    ham = B.make_hamiltonian("heisenberg", L, L, False, True, 1.0, 0.0)
    cfg = api.ModelConfig(nL, H, True, "fp16")
    th, sd = torch.from_numpy(theta).cuda(), torch.from_numpy(s).cuda()
    e, _ = api.sym_local_energy2d(th, sd, cfg, ham)
    e1, _ = api.sym_local_energy2d(th, sd[:1].contiguous(), cfg, ham)
    api.sync()
    assert torch.equal(e1, e[:1])
    m = min(n, 3)
    ref = vmc.local_energy_sym(lambda x: oracle_mod.logpsi2d(th64, nL, H, L, L, x, u1=True), s[:m], 0, L,
                               marshall=True, J=1.0, h=0.0)
    _, _, diag = oracle_mod.connected(0, L, L, False, s[:m])
    assert np.all(np.abs(e[:m].cpu().numpy() - ref) <= 1e-3 * (np.abs(diag) + np.abs(ref - diag)))
