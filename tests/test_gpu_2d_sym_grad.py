"""Gradient of the c4v-symmetrised 2D training step at the widths whose products
run on the tensor cores (its image weights come from the same forward): against
central differences of the oracle's symmetrised FP64 log psi weighted by the
oracle's centred E_loc, components within 1e-3 of the largest and directions
within 1e-3 of the norms, as at hidden 32."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from fdcheck import check_energy_gradient  # noqa: E402
from oracle import vmc  # noqa: E402
from paper_2605_13807_gb300 import api, binding as B, inputs  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    yield


@pytest.mark.parametrize("H,n", [(64, 12), (128, 8), (256, 6)])
def test_gradient_of_a_symmetrised_step(oracle_mod, H, n):
    L, nL = 4, 3
    theta = inputs.glorot_params2d(nL, H, seed=H)
    th = torch.from_numpy(theta).cuda()
    ham = B.make_hamiltonian("heisenberg", L, L, False, True, 1.0, 0.0)
    u = torch.from_numpy(inputs.uniform(31, (n, L * L // 4)).astype(np.float32)).cuda()
    us = torch.from_numpy(inputs.uniform(32, (n,)).astype(np.float32)).cuda()
    out = api.vmc_step2d(th, api.ModelConfig(nL, H, True, "fp32"), ham, u, api.Adam(theta.size, "cuda"),
                         symmetrize=True, sym_uniforms=us)
    api.sync()
    s = out["spins"].cpu().numpy()
    th64 = theta.astype(np.float64)
    e = vmc.local_energy_sym(lambda x: oracle_mod.logpsi2d(th64, nL, H, L, L, x, u1=True), s, 0, L, marshall=True,
                             J=1.0, h=0.0)
    check_energy_gradient(out["grad"].cpu().numpy(), lambda t: vmc.logpsi_sym(
        lambda x: oracle_mod.logpsi2d(t, nL, H, L, L, x, u1=True), s, L), th64, e, seed=33, n_top=8, n_rand=8, n_dir=3)
