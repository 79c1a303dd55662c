"""FP32 chain forward at the edges of its windows (16 and 32 sites counted from
the end of the sequence): log psi and the resumed local energies against the
oracle, both window sizes, every width, odd and even numbers of 16-site chunks,
and site counts around the 64-bit words of the packed spins.

Tolerances are the stated ones of the FP32 path: |d log psi| <= 1e-5 + 1e-6
|log psi|, E_loc 1e-3 of |diag| + |E_loc - diag| (2e-5 of it here: a ratio
exp(d log psi) carries the rounding of two log psi, at most 2e-5)."""
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


@pytest.mark.parametrize("H,nL", [(32, 3), (64, 2), (128, 3)])
@pytest.mark.parametrize("N,u1", [(2, False), (15, False), (16, True), (17, False), (32, True), (33, False),
                                  (48, True), (63, False), (65, False), (128, True)])
def test_windows_match_the_oracle(oracle_mod, H, nL, N, u1):
    theta = inputs.random_params(nL, H, seed=N + H)
    n = 7
    spins = inputs.zero_magnetisation_spins(3, n, N) if u1 else inputs.random_spins(3, n, N)
    kind = "heisenberg" if u1 else "tfim"
    ham = B.make_hamiltonian(kind, N, 1, False, True, 1.0, 0.7)
    ref = oracle_mod.logpsi(theta, nL, H, spins, u1=u1)
    k = oracle_mod.HEISENBERG if u1 else oracle_mod.TFIM
    rel = oracle_mod.local_energy(theta, nL, H, spins, k, N, 1, u1=u1, h=0.7)
    _, _, diag = oracle_mod.connected(k, N, 1, False, spins)
    th, s = torch.from_numpy(theta).cuda(), torch.from_numpy(spins).cuda()
    cfg = api.ModelConfig(nL, H, u1, "fp32")
    try:
        for shape in (32, 16):
            api.set_fwd_shape("fp32", shape)
            lp = api.logpsi(th, s, cfg)
            el, _ = api.local_energy(th, s, cfg, ham)
            api.sync()
            assert np.all(np.abs(lp.cpu().numpy() - ref) <= 1e-5 + 1e-6 * np.abs(ref))
            scale = np.abs(diag) + np.abs(rel - diag)
            assert np.all(np.abs(el.cpu().numpy() - rel) <= 2e-5 * scale + 1e-6)
    finally:
        api.set_fwd_shape("fp32", 0)
