"""BF16 chain forward with sequences that start in mid-chunk: chunk boundaries
counted from the end of the sequence in groups of 8 sites.  Site counts at and
around every offset (0, 8, 16, 24), whole forwards and resumed local energies,
both forward shapes, and a batch that mixes offsets.

Tolerances are the stated ones of the BF16 path: |d log psi| <= 2e-2 + 2e-5
|log psi|, E_loc 1e-3 of |diag| + |E_loc - diag| with a factor 2 for the random
parameters (every entry nonzero).  The two shapes agree bit for bit."""
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


@pytest.mark.parametrize("N,u1", [(1, False), (2, True), (8, True), (9, False), (24, True), (25, False), (31, False),
                                  (32, True), (33, False), (40, True), (57, False), (64, True), (72, True),
                                  (100, True), (130, False), (400, True)])
def test_offsets_match_the_oracle(oracle_mod, N, u1):
    nL, H, n = 3, 128, 5
    theta = inputs.glorot_params(nL, H, seed=N)
    spins = inputs.zero_magnetisation_spins(3, n, N) if u1 else inputs.random_spins(3, n, N)
    kind = "heisenberg" if u1 else "tfim"
    ham = B.make_hamiltonian(kind, N, 1, False, True, 1.0, 0.7)
    ref = oracle_mod.logpsi(theta, nL, H, spins, u1=u1)
    k = oracle_mod.HEISENBERG if u1 else oracle_mod.TFIM
    rel = oracle_mod.local_energy(theta, nL, H, spins, k, N, 1, u1=u1, h=0.7)
    _, _, diag = oracle_mod.connected(k, N, 1, False, spins)
    th, s = torch.from_numpy(theta).cuda(), torch.from_numpy(spins).cuda()
    cfg = api.ModelConfig(nL, H, u1, "bf16")
    got = []
    try:
        for shape in (1, 2):
            api.set_fwd_shape("bf16", shape)
            lp = api.logpsi(th, s, cfg)
            el, _ = api.local_energy(th, s, cfg, ham)
            api.sync()
            got.append((lp.clone(), el.clone()))
    finally:
        api.set_fwd_shape("bf16", 0)
    for lp, el in got:
        assert torch.equal(lp, got[0][0]) and torch.equal(el, got[0][1])
        assert np.all(np.abs(lp.cpu().numpy() - ref) <= 2e-2 + 2e-5 * np.abs(ref))
        scale = np.abs(diag) + np.abs(rel - diag)
        assert np.all(np.abs(el.cpu().numpy() - rel) <= 2e-3 * scale + 1e-6)


def test_batch_of_mixed_offsets_equals_single_calls():
    nL, H = 3, 128
    theta = torch.from_numpy(inputs.glorot_params(nL, H, seed=0)).cuda()
    cfg = api.ModelConfig(nL, H, False, "bf16")
    items = []
    for Lx, Ly in ((8, 8), (10, 10), (6, 5), (7, 3)):
        u1 = Lx * Ly % 2 == 0
        s = (inputs.neel_like_spins if u1 else lambda seed, n, a, b: inputs.random_spins(seed, n, a * b))(4, 9, Lx, Ly)
        ham = B.make_hamiltonian("heisenberg" if u1 else "tfim", Lx, Ly, False, True, 1.0, 0.9)
        items.append((torch.from_numpy(s).cuda(), ham, u1))
    outs = api.step_batch(theta, items, cfg, want=("logpsi", "eloc"))
    for (s, ham, u1), o in zip(items, outs):
        c = api.ModelConfig(nL, H, u1, "bf16")
        assert torch.equal(o["logpsi"], api.logpsi(theta, s, c))
        assert torch.equal(o["eloc"], api.local_energy(theta, s, c, ham)[0])
    api.sync()
