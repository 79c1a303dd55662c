"""Gradients when the layer arrays do not fit: ragged batches of samples, samples
that are recomputed chunk by chunk, a step that mixes the two, and a workspace
without room for the first batch (psr_context_set_memory).

Rows of the chain model against the FP64 oracle, of the LRU and 2D models
against central differences of the oracle's log psi along random directions
(unit directions, eps 1e-4: good to 1e-8).  Tolerance 2e-5 of a row's norm, as
for the same gradients in one batch (some hundred FP32 roundings of 2^-24 along
a site's path, about 1e-6); a weighted sum 2e-5 of the weighted norms."""
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


@pytest.fixture(autouse=True)
def _defaults():
    yield
    B.psr_context_set_memory(api._ctx())


def _sample_bytes(model, nL, H, N):
    """Bytes of layer arrays of one sample."""
    if model == "2d":
        return 4 * (N // 4) * ((5 * nL + 4) * H + 97)
    return 4 * N * (((8 * nL + 4) if model == "lru" else (5 * nL + 2)) * H + 1)


def _case(oracle_mod, model, nL, H, n, Lx, Ly, u1):
    N = Lx * Ly
    spins = inputs.zero_magnetisation_spins(5, n, N) if u1 else inputs.random_spins(5, n, N)
    seed = nL * 100 + H
    if model == "chain":
        theta = inputs.random_params(nL, H, seed=seed)
        _, rows = oracle_mod.grad(theta, nL, H, spins, u1=u1)
        return theta, spins, rows, None
    if model == "lru":
        theta = inputs.lru_params(nL, H, seed=seed)
        f = lambda t: oracle_mod.logpsi_lru(t, nL, H, spins, u1=u1)
    else:
        theta = inputs.glorot_params2d(nL, H, seed=seed)
        f = lambda t: oracle_mod.logpsi2d(t, nL, H, Lx, Ly, spins, u1=u1)
    rng = np.random.default_rng(nL)
    dirs = rng.standard_normal((3, theta.size))
    dirs /= np.linalg.norm(dirs, axis=1)[:, None]
    eps, t64 = 1e-4, theta.astype(np.float64)
    return theta, spins, dirs, np.array([(f(t64 + eps * d) - f(t64 - eps * d)) / (2 * eps) for d in dirs])


def _grad(model, th, s, cfg, Lx, Ly, w=None):
    if model == "2d":
        return api.grad2d(th, s, cfg, Lx, Ly, dout=w)
    return (api.grad_lru if model == "lru" else api.grad)(th, s, cfg, dout=w)


def _check(oracle_mod, model, nL, H, n, Lx, Ly, u1, prec, batch):
    theta, spins, ref, fd = _case(oracle_mod, model, nL, H, n, Lx, Ly, u1)
    cfg = api.ModelConfig(nL, H, u1, prec)
    th, s = torch.from_numpy(theta).cuda(), torch.from_numpy(spins).cuda()
    w = np.linspace(-1.0, 1.5, n).astype(np.float32)
    wt = torch.from_numpy(w).cuda()
    whole = _grad(model, th, s, cfg, Lx, Ly).clone()
    B.psr_context_set_memory(api._ctx(), grad_bytes=batch * _sample_bytes(model, nL, H, Lx * Ly))
    rows = _grad(model, th, s, cfg, Lx, Ly)
    tot = _grad(model, th, s, cfg, Lx, Ly, wt)
    api.sync()
    if batch > 0:
        assert torch.equal(rows, whole)  # a row does not depend on its batch
    r = rows.cpu().numpy().astype(np.float64)
    norms = np.linalg.norm(r, axis=1)
    if fd is None:
        assert np.all(np.linalg.norm(r - ref, axis=1) <= 2e-5 * np.linalg.norm(ref, axis=1))
        exact = w.astype(np.float64) @ ref
    else:
        for d, f in zip(ref, fd):
            assert np.all(np.abs(r @ d - f) <= 2e-5 * norms + 1e-7)
        exact = w.astype(np.float64) @ r
    assert np.linalg.norm(tot.cpu().numpy() - exact) <= 2e-5 * np.sum(np.abs(w) * norms) + 1e-12


@pytest.mark.parametrize("model,nL,H,Lx,Ly,u1,prec", [
    ("chain", 3, 32, 43, 1, False, "fp32"), ("chain", 2, 64, 20, 1, True, "fp32"), ("chain", 3, 128, 33, 1, False, "fp32"),
    ("chain", 3, 128, 6, 6, True, "bf16"), ("lru", 3, 64, 37, 1, False, "fp32"), ("lru", 2, 32, 129, 1, False, "fp32"),
    ("2d", 3, 64, 6, 4, True, "fp32"), ("2d", 2, 256, 4, 4, False, "fp32")])
@pytest.mark.parametrize("n,batch", [(7, 3), (5, 1), (6, 2)])
def test_batches(oracle_mod, model, nL, H, Lx, Ly, u1, prec, n, batch):
    _check(oracle_mod, model, nL, H, n, Lx, Ly, u1, prec, batch)


@pytest.mark.parametrize("model,nL,H,n,Lx,Ly,u1,prec", [
    ("chain", 1, 32, 1, 1, 1, False, "fp32"), ("chain", 3, 64, 3, 7, 1, False, "fp32"),
    ("chain", 2, 32, 2, 64, 1, True, "fp32"), ("chain", 4, 32, 5, 103, 1, False, "fp32"),
    ("chain", 3, 128, 4, 129, 1, False, "fp32"), ("chain", 3, 64, 3, 43, 1, False, "fp32"),
    ("chain", 3, 128, 3, 34, 1, True, "bf16"), ("lru", 3, 64, 3, 43, 1, False, "fp32"),
    ("lru", 2, 32, 2, 64, 1, True, "fp32"), ("lru", 3, 128, 2, 65, 1, False, "fp32"),
    ("2d", 2, 32, 3, 18, 2, False, "fp32"), ("2d", 3, 128, 3, 6, 6, True, "fp32"), ("2d", 3, 256, 2, 4, 6, False, "fp32")])
def test_recomputed_chunks(oracle_mod, model, nL, H, n, Lx, Ly, u1, prec):
    _check(oracle_mod, model, nL, H, n, Lx, Ly, u1, prec, 0)


def test_bf16_rows_against_the_recompute_kernel():
    """Two implementations that share no product, scan or readout."""
    theta = torch.from_numpy(inputs.glorot_params(3, 128, seed=0)).cuda()
    s = torch.from_numpy(inputs.neel_like_spins(11, 40, 12, 12)).cuda()
    rows = api.grad(theta, s, api.ModelConfig(3, 128, True, "bf16")).double()
    B.psr_context_set_memory(api._ctx(), grad_bytes=0)
    ref = api.grad(theta, s, api.ModelConfig(3, 128, True, "fp32")).double()
    api.sync()
    assert torch.all((rows - ref).norm(dim=1) <= 1e-4 * ref.norm(dim=1))
    assert torch.all((rows - ref).abs().amax(1) <= 1e-4 * ref.abs().amax(1))


@pytest.mark.parametrize("prec,H,graphs", [("fp32", 32, False), ("fp32", 64, True), ("bf16", 128, False)])
def test_a_step_with_layered_and_recomputed_items(oracle_mod, prec, H, graphs):
    nL = 3
    theta = inputs.glorot_params(nL, H, seed=H)
    th = torch.from_numpy(theta).cuda()
    sets = [(5, 4, 4), (3, 10, 7), (4, 6, 6), (2, 10, 10)]  # n, Lx, Ly
    batch, spins = [], []
    for k, (n, Lx, Ly) in enumerate(sets):
        u1 = Lx * Ly % 2 == 0
        s = inputs.zero_magnetisation_spins(k, n, Lx * Ly) if u1 else inputs.random_spins(k, n, Lx * Ly)
        spins.append(s)
        batch.append((torch.from_numpy(s).cuda(), B.make_hamiltonian("tfim", Lx, Ly, False, True, 1.0, 0.7), u1))
    cfg = api.ModelConfig(nL, H, False, prec)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = api._ctx()
        # room for a sample of 36 sites (two of 16), not for 70 or 100
        B.psr_context_set_memory(ctx, grad_bytes=_sample_bytes("chain", nL, H, 36))
        B.psr_context_set_graphs(ctx, graphs)
        for _ in range(2):
            outs = api.step_batch(th, batch, cfg)
        single = [api.grad(th, s, api.ModelConfig(nL, H, u1, prec)) for s, _, u1 in batch]
        api.sync()
        B.psr_context_set_graphs(ctx, False)
        B.psr_context_set_memory(ctx)
    for (s, _, u1), o, g, sp in zip(batch, outs, single, spins):
        assert torch.equal(o["grad"], g)
        if prec != "fp32":
            continue  # two-part operands: held to the oracle in test_gpu_grad_tc.py
        _, ref = oracle_mod.grad(theta, nL, H, sp, u1=u1)
        d = np.linalg.norm(o["grad"].cpu().numpy() - ref, axis=1)
        assert np.all(d <= 2e-5 * np.linalg.norm(ref, axis=1))


@pytest.mark.parametrize("model,H,Lx,Ly", [("chain", 64, 100, 1), ("lru", 64, 100, 1), ("2d", 64, 10, 10)])
@pytest.mark.parametrize("weighted", [False, True])
def test_a_batch_without_room_is_halved_once(model, H, Lx, Ly, weighted):
    nL, n = 3, 64
    N = Lx * Ly
    theta = {"chain": inputs.glorot_params, "lru": inputs.lru_params, "2d": inputs.glorot_params2d}[model](nL, H, 1)
    th, s = torch.from_numpy(theta).cuda(), torch.from_numpy(inputs.random_spins(2, n, N)).cuda()
    w = torch.linspace(-1, 1, n, device="cuda") if weighted else None
    cfg = api.ModelConfig(nL, H, False, "fp32")
    ref = _grad(model, th, s, cfg, Lx, Ly, w).clone()
    ctx = api._ctx()
    one = _sample_bytes(model, nL, H, N)
    B.psr_context_set_memory(ctx, workspace_bytes=n * one * 3 // 5)
    got = _grad(model, th, s, cfg, Lx, Ly, w).clone()
    size, gen, fit = B.psr_context_workspace(ctx)
    assert size <= n * one * 3 // 5 and fit < n * one and fit >= n // 4 * one
    again = _grad(model, th, s, cfg, Lx, Ly, w)
    api.sync()
    assert B.psr_context_workspace(ctx) == (size, gen, fit)
    assert torch.equal(got, again)
    if weighted:
        assert (got - ref).norm() <= 1e-5 * ref.norm()
    else:
        assert torch.equal(got, ref)
    B.psr_context_set_memory(ctx, workspace_bytes=1 << 10)
    with pytest.raises(B.PsrError) as e:
        _grad(model, th, s, cfg, Lx, Ly, w)
    assert e.value.code == B.PSR_ENOMEM
    # nothing fitted, so nothing was learned
    assert B.psr_context_workspace(ctx)[2] == 2 << 30


def test_a_step_without_room_is_halved_once():
    nL, H, n, L = 3, 64, 48, 10
    theta = torch.from_numpy(inputs.glorot_params(nL, H, seed=3)).cuda()
    s = torch.from_numpy(inputs.zero_magnetisation_spins(4, n, L * L)).cuda()
    ham = B.make_hamiltonian("heisenberg", L, L, False, True, 1.0, 0.0)
    cfg = api.ModelConfig(nL, H, True, "fp32")
    ref = api.step_batch(theta, [(s, ham, True)], cfg)[0]
    ctx = api._ctx()
    one = _sample_bytes("chain", nL, H, L * L)
    B.psr_context_set_memory(ctx, workspace_bytes=n * one * 3 // 4)
    got = api.step_batch(theta, [(s, ham, True)], cfg)[0]
    state = B.psr_context_workspace(ctx)
    assert state[2] < n * one
    again = api.step_batch(theta, [(s, ham, True)], cfg)[0]
    api.sync()
    assert B.psr_context_workspace(ctx) == state
    for k in ("logpsi", "eloc", "grad"):
        assert torch.equal(got[k], ref[k]) and torch.equal(again[k], ref[k])


def test_a_symmetrised_2d_step_in_batches():
    """Above one batch the image weights come from a forward of their own."""
    L, nL, H, n = 6, 3, 128, 40
    theta = torch.from_numpy(inputs.glorot_params2d(nL, H, 7)).cuda()
    ham = B.make_hamiltonian("heisenberg", L, L, False, True, 1.0, 0.0)
    cfg = api.ModelConfig(nL, H, True, "fp32")
    u, us = torch.rand(n, L * L // 4, device="cuda"), torch.rand(n, device="cuda")

    def step():
        return api.vmc_step2d(theta, cfg, ham, u, api.Adam(theta.numel(), "cuda"), symmetrize=True, sym_uniforms=us)

    a = step()
    B.psr_context_set_memory(api._ctx(), grad_bytes=96 * _sample_bytes("2d", nL, H, L * L))
    b = step()
    api.sync()
    assert torch.equal(a["spins"], b["spins"]) and torch.equal(a["eloc"], b["eloc"])
    # the weights 2/n (E - mean) x softmax(2 log psi) differ by 2 |d log psi| <= 2 (1e-5 + 1e-6 |log psi|), the
    # stated FP32 bound of a log psi, so the gradient by as much of the terms' norms, which add up to a few times its own
    assert (a["grad"] - b["grad"]).norm() <= 2e-4 * b["grad"].norm()


def test_memory_arguments():
    ctx = api._ctx()
    with pytest.raises(B.PsrError):
        B.psr_context_set_memory(0)
    B.psr_context_set_memory(ctx, grad_bytes=12345)
    assert B.psr_context_workspace(ctx)[2] == 12345
    B.psr_context_set_memory(ctx)
    assert B.psr_context_workspace(ctx)[2] == 2 << 30
