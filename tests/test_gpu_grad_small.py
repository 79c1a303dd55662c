"""Gradients of few sites, whose FP32 products run on small tiles: the O_k rows of
a sample have the bits that they have in a large batch (wide tiles), around
the tiles' edges, and the weighted sum over short ranges agrees with the rows
(2e-5 of the sum of their norms: FP32 rounding, about 1e-6)."""
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


def _grad(model, th, s, cfg, Lx, Ly, w=None):
    if model == "2d":
        return api.grad2d(th, s, cfg, Lx, Ly, dout=w)
    return (api.grad_lru if model == "lru" else api.grad)(th, s, cfg, dout=w)


# sites (patches) of the small batches: 1 to 3 tiles of 32, a range of 64 and
# its neighbours; of the large one: more than 128 wide tiles of 128
@pytest.mark.parametrize("model,H,Lx,Ly", [
    ("chain", 32, 16, 1), ("chain", 64, 33, 1), ("chain", 128, 21, 1), ("lru", 32, 31, 1), ("lru", 64, 32, 1),
    ("lru", 128, 11, 1), ("2d", 32, 6, 4), ("2d", 64, 4, 4), ("2d", 128, 10, 2), ("2d", 256, 6, 6)])
def test_rows_have_the_bits_of_a_large_batch(model, H, Lx, Ly):
    N, nL = Lx * Ly, 3
    sites = N // 4 if model == "2d" else N
    n = 20000 // sites
    theta = {"chain": inputs.glorot_params, "lru": inputs.lru_params, "2d": inputs.glorot_params2d}[model](nL, H, 1)
    th, s = torch.from_numpy(theta).cuda(), torch.from_numpy(inputs.random_spins(2, n, N)).cuda()
    cfg = api.ModelConfig(nL, H, False, "fp32")
    rows = _grad(model, th, s, cfg, Lx, Ly)
    for k in (1, 2, 3, 5, 64 // sites + 1, 4096 // sites):
        part = s[7:7 + k].contiguous()
        assert torch.equal(_grad(model, th, part, cfg, Lx, Ly), rows[7:7 + k]), k
        w = torch.linspace(-1.0, 1.5, k, device="cuda")
        tot = _grad(model, th, part, cfg, Lx, Ly, w).double()
        ref = w.double() @ rows[7:7 + k].double()
        api.sync()
        bound = 2e-5 * float((w.abs().double() * rows[7:7 + k].double().norm(dim=1)).sum())
        assert float((tot - ref).norm()) <= bound, k
