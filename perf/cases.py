"""What the performance of this library is measured on.

Each case is one call (or one step) that a variational Monte Carlo program
makes through `paper_2605_13807_gb300.api`, with device arrays in and out:

  logpsi      log psi of many configurations          (chain minGRU)
  eloc        local energies of samples               (chain minGRU, LRU, 2D)
  grad_sum    log psi and its weighted gradient through torch autograd
              (chain minGRU) or the gradient call     (LRU)
  ok_rows     per-sample O_k rows                     (chain minGRU)
  step        log psi + E_loc + O_k rows in one call  (chain minGRU)
  sample      exact samples and their log psi         (chain minGRU, LRU, 2D)
  scan        the recurrence h_t = a_t h_{t-1} + b_t over arrays in memory
  vmc_step    a whole c4v-symmetrised training step   (2D patched minGRU)

Sizes: the chains of 16, 100 and 256 sites, the 10x10 to 52x52 lattices and
the model widths that the tests, the benchmark and the paper's tables use.
The FP64 statistics that some calls also write (mean, variance, error of the
E_loc values) are sums of outputs that are returned whole and are left out.
"""
import math

import numpy as np
import torch

from paper_2605_13807_gb300 import api, binding, inputs

_LAYERS = 3  # the depth of every model of the paper's runs


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest call: amplitudes of a short chain in FP32 (checks against
        # exact diagonalisation, the first steps of iterative training)
        dict(name="logpsi_chain16_fp32", kind="logpsi", model="chain", hidden=32, precision="fp32",
             Lx=16, Ly=1, n=1024, u1=False),
        # local energies of a periodic Heisenberg chain, the plain FP32 path
        dict(name="eloc_chain100_fp32", kind="eloc", model="chain", hidden=64, precision="fp32",
             Lx=100, Ly=1, n=1024, u1=True, ham="heisenberg", pbc=True),
        # the energy gradient of that chain: a weighted sum over all samples,
        # through torch autograd
        dict(name="grad_sum_chain100_fp32", kind="grad_sum", model="chain", hidden=64, precision="fp32",
             Lx=100, Ly=1, n=4096, u1=True),
        # local energies of the 10x10 lattice on the tensor cores
        dict(name="eloc_square10_bf16", kind="eloc", model="chain", hidden=128, precision="bf16",
             Lx=10, Ly=10, n=2048, u1=True, ham="heisenberg", pbc=False),
        # O_k rows of the 10x10 lattice, as a covariance or SR solve reads them
        dict(name="ok_rows_square10_bf16", kind="ok_rows", model="chain", hidden=128, precision="bf16",
             Lx=10, Ly=10, n=2048, u1=True),
        # the headline workload, all outputs of a step at 52x52, the largest
        # call (128 of its samples)
        dict(name="step_square52_bf16", kind="step", model="chain", hidden=128, precision="bf16",
             Lx=52, Ly=52, n=128, u1=True, ham="heisenberg", pbc=False),
        # exact samples of the 10x10 lattice, one training step's worth
        dict(name="sample_square10_bf16", kind="sample", model="chain", hidden=128, precision="bf16",
             Lx=10, Ly=10, n=1024, u1=True),
        # the recurrence of one layer of the 52x52 model for the paper's 200 samples
        dict(name="scan_square52", kind="scan", n=200, N=52 * 52, hidden=128),
        # the paper's 1D model (Table I): local energies and gradient of the
        # 256-site transverse-field Ising chain, 1024 samples
        dict(name="eloc_lru256_fp16", kind="eloc", model="lru", hidden=64, precision="fp16",
             Lx=256, Ly=1, n=1024, u1=False, ham="tfim", pbc=False),
        dict(name="grad_sum_lru256", kind="grad_sum", model="lru", hidden=64, precision="fp32",
             Lx=256, Ly=1, n=1024, u1=False),
        # the paper's 2D model (Table V: width 256, 200 samples): local energies
        # at 16x16, and a whole c4v-symmetrised training step at 10x10
        dict(name="eloc_patched16_fp16", kind="eloc", model="2d", hidden=256, precision="fp16",
             Lx=16, Ly=16, n=200, u1=True, ham="heisenberg", pbc=False),
        dict(name="vmc_step_patched10_fp16", kind="vmc_step", model="2d", hidden=256, precision="fp16",
             Lx=10, Ly=10, n=200, u1=True, ham="heisenberg", pbc=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same kinds, over the whole range of sizes."""
    while True:
        c = _draw(rng)
        w = work(c)
        if (w["flops"] <= _MOST_FLOPS[_rate(c)] and w["bytes"] <= 5e9
                and c["n"] * _param_count(c) * 4 <= 3e9 * (1 if c["kind"] in ("ok_rows", "step") else 1e9)):
            return c


# What keeps a drawn case under the largest listed one's time, by the unit
# that runs its products: tensor cores, FP32 lanes, the FP32 samplers' and
# gradients' dependent chains.
_MOST_FLOPS = {"tensor": 5e13, "fp32": 1.2e12, "chain": 1e12}


def _rate(c):
    if c["kind"] in ("sample", "grad_sum", "vmc_step"):
        return "tensor" if c["kind"] == "vmc_step" else "chain"
    return "fp32" if c.get("precision") == "fp32" else "tensor"


def _draw(rng):
    kind = rng.choice(["logpsi", "eloc", "eloc", "grad_sum", "ok_rows", "step", "sample", "scan", "eloc", "grad_sum",
                       "eloc", "vmc_step"])
    if kind == "scan":
        return dict(kind=kind, n=_log_int(rng, 8, 2048), N=_log_int(rng, 64, 2704), hidden=rng.choice([32, 64, 128]))
    if kind == "vmc_step":
        L = rng.choice([6, 8, 10])
        return dict(kind=kind, model="2d", hidden=rng.choice([128, 256]), precision="fp16", Lx=L, Ly=L,
                    n=rng.randint(50, 200), u1=True, ham="heisenberg", pbc=False)
    models = {"logpsi": ["chain", "lru", "2d"], "eloc": ["chain", "chain", "lru", "2d"], "grad_sum": ["chain", "lru"],
              "ok_rows": ["chain"], "step": ["chain"], "sample": ["chain", "lru", "2d"]}[kind]
    model = rng.choice(models)
    c = dict(kind=kind, model=model)
    if model == "chain":
        tensor = kind in ("ok_rows", "step") or (kind != "grad_sum" and rng.random() < 0.6)
        c.update(precision="bf16" if tensor else "fp32", hidden=128 if tensor else rng.choice([32, 64, 128]))
        square = tensor or rng.random() < 0.4
    elif model == "lru":
        c.update(precision="fp32" if kind == "grad_sum" else rng.choice(["fp16", "fp16", "bf16"]), hidden=64)
        square = False
    else:
        c.update(precision="fp32" if kind == "sample" else "fp16", hidden=rng.choice([128, 256]))
        square = True
    if square:
        Lx = _log_int(rng, 5, 52 if kind in ("step", "logpsi", "ok_rows") else 24)
        Ly = max(2, Lx + rng.choice([0, 0, 0, -1, 1]))
        if model == "2d":
            Lx, Ly = 2 * (Lx // 2), 2 * (Ly // 2)
        Lx = max(Lx, 4)
    else:
        Lx, Ly = _log_int(rng, 12, 256), 1
    c.update(Lx=Lx, Ly=Ly, n=_log_int(rng, 24, 8192))
    c["u1"] = Lx * Ly % 2 == 0 and rng.random() < 0.7
    if kind in ("eloc", "step"):
        c["ham"] = "heisenberg" if c["u1"] else "tfim"
        c["pbc"] = Lx % 2 == 0 and Ly % 2 == 0 or Ly == 1 and Lx % 2 == 0
        c["pbc"] = bool(c["pbc"] and rng.random() < 0.3)
    return c


# ----------------------------------------------------------------- the inputs

def _glorot(shapes, seed):
    parts, off = [], 0
    for _, shape, weight in shapes:
        k = int(np.prod(shape))
        lim = math.sqrt(6.0 / sum(shape)) if weight else 0.0
        parts.append((2.0 * inputs.uniform(seed, (k,), offset=off) - 1.0) * lim)
        off += k
    return np.concatenate(parts).astype(np.float32)


def _shapes(c):
    """(name, shape) of every tensor in the flat parameter vector."""
    H = c["hidden"]
    if c["model"] == "lru":
        return [(s[0], s[1]) for s in inputs.param_shapes_lru(_LAYERS, H)]
    f = inputs.param_shapes2d if c["model"] == "2d" else inputs.param_shapes
    return [(s[0], s[1]) for s in f(_LAYERS, H)]


def _param_count(c):
    return 0 if c["kind"] == "scan" else sum(int(np.prod(s)) for _, s in _shapes(c))


def _theta(c, seed):
    H = c["hidden"]
    if c["model"] == "lru":
        return inputs.lru_params(_LAYERS, H, seed)
    if c["model"] == "2d":
        return inputs.glorot_params2d(_LAYERS, H, seed)
    return inputs.glorot_params(_LAYERS, H, seed)


def _spins(c, seed):
    """Samples as a training run meets them: antiferromagnetic on lattices, at
    zero magnetisation where the model keeps it, independent spins otherwise."""
    n, N = c["n"], c["Lx"] * c["Ly"]
    if not c["u1"]:
        return inputs.random_spins(seed, n, N)
    if c["Ly"] == 1:
        return inputs.zero_magnetisation_spins(seed, n, N)
    return inputs.neel_like_spins(seed, n, c["Lx"], c["Ly"])


def _data(c, seed):
    """The arrays of a case, made from the seed alone: name -> device tensor."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    rand = lambda *shape: torch.rand(shape, generator=g, device=dev, dtype=torch.float32)
    if c["kind"] == "scan":
        a, b, h0 = inputs.scan_inputs_device(seed, c["n"], c["N"], c["hidden"], dev)
        return dict(a=a, b=b, h0=h0)
    d = dict(theta=torch.from_numpy(_theta(c, seed)).to(dev))
    n, N = c["n"], c["Lx"] * c["Ly"]
    if c["kind"] in ("sample", "vmc_step"):
        d["uniforms"] = rand(n, N // 4 if c["model"] == "2d" else N)
    else:
        d["spins"] = torch.from_numpy(_spins(c, seed)).to(dev)
    if c["kind"] == "grad_sum":
        # 2/n (E_loc - mean) of a step: centred, of the order of 1/n
        w = torch.randn((n,), generator=g, device=dev, dtype=torch.float32)
        d["weights"] = (w - w.mean()) * (2.0 / n)
    if c["kind"] == "vmc_step":
        d["picks"] = rand(n)
        # moments of a run that has been going for a while
        d["m"] = (rand(d["theta"].numel()) - 0.5) * 2e-2
        d["v"] = rand(d["theta"].numel()) * 1e-4 + 1e-6
    return d


_ADAM_STEP = 100


def prepare(case, seed):
    c, d = case, _data(case, seed)
    s = dict(d, case=c)
    if c["kind"] == "scan":
        return s
    s["cfg"] = api.ModelConfig(_LAYERS, c["hidden"], c["u1"], c["precision"])
    if "ham" in c:
        s["ham"] = binding.make_hamiltonian(c["ham"], c["Lx"], c["Ly"], c["pbc"], True, 1.0, _field(c))
    if c["kind"] == "grad_sum" and c["model"] == "chain":
        s["theta"].requires_grad_(True)
    if c["kind"] == "vmc_step":
        s["adam"] = api.Adam(d["theta"].numel(), d["theta"].device)
        s["adam"].m, s["adam"].v, s["adam"].step = d["m"], d["v"], _ADAM_STEP
    return s


def _field(c):
    """Transverse field: critical in one and in two dimensions."""
    return 0.0 if c["ham"] == "heisenberg" else 1.0 if c["Ly"] == 1 else 3.044


def run(state):
    c, cfg = state["case"], state.get("cfg")
    kind, model = c["kind"], c.get("model")
    if kind == "scan":
        return api.scan(state["a"], state["b"], state["h0"])
    theta = state["theta"]
    if kind == "logpsi":
        if model == "2d":
            return api.logpsi2d(theta, state["spins"], cfg, c["Lx"], c["Ly"])
        return (api.logpsi_lru if model == "lru" else api.logpsi)(theta, state["spins"], cfg)
    if kind == "eloc":
        f = {"chain": api.local_energy, "lru": api.local_energy_lru, "2d": api.local_energy2d}[model]
        return f(theta, state["spins"], cfg, state["ham"])[0]
    if kind == "grad_sum":
        if model == "lru":
            return api.grad_lru(theta, state["spins"], cfg, dout=state["weights"])
        lp = api.LogPsi.apply(theta, state["spins"], cfg)
        (g,) = torch.autograd.grad(lp, theta, grad_outputs=state["weights"])
        return dict(logpsi=lp.detach(), grad=g)
    if kind == "ok_rows":
        return api.grad(theta, state["spins"], cfg)
    if kind == "step":
        o = api.step_batch(theta, [(state["spins"], state["ham"], c["u1"])], cfg)[0]
        return dict(logpsi=o["logpsi"], eloc=o["eloc"], grad=o["grad"])
    if kind == "sample":
        if model == "2d":
            s, lp = api.sample2d(theta, state["uniforms"], cfg, c["Lx"], c["Ly"])
        else:
            s, lp = (api.sample_lru if model == "lru" else api.sample)(theta, state["uniforms"], cfg)
        return dict(spins=s, logpsi=lp)
    o = api.vmc_step2d(theta, cfg, state["ham"], state["uniforms"], state["adam"], symmetrize=True,
                       sym_uniforms=state["picks"])
    return dict(theta=o["theta"], spins=o["spins"], eloc=o["eloc"], grad=o["grad"], m=state["adam"].m,
                v=state["adam"].v)


# ------------------------------------------------------------------- the work

def _flops_per_site(c):
    """Products of one evaluated site (one patch of the 2D model)."""
    H = c["hidden"]
    return {"chain": 18, "lru": 32, "2d": 24}[c["model"]] * H * H


def _connected_per_sample(c):
    Lx, Ly = c["Lx"], c["Ly"]
    if c["ham"] == "tfim":
        return Lx * Ly
    wrap = lambda L: 1 if c["pbc"] and L >= 3 else 0
    bonds = Ly * (Lx - 1 + wrap(Lx)) + Lx * (Ly - 1 + wrap(Ly))
    return bonds * (0.5 if Ly == 1 else 0.72)


def work(case):
    c = case
    n = c["n"]
    if c["kind"] == "scan":
        e = n * c["N"] * c["hidden"]
        return dict(bytes=12 * e + 4 * n * c["hidden"], flops=2 * e)
    N, P = c["Lx"] * c["Ly"], _param_count(c)
    sites = N // 4 if c["model"] == "2d" else N
    site = _flops_per_site(c)
    # a connected configuration differs from its sample from the first flipped
    # site on: half of the sites on average
    connected = n * _connected_per_sample(c) * sites * 0.5 if "ham" in c else 0
    b = 4 * P + n * N
    f = {"logpsi": n * sites, "eloc": n * sites + connected, "grad_sum": 3 * n * sites, "ok_rows": 3 * n * sites,
         "step": 3 * n * sites + connected, "sample": n * sites, "vmc_step": n * sites * (1 + 8 * 3) + 8 * connected}
    if c["kind"] in ("ok_rows", "step"):
        b += 4 * n * P
    if c["kind"] in ("sample", "vmc_step"):
        b += 4 * n * sites
    if c["kind"] == "grad_sum":
        b += 4 * P
    if c["kind"] == "vmc_step":
        b += 4 * 6 * P
    return dict(bytes=b + 4 * n, flops=f[c["kind"]] * site)


# ------------------------------------------------- the same in plain torch, FP64

_MOST_EXACT = 1.2e13  # FP64 operations of a case that stay well under 20 seconds


def _exact_flops(c):
    """Whole forwards of every connected configuration, nothing shared."""
    sites = c["Lx"] * c["Ly"] // (4 if c["model"] == "2d" else 1)
    per = 6 + (_connected_per_sample(c) if "ham" in c else 0)
    images = 8 if c["kind"] == "vmc_step" else 1
    return c["n"] * per * sites * _flops_per_site(c) * images


def _tensors(c, theta):
    out, off = {}, 0
    for name, shape in _shapes(c):
        k = int(np.prod(shape))
        out[name] = theta[off:off + k].reshape(shape)
        off += k
    return out


def _onehot_prev(s):
    """[n, N, 2] one-hot of the spin before each site, zero at the first."""
    x = torch.nn.functional.one_hot(s.long(), 2).to(torch.float64)
    return torch.cat([torch.zeros_like(x[:, :1]), x[:, :-1]], 1)


def _two_way(d, s, u1):
    """log psi from the logit differences d [n, N] of the spins s."""
    sf = s.to(torch.float64)
    lp = -torch.nn.functional.softplus(torch.where(s.bool(), -d, d))
    if u1:
        N = s.shape[1]
        up = torch.cumsum(sf, 1) - sf
        down = torch.arange(N, device=s.device, dtype=torch.float64) - up
        full_up, full_down = up >= N // 2, down >= N // 2
        lp = torch.where(full_up, torch.where(s.bool(), -math.inf, 0.0),
                         torch.where(full_down, torch.where(s.bool(), 0.0, -math.inf), lp))
    return 0.5 * lp.sum(1)


def _scan64(a, b, h):
    out = []
    for t in range(a.shape[1]):
        h = a[:, t] * h + b[:, t]
        out.append(h)
    return torch.stack(out, 1)


def _chain64(c, p, s, linear=torch.nn.functional.linear):
    """log psi of the chain minGRU; `linear` may record what it is given."""
    u, below = _onehot_prev(s), None
    for l in range(_LAYERS):
        a = torch.sigmoid(linear(u, p["W_z%d" % l], p["b_z%d" % l]))
        h = _scan64(a, (1 - a) * linear(u, p["W_h%d" % l], p["b_h%d" % l]), torch.zeros_like(a[:, 0]))
        y = linear(h, p["C%d" % l]) + linear(u, p["D%d" % l])
        if l >= 2:
            y = y + below
        u, below = torch.nn.functional.gelu(y), h
    logits = linear(u, p["W_o"], p["b_o"])
    return _two_way(logits[..., 1] - logits[..., 0], s, c["u1"])


def _lru64(c, p, s):
    linear = torch.nn.functional.linear
    u = _onehot_prev(s)
    for l in range(_LAYERS):
        q = lambda k: p["%s%d" % (k, l)]
        r, ph = torch.exp(-torch.exp(q("nu"))), torch.exp(q("theta"))
        lre, lim, g = r * torch.cos(ph), r * torch.sin(ph), torch.exp(q("gamma"))
        bre, bim = g * linear(u, q("B_re")), g * linear(u, q("B_im"))
        hre, him, outs = torch.zeros_like(bre[:, 0]), torch.zeros_like(bre[:, 0]), []
        for t in range(s.shape[1]):
            hre, him = lre * hre - lim * him + bre[:, t], lre * him + lim * hre + bim[:, t]
            outs.append((hre, him))
        y = linear(torch.stack([o[0] for o in outs], 1), q("C_re")) - linear(
            torch.stack([o[1] for o in outs], 1), q("C_im"))
        y = y + (linear(u, q("D")) if l == 0 else q("D") * u)
        x = linear(y, q("W_a"), q("b_a")) * torch.sigmoid(linear(y, q("W_g"), q("b_g")))
        u = x if l == 0 else x + u
    logits = linear(u, p["W_o"], p["b_o"])
    return _two_way(logits[..., 1] - logits[..., 0], s, c["u1"])


def _seq_pos(Lx, i, j):
    return j * Lx + (i if j % 2 == 0 else Lx - 1 - i)


def _patch_sites(c):
    """[Np, 4] sequence positions of the spins of every patch in path order."""
    Px, Py = c["Lx"] // 2, c["Ly"] // 2
    path = [(k if j % 2 == 0 else Px - 1 - k, j) for j in range(Py) for k in range(Px)]
    return torch.tensor([[_seq_pos(c["Lx"], 2 * i + dx, 2 * j + dy) for dy in (0, 1) for dx in (0, 1)]
                         for i, j in path], device="cuda")


def _patch_mask(c, ups, t):
    """[..., 16] values allowed after `ups` of the first t patches' spins."""
    pop = torch.tensor([bin(v).count("1") for v in range(16)], device="cuda")
    half = c["Lx"] * c["Ly"] // 2
    if not c["u1"]:
        return torch.ones(ups.shape + (16,), dtype=torch.bool, device="cuda")
    return (ups[..., None] + pop <= half) & (4 * t - ups[..., None] + 4 - pop <= half)


def _patched64(c, p, s, draws=None):
    """log psi of the 2D patched minGRU, patch by patch along the path; with
    `draws` [n, Np] the spins are drawn on the way and returned too."""
    linear, gelu = torch.nn.functional.linear, torch.nn.functional.gelu
    Px, Py, H = c["Lx"] // 2, c["Ly"] // 2, c["hidden"]
    where = _patch_sites(c)
    n = draws.shape[0] if s is None else s.shape[0]
    zero = torch.zeros((n, H), dtype=torch.float64, device="cuda")
    none = torch.zeros((n, 16), dtype=torch.float64, device="cuda")
    ups = torch.zeros(n, dtype=torch.long, device="cuda")
    bit = torch.tensor([1, 2, 4, 8], device="cuda")
    spins = torch.zeros((n, c["Lx"] * c["Ly"]), dtype=torch.uint8, device="cuda") if s is None else s
    above, above_v = [[zero] * _LAYERS for _ in range(Px)], [none] * Px
    total = 0.0
    for t in range(Px * Py):
        j, k = divmod(t, Px)
        i = k if j % 2 == 0 else Px - 1 - k
        if k == 0:
            left, left_v = [zero] * _LAYERS, none
        u, states = torch.cat([left_v, above_v[i]], 1), []
        for l in range(_LAYERS):
            q = lambda w: p["%s%d" % (w, l)]
            z = torch.sigmoid(linear(u, q("W_z"), q("b_z")))
            h = z * left[l] + (1 - z) * linear(torch.cat([u, above[i][l]], 1), q("W_h"), q("b_h"))
            y = linear(h, q("C")) + linear(u, q("D"))
            if l >= 2:
                y = y + states[l - 1]
            u = gelu(y)
            states.append(h)
        ok = _patch_mask(c, ups, t)
        lp = torch.log_softmax(torch.where(ok, linear(u, p["W_o"], p["b_o"]), -math.inf), 1)
        if s is None:
            over = (torch.cumsum(lp.exp(), 1) > draws[:, t:t + 1]) & ok
            last = 15 - ok.flip(1).int().argmax(1)
            v = torch.where(over.any(1), over.int().argmax(1), last)
            spins[:, where[t]] = ((v[:, None] & bit) > 0).to(torch.uint8)
        else:
            v = (s[:, where[t]].long() * bit).sum(1)
        total = total + lp.gather(1, v[:, None])[:, 0]
        ups = ups + ((v[:, None] & bit) > 0).sum(1)
        above[i], left = states, states
        left_v = torch.nn.functional.one_hot(v, 16).to(torch.float64)
        above_v[i] = left_v
    return (0.5 * total, spins) if s is None else 0.5 * total


_MODELS = {"chain": _chain64, "lru": _lru64, "2d": _patched64}


def _in_parts(c, f, s, most=1 << 20):
    """f over parts of the configurations, about `most` sites at a time."""
    k = max(1, most // s.shape[1])
    return torch.cat([f(s[i:i + k]) for i in range(0, s.shape[0], k)])


def _bonds(c):
    Lx, Ly, out = c["Lx"], c["Ly"], []
    for j in range(Ly):
        for i in range(Lx):
            for a, b in ((i + 1, j), (i, j + 1)):
                if c["pbc"]:
                    a, b = a % Lx if Lx >= 3 else a, b % Ly if Ly >= 3 else b
                if a < Lx and b < Ly and (a, b) != (i, j):
                    out.append((_seq_pos(Lx, i, j), _seq_pos(Lx, a, b)))
    return torch.tensor(out, device="cuda").reshape(-1, 2)


def _eloc64(c, logpsi, s):
    """diag + sum over connected configurations of c psi(s') / psi(s), J = 1."""
    n, N = s.shape
    bonds = _bonds(c)
    sp, sq = s[:, bonds[:, 0]], s[:, bonds[:, 1]]
    z = torch.where(sp == sq, 1.0, -1.0).to(torch.float64).sum(1)
    if c["ham"] == "heisenberg":
        at, which = torch.nonzero(sp != sq, as_tuple=True)
        flips, diag, coeff = bonds[which], 0.25 * z, -0.5
    else:
        at = torch.arange(n, device="cuda").repeat_interleave(N)
        flips, diag, coeff = torch.arange(N, device="cuda").repeat(n)[:, None], -z, -_field(c)
    base = logpsi(s)
    out = diag.clone()
    step = max(1, (1 << 25) // N)
    for i in range(0, at.numel(), step):
        smp = at[i:i + step]
        x = s[smp]
        x.scatter_(1, flips[i:i + step], 1 - x.gather(1, flips[i:i + step]))
        out.index_add_(0, smp, coeff * torch.exp(logpsi(x) - base[smp]))
    return out


def _rows64(c, theta, s):
    """(log psi, per-sample gradient rows) of the chain: gradients of every
    linear map's output by autograd, then a sum over sites for each sample."""
    p, seen = _tensors(c, theta), []

    def linear(u, W, b=None):
        y = torch.nn.functional.linear(u, W, b).requires_grad_(True)
        seen.append((u.detach(), y, b is not None))
        return y

    lp = _chain64(c, p, s, linear)
    gs = torch.autograd.grad(lp.sum(), [y for _, y, _ in seen])
    rows = []
    for (u, _, bias), g in zip(seen, gs):
        rows.append(torch.einsum("nth,ntk->nhk", g, u).flatten(1))
        if bias:
            rows.append(g.sum(1))
    return lp.detach(), torch.cat(rows, 1)


def _images(L):
    """[8, L * L] source positions of the images of a configuration under c4v."""
    m = L - 1
    ops = [lambda i, j: (i, j), lambda i, j: (m - j, i), lambda i, j: (m - i, m - j), lambda i, j: (j, m - i),
           lambda i, j: (m - i, j), lambda i, j: (i, m - j), lambda i, j: (j, i), lambda i, j: (m - j, m - i)]
    maps = torch.empty((8, L * L), dtype=torch.long)
    for g, op in enumerate(ops):
        for j in range(L):
            for i in range(L):
                maps[g, _seq_pos(L, *op(i, j))] = _seq_pos(L, i, j)
    return maps.cuda()


def _vmc64(c, d, theta):
    p, maps = _tensors(c, theta), _images(c["Lx"])
    drawn = _patched64(c, p, None, d["uniforms"].double())[1]
    pick = torch.clamp((8.0 * d["picks"]).floor().long(), 0, 7)
    s = drawn.gather(1, maps[pick])
    log8 = math.log(8.0)
    plain = lambda x: _in_parts(c, lambda y: _patched64(c, p, y), x)
    sym = lambda x: 0.5 * (torch.logsumexp(torch.stack([2 * plain(x[:, m]) for m in maps]), 0) - log8)
    eloc = _eloc64(c, sym, s)
    w = 2.0 / c["n"] * (eloc - eloc.mean())
    t = theta.clone().requires_grad_(True)
    q = _tensors(c, t)
    lp = torch.stack([_patched64(c, q, s[:, m]) for m in maps])
    (g,) = torch.autograd.grad((0.5 * torch.logsumexp(2 * lp, 0) * w).sum(), t)
    b1, b2, k = 0.9, 0.999, _ADAM_STEP + 1
    m, v = b1 * d["m"].double() + (1 - b1) * g, b2 * d["v"].double() + (1 - b2) * g * g
    new = theta - 1e-3 * (m / (1 - b1 ** k)) / (torch.sqrt(v / (1 - b2 ** k)) + 1e-8)
    return dict(theta=new, spins=None, eloc=eloc, grad=g, m=m, v=v)


def exact(case, seed):
    c = case
    d = _data(c, seed)
    if c["kind"] == "scan":
        return _scan64(d["a"].double(), d["b"].double(), d["h0"].double())
    kind, theta = c["kind"], d["theta"].double()
    small = _exact_flops(c) <= _MOST_EXACT
    if kind == "vmc_step":
        return _vmc64(c, d, theta) if small else None
    if kind == "sample":
        return None  # the draws decide what log psi is of
    s = d["spins"]
    if kind == "step":
        lp, rows = _rows64(c, theta, s)
        p = _tensors(c, theta)
        f = lambda x: _in_parts(c, lambda y: _chain64(c, p, y), x)
        return dict(logpsi=lp, eloc=_eloc64(c, f, s) if small else None, grad=rows)
    if not small:
        return None
    if kind == "ok_rows":
        k = max(1, (1 << 19) // s.shape[1])
        return torch.cat([_rows64(c, theta, s[i:i + k])[1] for i in range(0, s.shape[0], k)])
    if kind == "grad_sum":
        t = theta.clone().requires_grad_(True)
        total, lps, k = torch.zeros_like(theta), [], max(1, (1 << 19) // s.shape[1])
        for i in range(0, s.shape[0], k):
            lp = _MODELS[c["model"]](c, _tensors(c, t), s[i:i + k])
            (g,) = torch.autograd.grad((lp * d["weights"][i:i + k].double()).sum(), t)
            total += g
            lps.append(lp.detach())
        return total if c["model"] == "lru" else dict(logpsi=torch.cat(lps), grad=total)
    p = _tensors(c, theta)
    f = lambda x: _in_parts(c, lambda y: _MODELS[c["model"]](c, p, y), x)
    return f(s) if kind == "logpsi" else _eloc64(c, f, s)
