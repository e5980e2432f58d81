"""The calls this library is used for, as timed cases.

A case is one pass of a user's program through the public binding
(``paper_2206_02937_gb300``): a particle-in-cell code's collision step (binning
and scattering), its No-Time-Counter form, inference and training of the
surrogate networks, and a served mix of pre-paired batches.  The inputs are the
synthetic particle sets of the benchmark and the tests (log-normal 2D cells of
Maxwell-Juttner electrons and Planck photons, 3D cells of power-law electrons
and a photon beam, log-uniform surrogate samples), drawn on the GPU from the
seed.

``exact`` gives the same results in 64-bit torch arithmetic, written from the
method's definition (the header ``include/compton.h``): Philox4x32-10, the order
by (cell, key, id), the Klein-Nishina cross section and angular cumulative, the
textbook boosts, the networks, their gradients and Adam.
"""
from __future__ import annotations

import math
import time

import numpy as np
import torch

import paper_2206_02937_gb300 as cg

DEV = "cuda"
F64 = torch.float64
DT = 0.05                     # time step of every workload of the benchmark
STEP = 3                      # the step counter of the timed step
LR = 1e-3                     # the paper's learning rate
FEATURES = (1.0, 7.0, 1e-4, 10.0)
MODES = {"plain": cg.MODE_PLAIN, "fp32": cg.MODE_MLP_FP32, "bf16": cg.MODE_MLP_BF16, "fp8": cg.MODE_MLP_FP8,
         "pnet": cg.MODE_PNET}
MLP_SHAPES = ((64, 6), (64, 64), (64, 64), (64, 64), (1, 64))
PNET_SHAPES = ((9, 9), (12, 9), (9, 12), (1, 9))


# --------------------------------------------------------------------------
# The cases
# --------------------------------------------------------------------------
def listed():
    return [
        # a 1D run's step (64 cells of 64 + 64): a call whose time is its launches
        _step("step_1d_64", nx=64, ny=1, ppc=64, plasma="mono", order="cells"),
        # the benchmark's step: 512 x 512 cells, input in cell order (particles that kept their cells)
        _step("step_2d_512", nx=512, ny=512, ppc=64, plasma="thermal", order="cells"),
        # the same plasma after a push in which one particle in ten crossed into a neighbouring cell
        _step("step_2d_512_moved", nx=512, ny=512, ppc=64, plasma="thermal", order="moved"),
        # a first step (particles in no order) with the network in place of the cross section; odd grid
        _step("step_2d_301_bf16", nx=301, ny=257, ppc=40, plasma="thermal", order="any", mode="bf16"),
        # 3D: two million cells of 16, power-law electrons up to gamma = 1e4 on a photon beam
        _step("step_3d_128", nx=128, ny=128 * 128, ppc=16, plasma="beam", order="cells"),
        # No-Time-Counter collisions of a 2D run
        _step("ntc_2d_256", nx=256, ny=256, ppc=64, plasma="thermal", order="cells", mode="ntc"),
        # the network object on a batch of pairs: the tensor-core precision on a large ragged batch ...
        {"name": "infer_bf16_4M", "kind": "infer", "mode": "bf16", "n": 4194301},
        # ... and the reference precision
        {"name": "infer_fp32_1M", "kind": "infer", "mode": "fp32", "n": 1000003},
        # training the network in minibatches of 8192, on the tensor cores and in the default precision
        {"name": "train_bf16_8192", "kind": "train", "mode": "bf16", "n": 8192, "steps": 8},
        {"name": "train_fp32_8192", "kind": "train", "mode": "fp32", "n": 8192, "steps": 4},
        # training the paper's own 9-12-9 network
        {"name": "train_pnet_8192", "kind": "train", "mode": "pnet", "n": 8192, "steps": 8},
        # batches of uneven size submitted together, half of them for the network
        {"name": "serve_24", "kind": "serve", "requests": 24, "lo": 1000, "hi": 1000000},
    ]


def _step(name, nx, ny, ppc, plasma, order, mode="plain", weights=False):
    return {"name": name, "kind": "step", "nx": nx, "ny": ny, "ppc": ppc, "plasma": plasma, "order": order,
            "mode": mode, "weights": weights}


def draw(rng):
    kind = rng.choice(["step"] * 5 + ["infer"] * 2 + ["train"] * 2 + ["serve"])
    if kind == "step":
        ppc = round(_log(rng, 6, 200))
        cells = _log(rng, 64, min(1 << 21, 16.0e6 / ppc))
        nx = max(8, min(1024, round(math.sqrt(cells) * rng.uniform(0.6, 1.6))))
        c = _step("", nx, max(1, round(cells / nx)), ppc, rng.choice(["thermal", "thermal", "beam"]),
                  rng.choice(["cells", "moved", "any"]),
                  rng.choice(["plain", "plain", "plain", "bf16", "fp8", "fp32", "pnet", "ntc"]))
        c["weights"] = c["mode"] != "ntc" and rng.random() < 0.2
    elif kind == "infer":
        mode = rng.choice(["bf16", "fp8", "fp32", "pnet"])
        c = {"kind": kind, "mode": mode, "n": round(_log(rng, 1000, 1e6 if mode == "fp32" else 4e6))}
    elif kind == "train":
        mode = rng.choice(["bf16", "fp32", "pnet"])
        c = {"kind": kind, "mode": mode, "n": round(_log(rng, 256, 65536 if mode == "bf16" else 20000)),
             "steps": rng.choice([2, 4])}
    else:
        lo = round(_log(rng, 500, 20000))
        c = {"kind": kind, "requests": rng.randrange(4, 25), "lo": lo, "hi": round(lo * _log(rng, 4, 100))}
    c.pop("name", None)
    return c


def _log(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def work(case):
    """What a pass cannot do without: every particle's (or sample's) words read
    once and written once; the networks' multiply-adds."""
    kind = case["kind"]
    if kind == "step":
        n = case["nx"] * case["ny"] * case["ppc"]
        # five words per particle (six with weights), both species, in and out
        by = 2 * 2 * n * (24 if case["weights"] else 20)
        cand = 1.0 - math.exp(-2.0 * DT)  # pairs whose uniform lies below the bound of every probability
        per = {"plain": 150, "ntc": 300, "pnet": 612}.get(case["mode"], 25472)
        return {"bytes": by, "flops": n * cand * per}
    if kind == "infer":
        return {"bytes": 28 * case["n"], "flops": case["n"] * (612 if case["mode"] == "pnet" else 25472)}
    if kind == "train":
        n, params = case["n"] * case["steps"], 337 if case["mode"] == "pnet" else 12993
        return {"bytes": 28 * n + case["steps"] * 24 * params,
                "flops": n * (1836 if case["mode"] == "pnet" else 75520)}
    n = sum(_sizes(case))
    return {"bytes": 48 * n, "flops": n * 25472 / 2}


def _sizes(case):
    """Request sizes spread over [lo, hi] by their logarithm, odd ones, small and large in turn."""
    r, span = case["requests"], case["hi"] / case["lo"]
    sizes = [int(case["lo"] * span ** ((i + 0.5) / r)) | 1 for i in range(r)]
    return [sizes[i // 2 if i % 2 == 0 else r - 1 - i // 2] for i in range(r)]


# --------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) + 1000)
    return g


def _uniform(g, *shape, lo=0.0, hi=1.0):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float32) * (hi - lo) + lo


def _isotropic(g, n):
    mu = _uniform(g, n, lo=-1.0, hi=1.0)
    phi = _uniform(g, n, hi=2.0 * math.pi)
    s = torch.sqrt(torch.clamp(1.0 - mu * mu, min=0.0))
    return torch.stack([s * torch.cos(phi), s * torch.sin(phi), mu])


def _maxwell_juttner(g, n):
    """|u| at temperature theta = 1, by Sobol's rejection method."""
    out, have = [], 0
    while have < n:
        x = torch.log(torch.clamp(_uniform(g, 4, int((n - have) * 1.7) + 64), min=1e-30))
        u = -(x[0] + x[1] + x[2])
        eta = u - x[3]
        u = u[eta * eta - u * u > 1.0]
        out.append(u)
        have += int(u.shape[0])
    return torch.cat(out)[:n]


def _planck(g, n, kt=1e-2):
    """Photon energies with density eps^2 / (exp(eps / kt) - 1)."""
    y = torch.linspace(1e-4, 40.0, 40001, device=DEV, dtype=F64)
    f = y * y / torch.expm1(y)
    cdf = torch.cumsum(f, 0) - 0.5 * (f + f[0])
    cdf = (cdf / cdf[-1]).float()
    r = _uniform(g, n)
    i = torch.clamp(torch.searchsorted(cdf, r), 1, cdf.shape[0] - 1)
    c0, c1 = cdf[i - 1], cdf[i]
    frac = torch.where(c1 > c0, (r - c0) / (c1 - c0), torch.zeros_like(r))
    yf = y.float()
    return kt * (yf[i - 1] + frac * (yf[i] - yf[i - 1]))


def _momenta(g, n, plasma):
    if plasma == "mono":  # gamma = 10 electrons, photons of energy 1e-3
        return math.sqrt(99.0) * _isotropic(g, n), 1e-3 * _isotropic(g, n)
    if plasma == "beam":  # dN/dgamma ~ gamma^-2 on [1, 1e4], photons of energy 1e-2 along +x
        gamma = 1.0 / (1.0 - _uniform(g, n) * (1.0 - 1e-4))
        k = torch.zeros(3, n, device=DEV)
        k[0] = 1e-2
        return torch.sqrt(torch.clamp(gamma * gamma - 1.0, min=0.0)) * _isotropic(g, n), k
    return _maxwell_juttner(g, n) * _isotropic(g, n), _planck(g, n) * _isotropic(g, n)


def _samples(g, n):
    """Surrogate samples: gamma log-uniform on [1, 1e3], eps log-uniform on [1e-4, 1], isotropic."""
    gamma = 10.0 ** _uniform(g, n, hi=3.0)
    eps = 10.0 ** _uniform(g, n, lo=-4.0, hi=0.0)
    u = torch.sqrt(torch.clamp(gamma * gamma - 1.0, min=0.0)) * _isotropic(g, n)
    return u.contiguous(), (eps * _isotropic(g, n)).contiguous()


def _plasma(case, seed):
    """Both species of a step: (ux, uy, uz, cell, id, weight or None) each."""
    g = _gen(seed)
    nx, cells, ppc = case["nx"], case["nx"] * case["ny"], case["ppc"]
    if case["plasma"] == "thermal":  # log-normal density, shared by both species; ppc per cell in the mean
        edges = torch.cumsum(torch.exp(0.5 * torch.randn(cells, generator=g, device=DEV)).to(F64), 0)
        edges = torch.floor(edges * (cells * ppc / float(edges[-1])) + 0.5).to(torch.int64)
        counts = torch.diff(edges, prepend=edges.new_zeros(1))
    else:
        counts = torch.full((cells,), ppc, device=DEV, dtype=torch.int64)
    base = torch.repeat_interleave(torch.arange(cells, device=DEV, dtype=torch.int32), counts)
    n = int(base.shape[0])
    species = []
    for mom in _momenta(g, n, case["plasma"]):
        cell = base.clone()
        if case["order"] == "any":
            cell = cell[torch.randperm(n, generator=g, device=DEV)]
        elif case["order"] == "moved":
            hop = torch.tensor([1, -1, nx, -nx], device=DEV, dtype=torch.int32)
            hop = hop[torch.randint(0, 4, (n,), generator=g, device=DEV)]
            cell = torch.where(_uniform(g, n) < 0.1, torch.remainder(cell + hop, cells).to(torch.int32), cell)
        ident = torch.randperm(n, generator=g, device=DEV).to(torch.int32)
        w = _uniform(g, n, lo=0.5, hi=2.0) / ppc if case["weights"] else None
        species.append([mom[0].contiguous(), mom[1].contiguous(), mom[2].contiguous(), cell.contiguous(), ident, w])
    return species


def _theta(shapes, seed, bias=0.0):
    """Glorot-uniform weights, zero biases but the output's."""
    rng = np.random.default_rng(int(seed) + 77)
    parts = []
    for o, i in shapes:
        lim = math.sqrt(6.0 / (o + i))
        parts += [rng.uniform(-lim, lim, o * i), np.zeros(o)]
    parts[-1][:] = bias
    return np.concatenate(parts).astype(np.float32)


def _served(case, seed):
    """The requests of a serving case: (u, k, mode) each."""
    g = _gen(seed)
    out = []
    for i, n in enumerate(_sizes(case)):
        u, k = _momenta(g, n, "thermal")
        out.append((u.contiguous(), k.contiguous(), "bf16" if (i // 2) % 2 else "plain"))
    return out


class _Context:
    """A library context, given back when its state is dropped."""

    def __init__(self, **config):
        self.ctx = cg.compton_init(**config)

    def __del__(self):
        try:
            cg.compton_destroy(self.ctx)
        except Exception:
            pass


def _w_over_v(case):
    return 1.0 / case["ppc"]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        e, g = (cg.Species(*s) for s in _plasma(case, seed))
        ctx = _Context(n_cells=case["nx"] * case["ny"], max_particles=e.n, w_over_v=_w_over_v(case), dt=DT,
                       seed=int(seed))
        _load(ctx.ctx, case["mode"], seed)
        return {"case": case, "ctx": ctx, "e": e, "g": g, "e_out": cg.Species.empty_like(e),
                "g_out": cg.Species.empty_like(g)}
    if kind == "infer":
        u, k = _samples(_gen(seed), case["n"])
        ctx = _Context(n_cells=1, max_particles=1, w_over_v=1.0, dt=DT, seed=int(seed))
        _load(ctx.ctx, case["mode"], seed)
        return {"case": case, "ctx": ctx, "u": u, "k": k, "r": torch.empty(case["n"], device=DEV)}
    if kind == "train":
        u, k, y, theta = _training_set(case, seed)
        ctx = _Context(n_cells=1, max_particles=1, w_over_v=1.0, dt=DT, seed=int(seed), max_train_batch=case["n"])
        if case["mode"] == "pnet":
            cg.compton_pnet_set_params(ctx.ctx, theta)
        else:
            cg.compton_mlp_set_params(ctx.ctx, theta)
            cg.compton_mlp_set_train_precision(ctx.ctx, MODES[case["mode"]])
        cuts = [slice(i * case["n"], (i + 1) * case["n"]) for i in range(case["steps"])]
        return {"case": case, "ctx": ctx, "batches": [(u[:, s], k[:, s], y[s]) for s in cuts]}
    requests = _served(case, seed)
    pairs = sum(int(u.shape[1]) for u, _, _ in requests)
    ctx = _Context(n_cells=1, max_particles=1, w_over_v=1.0, dt=DT, seed=int(seed))
    _load(ctx.ctx, "bf16", seed)
    cg.compton_serve_start(ctx.ctx, 40 * pairs + (1 << 20))
    return {"case": case, "ctx": ctx, "requests": requests,
            "out": [(torch.empty_like(u), torch.empty_like(k)) for u, k, _ in requests]}


def _load(ctx, mode, seed):
    if mode in ("bf16", "fp8", "fp32"):
        cg.compton_mlp_set_params(ctx, _theta(MLP_SHAPES, seed))
        if mode == "fp8":
            cg.compton_mlp_calibrate(ctx, *_samples(_gen(seed + 1), 16384))
    elif mode == "pnet":
        cg.compton_pnet_set_params(ctx, _theta(PNET_SHAPES, seed))


def _training_set(case, seed):
    n = case["n"] * case["steps"]
    u, k = _samples(_gen(seed), n)
    x, v = _invariants(u.to(F64), k.to(F64))
    y = (0.5 * _sigma(x) * v).float()
    if case["mode"] == "pnet":  # the output starts at the median target
        m = float(torch.quantile(y[:4096], 0.5))
        return u, k, y, _theta(PNET_SHAPES, seed, math.log(m / (1.0 - m)))
    return u, k, y, _theta(MLP_SHAPES, seed)


# --------------------------------------------------------------------------
# One pass
# --------------------------------------------------------------------------
PNET_ROW = (0.015625, 0.015625, 0.1)  # weights of both particles and P_max of an explicit row


def run(state):
    case, ctx = state["case"], state["ctx"].ctx
    kind, mode = case["kind"], case.get("mode")
    if kind == "step":
        e, g = state["e_out"], state["g_out"]
        pairs = cg.compton_bin_pairs(ctx, state["e"], state["g"], e, g, STEP)
        if mode == "ntc":
            cg.compton_scatter_step_ntc(ctx, e, g, pairs, STEP)
        else:
            cg.compton_scatter_step(ctx, e, g, pairs, MODES[mode], STEP)
        return [[s.ux, s.uy, s.uz, s.cell, s.id] + ([s.w] if case["weights"] else []) for s in (e, g)]
    if kind == "infer":
        if mode == "pnet":
            cg.compton_pnet_infer(ctx, state["u"], state["k"], *PNET_ROW, state["r"])
        else:
            cg.compton_mlp_infer(ctx, state["u"], state["k"], MODES[mode], state["r"])
        return state["r"]
    if kind == "train":
        last = len(state["batches"]) - 1
        for i, (u, k, y) in enumerate(state["batches"]):
            if mode == "pnet":
                loss = cg.compton_pnet_train_step(ctx, u, k, y, None, *PNET_ROW, LR, want_loss=i == last)
            else:
                loss = cg.compton_mlp_train_step(ctx, u, k, y, None, LR, want_loss=i == last)
        theta = cg.compton_pnet_get_params(ctx)[0] if mode == "pnet" else cg.compton_mlp_get_params(ctx)
        return [theta, loss]
    tickets = [cg.compton_submit(ctx, u, k, uo, ko, 1.0, 5000 + i, STEP, MODES[m])
               for i, ((u, k, m), (uo, ko)) in enumerate(zip(state["requests"], state["out"]))]
    hits = []
    for t in tickets:
        while (r := cg.compton_poll(ctx, t)) is None:
            time.sleep(2e-5)
        hits.append(r["scatters"])
    return [state["out"], sum(hits)]


# --------------------------------------------------------------------------
# The same results in 64 bits
# --------------------------------------------------------------------------
M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Four 32-bit words per counter (int64 tensors), Philox4x32-10 under key seed."""
    k0, k1 = seed & M32, (seed >> 32) & M32
    as_words = [torch.as_tensor(c, device=DEV, dtype=torch.int64) for c in (c0, c1, c2, c3)]
    c0, c1, c2, c3 = torch.broadcast_tensors(*as_words)
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57  # modulo 2^64
        c0, c1, c2, c3 = ((p1 >> 32) & M32) ^ c1 ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c3 ^ k1, p0 & M32
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1, c2, c3


def _invariants(u, k):
    """x (photon energy in the electron's rest frame) and v = 1 - beta cos psi."""
    uu, kk = (u * u).sum(0), (k * k).sum(0)
    un, eps, gamma = torch.sqrt(uu), torch.sqrt(kk), torch.sqrt(1.0 + uu)
    norm = torch.clamp(un * eps, min=1e-300)
    c = (u * k).sum(0) / norm
    s2 = (torch.linalg.cross(u, k, dim=0) / norm).square().sum(0)
    omc = torch.where(c > 0.0, s2 / (1.0 + torch.clamp(c, min=0.0)), 1.0 - c)
    v = 1.0 / (gamma * (gamma + un)) + un / gamma * omc
    v = torch.where((un > 0.0) & (eps > 0.0), v, torch.ones_like(v))
    return gamma * eps * v, v


def _cumulative(x, t):
    """Integral of the Klein-Nishina angular density over 1 - cos(theta') from 0 to t, in 3/8 sigma_T."""
    w = x * t
    a = t * (2.0 + w) / (2.0 * (1.0 + w) ** 2)
    z, q = w / (2.0 + w), t / (2.0 + w)
    z2 = z * z
    s1 = torch.zeros_like(w)
    for j in range(24, 0, -1):
        s1 = s1 * z2 + 1.0 / (2 * j + 1)
    s2 = 1.0 / (1.0 - z2) - s1
    series = a + 2.0 * q * (z2 * s1 + 1.0) - 4.0 * q * q * (z * s1 + 1.0 / (1.0 + z) - q * s2)
    xs = torch.clamp(x, min=1e-3)
    log = torch.log1p(w)
    closed = a + log / xs - ((2.0 * xs + 2.0) * log - w - (2.0 * xs + 1.0) * w / (1.0 + w)) / xs ** 3
    return torch.where(w < 1.0, series, closed)


def _sigma(x):
    return 0.375 * _cumulative(x, torch.full_like(x, 2.0))


def _angle(x, word):
    """cos(theta') and the energy ratio for the 24-bit uniform of a word."""
    target = ((word >> 8).to(F64) + 0.5) * 2.0 ** -24 * _cumulative(x, torch.full_like(x, 2.0))
    lo, hi = torch.zeros_like(x), torch.full_like(x, 2.0)
    for _ in range(56):
        mid = 0.5 * (lo + hi)
        below = _cumulative(x, mid) < target
        lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
    t = 0.5 * (lo + hi)
    return 1.0 - t, torch.sqrt(t * (2.0 - t)), 1.0 / (1.0 + x * t)


def _collide(u, k, x, word_angle, word_phi):
    """Both momenta after the collision of each pair."""
    cth, sth, ratio = _angle(x, word_angle)
    gamma = torch.sqrt(1.0 + (u * u).sum(0))
    eps = torch.sqrt((k * k).sum(0))
    r = k + u * ((u * k).sum(0) / (gamma + 1.0) - eps)
    n = r / torch.sqrt((r * r).sum(0))
    sg = torch.where(n[2] >= 0.0, 1.0, -1.0).to(F64)
    a = -1.0 / (sg + n[2])
    b = n[0] * n[1] * a
    b1 = torch.stack([1.0 + sg * n[0] * n[0] * a, sg * b, -sg * n[0]])
    b2 = torch.stack([b, sg + n[1] * n[1] * a, -n[1]])
    phi = 2.0 * math.pi * (word_phi >> 8).to(F64) * 2.0 ** -24
    e1 = x * ratio
    q = e1 * (cth * n + sth * (torch.cos(phi) * b1 + torch.sin(phi) * b2))
    k1 = q + u * ((u * q).sum(0) / (gamma + 1.0) + e1)
    return u + k - k1, k1


def _layers(theta, shapes):
    out, at = [], 0
    for o, i in shapes:
        out.append((theta[at:at + o * i].reshape(o, i), theta[at + o * i:at + o * i + o]))
        at += o * i + o
    return out


def _net_features(u, k, extra=()):
    su, nu, sk, nk = FEATURES
    f = [torch.sign(u) * torch.log1p(u.abs() / su) / nu, torch.sign(k) * torch.log1p(k.abs() / sk) / nk]
    n = u.shape[1]
    f += [(torch.as_tensor(w, device=DEV, dtype=F64).log() / 8.0).expand(n).reshape(1, n) for w in extra]
    return torch.cat(f).T


def _network(theta, f, pnet):
    """Output r of the network with parameters theta (float64) on features f (n, inputs)."""
    layers = _layers(theta, PNET_SHAPES if pnet else MLP_SHAPES)
    for w, b in layers[:-1]:
        f = f @ w.T + b
        f = torch.relu(f) if pnet else f * torch.sigmoid(f)
    w, b = layers[-1]
    return torch.sigmoid(f @ w.T + b)[:, 0]


def _theta64(shapes, seed, bias=0.0):
    return torch.from_numpy(_theta(shapes, seed, bias)).to(DEV).to(F64)


def _network_r(u, k, mode, seed, extra=()):
    """r by blocks of pairs (bounded memory)."""
    pnet = mode == "pnet"
    theta = _theta64(PNET_SHAPES if pnet else MLP_SHAPES, seed)
    out = []
    for a in range(0, u.shape[1], 1 << 20):
        s = slice(a, a + (1 << 20))
        row = [w[s] if torch.is_tensor(w) else w for w in extra] if pnet else ()
        out.append(_network(theta, _net_features(u[:, s], k[:, s], row), pnet))
    return torch.cat(out) if out else u.new_zeros(0)


def _probability(u, k, dens, mode, seed, weights):
    """P of each pair and its rest-frame energy."""
    x, v = _invariants(u, k)
    p = -torch.expm1(-dens * DT * _sigma(x) * v)
    p = torch.where((k * k).sum(0) > 0.0, p, torch.zeros_like(p))
    if mode != "plain":
        r = _network_r(u, k, mode, seed, (*weights, 2.0 * dens * DT))
        g2, e2 = 1.0 + (u * u).sum(0), (k * k).sum(0)
        inside = (g2 <= 1e6) & (e2 >= 1e-8) & (e2 <= 1.0)
        p = torch.where(inside, -torch.expm1(-2.0 * dens * DT * r), p)
    return p, x


def _resolve(u, k, dens, mode, net_seed, seed, step, weights=(1.0, 1.0), weighted=False):
    """The pairs (u, k) (3, n) in float64 after their trial and collision, in place; the collision count."""
    n = u.shape[1]
    hits = 0
    for a in range(0, n, 1 << 22):
        s = slice(a, min(n, a + (1 << 22)))
        p = torch.arange(s.start, s.stop, device=DEV)
        words = torch.stack(_philox(torch.div(p, 4, rounding_mode="floor"), step, 3, 0, seed))
        word = words.gather(0, (p % 4)[None])[0]
        u0 = (word >> 8).to(F64) * 2.0 ** -24
        d = dens[s] if torch.is_tensor(dens) else torch.full((s.stop - s.start,), dens, device=DEV, dtype=F64)
        ws = [w[s] if torch.is_tensor(w) else torch.full_like(d, w) for w in weights]
        near = torch.nonzero(u0 < -torch.expm1(-2.001 * d * DT))[:, 0]  # P is below this bound
        uc, kc = u[:, s][:, near], k[:, s][:, near]
        wc = [w[near] for w in ws]
        prob, x = _probability(uc, kc, d[near], mode, net_seed, wc)
        hit = torch.nonzero(u0[near] < prob)[:, 0]
        at = near[hit] + s.start
        r0, r1, r2, _ = _philox(at, step, 4, 0, seed)
        un, kn = _collide(uc[:, hit], kc[:, hit], x[hit], r0, r1)
        if weighted:  # the heavier partner takes its new momentum with probability w_light / w_heavy
            we, wg = wc[0][hit], wc[1][hit]
            uw = (r2 >> 8).to(F64) * 2.0 ** -24
            un = torch.where((we <= wg) | (uw * we < wg), un, uc[:, hit])
            kn = torch.where((wg <= we) | (uw * wg < we), kn, kc[:, hit])
        u[:, at], k[:, at] = un, kn
        hits += int(hit.shape[0])
    return hits


def _sorted_species(s, stream, seed):
    """A species in the order by (cell, key, id): momenta in float64, cell, id, weight."""
    cell, ident = s[3].to(torch.int64), s[4].to(torch.int64)
    by_id = torch.argsort(ident)
    key = _philox(ident, STEP, stream, 0, seed)[0]
    order = by_id[torch.argsort(((cell << 32) | key)[by_id], stable=True)]
    return [torch.stack([s[0], s[1], s[2]])[:, order].to(F64), s[3][order], s[4][order],
            None if s[5] is None else s[5][order]]


def _offsets(cell, cells):
    counts = torch.bincount(cell.to(torch.int64), minlength=cells)
    return counts, torch.cumsum(counts, 0) - counts


def _exact_step(case, seed):
    cells, mode = case["nx"] * case["ny"], case["mode"]
    e, g = _plasma(case, seed)
    e, g = _sorted_species(e, 1, seed), _sorted_species(g, 2, seed)
    ne, oe = _offsets(e[1], cells)
    ng, og = _offsets(g[1], cells)
    if mode == "ntc":
        _exact_ntc(e[0], g[0], ne, oe, ng, og, _w_over_v(case), seed)
    else:
        m = torch.minimum(ne, ng)
        c = torch.repeat_interleave(torch.arange(cells, device=DEV), m)
        rank = torch.arange(c.shape[0], device=DEV) - (torch.cumsum(m, 0) - m)[c]
        ie, ig = oe[c] + rank, og[c] + rank
        dens = torch.maximum(ne, ng)[c].to(F64)
        weights = (_w_over_v(case),) * 2
        if case["weights"]:
            weights = (e[3][ie].to(F64), g[3][ig].to(F64))
            dens = dens * torch.maximum(*weights)
        else:
            dens = dens * _w_over_v(case)
        u, k = e[0][:, ie], g[0][:, ig]
        _resolve(u, k, dens, mode, seed, seed, STEP, weights, case["weights"])
        e[0][:, ie], g[0][:, ig] = u, k
    return [[*s[0], s[1], s[2]] + ([s[3]] if case["weights"] else []) for s in (e, g)]


def _exact_ntc(u, k, ne, oe, ng, og, w_over_v, seed):
    """The candidates of every cell in order, one of each cell at a time."""
    c = torch.arange(ne.shape[0], device=DEV)
    uc = (_philox(c, STEP, 5, 0, seed)[0] >> 8).to(F64) * 2.0 ** -24
    count = torch.floor(ne.to(F64) * ng.to(F64) * w_over_v * 2.0 * DT + uc).to(torch.int64)
    count = torch.where((ne > 0) & (ng > 0), count, torch.zeros_like(count))
    c = c[torch.argsort(count, descending=True)]
    counts = count[c].tolist()
    live = len(counts)
    for j in range(counts[0] if counts else 0):
        while live and counts[live - 1] <= j:
            live -= 1
        cj = c[:live]
        r = _philox(cj, STEP, 6 | (j << 8), 0, seed)
        ie, ig = oe[cj] + ((r[0] * ne[cj]) >> 32), og[cj] + ((r[1] * ng[cj]) >> 32)
        x, v = _invariants(u[:, ie], k[:, ig])
        hit = torch.nonzero((r[2] >> 8).to(F64) * 2.0 ** -24 < 0.5 * _sigma(x) * v)[:, 0]
        if hit.shape[0]:
            ie, ig = ie[hit], ig[hit]
            phi = _philox(cj[hit], STEP, 7 | (j << 8), 0, seed)[0]
            u[:, ie], k[:, ig] = _collide(u[:, ie], k[:, ig], x[hit], r[3][hit], phi)


def _exact_train(case, seed):
    pnet = case["mode"] == "pnet"
    u, k, y, theta = _training_set(case, seed)
    f = _net_features(u.to(F64), k.to(F64), PNET_ROW if pnet else ())
    theta = torch.from_numpy(theta).to(DEV).to(F64).requires_grad_(True)
    m, v, loss = torch.zeros_like(theta), torch.zeros_like(theta), None
    for i in range(case["steps"]):
        s = slice(i * case["n"], (i + 1) * case["n"])
        loss = (_network(theta, f[s], pnet) - y[s].to(F64)).abs().mean()
        (grad,) = torch.autograd.grad(loss, theta)
        m, v = 0.9 * m + 0.1 * grad, 0.999 * v + 0.001 * grad * grad
        with torch.no_grad():
            theta -= LR * (m / (1.0 - 0.9 ** (i + 1))) / (torch.sqrt(v / (1.0 - 0.999 ** (i + 1))) + 1e-7)
    return [theta.detach(), float(loss)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        return _exact_step(case, seed)
    if kind == "infer":
        u, k = _samples(_gen(seed), case["n"])
        return _network_r(u.to(F64), k.to(F64), case["mode"], seed, PNET_ROW)
    if kind == "train":
        return _exact_train(case, seed)
    out, hits = [], 0
    for i, (u, k, mode) in enumerate(_served(case, seed)):
        u, k = u.to(F64), k.to(F64)
        hits += _resolve(u, k, 1.0, mode, seed, 5000 + i, STEP)
        out.append((u, k))
    return [out, hits]
