"""What the performance of this framework is measured on: cases, their inputs, one pass of each, and the
values a pass should give in 64 bits.

Kinds of cases:

* ``solve``: radiation fields of some cells on a set of grains, through heat_set_fields and heat_solve: the
  distributions P, the emissivity j and the energy ledger, as far as the case asks for them.  The grain sets,
  field models and sizes are those of ``paper_1311_4627_gb300.workloads``.
* ``predict``: the surrogate ensemble's emissivities (heat_surrogate_predict).
* ``grads``: loss and gradients of one surrogate member, forward and backward (heat_surrogate_grads).

``prepare`` makes the context (grid and grain set-up) and the buffers a program keeps, ``run`` is the call.
"""
import functools
import math

import numpy as np
import torch

from paper_1311_4627_gb300 import heat
from paper_1311_4627_gb300 import workloads as W

EMIS = {"none": heat.HEAT_EMIS_NONE, "f64": heat.HEAT_EMIS_F64, "bf16x3": heat.HEAT_EMIS_BF16X3,
        "tf32x3": heat.HEAT_EMIS_TF32X3}
HC = W.H_PLANCK * W.C_LIGHT


# ----------------------------------------------------------------------------------------- cases
def _solve(name, cells, grains, n_lambda, model, build, emis, **more):
    c = {"kind": "solve", "cells": cells, "grains": grains, "n_lambda": n_lambda, "model": model, "bins": 0,
         "build": build, "emis": emis, "P": False, "ledger": False, "sum_sizes": False, "j32": build == "f32",
         "u32": False, "point": False, "discrete": False, "host": False}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one cell's small grains, everything in FP64 (a radiative-transfer code asking
        # for one spectrum); latency and launches
        _solve("single_exact", 1, 8, 256, "carbonaceous", "f64", "f64", bins=128, P=True),
        # a handful of cells of the full grain set, mixed precision (an adaptive step's few new cells)
        _solve("few_mixed", 5, 64, 1024, "growing", "f32", "bf16x3"),
        # the ordinary production step: 4096 cells, the full grain set, mixed precision
        _solve("batched_mixed", 4096, 64, 1024, "growing", "f32", "bf16x3"),
        # odd sizes: cells, grains and wavelengths that fill no tile, FP32 fields, TF32 emissivity
        _solve("ragged_mixed", 1003, 37, 771, "growing", "f32", "tf32x3", u32=True),
        # the exact path on the full grain set (reference spectra, training data of the surrogate)
        _solve("batched_exact", 512, 64, 1024, "growing", "f64", "f64", P=True),
        # the paper's own point rule, exact, odd sizes
        _solve("point_exact", 203, 19, 500, "growing", "f64", "f64", P=True, point=True),
        # many bins and wavelengths per grain: the emissivity-heavy configuration, a slice of its cells
        _solve("emissivity_heavy", 4096, 32, 2048, "carbonaceous", "f32", "bf16x3", bins=512),
        # a slice of the volume run: host fields in, size-integrated spectra and the energy ledger out
        _solve("volume_slice", 4096, 80, 1024, "pair", "f32", "bf16x3", bins=512, sum_sizes=True, ledger=True,
               host=True),
        # thermal-discrete cooling of one cell's small grains
        _solve("single_discrete", 1, 8, 256, "carbonaceous", "f64", "f64", bins=128, P=True, discrete=True),
        # thermal-discrete cooling on the full grain set, a few cells
        _solve("batched_discrete", 8, 64, 1024, "growing", "f64", "f64", P=True, discrete=True),
        # the trained ensemble applied to a chunk of samples (odd count)
        {"name": "surrogate_predict", "kind": "predict", "n": 100003, "n_lambda": 1024, "members": 4},
        # training direction: forward and backward of one member on a batch
        {"name": "surrogate_grads", "kind": "grads", "n": 8192, "n_lambda": 1024},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "mixed", "mixed", "wide", "exact", "point", "volume", "discrete", "predict", "grads"])
    if kind == "small":  # few cells, either precision
        if rng.random() < 0.5:
            return _solve(None, rng.randint(1, 16), rng.randint(3, 16), rng.randint(128, 512), "carbonaceous", "f64",
                          "f64", bins=rng.randint(64, 256), P=True)
        return _solve(None, rng.randint(1, 16), rng.randint(8, 64), rng.randint(256, 1100), "growing", "f32",
                      rng.choice(["bf16x3", "tf32x3"]))
    if kind == "mixed":
        return _solve(None, _log_int(rng, 64, 4096), rng.randint(16, 64), rng.randint(300, 1024), "growing", "f32",
                      rng.choice(["bf16x3", "bf16x3", "tf32x3"]), u32=rng.random() < 0.3)
    if kind == "wide":
        return _solve(None, _log_int(rng, 256, 3000), rng.randint(8, 32), rng.randint(1024, 2048), "carbonaceous",
                      "f32", rng.choice(["bf16x3", "tf32x3"]), bins=rng.randint(300, 512))
    if kind == "exact":
        return _solve(None, _log_int(rng, 20, 512), rng.randint(8, 64), rng.randint(256, 1024), "growing", "f64",
                      "f64", P=True, ledger=rng.random() < 0.5)
    if kind == "point":
        return _solve(None, _log_int(rng, 2, 300), rng.randint(5, 24), rng.randint(256, 640), "growing", "f64",
                      "f64", P=True, point=True)
    if kind == "volume":
        return _solve(None, _log_int(rng, 128, 3000), 2 * rng.randint(5, 40), rng.randint(256, 1024), "pair", "f32",
                      "bf16x3", bins=rng.randint(128, 512), sum_sizes=True, ledger=True, host=rng.random() < 0.7)
    if kind == "discrete":
        if rng.random() < 0.5:
            return _solve(None, rng.randint(1, 64), rng.randint(2, 12), rng.randint(128, 512), "carbonaceous", "f64",
                          "f64", bins=rng.randint(48, 200), P=True, discrete=True)
        return _solve(None, rng.randint(1, 6), rng.randint(8, 48), rng.randint(256, 1024), "growing", "f64", "f64",
                      P=True, discrete=True)
    if kind == "predict":
        return {"kind": "predict", "n": _log_int(rng, 1000, 100000), "n_lambda": 64 * rng.randint(4, 16),
                "members": rng.randint(2, 6)}
    return {"kind": "grads", "n": 64 * _log_int(rng, 8, 128), "n_lambda": 64 * rng.randint(4, 16)}


# ----------------------------------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=8)
def _grains(model, grains, bins, n_lambda):
    """The wavelength grid and grain set of a case (no fields): the program's configuration."""
    lam = W.wavelength_grid(n_lambda)
    if model == "growing":  # both compositions in turn, 128-1024 bins growing with the radius
        radii = np.geomspace(3.5e-8, 1e-4, grains)
        comps = ["carbonaceous" if g % 2 == 0 else "silicate" for g in range(grains)]
        nb = [W.batched_bins(g, grains) for g in range(grains)]
    elif model == "pair":  # both compositions at the same radii
        radii = np.tile(np.geomspace(3.5e-8, 1e-4, grains // 2), 2)
        comps = ["carbonaceous"] * (grains // 2) + ["silicate"] * (grains // 2)
        nb = [bins] * grains
    else:  # one composition; few grains are the small ones
        radii = np.geomspace(3.5e-8, 250e-8 if grains <= 16 else 1e-4, grains)
        comps = ["carbonaceous"] * grains
        nb = [bins] * grains
    radii, comps, cabs, off, T, E, sw = W.make_grains(lam, radii, comps, nb)
    return W.Workload("%s %d" % (model, grains), lam, radii, comps, cabs, off, T, E, sw)


def _fields(case, seed, lam):
    """u [cells][n_lambda] FP64 on the host: the workloads' field model."""
    rng = np.random.Generator(np.random.PCG64(seed))
    n = case["cells"]
    lo, hi = (0.1, 100.0) if case["grains"] <= 16 else (1e-2, 1e4)
    chi = np.exp(rng.uniform(math.log(lo), math.log(hi), n))
    hard = rng.uniform(-1.0, 1.0, n)
    wts = 10.0 ** rng.uniform(-2.0, 0.0, (n, 3))
    u = W.three_bb_fields(lam, chi, hard, wts)
    return u.astype(np.float32) if case["u32"] else u


class _State:
    """A context and its buffers; the context goes with the state."""

    def __init__(self, case):
        self.case, self.ctx = case, None

    def __del__(self):
        if self.ctx is not None:
            heat.heat_destroy(self.ctx)
            self.ctx = None


def _stream():
    return torch.cuda.current_stream().cuda_stream


def prepare(case, seed):
    s = _State(case)
    if case["kind"] != "solve":
        return _prepare_surrogate(s, case, seed)
    wl = _grains(case["model"], case["grains"], case["bins"], case["n_lambda"])
    s.ctx = heat.heat_create_grid(0, wl.lam)
    heat.heat_set_grains(s.ctx, wl.radius, wl.cabs, wl.bin_off, wl.T, wl.E, wl.size_weight)
    u = torch.from_numpy(_fields(case, seed, wl.lam))
    cells, G, N = case["cells"], wl.n_grains, wl.n_lambda
    host = case["host"]
    where = {"pin_memory": True} if host else {"device": "cuda"}
    s.u = u.pin_memory() if host else u.cuda()
    s.P = torch.empty(cells, wl.total_bins, dtype=torch.float64, **where) if case["P"] else None
    shape = (cells, N) if case["sum_sizes"] else (cells, G, N)
    s.j = torch.empty(*shape, dtype=torch.float32 if case["j32"] else torch.float64, **where)
    s.ledger = torch.empty(cells, G, 2, dtype=torch.float64, **where) if case["ledger"] else None
    s.opts = heat.heat_default_opts(
        build=heat.HEAT_BUILD_F32 if case["build"] == "f32" else heat.HEAT_BUILD_F64, emis=EMIS[case["emis"]],
        j_dtype=heat.HEAT_F32 if case["j32"] else heat.HEAT_F64, size_integrate=case["sum_sizes"],
        host_io=1 if host else 0, heating=heat.HEAT_HEATING_POINT if case["point"] else heat.HEAT_HEATING_INTEGRAL,
        cooling=heat.HEAT_COOLING_DISCRETE if case["discrete"] else heat.HEAT_COOLING_CONTINUOUS,
        ledger_out=s.ledger)
    return s


def run(s):
    case = s.case
    st = _stream()
    if case["kind"] == "predict":
        heat.heat_surrogate_predict(s.ctx, s.X, s.lnp, case["n"], s.lnj, s.spread, st)
        return {"lnj": s.lnj, "spread": s.spread}
    if case["kind"] == "grads":
        loss = heat.heat_surrogate_grads(s.ctx, 0, s.X, s.T, case["n"], s.grads, st)
        return {"grads": s.grads, "loss": loss}
    heat.heat_set_fields(s.ctx, case["cells"], s.u, heat.HEAT_F32 if case["u32"] else heat.HEAT_F64,
                         0 if case["host"] else 1, st)
    heat.heat_solve(s.ctx, s.opts, s.P, s.j, st)
    out = {"j": s.j}
    if s.P is not None:
        out["P"] = s.P
    if s.ledger is not None:
        out["ledger"] = s.ledger
    return out


LAYERS = (128, 512, 512, 512, 512)  # the surrogate's inputs and hidden layers; then n_lambda outputs


def _weights(case, seed, member):
    """Flat FP32 parameters of a member (per layer W [out][in], then b), as a checkpoint would hold."""
    rng = np.random.Generator(np.random.PCG64([seed, member, 7]))
    dims = LAYERS + (case["n_lambda"],)
    flat = []
    for l in range(5):
        flat.append(rng.standard_normal(dims[l + 1] * dims[l], dtype=np.float32) *
                    np.float32(math.sqrt((2.0 if l < 4 else 1.0) / dims[l])))
        flat.append(0.02 * rng.standard_normal(dims[l + 1], dtype=np.float32))
    return np.concatenate(flat)


def _samples(case, seed):
    """Raw inputs (64 log band powers falling off towards the ends, ln radius, flag, ln of the total, zeros)
    and ln P_abs."""
    rng = np.random.Generator(np.random.PCG64([seed, 11]))
    n = case["n"]
    X = np.zeros((n, 128), dtype=np.float32)
    level = rng.uniform(-40.0, -25.0, (n, 1)).astype(np.float32)
    band = np.linspace(-1.0, 1.0, 64, dtype=np.float32)
    X[:, :64] = level - 6.0 * (band - rng.uniform(-0.5, 0.5, (n, 1)).astype(np.float32)) ** 2
    X[:, :64] += 0.3 * rng.standard_normal((n, 64), dtype=np.float32)
    X[:, 64] = rng.uniform(-17.0, -9.0, n)
    X[:, 65] = rng.integers(0, 2, n)
    X[:, 66] = level[:, 0] + 2.0
    return X, X[:, 66].copy()


def _targets(case, seed, rows):
    """Targets ln j - ln P_abs of some rows, masked (NaN) towards short wavelengths."""
    rng = np.random.Generator(np.random.PCG64([seed, 13]))
    N = case["n_lambda"]
    x = np.linspace(0.0, 1.0, N, dtype=np.float32)
    mid = rng.uniform(0.4, 0.7, (rows, 1)).astype(np.float32)
    Y = 10.0 - 60.0 * (x - mid) ** 2 + 0.1 * rng.standard_normal((rows, N), dtype=np.float32)
    Y[x[None, :] < mid - 0.35] = np.nan
    return Y


def _norm_inputs(case, seed):
    X, _ = _samples(dict(case, n=2048), seed + 1)
    return X, _targets(case, seed + 1, 2048)


def _prepare_surrogate(s, case, seed):
    N = case["n_lambda"]
    wl = _grains("carbonaceous", 2, 32, N)
    s.ctx = heat.heat_create_grid(0, wl.lam)
    heat.heat_set_grains(s.ctx, wl.radius, wl.cabs, wl.bin_off, wl.T, wl.E, wl.size_weight)
    members = case.get("members", 1)
    heat.heat_surrogate_init(s.ctx, members, None, seed)
    for m in range(members):
        heat.heat_surrogate_params(s.ctx, m, _weights(case, seed, m))
    Xf, Yf = (torch.from_numpy(v).cuda() for v in _norm_inputs(case, seed))
    heat.heat_surrogate_fit_norm(s.ctx, Xf, Yf, 2048, _stream())
    torch.cuda.synchronize()
    n = case["n"]
    if case["kind"] == "predict":
        X, lnp = _samples(case, seed)
        s.X, s.lnp = torch.from_numpy(X).cuda(), torch.from_numpy(lnp).cuda()
        s.lnj = torch.empty(n, N, dtype=torch.float32, device="cuda")
        s.spread = torch.empty(n, dtype=torch.float32, device="cuda")
    else:
        s.X, s.T = _standard_batch(case, seed)
        s.grads = torch.empty(_weights(case, seed, 0).size, dtype=torch.float32, device="cuda")
    return s


def _standard_batch(case, seed):
    """Standardised inputs and targets of a batch, on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, N = case["n"], case["n_lambda"]
    X = torch.randn(n, 128, generator=g, device="cuda")
    X[:, 67:] = 0.0
    T = torch.randn(n, N, generator=g, device="cuda")
    T[torch.rand(n, 1, generator=g, device="cuda") * 0.5 > torch.linspace(0.0, 1.0, N, device="cuda")] = math.nan
    return X, T


# ----------------------------------------------------------------------------------------- work
@functools.lru_cache(maxsize=64)
def _counts(model, grains, bins, n_lambda):
    """Per cell: band elements of the heating matrix (pairs a photon on the grid can join), bins, (bin,
    wavelength) pairs with emission, and the multiply-adds of the full stationary solve."""
    wl = _grains(model, grains, bins, n_lambda)
    band = rows = emit = full = 0
    for g in range(wl.n_grains):
        E, T = wl.E[wl.grain_slice(g)], wl.T[wl.grain_slice(g)]
        nb = len(E)
        elo = np.concatenate([[0.0], 0.5 * (E[1:] + E[:-1])])
        gap = np.tril(elo[:, None] - E[None, :], -1)
        band += int(np.count_nonzero((gap > 0.0) & (gap <= HC / wl.lam[0])))
        rows += nb
        x = HC / (wl.lam[None, :] * W.K_BOLTZ * T[:, None])
        emit += int(np.count_nonzero((E[:, None] >= HC / wl.lam[None, :]) & (x <= 745.0)))
        # state reduction inside the band of heating and cooling rates: M w^2, at most M^3 / 3
        w = np.count_nonzero((gap > 0.0) & (gap <= HC / wl.lam[0]), axis=1).max() + 1
        full += int(min(nb**3 / 3.0, nb * float(w) ** 2))
    return band, rows, emit, full


def work(case):
    if case["kind"] != "solve":
        N, n, m = case["n_lambda"], case["n"], case.get("members", 1)
        macs = 128 * 512 + 3 * 512 * 512 + 512 * N
        if case["kind"] == "predict":
            return {"bytes": 4.0 * n * (128 + 1 + N + 1) + 4.0 * m * macs, "flops": 2.0 * n * m * macs}
        return {"bytes": 4.0 * n * (128 + N) + 8.0 * macs, "flops": 2.0 * n * (3 * macs - 128 * 512)}
    band, rows, emit, full = _counts(case["model"], case["grains"], case["bins"], case["n_lambda"])
    c, G, N = case["cells"], case["grains"], case["n_lambda"]
    je = 4 if case["j32"] else 8
    out = c * N * je * (1 if case["sum_sizes"] else G)
    if case["P"]:
        out += 8 * c * rows
    if case["ledger"]:
        out += 16 * c * G
    u = c * N * (4 if case["u32"] else 8)
    # a band element: its integral (8 operations) and its multiply-add of the recursion, or the full solve
    flops = c * (8.0 * band + 2.0 * emit + (2.0 * full if case["discrete"] else 2.0 * (band + rows)))
    return {"bytes": float(u + out), "flops": flops}


# ----------------------------------------------------------------------------------------- exact values
# The method in plain torch, FP64, cells along the last axis.  Written from the equations: nothing of the
# framework's arithmetic is used.
_GLX, _GLW = np.polynomial.legendre.leggauss(16)


def _dev(x):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda")


def _e1(z):
    return torch.where(z == 0.0, torch.ones_like(z), torch.expm1(z) / torch.where(z == 0.0, torch.ones_like(z), z))


def _panels(wl, g):
    """Wavelength panels for integrals of C(lambda) f(lambda): the grid's segments and, beyond the grid,
    panels with the end segments' power laws.  Returns edges, and per panel C and slope at a reference."""
    lam, C = wl.lam, wl.cabs[g]
    s = np.diff(np.log(C)) / np.diff(np.log(lam))
    lo = np.exp(np.arange(math.log(lam[0]) - 3.2, math.log(lam[0]) - 1e-9, 0.02))
    hi = np.exp(math.log(lam[-1]) + 0.125 * np.arange(1, 201))
    edges = np.concatenate([lo, lam, hi])
    c0 = np.concatenate([np.full(len(lo), C[0]), C[:-1], np.full(200, C[-1])])
    l0 = np.concatenate([np.full(len(lo), lam[0]), lam[:-1], np.full(200, lam[-1])])
    sl = np.concatenate([np.full(len(lo), s[0]), s, np.full(200, s[-1])])
    return edges, c0, l0, sl


def _planck_lambda(lam, T):
    x = HC / (lam * W.K_BOLTZ * T)
    return torch.where(x > 745.0, torch.zeros_like(x),
                       2.0 * W.H_PLANCK * W.C_LIGHT**2 / lam**5 / torch.expm1(x.clamp(max=745.0)))


def _cooling(wl, g):
    """T_{f-1,f} of every bin f (0 for f = 0)."""
    E, T = _dev(wl.E[wl.grain_slice(g)]), _dev(wl.T[wl.grain_slice(g)])
    edges, c0, l0, sl = (_dev(v) for v in _panels(wl, g))
    gx, gw = _dev(_GLX), _dev(_GLW)
    out = torch.zeros_like(E)
    for b in range(1, len(E), 128):
        e, t = E[b:b + 128, None], T[b:b + 128, None]
        a = torch.log(torch.maximum(edges[None, :-1], torch.maximum(HC / e, HC / (800.0 * W.K_BOLTZ * t))))
        half = 0.5 * (torch.log(edges[None, 1:]) - a)
        lam = torch.exp((a + half)[..., None] + half[..., None] * gx)
        f = c0[None, :, None] * (lam / l0[None, :, None]) ** sl[None, :, None] * _planck_lambda(lam, t[..., None]) * lam
        p = ((f * gw).sum(-1) * half * (half > 0.0)).sum(-1)
        out[b:b + 128] = 4.0 * math.pi * p / (E[b:b + 128] - E[b - 1:b + 127][:p.numel()])
    return out


class _Cell:
    """Omega = u C of grain g on its log-log interpolant, for all cells: [n_lambda - 1][cells] tables."""

    def __init__(self, wl, g, ut, su):
        self.lam = _dev(wl.lam)
        C = _dev(wl.cabs[g])
        self.dl = torch.log(self.lam[1:] / self.lam[:-1])
        sC = torch.log(C[1:] / C[:-1]) / self.dl
        self.om = ut[:-1] * C[:-1, None]
        self.s = su + sC[:, None]
        l, d = self.lam[:-1, None], self.dl[:, None]
        self.seg1 = self.om * l * l * d * _e1((self.s + 2.0) * d)  # int Omega lambda over each segment
        self.seg0 = self.om * l * d * _e1((self.s + 1.0) * d)      # int Omega
        z = torch.zeros_like(ut[:1])
        self.pre1 = torch.cat([z, torch.cumsum(self.seg1, 0)])            # from the short end up to node n
        self.suf0 = torch.cat([torch.flip(torch.cumsum(torch.flip(self.seg0, [0]), 0), [0]), z])  # from node n on

    def seg(self, x):
        return (torch.searchsorted(self.lam, x, right=True) - 1).clamp(0, len(self.lam) - 2)

    def part(self, n, x, y, p):
        """int_x^y Omega lambda^p inside segment n (1-D n, x, y): [len(n)][cells]."""
        ln = self.lam[n]
        tx, dt = torch.log(x / ln)[:, None], torch.log(y / x)[:, None]
        q = self.s[n] + (p + 1.0)
        return self.om[n] * (ln ** (p + 1))[:, None] * torch.exp(q * tx) * dt * _e1(q * dt)

    def phi(self, x):
        """(1/h) int Omega lambda from the short end of the grid to x (clamped to the grid)."""
        x = x.clamp(self.lam[0], self.lam[-1])
        n = self.seg(x)
        return (self.pre1[n] + self.part(n, self.lam[n], x, 1)) / W.H_PLANCK

    def power_above(self, x):
        """c int Omega from x to the long end of the grid."""
        x = x.clamp(self.lam[0], self.lam[-1])
        n = self.seg(x)
        return W.C_LIGHT * (self.suf0[n + 1] + self.part(n, x, self.lam[n + 1], 0))

    def at(self, x):
        n = self.seg(x)
        return self.om[n] * (x / self.lam[n])[:, None] ** self.s[n]


def _bins(wl, g):
    E = _dev(wl.E[wl.grain_slice(g)])
    elo = torch.cat([torch.zeros_like(E[:1]), 0.5 * (E[1:] + E[:-1])])
    return E, elo


def _rescale(X, f):
    X[:f + 1] *= torch.where(X[f] > 2.0**800, X.new_full((), 2.0**-800), X.new_ones(()))


def _continuous(wl, g, cell, cool, point):
    """P [bins][cells] by the recursion X_f = sum_j B_fj X_j / T_{f-1,f}."""
    E, elo = _bins(wl, g)
    nb, M = len(E), len(E) - 1
    gap = (elo[:, None] - E[None, :]).tril(-1)
    reach = (gap > 0.0) & (gap <= HC / float(wl.lam[0]))
    reach = reach.cpu().numpy()
    first = np.where(reach.any(1), reach.argmax(1), np.arange(nb) - 1)  # the lowest j of each row's band
    X = torch.zeros(nb, cell.om.shape[1], dtype=torch.float64, device="cuda")
    X[0] = 1.0
    if point:
        u, j = torch.tril_indices(nb, nb, -1, device="cuda")
        x = HC / (E[u] - E[j])
        width = torch.cat([elo[1:] - elo[:-1], (E[M] - E[M - 1])[None]])
        fac = x**3 * width[u] / (W.H_PLANCK**2 * W.C_LIGHT)
        on = (x >= cell.lam[0]) & (x <= cell.lam[-1])
        B = torch.zeros(nb, nb, X.shape[1], dtype=torch.float64, device="cuda")
        B[u[on], j[on]] = cell.at(x[on]) * fac[on][:, None]
        B = torch.flip(torch.cumsum(torch.flip(B, [0]), 0), [0])
        for f in range(1, nb):
            X[f] = (B[f, :f] * X[:f]).sum(0) / cool[f]
            _rescale(X, f)
    else:
        soft = cell.power_above(HC / (elo[1:] - E[:-1])) / (E[1:] - E[:-1])[:, None]
        soft[HC / (elo[1:] - E[:-1]) >= cell.lam[-1]] = 0.0
        f = 1
        while f < nb:  # a few rows' elements at a time
            f1, count = f, 0
            while f1 < nb and (count == 0 or count + f1 - first[f1] <= 8192):
                count += f1 - first[f1]
                f1 += 1
            fs = np.repeat(np.arange(f, f1), [r - first[r] for r in range(f, f1)])
            js = np.concatenate([np.arange(first[r], r) for r in range(f, f1)])
            x = HC / (elo[torch.as_tensor(fs, device="cuda")] - E[torch.as_tensor(js, device="cuda")])
            B = cell.phi(x)
            B[x < cell.lam[0]] = 0.0
            e = 0
            for r in range(f, f1):
                w = r - first[r]
                X[r] = ((B[e:e + w] * X[first[r]:r]).sum(0) + soft[r - 1] * X[r - 1]) / cool[r]
                _rescale(X, r)
                e += w
            f = f1
    return X / X.sum(0)


def _discrete_cooling(wl, g):
    """T_lu [l][u] of thermal-discrete cooling: the power of photon energies E_u - e, e in bin l, over E_u - E_l."""
    E, elo = _bins(wl, g)
    T = _dev(wl.T[wl.grain_slice(g)])
    nb = len(E)
    edges, c0, l0, sl = (_dev(v) for v in _panels(wl, g))
    node_e = torch.flip(HC / edges, [0])  # ascending photon energies of the panel edges
    gx, gw = _dev(_GLX), _dev(_GLW)
    out = torch.zeros(nb, nb, dtype=torch.float64, device="cuda")
    for u0 in range(1, nb, 64):
        us = torch.arange(u0, min(u0 + 64, nb), device="cuda")
        u = torch.repeat_interleave(us, us)
        l = torch.cat([torch.arange(int(k), device="cuda") for k in us])
        top = l == u - 1
        width = torch.where(top, E[u] - elo[l], elo[(l + 1).clamp(max=nb - 1)] - elo[l])
        e_hi = E[u] - elo[l]                                   # photon energy at the window's lower end
        e_lo = torch.where(top, torch.zeros_like(e_hi), E[u] - elo[(l + 1).clamp(max=nb - 1)])
        k0 = torch.searchsorted(node_e, e_lo.contiguous(), right=True)  # first edge above e_lo
        k1 = torch.searchsorted(node_e, e_hi.contiguous(), right=False)  # first edge at or above e_hi
        n = (k1 - k0).clamp(min=0) + 1
        wi = torch.repeat_interleave(torch.arange(len(n), device="cuda"), n)
        i = torch.arange(len(wi), device="cuda") - torch.repeat_interleave(torch.cumsum(n, 0) - n, n)
        off = (E[u] - elo[l])[wi]
        # offsets of the piece in the grain's final energy, from the window's lower end; pieces by edge, high first
        ka = (k1[wi] - i).clamp(0, len(node_e) - 1)
        kb = (k1[wi] - i - 1).clamp(0, len(node_e) - 1)
        a = torch.where(i == 0, torch.zeros_like(off), off - node_e[ka])
        b = torch.where(i == n[wi] - 1, width[wi], off - node_e[kb])
        half = 0.5 * (b - a)
        eps = off[:, None] - ((a + half)[:, None] + half[:, None] * gx)
        eps = eps.clamp(min=1e-30 * float(E[-1]))
        lam = HC / eps
        seg = (torch.searchsorted(edges, lam.contiguous(), right=True) - 1).clamp(0, len(c0) - 1)
        x = eps / (W.K_BOLTZ * T[u][wi][:, None])
        f = c0[seg] * (lam / l0[seg]) ** sl[seg] * eps**3 / torch.expm1(x.clamp(max=745.0))
        f = torch.where((x > 745.0) | (lam > edges[-1]), torch.zeros_like(f), f)
        p = torch.zeros(len(n), dtype=torch.float64, device="cuda").index_add_(0, wi, (f * gw).sum(1) * half)
        out[l, u] = 8.0 * math.pi / (W.H_PLANCK**3 * W.C_LIGHT**2) * p / (E[u] - E[l])
    return out


def _discrete(wl, g, cell):
    """P [bins][cells]: the stationary state of the full rate matrix, by state reduction."""
    E, elo = _bins(wl, g)
    nb, M, cells = len(E), len(E) - 1, cell.om.shape[1]
    D = _discrete_cooling(wl, g)
    q = torch.zeros(cells, nb, nb, dtype=torch.float64, device="cuda")  # rate from row to column
    q += D.t()[None]
    for i in range(M):
        b = HC / (elo[i + 1:] - E[i])
        a = torch.cat([b[1:], b.new_zeros(1)])
        ca, cb = a.clamp(cell.lam[0], cell.lam[-1]), b.clamp(cell.lam[0], cell.lam[-1])
        na, nz = cell.seg(ca), cell.seg(cb)
        same = cell.part(na, ca, cb, 1)
        across = (cell.part(na, ca, cell.lam[na + 1], 1) + (cell.pre1[nz] - cell.pre1[na + 1]) +
                  cell.part(nz, cell.lam[nz], cb, 1))
        v = torch.where((na == nz)[:, None], same, across) / W.H_PLANCK
        v[cb <= ca] = 0.0
        if float(b[0]) < float(cell.lam[-1]):
            v[0] += cell.power_above(b[:1])[0] / (E[i + 1] - E[i])
        q[:, i, i + 1:] = v.t()
    s = torch.ones(nb, cells, dtype=torch.float64, device="cuda")
    for n in range(M, 0, -1):
        s[n] = q[:, n, :n].sum(1)
        q[:, :n, :n] += q[:, :n, n, None] * (q[:, n, None, :n] / s[n][:, None, None])
    X = torch.zeros(nb, cells, dtype=torch.float64, device="cuda")
    X[0] = 1.0
    for n in range(1, nb):
        X[n] = (X[:n] * q[:, :n, n].t()).sum(0) / s[n]
        _rescale(X, n)
    return X / X.sum(0)


def _exact_solve(case, seed):
    wl = _grains(case["model"], case["grains"], case["bins"], case["n_lambda"])
    u = _dev(_fields(case, seed, wl.lam).astype(np.float64))
    cells, G, N = case["cells"], wl.n_grains, wl.n_lambda
    lam = _dev(wl.lam)
    ut = u.t().contiguous()
    su = torch.log(ut[1:] / ut[:-1]) / torch.log(lam[1:] / lam[:-1])[:, None]
    j = torch.zeros((cells, N) if case["sum_sizes"] else (cells, G, N), dtype=torch.float64, device="cuda")
    P = torch.zeros(cells, wl.total_bins, dtype=torch.float64, device="cuda") if case["P"] else None
    led = torch.zeros(cells, G, 2, dtype=torch.float64, device="cuda") if case["ledger"] else None
    for g in range(G):
        sl = wl.grain_slice(g)
        E, T = _dev(wl.E[sl]), _dev(wl.T[sl])
        K = _dev(wl.cabs[g])[None, :] * _planck_lambda(lam[None, :], T[:, None])
        K[E[:, None] < HC / lam[None, :]] = 0.0
        cool = None if case["discrete"] else _cooling(wl, g)
        if case["ledger"] and cool is None:
            cool = _cooling(wl, g)
        step = max(1, int(2.0e9 / 8 / len(E) ** 2)) if case["point"] or case["discrete"] else 4096
        for c0 in range(0, cells, step):
            c1 = min(cells, c0 + step)
            cell = _Cell(wl, g, ut[:, c0:c1], su[:, c0:c1])
            if case["discrete"]:
                p = _discrete(wl, g, cell)
            else:
                p = _continuous(wl, g, cell, cool, case["point"])
            jg = p.t() @ K
            if case["sum_sizes"]:
                j[c0:c1] += float(wl.size_weight[g]) * jg
            else:
                j[c0:c1, g] = jg
            if P is not None:
                P[c0:c1, sl] = p.t()
            if led is not None:
                led[c0:c1, g, 0] = W.C_LIGHT * cell.suf0[0]
                led[c0:c1, g, 1] = (p[1:] * (cool[1:] * (E[1:] - E[:-1]))[:, None]).sum(0)
    out = {"j": j}
    if P is not None:
        out["P"] = P
    if led is not None:
        out["ledger"] = led
    return out


def _layers(flat, N):
    dims, k, out = LAYERS + (N,), 0, []
    for l in range(5):
        w = flat[k:k + dims[l + 1] * dims[l]].reshape(dims[l + 1], dims[l])
        k += w.size
        out.append((_dev(w), _dev(flat[k:k + dims[l + 1]])))
        k += dims[l + 1]
    return out


def _gelu(x):
    return 0.5 * x * (1.0 + torch.tanh(math.sqrt(2.0 / math.pi) * (x + 0.044715 * x**3)))


def _exact_predict(case, seed):
    X, lnp = _samples(case, seed)
    Xf, Yf = (_dev(v) for v in _norm_inputs(case, seed))
    stats = []
    for A in (Xf, Yf):
        ok = ~torch.isnan(A)
        n = ok.sum(0).to(torch.float64)
        mu = torch.where(ok, A, 0.0).sum(0) / n
        var = torch.where(ok, A * A, 0.0).sum(0) / n - mu * mu
        mu = torch.where(n > 0, mu, torch.zeros_like(mu))
        stats.append((mu, torch.where((n > 1) & (var > 1e-12), torch.sqrt(var.clamp(min=0.0)), torch.ones_like(var))))
    (xm, xs), (ym, ys) = stats
    nets = [_layers(_weights(case, seed, m), case["n_lambda"]) for m in range(case["members"])]
    lnj = torch.empty(case["n"], case["n_lambda"], dtype=torch.float64, device="cuda")
    spread = torch.empty(case["n"], dtype=torch.float64, device="cuda")
    for b in range(0, case["n"], 16384):
        x = (_dev(X[b:b + 16384]) - xm) / xs
        ys_m = []
        for net in nets:
            a = x
            for l, (w, c) in enumerate(net):
                a = a @ w.t() + c
                a = _gelu(a) if l < 4 else a
            ys_m.append(a * ys + ym)
        y = torch.stack(ys_m)
        mean = y.mean(0)
        lnj[b:b + 16384] = mean + _dev(lnp[b:b + 16384])[:, None]
        sd = torch.sqrt(((y - mean) ** 2).sum(0) / (len(nets) - 1))
        thr = mean.max(1, keepdim=True).values + math.log(1e-6)
        spread[b:b + 16384] = torch.where(mean > thr, sd, torch.zeros_like(sd)).max(1).values
    return {"lnj": lnj, "spread": spread}


def _exact_grads(case, seed):
    X, T = _standard_batch(case, seed)
    X, T = X.double(), T.double()
    net = _layers(_weights(case, seed, 0), case["n_lambda"])
    ps = [p.requires_grad_() for wb in net for p in wb]
    a = X
    for l, (w, c) in enumerate(net):
        a = a @ w.t() + c
        a = _gelu(a) if l < 4 else a
    ok = ~torch.isnan(T)
    loss = torch.where(ok, a - torch.where(ok, T, 0.0), 0.0).square().sum() / ok.sum()
    grads = torch.autograd.grad(loss, ps)
    return {"grads": torch.cat([g.reshape(-1) for g in grads]), "loss": float(loss.detach())}


def exact(case, seed):
    if case["kind"] == "predict":
        return _exact_predict(case, seed)
    if case["kind"] == "grads":
        return _exact_grads(case, seed)
    return _exact_solve(case, seed)
