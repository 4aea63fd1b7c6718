"""The calls of libhlb whose time counts, each as a program that uses the library makes it.

A program holds a handle with its velocity sets, grid, walls and forces, puts a state into it, steps, and reads the
state or the moments back.  A case is such a handle plus what one pass does: ``kind`` "steps" (hlb_step of ``steps``
RK-3 steps, then hlb_get_state_dev of the whole state) or "moments" (hlb_moments_dev of a state that the handle holds).
``prepare`` makes the handle and a seeded state on the GPU, ``run`` is the pass, ``exact`` the same pass in 64 bits with
torch alone: quadratures, force matrices, equilibria and the step are written out below from the method.

The listed cases:
  channel_fp64       the plain method in FP64: 64 cells, 32 velocities, upwind2, the smallest run there is; it is stepped
                     thousands of times, so latency and launches are all of it
  stretched_channel  one 1D FP32 channel (512 cells on a tanh-stretched grid, 128 velocities, WENO-5), an ordinary 1D run
  transition_q200    the order-200 half-range set with collisions at three Knudsen numbers (FP64, 24 cells each)
  ballistic_q200     the order-200 set without collisions, the eight cases of the ballistic convergence figure (FP64)
  fp64_2d            a 2D FP64 run of odd size, the reference a user checks an FP32 run against
  channels_rounded   37 seeded FP32 channels in one handle with stochastic rounding, a small parameter study run long
  field_2d           a ragged 2D FP32 channel with a per-node acceleration field (a potential) on a stretched grid
  box_2d             the 256 x 256 box, 512 velocities, FP32
  long_channel       131072 cells x 512 velocities, FP32, the largest 1D run
  batched            4096 seeded FP32 channels of three velocity sets in one handle, autotuned once
  large_2d           the 1024 x 512 channel with 1024 velocities (537M values), FP32, autotuned once
  moments_large      reading n, u, T and q of that channel's state
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1708_03249_gb300 import hlb
from paper_1708_03249_gb300 import workloads as W

_ADV = {"weno5": W.WENO5, "upwind2": W.UPWIND2}
_PREC = {"fp64": W.FP64, "fp32": W.FP32}

_DEFAULT = dict(kind="steps", set="single", Qx=4, Qy=0, Qz=0, Nx_eq=-1, nx=64, ny=1, Lx=1.0, Ly=1.0, stretch_A=0.0,
                advection="weno5", precision="fp32", cfl=0.5, dt=0.0, T_left=1.0, T_right=1.0, ax=0.0, ay=0.0, az=0.0,
                Kn=1.0, collisionless=False, full_range_x=False, ninst=1, cells_most=1024, field=False,
                stochastic=False, tune=False, steps=1)


def _case(**kw):
    unknown = set(kw) - set(_DEFAULT) - {"name"}
    if unknown:
        raise KeyError(f"unknown fields {sorted(unknown)}")
    return {**_DEFAULT, **kw}


def listed():
    g = W.gravity
    return [
        _case(name="channel_fp64", Qx=4, Qy=4, nx=64, advection="upwind2", precision="fp64", Kn=0.1, ax=-0.1, steps=60),
        _case(name="stretched_channel", Qx=8, Qy=8, nx=512, stretch_A=0.9, T_left=0.5, T_right=1.5, Kn=0.1, steps=30,
              **g(0.5, 30.0)),
        _case(name="transition_q200", set="transition", Qx=200, Nx_eq=20, nx=24, stretch_A=0.99, precision="fp64",
              dt=1e-4, T_left=1.0, T_right=1.2, ax=-0.1, ninst=3, steps=30),
        _case(name="ballistic_q200", set="ballistic", Qx=200, Nx_eq=20, nx=24, stretch_A=0.99, precision="fp64",
              dt=1e-4, collisionless=True, ninst=8, steps=30),
        _case(name="fp64_2d", Qx=8, Qy=8, nx=95, ny=61, Ly=0.6, precision="fp64", T_left=1.0, T_right=1.5, Kn=0.2,
              steps=3, **g(0.3, 40.0)),
        _case(name="channels_rounded", set="batch", ninst=37, stochastic=True, steps=30),
        _case(name="field_2d", Qx=8, Qy=8, nx=317, ny=203, Ly=0.7, stretch_A=0.5, T_left=0.9, T_right=1.3, Kn=0.3,
              field=True, steps=6, **g(0.2, 60.0)),
        _case(name="box_2d", Qx=16, Qy=16, nx=256, ny=256, T_left=1.0, T_right=1.2, Kn=0.05, steps=6, **g(0.2, 45.0)),
        _case(name="long_channel", Qx=16, Qy=16, nx=131072, T_left=1.0, T_right=1.5, Kn=0.1, ax=-0.3, ay=-0.2, steps=6),
        _case(name="batched", set="batch", ninst=4096, tune=True, steps=3),
        _case(name="large_2d", Qx=8, Qy=8, Qz=8, nx=1024, ny=512, Ly=0.5, T_left=1.0, T_right=2.0, ax=-0.3, ay=-0.3,
              Kn=0.5, tune=True, steps=3),
        _case(name="moments_large", kind="moments", Qx=8, Qy=8, Qz=8, nx=1024, ny=512, Ly=0.5, T_left=1.0, T_right=2.0,
              ax=-0.3, ay=-0.3, Kn=0.5),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    phys = dict(T_left=round(rng.uniform(0.6, 1.5), 3), T_right=round(rng.uniform(0.6, 1.5), 3),
                Kn=round(math.exp(rng.uniform(math.log(0.02), math.log(10.0))), 4), ax=-round(rng.uniform(0.0, 0.6), 3),
                ay=-round(rng.uniform(0.0, 0.6), 3), collisionless=rng.random() < 0.1)
    stretch = round(rng.uniform(0.3, 0.95), 3) if rng.random() < 0.4 else 0.0
    adv = "weno5" if rng.random() < 0.75 else "upwind2"
    family = rng.choice(["channel_fp64", "channel", "channel", "plane", "plane", "plane_z", "plane_fp64", "batch",
                         "q200", "moments"])
    if family == "channel_fp64":
        Q = rng.choice((4, 8, 16))
        return _case(Qx=Q, Qy=Q, nx=size(24, 2048), stretch_A=stretch, advection=adv, precision="fp64", steps=30, **phys)
    if family == "channel":
        Q = rng.choice((4, 8, 16))
        full = rng.random() < 0.15
        nx = size(32, 131072)
        return _case(Qx=2 * Q if full else Q, Qy=Q, nx=nx, stretch_A=stretch, advection=adv, full_range_x=full,
                     stochastic=rng.random() < 0.2, field=rng.random() < 0.15, steps=30 if nx < 4096 else 6, **phys)
    if family == "plane":
        Q = rng.choice((4, 8, 16))
        nx, ny = size(24, 600), size(12, 600)
        return _case(Qx=Q, Qy=Q, nx=nx, ny=ny, Ly=round(rng.uniform(0.3, 1.0), 3), stretch_A=stretch, advection=adv,
                     field=rng.random() < 0.25, stochastic=rng.random() < 0.2, steps=6, **phys)
    if family == "plane_z":
        Q, Qz = rng.choice(((4, 4), (8, 4), (8, 8)))
        return _case(Qx=Q, Qy=Q, Qz=Qz, nx=size(24, 500), ny=size(12, 300), Ly=round(rng.uniform(0.3, 1.0), 3),
                     advection=adv, az=-0.2 if rng.random() < 0.25 else 0.0, steps=3, **phys)
    if family == "plane_fp64":
        Q = rng.choice((4, 8))
        return _case(Qx=Q, Qy=Q, nx=size(24, 160), ny=size(8, 100), Ly=round(rng.uniform(0.3, 1.0), 3),
                     stretch_A=stretch, advection=adv, precision="fp64", steps=3, **phys)
    if family == "batch":
        return _case(set="batch", ninst=size(8, 2500), cells_most=rng.choice((200, 1024)), steps=6,
                     stochastic=rng.random() < 0.25)
    if family == "q200":
        if rng.random() < 0.5:
            return _case(set="ballistic", Qx=rng.choice((64, 100, 200)), Nx_eq=20, nx=24, stretch_A=0.99,
                         precision="fp64", dt=1e-4, collisionless=True, ninst=rng.randint(1, 8), steps=15)
        return _case(set="transition", Qx=rng.choice((64, 100, 200)), Nx_eq=rng.choice((12, 20)), nx=rng.randint(16, 40),
                     stretch_A=0.99, precision="fp64", dt=1e-4, T_left=1.0, T_right=1.2, ax=-0.1, ninst=rng.randint(1, 3),
                     steps=15)
    Q, Qz = rng.choice(((4, 0), (8, 0), (16, 0), (8, 8)))
    return _case(kind="moments", Qx=Q, Qy=Q, Qz=Qz, nx=size(32, 1024), ny=size(8, 400), Ly=0.5,
                 precision="fp64" if rng.random() < 0.2 else "fp32", **phys)


# ---------------------------------------------------------------------------------------------------------------------
# the handle's configurations
# ---------------------------------------------------------------------------------------------------------------------
def _configs(c):
    if c["set"] == "batch":
        # no instance larger than cells_most (a study of short channels is drawn so)
        return [W.scaled(i, nx=min(i["nx"], c["cells_most"])) for i in W.batched_instances(c["ninst"])]
    if c["set"] == "ballistic":
        return [W.hhlb_ballistic(g, dT, Qx=c["Qx"], Nx_eq=c["Nx_eq"]) for g in W.HHLB_BALLISTIC_G
                for dT in W.HHLB_BALLISTIC_DT][:c["ninst"]]
    base = W.make(Qx=c["Qx"], Qy=c["Qy"], Qz=c["Qz"], Nx_eq=c["Nx_eq"], nx=c["nx"], ny=c["ny"], Lx=c["Lx"], Ly=c["Ly"],
                  stretch_A=c["stretch_A"], advection=_ADV[c["advection"]], precision=_PREC[c["precision"]],
                  cfl=c["cfl"], dt=c["dt"], T_left=c["T_left"], T_right=c["T_right"], ax=c["ax"], ay=c["ay"],
                  az=c["az"], Kn=math.inf if c["collisionless"] else c["Kn"],
                  x_basis=W.X_FULL if c["full_range_x"] else W.X_HALF)
    if c["set"] == "transition":
        return [W.scaled(base, Kn=k) for k in (0.1, 0.5, 1.0)[:c["ninst"]]]
    return [base]


def _velocities(cfg):
    nx = cfg["Qx"] if cfg["x_basis"] == W.X_FULL else 2 * cfg["Qx"]
    return nx, max(cfg["Qy"], 1), max(cfg["Qz"], 1)


def _values(cfg):
    a, b, d = _velocities(cfg)
    return a * b * d * cfg["nx"] * cfg["ny"]


# ---------------------------------------------------------------------------------------------------------------------
# the pass
# ---------------------------------------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _stream():
    """The program's one stream: every handle enqueues on it, so that passes follow one another."""
    return torch.cuda.Stream()


def prepare(case, seed):
    cfgs = _configs(case)
    stream = _stream()
    h = hlb.Handle(cfgs, stream=stream.cuda_stream)
    if case["field"]:
        for i, cfg in enumerate(cfgs):
            ax, ay = _field(cfg)
            h.set_force_field(i, ax, ay)
    if case["stochastic"]:
        h.set_rounding(True)
    f0 = _initial(case, cfgs, seed)
    torch.cuda.synchronize()
    h.set_state_dev(f0.data_ptr(), h.state_bytes)
    if case["tune"]:
        h.autotune()
    if case["kind"] == "moments":
        out = {k: torch.empty((h.nodes, 3) if k == "u" else h.nodes, dtype=torch.float64, device="cuda")
               for k in ("n", "u", "T", "q")}
    else:
        out = {"f": torch.empty_like(f0)}
    stream.synchronize()
    return {"handle": h, "out": out, "kind": case["kind"], "steps": case["steps"]}


def run(state):
    h, out = state["handle"], state["out"]
    if state["kind"] == "moments":
        h.moments_dev(out["n"].data_ptr(), out["u"].data_ptr(), out["T"].data_ptr(), out["q"].data_ptr())
    else:
        h.step(state["steps"])
        h.get_state_dev(out["f"].data_ptr(), h.state_bytes)
    return out


def work(case):
    """Bytes: the state read once, and the state (or the moments) written once.  Flops: per node-velocity and stage the
    force term's dot products, 60 (WENO-5) or 4 (upwind2) per spatial axis and about 20 for equilibrium, relaxation and
    RK-3; moments 18 per node-velocity."""
    nbytes = flops = 0
    for cfg in _configs(case):
        values = _values(cfg)
        size = 8 if cfg["precision"] == W.FP64 else 4
        nodes = cfg["nx"] * cfg["ny"]
        if case["kind"] == "moments":
            nbytes += values * size + 48 * nodes
            flops += 18 * values
            continue
        nbytes += 2 * values * size
        a, b, d = _velocities(cfg)
        unit = 20 + (2 if cfg["ny"] > 1 else 1) * (60 if cfg["advection"] == W.WENO5 else 4)
        unit += 2 * a * (cfg["ax"] != 0.0) + 2 * b * (cfg["ay"] != 0.0 and b > 1) + 2 * d * (cfg["az"] != 0.0 and d > 1)
        flops += 3 * case["steps"] * values * unit
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------------------------------------------------
# inputs: a gas between its walls' temperatures with a density wave, moving slowly, and 1 % of seeded noise per value
# ---------------------------------------------------------------------------------------------------------------------
_TABLE = 65


def _initial(case, cfgs, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) & 0x7FFFFFFF)
    r = np.random.default_rng(int(seed) & 0x7FFFFFFF)
    ux, uy = r.uniform(-0.05, 0.05, 2)
    phase, waves = r.uniform(0, 2 * math.pi), int(r.integers(1, 4))
    dtype = torch.float64 if cfgs[0]["precision"] == W.FP64 else torch.float32
    out = torch.empty(sum(_values(c) for c in cfgs), dtype=dtype, device="cuda")
    high = cfgs[0]["Qx"] > 32            # the order-200 runs start from a gas at T = 1
    t_lo = 0.97 if high else min(min(c["T_left"], c["T_right"]) for c in cfgs)
    t_hi = 1.03 if high else max(max(c["T_left"], c["T_right"]) for c in cfgs) + 1e-3
    at, tables = 0, {}
    for c in cfgs:
        key = (c["Qx"], c["Qy"], c["Qz"], c["Nx_eq"], c["x_basis"])
        if key not in tables:
            T = torch.linspace(t_lo, t_hi, _TABLE, dtype=torch.float64, device="cuda")
            u = torch.zeros((_TABLE, 3), dtype=torch.float64, device="cuda")
            u[:, 0], u[:, 1] = float(ux), float(uy) * (c["Qy"] > 0)
            tables[key] = _Axes.of(c).equilibrium(torch.ones_like(T), u, T).reshape(_TABLE, -1).to(dtype)
        tab = tables[key]
        x = (torch.arange(c["nx"], device="cuda", dtype=torch.float64) + 0.5) / c["nx"]
        y = (torch.arange(c["ny"], device="cuda", dtype=torch.float64) + 0.5) / c["ny"]
        T = t_lo + (t_hi - t_lo) * x if high else c["T_left"] + (c["T_right"] - c["T_left"]) * x
        w = (T - t_lo) / (t_hi - t_lo) * (_TABLE - 1)
        k = w.floor().clamp(0, _TABLE - 2)
        w, k = (w - k).to(dtype)[:, None], k.long()
        line = tab[k] * (1 - w) + tab[k + 1] * w
        n = 1 + 0.1 * torch.sin(2 * math.pi * (waves * x[None, :] + y[:, None] * (c["ny"] > 1)) + phase)
        v = out[at:at + _values(c)].view(c["ny"], c["nx"], -1)
        v.uniform_(0.99, 1.01, generator=gen)
        v *= n.to(dtype)[:, :, None]
        v *= line[None]
        at += _values(c)
    return out


def _field(cfg):
    """A smooth acceleration field: minus the gradient of a periodic potential."""
    x = (np.arange(cfg["nx"]) + 0.5) / cfg["nx"]
    y = (np.arange(cfg["ny"]) + 0.5) / cfg["ny"]
    ax = 0.3 * np.sin(2 * math.pi * x)[None, :] * (1 + 0.5 * np.cos(2 * math.pi * y))[:, None]
    ay = 0.2 * np.cos(2 * math.pi * x)[None, :] * np.sin(2 * math.pi * y)[:, None]
    return ax, ay if cfg["Qy"] else None


# ---------------------------------------------------------------------------------------------------------------------
# the method in 64 bits: quadratures, force matrices, projected equilibria
# ---------------------------------------------------------------------------------------------------------------------
def _panels(hi, width, points):
    g, w = np.polynomial.legendre.leggauss(points)
    n = int(math.ceil(hi / width))
    p = ((np.arange(n)[:, None] + 0.5 * (1 + g)[None, :]) * width).ravel()
    return p, np.tile(0.5 * width * w, n)


def _orthonormal(alpha, beta, x, n):
    """h_0 .. h_{n-1} at x from the recurrence sqrt(b_{l+1}) h_{l+1} = (x - a_l) h_l - sqrt(b_l) h_{l-1}, b_0 the mass."""
    h = np.zeros((n,) + np.shape(x))
    h[0] = 1.0 / math.sqrt(beta[0])
    for i in range(1, n):
        h[i] = (x - alpha[i - 1]) * h[i - 1] - (math.sqrt(beta[i - 1]) * h[i - 2] if i > 1 else 0.0)
        h[i] /= math.sqrt(beta[i])
    return h


@functools.lru_cache(maxsize=None)
def _half_range(Q):
    """Recurrence, nodes and weights of the weight exp(-p^2/2)/sqrt(2 pi) on [0, inf): discretised Stieltjes."""
    p, w = _panels(46.0, 0.5, 60)
    v = np.sqrt(w * np.exp(-p * p / 2) / math.sqrt(2 * math.pi))
    alpha, beta = np.zeros(Q + 1), np.zeros(Q + 1)
    beta[0] = v @ v
    cur, old = v / math.sqrt(beta[0]), np.zeros_like(v)
    for i in range(Q + 1):
        alpha[i] = cur @ (p * cur)
        nxt = (p - alpha[i]) * cur - (math.sqrt(beta[i]) * old if i else 0.0)
        if i < Q:
            beta[i + 1] = nxt @ nxt
            cur, old = nxt / math.sqrt(beta[i + 1]), cur
    J = np.diag(alpha[:Q]) + np.diag(np.sqrt(beta[1:Q]), 1) + np.diag(np.sqrt(beta[1:Q]), -1)
    z = np.linalg.eigvalsh(J)
    h = _orthonormal(alpha, beta, z, Q)
    return alpha, beta, z, 1.0 / (h * h).sum(0)


def _half_force(Q):
    """(K f)_k = d_p f at the nodes, the jump at p = 0 shared between the halves.  With f = omega sum_l F_l h_l on each
    half, F'_l = -+ [int f h_l' + h_l(0) (f(0+) + f(0-)) / 2]; int f h_l' through the derivative's expansion."""
    alpha, beta, z, w = _half_range(Q)
    H, h0 = _orthonormal(alpha, beta, z, Q), _orthonormal(alpha, beta, np.zeros(1), Q)[:, 0]
    om0 = 1.0 / math.sqrt(2 * math.pi)
    lead = 1.0 / np.sqrt(np.cumprod(beta[:Q]))
    tail = np.zeros_like(H)              # tail[l] = sum_{s > l} h_s(0) h_s(z_k)
    for i in range(Q - 2, -1, -1):
        tail[i] = tail[i + 1] + h0[i + 1] * H[i + 1]
    same = np.zeros((Q, Q))
    for i in range(Q - 1):
        same += np.outer(om0 * h0[i] * tail[i] - lead[i] / lead[i + 1] * H[i + 1], H[i])
    phi0 = h0 @ H
    jump = 0.5 * om0 * np.outer(phi0, phi0)
    K = np.empty((2 * Q, 2 * Q))
    K[:Q, :Q], K[:Q, Q:] = w[:, None] * (same - jump), -w[:, None] * jump
    K[Q:, Q:], K[Q:, :Q] = -K[:Q, :Q], -K[:Q, Q:]
    return K


@functools.lru_cache(maxsize=None)
def _full_range(Q):
    z, w = np.polynomial.hermite_e.hermegauss(Q)
    w = w / math.sqrt(2 * math.pi)
    He = np.zeros((Q, Q))
    He[0] = 1.0
    if Q > 1:
        He[1] = z
    for i in range(1, Q - 1):
        He[i + 1] = z * He[i] - i * He[i - 1]
    K = np.zeros((Q, Q))
    for i in range(Q - 1):
        K -= np.outer(w * He[i + 1], He[i]) / math.factorial(i)
    return z, w, He, K


class _Axes:
    """Momenta, weights, force matrices and equilibrium of one velocity set, on the GPU in 64 bits."""

    _kept: dict = {}

    @classmethod
    def of(cls, c):
        key = (c["Qx"], c["Qy"], c["Qz"], c["Nx_eq"], c["x_basis"])
        if key not in cls._kept:
            cls._kept[key] = cls(c)
        return cls._kept[key]

    def __init__(self, c):
        def up(a):
            return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")

        Q, self.full = c["Qx"], c["x_basis"] == W.X_FULL
        self.N = (Q if c["Nx_eq"] < 0 else c["Nx_eq"] + 1) - 1
        self.D = 1 + (c["Qy"] > 0) + (c["Qz"] > 0)
        if self.full:
            z, w, He, K = _full_range(Q)
            o = np.concatenate([np.arange(Q // 2, Q), np.arange(Q // 2 - 1, -1, -1)])
            self.px, self.wx, self.Kx, self.Hx = up(z[o]), up(w[o]), up(K[o][:, o]), up(He[:, o])
            self.half = Q // 2
        else:
            self.alpha, self.beta, z, w = _half_range(Q)
            self.px, self.wx, self.Kx = up(np.concatenate([z, -z])), up(np.concatenate([w, w])), up(_half_force(Q))
            self.Hx = up(_orthonormal(self.alpha, self.beta, z, self.N + 1))
            self.half = Q
        self.other = []
        for q in (c["Qy"], c["Qz"]):
            if q:
                z, w, He, K = _full_range(q)
                self.other.append((up(z), up(w), up(He), up(K)))
            else:
                self.other.append((up([0.0]), up([1.0]), None, up([[0.0]])))
        self.shape = (self.other[1][0].numel(), self.other[0][0].numel(), self.px.numel())

    @staticmethod
    def _full_g(u, T, w, He, N):
        G = [torch.ones_like(u), u]
        for i in range(1, N):
            G.append(u * G[i] + i * (T - 1) * G[i - 1])
        g = torch.zeros(u.shape + w.shape, dtype=torch.float64, device=u.device)
        for i in range(N + 1):
            g += G[i][..., None] * (w * He[i] / math.factorial(i))
        return g

    def gx(self, u, T):
        if self.full:
            return self._full_g(u, T, self.wx, self.Hx, self.N)
        t_lo, t_hi, u_hi = float(T.min()), float(T.max()), float(u.abs().max())
        p, w = _panels(u_hi + 15 * math.sqrt(t_hi), 0.5 * math.sqrt(t_lo), 16)
        H = torch.as_tensor((_orthonormal(self.alpha, self.beta, p, self.N + 1) * w).T.copy(), device="cuda")
        p = torch.as_tensor(p, device="cuda")
        out = torch.empty(u.shape + (2 * self.half,), dtype=torch.float64, device="cuda")
        for a in range(0, u.shape[0], 65536):
            s = slice(a, a + 65536)
            norm = 1 / torch.sqrt(2 * math.pi * T[s])
            for sign, part in ((1.0, slice(0, self.half)), (-1.0, slice(self.half, None))):
                e = torch.exp((p - sign * u[s, None]).square_() / (-2 * T[s, None]))
                out[s, part] = ((e @ H) * norm[:, None]) @ (self.Hx * self.wx[:self.half])
        return out

    def factors(self, n, u, T):
        f = [n[:, None] * self.gx(u[:, 0], T)]
        for k, (z, w, He, _) in enumerate(self.other):
            f.append(self._full_g(u[:, 1 + k], T, w, He, z.numel() - 1) if He is not None else
                     torch.ones((n.shape[0], 1), dtype=torch.float64, device="cuda"))
        return f

    def equilibrium(self, n, u, T):
        gx, gy, gz = self.factors(n, u, T)
        return gz[:, :, None, None] * gy[:, None, :, None] * gx[:, None, None, :]

    def moments(self, f):
        """n, u, T, q_x of f[cells, kz, jy, ix]."""
        py, pz = self.other[0][0], self.other[1][0]
        n = f.sum((1, 2, 3))
        j = torch.stack([(f.sum((1, 2)) @ self.px), f.sum((1, 3)) @ py, f.sum((2, 3)) @ pz], 1)
        u = j / n[:, None]
        E = f.sum((1, 2)) @ self.px.square() + f.sum((1, 3)) @ py.square() + f.sum((2, 3)) @ pz.square()
        T = (E - n * u.square().sum(1)) / (self.D * n)
        q = torch.empty_like(n)
        for a in range(0, n.shape[0], 65536):
            s = slice(a, a + 65536)
            cx = self.px[None, :] - u[s, 0, None]
            cy = (py[None, :] - u[s, 1, None]).square() if self.other[0][2] is not None else torch.zeros_like(u[s, :1])
            cz = (pz[None, :] - u[s, 2, None]).square() if self.other[1][2] is not None else torch.zeros_like(u[s, :1])
            g = f[s]
            q[s] = 0.5 * ((g.sum((1, 2)) * cx.pow(3)).sum(1) +
                          ((g.sum(1) @ cx[:, :, None]).squeeze(2) * cy).sum(1) +
                          ((g.sum(2) @ cx[:, :, None]).squeeze(2) * cz).sum(1))
        return n, u, T, q


def _weno5(a, b, c, d, e):
    """Upwind face value of the stencil a..e (face between c and d), no epsilon: a vanishing indicator takes all weight."""
    m = torch.maximum(torch.maximum(a.abs(), b.abs()), torch.maximum(torch.maximum(c.abs(), d.abs()), e.abs()))
    m = torch.where(m > 0, m, torch.ones_like(m))
    A, B, C, D, E = a / m, b / m, c / m, d / m, e / m
    s = [13 / 12 * (A - 2 * B + C).square() + 0.25 * (A - 4 * B + 3 * C).square(),
         13 / 12 * (B - 2 * C + D).square() + 0.25 * (B - D).square(),
         13 / 12 * (C - 2 * D + E).square() + 0.25 * (3 * C - 4 * D + E).square()]
    low = torch.minimum(s[0], torch.minimum(s[1], s[2]))
    w = [k * torch.where(low > 0, low / x, (x == 0).to(x.dtype)).nan_to_num(0.0).square() for k, x in zip((0.1, 0.6, 0.3), s)]
    del s, low
    top = w[0] * (2 * A - 7 * B + 11 * C) + w[1] * (5 * C - B + 2 * D) + w[2] * (2 * C + 5 * D - E)
    return top / (6 * (w[0] + w[1] + w[2])) * m


def _face(adv, a, b, c, d, e):
    return _weno5(a, b, c, d, e) if adv == W.WENO5 else 1.5 * c - 0.5 * b


class _Group:
    """The instances of one velocity set and scheme, their cells flattened; every row gets three ghosts at each wall."""

    def __init__(self, cfgs, fields):
        self.ax = _Axes.of(cfgs[0])
        self.adv = cfgs[0]["advection"]
        cells, ext, inv_dx, per_cell = 0, [], [], {k: [] for k in ("dt", "inv_Kn", "ax", "ay", "az")}
        lines = []
        self.two_d = cfgs[0]["ny"] > 1
        self.rows = (cfgs[0]["ny"], cfgs[0]["nx"]) if self.two_d else None
        # the walls' Maxwellians (rows of a 2D instance share them)
        walls = torch.as_tensor([c["T_left"] for c in cfgs] + [c["T_right"] for c in cfgs], dtype=torch.float64, device="cuda")
        walls = self.ax.equilibrium(torch.ones_like(walls), walls.new_zeros((walls.numel(), 3)), walls)
        self.gl, self.gr = walls[:len(cfgs)], walls[len(cfgs):]
        px_hi = float(self.ax.px.abs().max())
        py_hi = float(self.ax.other[0][0].abs().max())
        slots = 0
        for c in cfgs:
            nx, ny = c["nx"], c["ny"]
            if c["stretch_A"] > 0:
                step = 2 * math.atanh(c["stretch_A"]) / nx
                edge = c["Lx"] / 2 + c["Lx"] / (2 * c["stretch_A"]) * np.tanh((np.arange(nx + 1) - nx / 2) * step)
            else:
                edge = np.linspace(0.0, c["Lx"], nx + 1)
            dx = np.diff(edge)
            self.inv_dy = ny / c["Ly"]
            rate = px_hi / dx.min() + (py_hi * self.inv_dy if ny > 1 else 0.0)
            fa = fields.get(id(c), (0.0, 0.0))
            for k, v in (("dt", c["dt"] if c["dt"] > 0 else c["cfl"] / rate),
                         ("inv_Kn", 0.0 if math.isinf(c["Kn"]) else 1 / c["Kn"]), ("ax", c["ax"] + fa[0]),
                         ("ay", c["ay"] + (0.0 if fa[1] is None else fa[1])), ("az", c["az"])):
                per_cell[k].append(np.broadcast_to(np.asarray(v, dtype=np.float64), (ny, nx)).ravel())
            inv_dx.append(np.tile(1 / dx, ny))
            for y in range(ny):
                lines.append((cells + y * nx, nx, slots))
                ext.append(np.arange(nx) + slots + 3)
                slots += nx + 6
            cells += nx * ny

        def up(a, dtype=torch.float64):
            return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")

        self.slots = slots
        self.ext = up(np.concatenate(ext), torch.long)
        self.inv_dx = up(np.concatenate(inv_dx))
        self.p = {k: up(np.concatenate(v)) for k, v in per_cell.items()}
        L = np.array(lines)
        self.left = [up(L[:, 0] + i, torch.long) for i in range(3)]
        self.right = [up(L[:, 0] + L[:, 1] - 1 - i, torch.long) for i in range(3)]
        self.ghost_l = [up(L[:, 2] + 2 - i, torch.long) for i in range(3)]
        self.ghost_r = [up(L[:, 2] + L[:, 1] + 3 + i, torch.long) for i in range(3)]

    def rate(self, f):
        """L[f] of f[cells, kz, jy, ix]."""
        A, h = self.ax, self.ax.half
        collide = bool((self.p["inv_Kn"] != 0).any())
        L = torch.zeros_like(f)
        if collide:
            n, u, T, _ = A.moments(f)
            gx, gy, gz = A.factors(n, u, T)
            itau = (n * self.p["inv_Kn"])[:, None, None]
        # walls: the incident fluxes over the whole velocity set fix the emitted densities
        flux = {}
        for side, cells, part in (("l", self.left, slice(h, None)), ("r", self.right, slice(0, h))):
            f0, f1, f2 = (f[i][..., part] for i in cells)
            d, e = 3 * f0 - 3 * f1 + f2, 6 * f0 - 8 * f1 + 3 * f2
            flux[side] = (_face(self.adv, f2, f1, f0, d, e) * A.px[part]).sum((1, 2, 3))
        den_l = (self.gl[..., :h] * A.px[:h]).sum((1, 2, 3))
        den_r = (self.gr[..., h:] * A.px[h:]).sum((1, 2, 3))
        nl, nr = (-flux["l"] / den_l)[:, None, None], (-flux["r"] / den_r)[:, None, None]
        for kz in range(f.shape[1]):
            s = f[:, kz]
            E = torch.zeros((self.slots,) + s.shape[1:], dtype=f.dtype, device=f.device)
            E[self.ext] = s
            l0, l1, l2 = (s[i][..., h:] for i in self.left)
            r0, r1, r2 = (s[i][..., :h] for i in self.right)
            for i in range(3):
                E[self.ghost_l[i], :, :h] = nl * self.gl[:, kz, :, :h]
                E[self.ghost_r[i], :, h:] = nr * self.gr[:, kz, :, h:]
            E[self.ghost_l[0], :, h:], E[self.ghost_l[1], :, h:] = 3 * l0 - 3 * l1 + l2, 6 * l0 - 8 * l1 + 3 * l2
            E[self.ghost_r[0], :, :h], E[self.ghost_r[1], :, :h] = 3 * r0 - 3 * r1 + r2, 6 * r0 - 8 * r1 + 3 * r2
            for part, mirrored in ((slice(0, h), False), (slice(h, None), True)):
                e = E[..., part]
                F = torch.zeros_like(e)              # F[i]: the face between slots i and i + 1
                m = self.slots
                if mirrored:
                    F[1:m - 3] = _face(self.adv, e[4:], e[3:m - 1], e[2:m - 2], e[1:m - 3], e[:m - 4])
                else:
                    F[2:m - 2] = _face(self.adv, e[:m - 4], e[1:m - 3], e[2:m - 2], e[3:m - 1], e[4:])
                L[:, kz, :, part] -= (F[self.ext] - F[self.ext - 1]) * self.inv_dx[:, None, None] * A.px[part]
                del e, F
            del E
            if self.two_d:
                py, g = A.other[0][0], s.reshape(self.rows + s.shape[1:])
                for j in range(py.numel()):
                    up = float(py[j]) > 0
                    q = [g[:, :, j].roll(-k if up else k, 0) for k in range(-2, 3)]
                    G = _face(self.adv, *(q if up else [x.roll(-1, 0) for x in q]))      # the face above each row
                    L[:, kz, j] -= ((G - G.roll(1, 0)) * (self.inv_dy * py[j])).reshape(s.shape[0], -1)
            kf = (s @ A.Kx.T) * self.p["ax"][:, None, None]
            if A.other[0][2] is not None:
                kf += torch.einsum("jk,ckx->cjx", A.other[0][3], s) * self.p["ay"][:, None, None]
            if A.other[1][2] is not None and bool((self.p["az"] != 0).any()):
                kf += torch.einsum("k,ckjx->cjx", A.other[1][3][kz], f) * self.p["az"][:, None, None]
            L[:, kz] -= kf
            if collide:
                L[:, kz] -= (s - gz[:, kz, None, None] * gy[:, :, None] * gx[:, None, :]) * itau
        return L

    def step(self, f):
        dt = self.p["dt"][:, None, None, None]
        f1 = self.rate(f).mul_(dt).add_(f)
        f2 = self.rate(f1).mul_(dt).add_(f1).mul_(0.25).add_(f, alpha=0.75)
        del f1
        return self.rate(f2).mul_(dt).add_(f2).mul_(2 / 3).add_(f, alpha=1 / 3)


def exact(case, seed):
    cfgs = _configs(case)
    f0 = _initial(case, cfgs, seed).double()
    fields = {id(c): _field(c) for c in cfgs} if case["field"] else {}
    groups: dict = {}
    at = 0
    for c in cfgs:
        groups.setdefault((c["Qx"], c["Qy"], c["Qz"], c["Nx_eq"], c["advection"], c["x_basis"]), []).append((c, at))
        at += _values(c)
    if case["kind"] == "moments":
        n, u, T, q = _Axes.of(cfgs[0]).moments(f0.view((-1,) + _Axes.of(cfgs[0]).shape))
        return {"n": n, "u": u, "T": T, "q": q}
    for members in groups.values():
        grp = _Group([c for c, _ in members], fields)
        f = torch.cat([f0[a:a + _values(c)] for c, a in members]).view((-1,) + grp.ax.shape)
        for _ in range(case["steps"]):
            f = grp.step(f)
        f = f.reshape(-1)
        b = 0
        for c, a in members:
            f0[a:a + _values(c)] = f[b:b + _values(c)]
            b += _values(c)
        del f, grp
    return {"f": f0}
