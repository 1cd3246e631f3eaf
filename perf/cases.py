"""Workloads of the solver library as a program calls it: short Crank-Nicolson
trajectories (symmetric and not, every arithmetic path, one problem and many,
state on the device and on the host) and the warm-start network's training
step and prediction.

  listed()            the named workloads
  draw(rng)           one more of the same ranges
  prepare(case, seed) inputs, problems and buffers a program has in hand
  run(state)          one pass through the public entry points
  work(case)          bytes and operations of one pass that cannot be avoided
  exact(case, seed)   the same results in 64-bit arithmetic with plain torch
"""
from __future__ import annotations

import math
import random
from decimal import Decimal, localcontext

import numpy as np
import torch

from paper_2511_21198_gb300 import tfde as T
from paper_2511_21198_gb300 import warmstart as W

DEV = "cuda"


# ------------------------------------------------------------------ the list
def march(name, n, delta, kp, km, steps, dt, tol, mixed=True, source=False, order=0, host=False):
    c = {"kind": "march", "mixed": mixed, "source": source, "order": order, "host": host, "steps": steps, "dt": dt,
         "tol": tol}
    for a in range(3):
        c |= {f"n{a}": n[a], f"delta{a}": delta[a], f"kp{a}": kp[a], f"km{a}": km[a]}
    return {"name": name, **c} if name else c


def batch(name, count, layout, largest, symmetric, steps, tol):
    c = {"kind": "batch", "count": count, "layout": layout, "largest": largest, "symmetric": symmetric,
         "steps": steps, "dt": 0.1, "tol": tol}
    return {"name": name, **c} if name else c


def network(name, train, n, samples):
    c = {"kind": "train" if train else "predict", "samples": samples}
    c |= {f"n{a}": n[a] for a in range(3)}
    return {"name": name, **c} if name else c


# Tolerances: the paper's 1e-9 where it leaves the solution within a few 1e-10 of the discrete one, 1e-10 (what the
# network's training trajectories are computed with) otherwise.
SYM = ((1.0,) * 3, (1.0,) * 3)
SKEW = ((1.0,) * 3, (0.5,) * 3)


def listed():
    return [
        # the smallest workload of the benchmark: every step in FP64, bound by latency
        march("fp64_sym_16", (16,) * 3, (0.5,) * 3, *SYM, 16, 1 / 16, 1e-9, mixed=False, source=True),
        # the FP64 path at an ordinary size, non-symmetric: what the mixed path is compared with
        march("fp64_skew_64", (64,) * 3, (0.3, 0.6, 0.8), *SKEW, 4, 1 / 50, 1e-9, mixed=False),
        # a small uneven grid on the tensor-core path, default guess: a parameter study's inner call
        march("mixed_skew_40x32x24", (40, 32, 24), (0.3, 0.6, 0.8), *SKEW, 8, 1 / 50, 1e-10),
        # the non-symmetric benchmark workload (PGMRES)
        march("mixed_skew_128", (128,) * 3, (0.3, 0.6, 0.8), *SKEW, 10, 1 / 50, 1e-10, order=3),
        # the headline workload (PCG, manufactured source)
        march("mixed_sym_256", (256,) * 3, (0.7,) * 3, *SYM, 10, 1 / 20, 1e-9, source=True, order=3),
        # the same solver for a program that keeps its state in host memory
        march("host_sym_192", (192,) * 3, (0.7,) * 3, *SYM, 6, 1 / 20, 1e-9, source=True, order=3, host=True),
        # the paper's own grids, n + 1 a power of two: no axis is a multiple of eight
        march("mixed_sym_127", (127,) * 3, (0.7,) * 3, *SYM, 6, 1 / 16, 1e-9, source=True, order=3),
        # a ragged uneven grid, non-symmetric
        march("mixed_skew_90x75x110", (90, 75, 110), (0.4, 0.5, 0.7), *SKEW, 5, 1 / 50, 1e-10),
        # the paper's two-dimensional example at its largest grid
        march("plane_skew_511", (511, 511, 0), (0.4, 0.5, 0.5), (19.0, 21.0, 1.0), (21.0, 23.0, 1.0), 6, 1 / 64, 1e-9,
              source=True),
        # the batched workload of the benchmark: 64 uneven non-symmetric problems
        batch("batch_skew_64", 64, 4, 128, False, 4, 1e-10),
        # one optimiser step of the warm-start network: a mini-batch of eight samples
        network("train_64", True, (64,) * 3, 8),
        # the network's proposal of an initial guess on a finer grid than it was trained on
        network("predict_128", False, (128,) * 3, 1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["fp64", "mixed", "mixed", "mixed", "ragged", "ragged", "plane", "batch", "train", "predict"])
    delta = tuple(round(rng.uniform(0.1, 0.9), 3) for _ in range(3))
    kp = tuple(round(rng.uniform(0.5, 2.0), 3) for _ in range(3))
    sym = rng.random() < 0.5
    km = kp if sym else tuple(round(rng.uniform(0.5, 2.0), 3) for _ in range(3))
    source, order = rng.random() < 0.5, rng.choice([0, 3, 3])
    steps, dt = rng.randint(3, 10), rng.choice([1 / 10, 1 / 20, 1 / 50])
    if kind == "fp64":
        return march(None, tuple(_log(rng, 12, 96) for _ in range(3)), delta, kp, km, min(steps, 5), dt, 1e-10,
                     mixed=False, source=source)
    if kind == "mixed":
        n = tuple(8 * _log(rng, 2, 36) for _ in range(3))
        while points(n) > 256 ** 3:
            n = tuple(8 * _log(rng, 2, 36) for _ in range(3))
        return march(None, n, delta, kp, km, steps, dt, 1e-10, source=source, order=order, host=rng.random() < 0.2)
    if kind == "ragged":
        n = tuple(_log(rng, 15, 150) for _ in range(3))
        return march(None, n, delta, kp, km, min(steps, 5), dt, 1e-10, source=source, order=order)
    if kind == "plane":
        return march(None, (_log(rng, 60, 600), _log(rng, 60, 600), 0), delta, kp, km, min(steps, 5), dt, 1e-10,
                     source=source)
    if kind == "batch":
        return batch(None, rng.randint(4, 48), rng.randint(0, 1 << 20), rng.choice([48, 96, 128]), sym,
                     rng.randint(2, 4), 1e-10)
    if kind == "train":
        return network(None, True, tuple(_log(rng, 16, 80) for _ in range(3)), rng.randint(2, 8))
    return network(None, False, tuple(_log(rng, 16, 160) for _ in range(3)), rng.randint(1, 3))


def grid(case):
    return tuple(case[f"n{a}"] for a in range(3))


def points(n):
    return n[0] * n[1] * max(1, n[2])


def batch_grids(case):
    r = random.Random(case["layout"])
    sizes = [n for n in (32, 48, 64, 96, 128) if n <= case["largest"]]
    return [(r.choice(sizes),) * 3 for _ in range(case["count"])]


def work(case):
    """Each step reads and writes the state once (FP64); the network reads the
    levels it is given and does the products of its four convolutions (and,
    for a training sample, of the two gradients of each)."""
    if case["kind"] == "march":
        return {"bytes": 16.0 * case["steps"] * points(grid(case)), "flops": 0}
    if case["kind"] == "batch":
        return {"bytes": 16.0 * case["steps"] * sum(points(n) for n in batch_grids(case)), "flops": 0}
    N, s = points(grid(case)), case["samples"]
    forward = 2.0 * 27 * (13 * 16 + 2 * 16 * 16 + 16) * N
    if case["kind"] == "train":
        return {"bytes": 40.0 * N * s, "flops": s * (3 * forward - 2.0 * 27 * 13 * 16 * N)}
    return {"bytes": 40.0 * N * s, "flops": s * forward}


# ------------------------------------------------------------------ inputs
def generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 17)


def smoothed(shape, g, passes=4):
    """Uniform noise smoothed by [1, 2, 1] / 4 per axis with zero exterior, largest value 1."""
    u = torch.rand(shape, generator=g, device=DEV, dtype=torch.float64)
    for _ in range(passes):
        for ax in range(3):
            if shape[ax] == 1:
                continue
            m = shape[ax]
            v = 0.5 * u
            v.narrow(ax, 1, m - 1).add_(u.narrow(ax, 0, m - 1), alpha=0.25)
            v.narrow(ax, 0, m - 1).add_(u.narrow(ax, 1, m - 1), alpha=0.25)
            u = v
    return (u / u.abs().max()).contiguous()


def profile(n):
    """Nodal values of P(x) P(y) P(z), P(s) = s^2 (1 - s)^2 (P(x) P(y) in two dimensions)."""
    out = torch.ones((1, 1, 1), device=DEV, dtype=torch.float64)
    for a in range(3):
        if n[a] > 0:
            s = torch.arange(1, n[a] + 1, device=DEV, dtype=torch.float64) / (n[a] + 1)
            view = [1, 1, 1]
            view[2 - a] = n[a]
            out = out * (s * s * (1 - s) ** 2).view(view)
    return out.contiguous()


def initial(case, seed):
    """(u^0, amplitude, t_0): the manufactured solution's initial data, scaled
    and shifted in time, with a source; smoothed noise without."""
    n, r = grid(case), random.Random(seed)
    if case["source"]:
        amp, t0 = r.uniform(0.5, 4.0), r.uniform(0.0, 0.5)
        return profile(n) * (amp * math.exp(-t0)), amp, t0
    return smoothed((max(1, n[2]), n[1], n[0]), generator(seed)), 0.0, 0.0


def coefficients(case):
    return tuple(tuple(case[f"{k}{a}"] for a in range(3)) for k in ("delta", "kp", "km"))


def batch_coefficients(case, seed):
    r = random.Random(seed * 31 + 5)
    out = []
    for _ in range(case["count"]):
        delta = tuple(r.uniform(0.1, 0.9) for _ in range(3))
        kp = tuple(r.uniform(0.5, 2.0) for _ in range(3))
        out.append((delta, kp, kp if case["symmetric"] else tuple(r.uniform(0.5, 2.0) for _ in range(3))))
    return out


def network_inputs(case, seed):
    """Parameters, nine constants and, per sample, four consecutive levels of a
    slowly varying state with a source term."""
    n = grid(case)
    shape = (n[2], n[1], n[0])
    g, r = generator(seed), random.Random(seed)
    out = []
    for _ in range(case["samples"]):
        levels = [smoothed(shape, g)]
        for d in (0.1, 0.08, 0.07):
            levels.append(levels[-1] * (1 - d) + 0.2 * d * smoothed(shape, g))
        delta = [r.uniform(0.1, 0.9) for _ in range(3)]
        out.append((levels, 0.01 * smoothed(shape, g), delta + [r.uniform(-1.0, 3.0) for _ in range(6)]))
    return W.init_params(seed % 100003), out


class State:
    """What a program keeps between calls; releases the library's objects with itself."""

    def __init__(self, case):
        self.case, self.problem, self.batch, self.net = case, None, None, None

    def __del__(self):
        if self.problem is not None:
            T.tfde_destroy(self.problem)
        if self.batch is not None:
            T.tfde_batch_destroy(self.batch)
        if self.net is not None:
            T.tfde_cnn_destroy(self.net)


def prepare(case, seed):
    s = State(case)
    if case["kind"] == "march":
        delta, kp, km = coefficients(case)
        prm = T.make_params(grid(case), delta, kp, km, case["dt"])
        s.problem = T.tfde_assemble(prm, T.TFDE_MIXED if case["mixed"] else T.TFDE_FP64)
        T.tfde_set_guess_order(s.problem, case["order"])
        s.u0, s.amp, s.t0 = initial(case, seed)
        s.u = torch.empty_like(s.u0)
        s.F = torch.empty_like(s.u0) if case["source"] else None
        if case["host"]:
            s.first = s.u0.cpu().pin_memory()
            s.levels = [torch.empty_like(s.first).pin_memory() for _ in range(2)]
    elif case["kind"] == "batch":
        prm = [T.make_params(n, *c, case["dt"]) for n, c in zip(batch_grids(case), batch_coefficients(case, seed))]
        s.batch = T.tfde_batch_create(prm, 20)
        T.tfde_batch_set_guess_order(s.batch, 3)
        g = generator(seed)
        s.u0 = [smoothed(n, g) for n in batch_grids(case)]
        s.u = [torch.empty_like(u) for u in s.u0]
    else:
        s.params, s.samples = network_inputs(case, seed)
        s.net = T.tfde_cnn_create(grid(case))
        T.tfde_cnn_set_params(s.net, s.params)
        s.out = [torch.empty_like(levels[0]) for levels, _, _ in s.samples]
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    case = s.case
    if case["kind"] == "march":
        if not case["host"]:
            s.u.copy_(s.u0)
        given = s.first if case["host"] else None
        for m in range(case["steps"]):
            if s.F is not None:
                f = -s.amp * math.exp(-(s.t0 + (m + 0.5) * case["dt"]))
                T.tfde_source_example2(s.problem, f, f, s.F)
            if case["host"]:
                T.tfde_cn_advance_host(s.problem, given, s.levels[m % 2], s.u, s.F, m == 0, case["tol"])
                given = s.levels[m % 2]
            else:
                T.tfde_cn_advance(s.problem, s.u, s.F, m == 0, case["tol"])
        return given if case["host"] else s.u
    if case["kind"] == "batch":
        for u, u0 in zip(s.u, s.u0):
            u.copy_(u0)
        for m in range(case["steps"]):
            T.tfde_batch_cn_advance(s.batch, s.u, None, m == 0, case["tol"])
        return s.u
    if case["kind"] == "train":
        # from a given checkpoint: the gradients of the mini-batch and the updated parameters
        T.tfde_cnn_set_params(s.net, s.params)
        loss = [T.tfde_cnn_accumulate_hist(s.net, lv[2], lv[1], lv[0], F, c, lv[3]) for lv, F, c in s.samples]
        grads = T.tfde_cnn_get_grads(s.net)
        T.tfde_cnn_adam_step(s.net, 1e-3)
        return {"loss": np.array(loss), "grads": grads, "params": T.tfde_cnn_get_params(s.net)}
    for (lv, F, c), x0 in zip(s.samples, s.out):
        T.tfde_cnn_predict_hist(s.net, lv[2], lv[1], lv[0], F, c, x0)
    return s.out


# ------------------------------------------------------------------ 64 bits
def generator_q(delta, n):
    """q_0..q_n: first differences of s_k, the second differences of (k + 1/2)^delta."""
    with localcontext() as ctx:
        ctx.prec = 45
        d = Decimal(delta)
        p = [(Decimal(2 * k + 1) / 2) ** d for k in range(n + 1)]
        s = [p[0], p[1] - 2 * p[0]] + [p[k] - 2 * p[k - 1] + p[k - 2] for k in range(2, n + 1)]
        return [float(-s[0])] + [float(s[k - 1] - s[k]) for k in range(1, n + 1)]


class Axis:
    """Stiffness eta B, mass A, the sine transform S and the eigenvalues of one axis."""

    def __init__(self, n, delta, kp, km, dt):
        f = dict(device=DEV, dtype=torch.float64)
        i = torch.arange(n, device=DEV)
        eta = dt / (2 * math.gamma(delta + 1) * (1 / (n + 1)) ** (2 - delta))
        q = generator_q(delta, n)
        at = i[:, None] - i[None, :] + 1
        Tm = torch.where(at >= 0, torch.tensor(q, **f)[at.clamp(0, n)], torch.zeros((), **f))
        self.B = eta * (kp * Tm + km * Tm.T)
        near = (i[:, None] - i[None, :]).abs()
        self.A = ((near == 0) * 6.0 + (near == 1) * 1.0).to(torch.float64) / 8
        k = torch.arange(1, n + 1, **f)
        th = k * (math.pi / (n + 1))
        self.S = math.sqrt(2 / (n + 1)) * torch.sin((k[:, None] * k[None, :] % (2 * (n + 1))) * (math.pi / (n + 1)))
        self.mu = (6 + 2 * torch.cos(th)) / 8
        j = torch.arange(n, **f)
        t = torch.tensor([q[1]] + ([q[0] + q[2]] if n > 1 else []) + [q[m + 1] for m in range(2, n)], **f)
        self.lam = eta * (kp + km) * (torch.cos(th[:, None] * j[None, :]) @ t)


class Point:
    """The absent third axis of a two-dimensional problem."""

    def __init__(self):
        one = torch.ones((1, 1), device=DEV, dtype=torch.float64)
        self.A, self.S, self.B, self.mu, self.lam = one, one, 0 * one, one[0], 0 * one[0]


def along(M, v, a):
    if a == 0:
        return v @ M.T
    if a == 1:
        return torch.matmul(M, v)
    return (M @ v.reshape(v.shape[0], -1)).view(v.shape)


class System:
    def __init__(self, n, delta, kp, km, dt):
        self.dt, self.n, self.delta, self.kp, self.km = dt, n, delta, kp, km
        self.ax = [Axis(n[a], delta[a], kp[a], km[a], dt) if n[a] > 0 else Point() for a in range(3)]
        m = [self.ax[a].mu.view([-1 if 2 - a == i else 1 for i in range(3)]) for a in range(3)]
        e = [self.ax[a].lam.view([-1 if 2 - a == i else 1 for i in range(3)]) for a in range(3)]
        lam = m[2] * m[1] * m[0] + m[2] * m[1] * e[0] + m[2] * e[1] * m[0] + e[2] * m[1] * m[0]
        # the preconditioner and the inner Krylov vectors in 32 bits: refinement supplies the rest
        self.lam32, self.S32 = lam.float(), [x.S.float() for x in self.ax]
        self.op32 = [(x.A.float(), x.B.float()) for x in self.ax]
        self.op64 = [(x.A, x.B) for x in self.ax]

    @staticmethod
    def terms(ops, v):
        """(A_N v, K v)"""
        (A0, B0), (A1, B1), (A2, B2) = ops
        a = along(A0, v, 0)
        xy = along(A1, a, 1)
        stiff = along(A2, along(A1, along(B0, v, 0), 1) + along(B1, a, 1), 2) + along(B2, xy, 2)
        return along(A2, xy, 2), stiff

    def precondition(self, r):
        for a in range(3):
            r = along(self.S32[a], r, a)
        r = r / self.lam32
        for a in range(3):
            r = along(self.S32[a], r, a)
        return r

    def correct(self, r, steps=14):
        """An approximate A^{-1} r by GMRES on 32-bit vectors, preconditioned from the right."""
        beta = float(r.norm())
        V = torch.empty((steps + 1, r.numel()), device=DEV, dtype=torch.float32)
        V[0] = (r / beta).float().view(-1)
        H = torch.zeros((steps + 1, steps), device=DEV, dtype=torch.float64)
        for j in range(steps):
            mass, stiff = self.terms(self.op32, self.precondition(V[j].view(r.shape)))
            w = (mass + stiff).view(-1)
            for _ in range(2):
                h = V[:j + 1] @ w
                w = w - V[:j + 1].T @ h
                H[:j + 1, j] += h.double()
            H[j + 1, j] = w.double().norm()
            V[j + 1] = w / H[j + 1, j].clamp_min(1e-30).float()
        e = torch.zeros((steps + 1, 1), device=DEV, dtype=torch.float64)
        e[0] = beta
        y = torch.linalg.lstsq(H.cpu(), e.cpu(), driver="gelsd").solution[:, 0].to(DEV)
        scale = float(y.abs().max())
        x = V[:steps].T @ (y / scale).float()
        return self.precondition(x.view(r.shape)).double() * scale

    def advance(self, u, F):
        mass, stiff = self.terms(self.op64, u)
        b = mass - stiff + (0 if F is None else self.dt * F)
        x, best = u.clone(), None
        for _ in range(8):
            mass, stiff = self.terms(self.op64, x)
            r = b - mass - stiff
            rel = float(r.norm() / b.norm())
            if best is not None and rel > 0.5 * best[0]:
                break
            best = (rel, x)
            if rel < 1e-14:
                break
            x = x + self.correct(r)
        return best[1]

    def averages(self, f):
        """Cell averages of f (P P P + S P P + P S P + P P S): the factors' exact integrals."""
        def power(p, left, n):
            """Mean of s^p (left) or (1 - s)^p over the cells around the nodes."""
            h = 1.0 / (n + 1)
            c = (torch.arange(1, n + 1, device=DEV, dtype=torch.float64) * h)
            c = c if left else 1 - c
            return ((c + h / 2) ** (p + 1) - (c - h / 2) ** (p + 1)) / ((p + 1) * h)

        P, S = [], []
        for a in range(3):
            n, d = self.n[a], self.delta[a]
            view = [-1 if 2 - a == i else 1 for i in range(3)]
            if n == 0:
                P.append(torch.ones((1, 1, 1), device=DEV, dtype=torch.float64))
                S.append(torch.zeros((1, 1, 1), device=DEV, dtype=torch.float64))
                continue
            P.append((power(2, True, n) - 2 * power(3, True, n) + power(4, True, n)).view(view))
            acc = 0
            for k in range(3):
                w = (-1) ** k * math.comb(2, k) * math.gamma(5 - k) / math.gamma(3 - k + d)
                acc = acc + w * (self.kp[a] * power(2 - k + d, True, n) + self.km[a] * power(2 - k + d, False, n))
            S.append(acc.view(view))
        return f * (P[2] * P[1] * P[0] + P[2] * P[1] * S[0] + P[2] * S[1] * P[0] + S[2] * P[1] * P[0])

    def march(self, u, steps, amp=None, t0=0.0):
        base = None if amp is None else self.averages(1.0)
        for m in range(steps):
            F = None if amp is None else -amp * math.exp(-(t0 + (m + 0.5) * self.dt)) * base
            u = self.advance(u, F)
        return u


def convolve(x, Wl, b):
    """3 x 3 x 3 convolution with zero padding: x (cin, n3, n2, n1), Wl (cout, cin, 27)."""
    z, y, w = x.shape[1:]
    p = torch.nn.functional.pad(x, (1, 1, 1, 1, 1, 1))
    out = b.view(-1, 1).expand(-1, z * y * w)
    for t in range(27):
        v = p[:, t // 9:t // 9 + z, t // 3 % 3:t // 3 % 3 + y, t % 3:t % 3 + w]
        out = out + Wl[:, :, t] @ v.reshape(x.shape[0], -1)
    return out.view(-1, z, y, w)


def network64(flat, levels, F, c):
    """(base, s, output) of the network at the third of the four levels."""
    u, u1, u2 = levels[2], levels[1], levels[0]
    s = u.abs().max()
    x = torch.stack([u / s, F / s] + [torch.full_like(u, v) for v in c] + [(u - u1) / s, (u - 2 * u1 + u2) / s])
    for l in range(4):
        blk = flat[l * W.PSZ:(l + 1) * W.PSZ]
        co, ci = W.CHANNELS[l + 1], W.CHANNELS[l]
        x = convolve(x, blk[:W.WSZ].view(16, 16, 27)[:co, :ci], blk[W.WSZ:W.WSZ + co])
        x = torch.relu(x) if l < 3 else x
    return 3 * u - 3 * u1 + u2, s, x[0]


def exact(case, seed):
    if case["kind"] == "march":
        A = System(grid(case), *coefficients(case), case["dt"])
        u0, amp, t0 = initial(case, seed)
        u = A.march(u0, case["steps"], amp if case["source"] else None, t0)
        return u.cpu() if case["host"] else u
    if case["kind"] == "batch":
        g, out = generator(seed), []
        for n, c in zip(batch_grids(case), batch_coefficients(case, seed)):
            out.append(System(n, *c, case["dt"]).march(smoothed(n, g), case["steps"]))
        return out
    params, samples = network_inputs(case, seed)
    flat = torch.tensor(params, device=DEV, dtype=torch.float64, requires_grad=case["kind"] == "train")
    if case["kind"] == "predict":
        out = []
        for lv, F, c in samples:
            base, s, y = network64(flat, lv, F, c)
            out.append(base + s * y)
        return out
    loss = []
    for lv, F, c in samples:
        base, s, y = network64(flat, lv, F, c)
        e = (y - (lv[3] - base) / s).square().mean()
        e.backward()
        loss.append(float(e.detach()))
    grads = flat.grad
    g = grads / len(samples)
    updated = flat.detach() - 1e-3 * g / (g.abs() + 1e-8)
    return {"loss": np.array(loss), "grads": grads.cpu().numpy(), "params": updated.cpu().numpy()}
