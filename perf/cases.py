"""What programs built on this package have it do, as cases that can be timed and compared.

Each case is one call (or one short sequence of calls) of the public API on a seeded
synthetic population with the shape of one of the three flows of
paper_2606_15622_gb300/populations.py, drawn here on the GPU:

  couette   every cell holds `ppc` particles of a Maxwellian
  cavity    Poisson(`ppc`) particles, skewed and stressed distributions, 10 % bimodal cells
  cylinder  log-normal counts around `ppc` (2 to 2000 a cell, an uneven total): Mach-10 free stream, hot
            post-shock layer, two-temperature shock cells, rarefied wake, near-empty body

Cells with fewer than MIN_PARTICLES particles take the linear drift, as a program sets
that does not want coefficients from a handful of particles.
"""

import functools
import math
import os

import torch

import paper_2606_15622_gb300 as package
from paper_2606_15622_gb300 import api, autograd, surrogate

MIN_PARTICLES = 8
EPS2 = 1e-3
DT = 0.1
MAX_PARTICLES = 12_000_000
WEIGHTS = os.path.join(os.path.dirname(package.__file__), "weights")


def listed():
    return [
        # A one-dimensional flow's cells, the smallest population that the benchmark knows:
        # latency and launches count.
        {"name": "couette_exact_fp64", "op": "exact", "flow": "couette", "cells": 400, "ppc": 100, "prec": "fp64"},
        # The exact closure of an ordinary flow in its fast mode (FP32 velocities and moments).
        {"name": "cavity_exact_fp32", "op": "exact", "flow": "cavity", "cells": 16384, "ppc": 50, "prec": "fp32"},
        # The same call on the largest flow, in both precisions.
        {"name": "cylinder_exact_fp32", "op": "exact", "flow": "cylinder", "cells": 131072, "ppc": 91, "prec": "fp32"},
        {"name": "cylinder_exact_fp64", "op": "exact", "flow": "cylinder", "cells": 131072, "ppc": 91, "prec": "fp64"},
        # A loss through the closure: forward and backward in FP64 with autograd.
        {"name": "cavity_gradient_fp64", "op": "gradient", "flow": "cavity", "cells": 16384, "ppc": 50, "prec": "fp64"},
        # Solve keeping its factors, then the adjoint from them down to FP32 velocities.
        {"name": "cylinder_adjoint_fp32", "op": "adjoint", "flow": "cylinder", "cells": 131072, "ppc": 91, "prec": "fp32"},
        # The collision step of the particles with the library's own noise.
        {"name": "cylinder_update_fp32", "op": "update", "flow": "cylinder", "cells": 131072, "ppc": 91, "prec": "fp32"},
        # Inference of the learned closure on a batch of a million cells.
        {"name": "learned_closure_1m", "op": "learned", "flow": "cavity", "cells": 1048576, "ppc": 50, "prec": "fp32"},
        # One step of a flow solver: particles that moved a little are sorted by cell, closed and updated.
        {"name": "cylinder_step_exact", "op": "step", "flow": "cylinder", "cells": 131072, "ppc": 91, "prec": "fp32",
         "net": False, "moved": 0.03},
        # The same with the learned closure on low-order inputs, on an odd number of cells in any order.
        {"name": "cylinder_step_lite", "op": "step", "flow": "cylinder", "cells": 20011, "ppc": 60, "prec": "fp32",
         "net": True, "moved": 1.0},
        # One training step of the learned closure at the benchmark's batch size.
        {"name": "train_step_8192", "op": "train", "flow": "cavity", "cells": 8192, "ppc": 50, "prec": "fp32"},
        # A step on velocities in host memory: closure, learned closure, adjoint and update, copies overlapped.
        {"name": "cylinder_host_step", "op": "host", "flow": "cylinder", "cells": 131072, "ppc": 91, "prec": "fp32"},
    ]


def draw(rng):
    op = rng.choice(["exact", "exact", "exact", "gradient", "adjoint", "update", "learned", "step", "step", "train",
                     "host"])
    flow = rng.choice(["couette", "cavity", "cylinder"])
    prec = "fp64" if op == "gradient" or op == "exact" and rng.random() < 0.5 else "fp32"
    ppc = round(math.exp(rng.uniform(math.log(12), math.log(200))))
    lo, hi = {"train": (256, 8192), "learned": (300, 1048576), "gradient": (100, 16384)}.get(op, (100, 131072))
    cells = round(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    if op == "learned":
        ppc = min(ppc, 50)
    elif cells * ppc > MAX_PARTICLES * 0.99:
        cells = int(MAX_PARTICLES * 0.99) // ppc
    case = {"op": op, "flow": flow, "cells": cells, "ppc": ppc, "prec": prec}
    if op == "step":
        case.update(net=rng.random() < 0.5, moved=rng.choice([0.0, 0.03, 0.3, 1.0]))
    return case


# ---- populations -----------------------------------------------------------
def fill(counts, total, lo, hi, g):
    """Moves the cells' counts (in place, within [lo, hi]) one by one until they add up to total."""
    while left := total - int(counts.sum()):
        step = 1 if left > 0 else -1
        may = ((counts < hi) if left > 0 else (counts > lo)).nonzero()[:, 0]
        may = may[torch.randperm(may.numel(), generator=g, device="cuda")]
        counts[may[:abs(left)]] += step


def population(case, seed, n_cells=None):
    """Velocities [3, n_particles] (float64, sorted by cell), offsets, tau on the GPU."""
    n, ppc, flow = n_cells or case["cells"], case["ppc"], case["flow"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    d = dict(device="cuda", dtype=torch.float64)
    uni = lambda lo, hi: lo + (hi - lo) * torch.rand(n, generator=g, **d)  # noqa: E731
    i = torch.arange(n, **d)
    mean = torch.zeros(3, n, **d)
    if flow == "couette":
        dens, theta = uni(0.8, 1.2), uni(0.8, 1.2)
        mean[0] = i / max(n - 1, 1) - 0.5
        counts = torch.full((n,), ppc, device="cuda")
    elif flow == "cavity":
        nx = max(1, math.isqrt(n))
        x, y = (i % nx + 0.5) / nx, (i // nx + 0.5) / math.ceil(n / nx)
        dens = 1 + 0.2 * torch.sin(math.pi * x) * torch.cos(math.pi * y)
        theta = 1 + 2 * torch.exp(-((x - 0.7) ** 2 + (y - 0.75) ** 2) / (2 * 0.18**2))
        mean[0] = y**6 - 0.15 * torch.sin(math.pi * y) * torch.sin(math.pi * x)
        mean[1] = 0.15 * torch.sin(2 * math.pi * x) * torch.sin(math.pi * y)
        counts = torch.poisson(torch.full((n,), float(ppc), **d), generator=g).clamp(8, 400).long()
        fill(counts, n * ppc, 8, 400, g)
    else:
        nx = max(2, math.isqrt(2 * n))
        ny = math.ceil(n / nx)
        R, u_inf = 28.0 * nx / 512, 10 * math.sqrt(5 / 3)
        dx, dy = i % nx + 0.5 - 0.75 * nx, i // nx + 0.5 - 0.5 * ny
        r, phi = torch.hypot(dx, dy), torch.atan2(dy.abs(), -dx)
        r_shock = R * (1 + 0.36 + 1.07 * phi**2)
        s = (torch.cos(phi.clamp(max=math.pi / 2)) ** 2).clamp(0.05, 1.0)
        h = ((r_shock - r) / (r_shock - R)).clamp(0, 1)
        body, post = r < R, (r >= R) & (r < r_shock) & (phi < 1.9)
        shock = (r >= r_shock) & (r < r_shock + max(1.0, 3.0 * nx / 512)) & (phi < 1.9)
        wake = (dx > 0) & (dy.abs() < R + 0.4 * dx) & (r >= R) & ~post & ~shock
        dens, theta = torch.ones(n, **d), torch.ones(n, **d)
        mean[0] = u_inf
        for at, density, temperature, ux in ((post, 1 + 4 * s * (0.6 + 0.4 * h), 1 + 39 * s * (0.7 + 0.3 * h),
                                              u_inf * (1 - 0.85 * s * (0.3 + 0.7 * h))),
                                             (shock, 1 + 2 * s, 1 + 20 * s, u_inf * (1 - 0.4 * s)),
                                             (wake, 0.25 + 0 * s, 3 + 0 * s, 0.2 * u_inf + 0 * s),
                                             (body, 0.05 + 0 * s, 2.5 + 0 * s, 0 * s)):
            dens, theta = torch.where(at, density, dens), torch.where(at, temperature, theta)
            mean[0] = torch.where(at, ux, mean[0])
        base = torch.exp(0.55 * torch.randn(n, generator=g, **d)) * dens**0.6
        counts = (base * (ppc * n / base.sum())).round().clamp(2, 2000).long()
        fill(counts, n * ppc - n // 3, 2, 2000, g)
    offsets = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(counts, 0, out=offsets[1:])
    cell = cells_of(offsets)
    c = torch.randn(3, cell.numel(), generator=g, **d)
    if flow == "cavity":
        skew = 0.1 * torch.randn(3, n, generator=g, **d)  # heat flux
        pull = 1 + 0.15 * (2 * torch.rand(3, n, generator=g, **d) - 1)  # stress
        e = torch.nn.functional.normalize(torch.randn(3, n, generator=g, **d), dim=0) * uni(0.5, 1.5)
        e = e * (uni(0, 1) < 0.1)  # bimodal cells: two Maxwellians at +/- e
        sign = (torch.rand(cell.numel(), generator=g, **d) < 0.5).double() * 2 - 1
        c = pull[:, cell] * (c + skew[:, cell] * (c * c - 1) + sign * e[:, cell])
    elif flow == "cylinder":
        beam = shock[cell] & (torch.rand(cell.numel(), generator=g, **d) < 0.5)
        c = torch.where(beam, (c + torch.tensor([[1.0], [0.0], [0.0]], **d) * (u_inf - mean[0, cell])) /
                        theta.sqrt()[cell], c)
    return mean[:, cell] + theta.sqrt()[cell] * c, offsets, 1 / dens


def rounded(case, v):
    return v if case["prec"] == "fp64" else v.float()


def cells_of(offsets):
    return torch.repeat_interleave(torch.arange(offsets.numel() - 1, device="cuda"), offsets.diff())


def sums(x, offsets):
    return torch.segment_reduce(x, "sum", lengths=offsets.diff(), unsafe=True, initial=0.0)


PAIRS = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]
TRIPLES = [(0, 0, 0), (0, 0, 1), (0, 0, 2), (0, 1, 1), (0, 1, 2), (0, 2, 2), (1, 1, 1), (1, 1, 2), (1, 2, 2),
           (2, 2, 2)]


def monomials(c):
    """The 25 functions of the moment vector (from its slot 5 on) and |c|^6."""
    r2 = c[0] * c[0] + c[1] * c[1] + c[2] * c[2]
    for i, j in PAIRS:
        yield c[i] * c[j]
    for i, j, k in TRIPLES:
        yield c[i] * c[j] * c[k]
    for i, j in PAIRS:
        yield r2 * c[i] * c[j]
    for i in range(3):
        yield r2 * r2 * c[i]
    yield r2 * r2 * r2


def moments64(v, offsets):
    """Moment vectors [n, 30] and <|c|^6> [n] of v in 64 bits."""
    v, n = v.double(), offsets.diff().double()
    k = n.clamp(min=1)
    U = torch.stack([sums(v[d], offsets) / k for d in range(3)])
    c = v - U[:, cells_of(offsets)]
    m = [sums(x, offsets) / k for x in monomials(c)]
    theta = (m[0] + m[3] + m[5]) / 3
    return torch.stack([n, *U, theta, *m[:25]], 1).contiguous(), m[25].contiguous()


def few(m):
    return m[:, 0] < MIN_PARTICLES


def sym(a, b):
    return PAIRS.index((min(a, b), max(a, b)))


def system64(m, tau):
    """The moment-matching system A Y = r of every cell (fpclosure.h)."""
    n = m.shape[0]
    u = lambda i, j: m[:, 5 + sym(i, j)]  # noqa: E731
    u3 = lambda i, j, k: m[:, 11 + TRIPLES.index(tuple(sorted((i, j, k))))]  # noqa: E731
    w = lambda i, j: m[:, 21 + sym(i, j)]  # noqa: E731
    th, zero = m[:, 4], torch.zeros_like(m[:, 4])
    b = [u3(i, 0, 0) + u3(i, 1, 1) + u3(i, 2, 2) for i in range(3)]
    s4, eps2 = w(0, 0) + w(1, 1) + w(2, 2), EPS2 / (tau * th)
    A, r = [[zero] * 9 for _ in range(9)], [zero] * 9

    def add(row, col, x):
        A[row][col] = A[row][col] + x

    for i, j in PAIRS:
        row = sym(i, j)
        for k in range(3):
            add(row, sym(i, k), u(k, j))
            add(row, sym(j, k), u(k, i))
        add(row, 6 + i, b[j])
        add(row, 6 + j, b[i])
        r[row] = -2 / tau * u(i, j) + 2 * eps2 * w(i, j)
    for i in range(3):
        row = 6 + i
        for l in range(3):
            add(row, sym(i, l), b[l])
            for k in range(3):
                add(row, sym(k, l), 2 * u3(i, k, l))
            add(row, 6 + l, 2 * (w(l, i) - 3 * th * u(l, i)))
        add(row, 6 + i, s4 - 9 * th * th)
        ub = u(i, 0) * b[0] + u(i, 1) * b[1] + u(i, 2) * b[2]
        r[row] = -4 / (3 * tau) * b[i] + eps2 * (3 * m[:, 27 + i] - 3 * th * b[i] - 2 * ub)
    return torch.stack([x for row in A for x in row], 1).view(n, 9, 9), torch.stack(r, 1)


def linear_drift(tau):
    y = torch.zeros(tau.numel(), 9, device="cuda", dtype=torch.float64)
    y[:, [0, 3, 5]] = (-1 / tau)[:, None]
    return y


def coeffs64(m, tau):
    A, r = system64(m, tau)
    skip = few(m)
    A = torch.where(skip[:, None, None], torch.eye(9, device="cuda", dtype=torch.float64), A)
    y = torch.linalg.solve(A, r.unsqueeze(2)).squeeze(2)
    return torch.where(skip[:, None], linear_drift(tau), y).contiguous()


def gradient64(v, offsets, tau, m, gY, gm_in=None):
    """Loss gradient with respect to the moments and the velocities."""
    leaf = m.clone().requires_grad_()
    A, r = system64(leaf, tau)
    skip = few(m)
    A = torch.where(skip[:, None, None], torch.eye(9, device="cuda", dtype=torch.float64), A)
    r = torch.where(skip[:, None], torch.zeros_like(r), r)
    gm, = torch.autograd.grad(torch.linalg.solve(A, r.unsqueeze(2)).squeeze(2), leaf, gY)
    if gm_in is not None:
        gm = gm + gm_in
    cell, n = cells_of(offsets), m[:, 0].clamp(min=1)
    c = (v.double() - m[:, 1:4].T[:, cell]).requires_grad_()
    loss = ((c * c).sum(0) / 3 * gm[cell, 4]).sum()
    for k, x in enumerate(monomials(c)):
        if k < 25:
            loss = loss + (x * gm[cell, 5 + k]).sum()
    h, = torch.autograd.grad(loss, c)
    gv = torch.stack([(h[d] - (sums(h[d], offsets) / n)[cell] + gm[cell, 1 + d]) / n[cell] for d in range(3)])
    return gm, gv


# ---- the velocity update in 64 bits ----------------------------------------
def noise64(n, seed, step):
    """The library's standard normals [3, n]: a Philox4x32-10 word stream through the
    inverse normal distribution function (fpclosure.h)."""
    M = 0xFFFFFFFF
    blk = torch.arange((3 * n + 3) // 4, device="cuda")
    x = [blk & M, blk >> 32, torch.full_like(blk, step & M), torch.full_like(blk, step >> 32)]
    k0, k1 = seed & M, seed >> 32
    for r in range(10):
        p0, p1 = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57
        x = [((p1 >> 32) & M) ^ x[1] ^ ((k0 + 0x9E3779B9 * r) & M), p1 & M,
             ((p0 >> 32) & M) ^ x[3] ^ ((k1 + 0xBB67AE85 * r) & M), p0 & M]
    words = torch.stack(x, 1).reshape(-1)[:3 * n]
    return torch.special.ndtri(((words >> 9).double() + 0.5) * 2.0**-23).view(n, 3).T


def update64(v, offsets, m, y, tau, seed, step):
    """(M^{n+1}, alpha); cells with too few particles take the linear model's step."""
    cell, th, k = cells_of(offsets), m[:, 4], m[:, 0].clamp(min=1)
    skip = few(m)
    C = y.clone()
    C[:, [0, 3, 5]] += (1 / tau)[:, None]
    C = torch.where(skip[:, None], torch.zeros_like(C), C)
    eps2 = torch.where(skip, torch.zeros_like(tau), EPS2 / (tau * th))
    c = v.double() - m[:, 1:4].T[:, cell]
    r2 = (c * c).sum(0)
    N = []
    for i in range(3):
        b = sum(m[:, 11 + TRIPLES.index(tuple(sorted((i, j, j))))] for j in range(3))
        N.append(sum(C[cell, sym(i, j)] * c[j] for j in range(3)) + C[cell, 6 + i] * (r2 - 3 * th[cell])
                 - eps2[cell] * (c[i] * r2 - b[cell]))
    nn = sums(N[0] * N[0] + N[1] * N[1] + N[2] * N[2], offsets) / k
    mn = sums(N[0] * c[0] + N[1] * c[1] + N[2] * c[2], offsets) / k
    a, om = torch.exp(-DT / tau), -torch.expm1(-DT / tau)
    alpha2 = 1 + tau / (3 * th) * (tau * om * om * nn + 2 * a * om * mn)
    alpha = torch.where(skip, torch.ones_like(tau), alpha2.sqrt())
    xi, noise = noise64(v.shape[1], seed, step), (th * om * (1 + a)).sqrt()
    new = [(c[i] * a[cell] + (om * tau)[cell] * N[i] + noise[cell] * xi[i]) / alpha[cell] + m[cell, 1 + i]
           for i in range(3)]
    return torch.stack(new), alpha


# ---- the learned closure in 64 bits ----------------------------------------
@functools.lru_cache(None)
def network(kind):
    return surrogate.Surrogate.load(os.path.join(WEIGHTS, f"surrogate_{kind}.fpw"))


def inputs64(m, tau, kind):
    th = m[:, 4:5]
    if kind == "full":
        return torch.cat([m[:, 5:11] / th, m[:, 11:21] / th**1.5, m[:, 21:27] / th**2, m[:, 27:30] / th**2.5], 1)
    u = m[:, 5:11]
    b = torch.stack([sum(m[:, 11 + TRIPLES.index(tuple(sorted((i, j, j))))] for j in range(3)) for i in range(3)], 1)
    full = torch.stack([u[:, sym(i, j)] for i in range(3) for j in range(3)], 1).view(-1, 3, 3)
    pi = u - th * torch.tensor([1.0, 0, 0, 1, 0, 1], device="cuda", dtype=torch.float64)
    return torch.cat([m[:, :1], th, m[:, 1:4], pi, b / 2, torch.linalg.det(full)[:, None], 1 / tau[:, None]], 1)


def standardised(s, f):
    x = torch.zeros(f.shape[0], surrogate.IN, device="cuda", dtype=torch.float64)
    x[:, :s.nfeat] = (f - s.x_mu[:s.nfeat].double()) / s.x_sigma[:s.nfeat].double()
    return x


def layers64(s):
    W, b = [], s.layer_views()[1]
    for l, view in enumerate(s.layer_views()[0]):
        k = surrogate.param_offset(0, l)
        W.append(s.shadow[k:k + view.numel()].view(view.shape).double())
    return W, [x.double() for x in b]


def forward64(W, b, x):
    for l in range(4):
        x = torch.nn.functional.silu(x @ W[l].T + b[l])
    return x @ W[4].T + b[4]


def learned64(s, m, tau, kind):
    f = torch.where(few(m)[:, None], torch.zeros(1, device="cuda", dtype=torch.float64), inputs64(m, tau, kind))
    t = torch.cat([forward64(*layers64(s), standardised(s, x)) for x in f.split(1 << 18)])[:, :9]
    t = t * s.y_sigma[:9].double() + s.y_mu[:9].double()
    y = t / tau[:, None]
    y[:, 6:] /= m[:, 4:5].sqrt()
    if kind == "full":  # cells outside the training box or off in energy are solved exactly
        pad = 0.5 * s.x_sigma[:25].double()
        out = ((f < s.x_min[:25].double() - pad) | (f > s.x_max[:25].double() + pad)).any(1)
        out |= energy64(t, f).abs() > 0.05
        y = torch.where(out[:, None], coeffs64(m, tau), y)
    return torch.where(few(m)[:, None], linear_drift(tau), y)


def aux64(f):
    """Normalised u (6), b (3) and s4 of the full inputs."""
    b = [sum(f[:, 6 + TRIPLES.index(tuple(sorted((i, j, j))))] for j in range(3)) for i in range(3)]
    return torch.stack([*f[:, :6].T, *b, f[:, 16] + f[:, 19] + f[:, 21]], 1)


def energy64(t, f):
    x = aux64(f)
    twice = torch.tensor([1.0, 2, 2, 1, 2, 1], device="cuda", dtype=torch.float64)
    return 1 + ((t[:, :6] * x[:, :6] * twice).sum(1) + (t[:, 6:9] * x[:, 6:9]).sum(1) - EPS2 * x[:, 9]) / 3


def train_inputs(case, seed):
    """BF16 inputs, targets and auxiliary rows of a batch, from the exact coefficients."""
    v, offsets, tau = population(case, seed)
    m, _ = moments64(v, offsets)
    y = coeffs64(m, tau)
    f = inputs64(m, tau, "full")
    t = y * tau[:, None]
    t[:, 6:] *= m[:, 4:5].sqrt()
    aux = torch.zeros(f.shape[0], 16, device="cuda")
    aux[:, :10] = aux64(f).float()
    return standardised(network("full"), f).bfloat16().contiguous(), t.float().contiguous(), aux


def train64(s, x, t, aux, scale, lr, weight, lam_drift, lam_energy):
    """(parameters, gradient, Adam's moments, loss sum) after the first step."""
    W, b = layers64(s)
    leaves = [a.requires_grad_() for pair in zip(W, b) for a in pair]
    o = forward64(W, b, x.double())[:, :9]
    mu, sd, t, aux = s.y_mu[:9].double(), s.y_sigma[:9].double(), t.double(), aux.double()
    p = mu + sd * o
    full = lambda q: torch.stack([q[:, sym(i, j)] for i in range(3) for j in range(3)], 1).view(-1, 3, 3)  # noqa: E731
    D, g, u, bh, s4 = full((p - t)[:, :6]), (p - t)[:, 6:], full(aux[:, :6]), aux[:, 6:9], aux[:, 9]
    drift = (D @ u @ D).diagonal(dim1=1, dim2=2).sum(1) + 2 * ((D @ bh[:, :, None])[:, :, 0] * g).sum(1) \
        + (g * g).sum(1) * (s4 - 9)
    twice = torch.tensor([1.0, 2, 2, 1, 2, 1], device="cuda", dtype=torch.float64)
    e = 1 + ((p[:, :6] * aux[:, :6] * twice).sum(1) + (p[:, 6:] * bh).sum(1) - EPS2 * s4) / 3
    rows = (weight * (o - (t - mu) / sd) ** 2).sum(1) + lam_drift * drift + lam_energy * e * e
    grads = torch.cat([a.reshape(-1) for a in torch.autograd.grad(rows.sum() * scale, leaves)])
    m, v = 0.1 * grads, 0.001 * grads * grads
    new = s.params.double() - lr * (m / 0.1) / ((v / 0.001).sqrt() + 1e-8)
    return [new, grads, m, v, rows.sum().detach().reshape(1)]


# ---- what a program has in hand, and the calls -------------------------------
class State:
    pass


def moved_cells(case, seed, offsets):
    """The cell of every particle before the sort: the last step's order with a share of the
    particles moved to a neighbouring cell, or (a share of 1) in any order."""
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    cell = cells_of(offsets)
    if case["moved"] >= 1:
        return cell[torch.randperm(cell.numel(), generator=g, device="cuda")].int()
    hop = torch.randint(-1, 2, (cell.numel(),), generator=g, device="cuda")
    hop = hop * (torch.rand(cell.numel(), generator=g, device="cuda") < case["moved"])
    return (cell + hop).clamp(0, case["cells"] - 1).int()


def prepare(case, seed):
    s, op = State(), case["op"]
    s.case, s.seed = case, seed
    s.params = api.default_params(min_particles=MIN_PARTICLES, eps2_hat=EPS2)
    if op == "train":
        s.x, s.t, s.aux = train_inputs(case, seed)
        s.trainer = surrogate.Trainer(surrogate.Surrogate.load(os.path.join(WEIGHTS, "surrogate_full.fpw")),
                                      batch=case["cells"])
        return s
    if op == "learned":  # the moments of a million cells, a quarter million at a time
        parts = []
        for c0 in range(0, case["cells"], 1 << 18):
            v, offsets, tau = population(case, seed + c0, min(1 << 18, case["cells"] - c0))
            parts.append((moments64(v, offsets)[0], tau))
        s.moments, s.tau = (torch.cat([p[k] for p in parts]).contiguous() for k in (0, 1))
        s.net = network("full")
        return s
    v, s.offsets, s.tau = population(case, seed)
    s.v = rounded(case, v)
    n, g = case["cells"], torch.Generator(device="cuda").manual_seed(seed + 2)
    f64 = dict(device="cuda", dtype=torch.float64)
    if op == "gradient":
        s.v.requires_grad_()
        s.gY = torch.randn(n, 9, generator=g, **f64)
        s.gM = 0.1 * torch.randn(n, 30, generator=g, **f64)
    elif op in ("adjoint", "update"):
        s.moments, s.m6 = moments64(s.v, s.offsets)
        if op == "adjoint":
            s.gY = torch.randn(n, 9, generator=g, **f64)
            s.lu = torch.empty(api.lu_doubles(n), **f64)
        else:
            s.coeffs = coeffs64(s.moments, s.tau)
            s.flags = few(s.moments).int() * api.FLAG_FEW
            s.v_out, s.alpha = torch.empty_like(s.v), torch.empty(n, **f64)
    elif op == "step":
        s.cell = moved_cells(case, seed, s.offsets)
        s.net = network("lite") if case["net"] else None
        need = api.lib().fp_collision_step_workspace_bytes(s.cell.numel(), n, api.V_F32, int(case["net"]))
        s.workspace = torch.empty(int(need), dtype=torch.uint8, device="cuda")
    elif op == "host":
        host = lambda t: torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)  # noqa: E731
        s.h_v, s.h_offsets, s.h_tau = host(s.v), host(s.offsets), host(s.tau)
        s.h_v_out = torch.empty(s.v.shape, dtype=s.v.dtype, pin_memory=True)
        s.h_coeffs = torch.empty((n, 9), dtype=torch.float64, pin_memory=True)
        s.h_flags = torch.empty(n, dtype=torch.int32, pin_memory=True)
        s.host_step = api.HostStep(n, s.v.shape[1], surrogate=network("full"), adjoint=True)
        del s.v
    return s


def run(s):
    case, op = s.case, s.case["op"]
    if op == "exact":
        return list(api.fp_closure_exact(s.v, s.offsets, s.tau, params=s.params, prec=case["prec"]))
    if op == "gradient":
        m, y, flags = autograd.closure(s.v, s.offsets, s.tau, prec=case["prec"], params=s.params)
        gv, = torch.autograd.grad([y, m], s.v, [s.gY, s.gM])
        return [m.detach(), y.detach(), flags, gv]
    if op == "adjoint":
        y, flags = api.fp_closure_solve(s.moments, s.tau, params=s.params, prec=case["prec"], lu_out=s.lu)
        gm, gv = api.fp_closure_backward(s.v, s.offsets, s.tau, s.moments, y, flags, s.gY, params=s.params, lu=s.lu)
        return [y, flags, gm, gv]
    if op == "update":
        v, alpha, flags = api.fp_velocity_update(s.v, s.offsets, s.moments, s.coeffs, s.tau, s.flags, DT,
                                                 params=s.params, seed=s.seed, step=7, alpha_out=s.alpha,
                                                 v_out=s.v_out, m6=s.m6)
        return [v, alpha, flags]
    if op == "learned":
        return list(s.net.closure(s.moments, s.tau, params=s.params, prec=case["prec"]))
    if op == "step":
        return list(api.fp_collision_step(s.cell, s.v, case["cells"], s.tau, DT, params=s.params, prec=case["prec"],
                                          net_lite=s.net.net() if s.net else None, seed=s.seed, step=7,
                                          workspace=s.workspace))
    if op == "train":
        t = s.trainer
        t.step(s.x, s.t, s.aux, 1.0 / case["cells"])
        return [t.s.params, t.grads, t.m, t.v, t.loss_acc]
    h = s.host_step
    h(s.h_v, s.h_offsets, s.h_tau, s.h_v_out, s.h_coeffs, s.h_flags, DT, params=s.params, prec=case["prec"],
      seed=s.seed, step=7)
    return [s.h_v_out, s.h_coeffs, s.h_flags, h.coeffs_s, h.flags_s, h.grad_moments, h.grad_v]


def exact(case, seed):
    s, op = prepare(case, seed), case["op"]
    if op == "train":
        t = s.trainer
        return train64(t.s, s.x, s.t, s.aux, 1.0 / case["cells"], t.lr,
                       torch.tensor(t.w, device="cuda").double(), t.lam_drift, t.lam_energy)
    if op == "learned":
        return [learned64(s.net, s.moments, s.tau, "full"), None]
    if op == "host":
        s.v, s.offsets, s.tau = s.h_v.cuda(), s.h_offsets.cuda(), s.h_tau.cuda()
    v, offsets, perm = s.v.detach(), s.offsets, None
    if op == "step":
        key, perm = torch.sort(s.cell.long(), stable=True)
        offsets = torch.searchsorted(key, torch.arange(case["cells"] + 1, device="cuda"))
        v = v[:, perm]
    m, _ = moments64(v, offsets)
    if op == "step" and case["net"]:
        y = learned64(s.net, m, s.tau, "lite")
    else:
        y = coeffs64(m, s.tau)
    if op == "exact":
        return [m, y, None]
    if op == "gradient":
        return [m, y, None, gradient64(v, offsets, s.tau, m, s.gY, s.gM)[1]]
    if op == "adjoint":
        return [y, None, *gradient64(v, offsets, s.tau, m, s.gY)]
    if op == "update":
        return [*update64(v, offsets, s.moments, s.coeffs, s.tau, seed, 7), None]
    new = update64(v, offsets, m, y, s.tau, seed, 7)[0]
    if op == "step":
        return [new, None, None, y, None]
    ones = torch.ones(case["cells"], 9, device="cuda", dtype=torch.float64)
    return [new, y, None, learned64(network("full"), m, s.tau, "full"), None,
            *gradient64(v, offsets, s.tau, m, ones)]


def work(case):
    """Bytes and operations of one pass: every input read once and every output written once;
    operations of the moments, of the 9 x 9 solve, of the update and of the network."""
    n = case["cells"]
    p, size = n * case["ppc"], 8 if case["prec"] == "fp64" else 4
    particles, vectors, coeffs, factors = 3 * size * p, 240 * n, 76 * n, 656 * n
    moments, solve, update, network_ = 61 * p, 658 * n, 110 * p, 110592 * n
    op = case["op"]
    if op == "exact":
        return {"bytes": particles + 16 * n + vectors + coeffs, "flops": moments + solve}
    if op == "gradient":
        return {"bytes": 2 * particles + 16 * n + 2 * vectors + 2 * coeffs, "flops": moments + 2 * solve + 120 * p}
    if op == "adjoint":
        return {"bytes": 2 * particles + 16 * n + 2 * vectors + 2 * coeffs, "flops": 2 * solve + 120 * p}
    if op == "update":
        return {"bytes": 2 * particles + 16 * n + vectors + 8 * n + coeffs + 12 * n, "flops": update}
    if op == "learned":
        return {"bytes": vectors + 8 * n + coeffs, "flops": network_}
    if op == "step":
        closure = network_ if case["net"] else solve
        return {"bytes": 2 * particles + 8 * p + 16 * n + coeffs, "flops": moments + closure + update}
    if op == "train":
        return {"bytes": n * (64 + 36 + 64) + 20 * 54000, "flops": 3 * network_}
    return {"bytes": 3 * particles + 16 * n + vectors + 2 * coeffs,
            "flops": moments + 3 * solve + network_ + update + 120 * p}
