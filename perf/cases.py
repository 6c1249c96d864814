"""What this library is timed on: the calls that a user's program makes, over the sizes it makes them with.

Every case is one system (or one batch of systems) in the box [0, 5]^D that the plans default to, evaluated by
one call of a public entry point of ``paper_2009_00767_gb300.binding``.  A program that uses the library keeps
its plan and its device buffers and calls again with new positions and charges, so ``prepare`` makes the inputs,
the plan and the output buffer, and ``run`` is the call alone, with the wait and the device-side checks that the
call does by default.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_2009_00767_gb300 import binding

BOX = 5.0
WEIGHTS = "paper_2009_00767_gb300/selector_gb300.bin"   # the trained selector that the package ships

# The Gaussian mixtures: 32 components, sigma log-uniform in the range of the clustered configuration.
GMM_K, GMM_LO, GMM_HI = 32, 0.01, 0.3


def listed():
    return [
        # The smallest call: the plain FP64 method on 4,096 charges, the size at which a result is checked by
        # hand against the direct sum.  Launches and latency count.
        dict(name="fp64_4k", kind="potential", precision="fp64", family="uniform", n=4096, levels=4, p=16),
        # The plain FP64 method at the size of the headline configuration, the judge of the mixed forms there.
        dict(name="fp64_1m", kind="potential", precision="fp64", family="uniform", n=1 << 20, levels=8, p=20),
        # The lower end of the selector's range, at the (levels, p) that it picks there: a time step of a small
        # particle simulation.
        dict(name="mixed_64k", kind="potential", precision="bf16x2", family="uniform", n=1 << 16, levels=6, p=12),
        # The headline configuration in the fastest form that meets 1e-6.
        dict(name="mixed_1m", kind="potential", precision="bf16x2", family="uniform", n=1 << 20, levels=8, p=20),
        # Potential and force field (what a particle simulation integrates) of an odd number of charges that
        # fill only a ring of the box, in the FP32-accurate tensor-core form.
        dict(name="field_200k", kind="field", precision="3xtf32", family="annulus", n=200003, levels=7, p=16),
        # The largest call: 2^24 clustered charges, finest squares from empty to thousands of charges.
        dict(name="clustered_16m", kind="potential", precision="bf16x2", family="gmm", n=1 << 24, levels=10, p=24),
        # The headline configuration called on pinned host arrays, copies included.
        dict(name="host_1m", kind="host", precision="bf16x2", family="uniform", n=1 << 20, levels=8, p=20),
        # The batched configuration: 1,024 systems of uneven size, half of them clustered, one graph replay.
        dict(name="batch_1024", kind="batch", precision="bf16x2", systems=1024, n_lo=1024, n_hi=262144, sizes=1, p=16),
        # The Lagrange-node form on the 3D Coulomb workload of the largest of the published tables.
        dict(name="lag3d_200k", kind="lagrange", form="node_f32", dim=3, n=200000, levels=3),
        # The Lagrange-node form in 2D at the headline number of charges.
        dict(name="lag2d_1m", kind="lagrange", form="node_f32", dim=2, n=1 << 20, levels=7),
        # The same method in FP64, on the workload of the smaller published table.
        dict(name="lag3d_80k_fp64", kind="lagrange", form="node_f64", dim=3, n=80000, levels=3),
        # The learned choice of (levels, p) for a system: occupancy statistics, then the network.
        dict(name="select_1m", kind="select", family="annulus", n=1 << 20),
    ]


def _depth(n):
    """The depth with about 16 charges in a finest square."""
    return max(2, round(math.log(n / 16.0, 4)))


def draw(rng):
    """One more case of the listed ones' ranges."""
    def size(lo, hi):
        return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))

    kind = rng.choice(["fp64", "mixed", "mixed", "mixed", "field", "host", "batch", "lagrange", "lagrange", "select"])
    if kind == "fp64":
        n = size(4096, 1 << 20)
        return dict(kind="potential", precision="fp64", family=rng.choice(["uniform", "annulus"]), n=n,
                    levels=_depth(n), p=rng.randint(8, 20))
    if kind == "mixed":
        n = size(1 << 14, 1 << 22)
        return dict(kind="potential", precision=rng.choice(["bf16x2", "bf16x2", "bf16x3", "3xtf32", "fp32"]),
                    family=rng.choice(["uniform", "annulus", "gmm"]), n=n, levels=_depth(n), p=rng.randint(8, 28))
    if kind == "field":
        n = size(1 << 14, 1 << 20)
        return dict(kind="field", precision=rng.choice(["bf16x2", "3xtf32", "fp32"]),
                    family=rng.choice(["uniform", "annulus"]), n=n, levels=_depth(n), p=rng.randint(8, 24))
    if kind == "host":
        n = size(1 << 16, 1 << 21)
        return dict(kind="host", precision="bf16x2", family="uniform", n=n, levels=_depth(n), p=rng.randint(8, 24))
    if kind == "batch":
        return dict(kind="batch", precision=rng.choice(["bf16x2", "fp32"]), systems=size(16, 512), n_lo=1024,
                    n_hi=size(4096, 262144), sizes=rng.randrange(1 << 20), p=16)
    if kind == "lagrange":
        form = rng.choice(["node_f32", "node_f32", "node_f64"])
        if rng.random() < 0.5:
            n = size(10000, 200000 if form == "node_f32" else 80000)
            levels = 2 if n < 25000 else 3
            return dict(kind="lagrange", form=form, dim=3, n=n, levels=levels)
        n = size(20000, 1 << 20 if form == "node_f32" else 200000)
        return dict(kind="lagrange", form=form, dim=2, n=n, levels=max(2, round(math.log(n / 64.0, 4))))
    return dict(kind="select", family=rng.choice(["uniform", "annulus", "gmm"]), n=size(1 << 16, 1 << 22))


# ------------------------------------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(n, g):
    return torch.rand(n, generator=g, dtype=torch.float64, device="cuda")


def _positions(family, n, g):
    """[n, 2] positions: uniform, a ring of radius 1..2 about the centre, or a Gaussian mixture redrawn into the box."""
    if family == "uniform":
        return BOX * torch.rand(n, 2, generator=g, dtype=torch.float64, device="cuda")
    if family == "annulus":
        r, t = 1.0 + _rand(n, g), 2.0 * math.pi * _rand(n, g)
        return torch.stack((2.5 + r * torch.cos(t), 2.5 + r * torch.sin(t)), 1).contiguous()
    centre = 0.5 + 4.0 * torch.rand(GMM_K, 2, generator=g, dtype=torch.float64, device="cuda")
    sigma = torch.exp(math.log(GMM_LO) + math.log(GMM_HI / GMM_LO) * _rand(GMM_K, g))
    comp = torch.randint(GMM_K, (n,), generator=g, device="cuda")
    xy = torch.empty(n, 2, dtype=torch.float64, device="cuda")
    todo = torch.arange(n, device="cuda")
    while todo.numel():
        c = comp[todo]
        z = torch.randn(todo.numel(), 2, generator=g, dtype=torch.float64, device="cuda")
        xy[todo] = centre[c] + sigma[c, None] * z
        p = xy[todo]
        todo = todo[((p < 0.0) | (p >= BOX)).any(1)]
    return xy


def _system(case, seed):
    """(positions, charges) of one system: q ~ U[-1, 1] in 2D, +-1 for the Lagrange-node form's experiments."""
    g = _gen(seed)
    n = case["n"]
    if case["kind"] == "lagrange":
        pos = BOX * torch.rand(n, case["dim"], generator=g, dtype=torch.float64, device="cuda")
        return pos, torch.where(_rand(n, g) < 0.5, -1.0, 1.0).to(torch.float64)
    return _positions(case["family"], n, g), 2.0 * _rand(n, g) - 1.0


def _batch_sizes(case):
    """Charges, depth and family of every system: a property of the plan, so of the case and not of the seed."""
    r = np.random.RandomState(case["sizes"])
    n = np.exp(r.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), case["systems"])).astype(np.int64)
    return n, np.array([_depth(int(v)) for v in n], dtype=np.int32), r.rand(case["systems"]) < 0.5


def _batch_system(case, seed):
    n, _, uniform = _batch_sizes(case)
    g = _gen(seed)
    xy = torch.cat([_positions("uniform" if u else "gmm", int(v), g) for v, u in zip(n, uniform)])
    return xy, 2.0 * _rand(int(n.sum()), g) - 1.0


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        xy, q = _batch_system(case, seed)
        n, levels, _ = _batch_sizes(case)
        plan = binding.Batch(n, levels, case["p"], BOX, case["precision"])
    elif kind == "select":
        xy, q = _system(case, seed)
        plan = binding.Selector()
        plan.load(WEIGHTS)
    elif kind == "lagrange":
        xy, q = _system(case, seed)
        plan = binding.LagPlan(case["dim"], case["n"], case["levels"], BOX, case["form"])
    else:
        xy, q = _system(case, seed)
        plan = binding.Plan(case["n"], case["levels"], case["p"], BOX, case["precision"])
    state = dict(kind=kind, plan=plan, xy=xy, q=q, phi=torch.empty_like(q))
    if kind == "host":
        for k in ("xy", "q", "phi"):
            state[k] = state[k].cpu().pin_memory()
    if kind == "field":
        state["field"] = torch.empty_like(xy)
    return state


def run(state):
    kind, plan = state["kind"], state["plan"]
    if kind == "field":
        return plan.potential_field(state["xy"], state["q"], state["phi"], state["field"])
    if kind == "host":
        return plan.potential_host(state["xy"], state["q"], state["phi"])
    if kind == "select":
        return {"features": plan.features(state["xy"]), "pick": plan.select(state["xy"])}
    return plan.potential(state["xy"], state["q"], state["phi"])


# ------------------------------------------------------------------------------------------------ work

def _pairs(n, levels, family, dim=2):
    """Unordered near-field pairs of n charges, in expectation: own and adjacent finest cells."""
    side = BOX / (1 << levels)
    near = min(BOX, 3.0 * side) ** dim
    if family == "annulus":
        density = 1.0 / (3.0 * math.pi) * 1.12   # the radius is uniform: the integral of density^2 is a little larger
    elif family == "gmm":
        own = (GMM_LO ** -2 - GMM_HI ** -2) / (2.0 * math.log(GMM_HI / GMM_LO)) / (4.0 * math.pi)
        density = (min(own, 1.0 / near) + (GMM_K - 1) / 16.0) / GMM_K
    else:
        density = BOX ** -dim
    return 0.5 * float(n) * n * density * near


def _far_flops(n, levels, coefficients, flops, dim=2):
    """Moments and local sums of every charge once, and each finest cell's interaction list once."""
    if levels < 2:
        return 0.0
    cells = min(float(n), float(1 << (dim * levels)))
    return 2.0 * flops * coefficients * n + flops * coefficients ** 2 * cells * (6 ** dim - 3 ** dim)


def work(case):
    kind = case["kind"]
    if kind == "select":
        return {"bytes": 16.0 * case["n"], "flops": 8.0 * case["n"]}
    if kind == "lagrange":
        n, dim = case["n"], case["dim"]
        return {"bytes": 8.0 * n * (dim + 2),
                "flops": (3.0 * dim + 5.0) * _pairs(n, case["levels"], "uniform", dim)
                + _far_flops(n, case["levels"], 4 ** dim, 2.0, dim)}
    pair = 16.0 if kind == "field" else 10.0
    if kind == "batch":
        n, levels, uniform = _batch_sizes(case)
        flops = sum(pair * _pairs(int(v), int(k), "uniform" if u else "gmm")
                    + _far_flops(int(v), int(k), case["p"] + 1, 8.0) for v, k, u in zip(n, levels, uniform))
        return {"bytes": 32.0 * float(n.sum()), "flops": flops}
    n = case["n"]
    return {"bytes": (48.0 if kind == "field" else 32.0) * n,
            "flops": pair * _pairs(n, case["levels"], case["family"]) + _far_flops(n, case["levels"], case["p"] + 1, 8.0)}


# ------------------------------------------------------------------------------------------------ values in 64 bits

MOST_PAIRS = 3e10   # ordered pairs that a reference sums directly


def _pair_sums(t, s, q, dim, field):
    """Kernel sums at targets t [..., T, D] from sources s [..., S, D] with charges q [..., S]; a pair at distance 0 adds 0."""
    d = t.unsqueeze(-2) - s.unsqueeze(-3)
    r2 = (d * d).sum(-1)
    apart = r2 > 0.0
    r2 = torch.where(apart, r2, 1.0)
    k = 0.5 * torch.log(r2) if dim == 2 else torch.rsqrt(r2)
    qa = torch.where(apart, q.unsqueeze(-2), 0.0)
    e = -(qa / r2).unsqueeze(-1).mul(d).sum(-2) if field else None
    return (qa * k).sum(-1), e


def _direct(xy, q, field):
    n, step = xy.shape[0], max(1, (1 << 25) // xy.shape[0])
    parts = [_pair_sums(xy[i:i + step], xy, q, xy.shape[1], field) for i in range(0, n, step)]
    return torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts]) if field else None


def _cells(pos, level):
    side = 1 << level
    cell = torch.floor(pos * side / BOX).long().clamp_(0, side - 1)
    return cell, sum(cell[:, a] * side ** a for a in range(pos.shape[1]))


def _near(pos, q, level, field):
    """Sums over the own and adjacent cells of `level`; None where the cells are too uneven for it."""
    n, dim = pos.shape
    side = 1 << level
    _, lin = _cells(pos, level)
    count = torch.bincount(lin, minlength=side ** dim)
    cap = int(count.max())
    full = torch.nonzero(count).flatten()
    if float(full.numel()) * cap * cap * 3 ** dim > MOST_PAIRS:
        return None
    order = torch.argsort(lin)
    start = torch.cumsum(count, 0) - count
    # slot [cell][place]: the charge there, or charge n, which is far away and zero
    place = torch.arange(n, device="cuda") - start[lin[order]]
    slots = torch.full((side ** dim + 1, cap), n, device="cuda")
    slots[lin[order], place] = order
    p1 = torch.cat((pos, torch.full((1, dim), -BOX, dtype=pos.dtype, device="cuda")))
    q1 = torch.cat((q, q.new_zeros(1)))
    phi, e = q.new_zeros(n + 1), p1.new_zeros(n + 1, dim) if field else None
    step = max(1, (1 << 24) // (cap * cap))
    for i in range(0, full.numel(), step):
        own = full[i:i + step]
        at = [(own // side ** a) % side for a in range(dim)]
        t = slots[own]
        for o in itertools.product((-1, 0, 1), repeat=dim):
            to = [a + b for a, b in zip(at, o)]
            inside = torch.stack([(c >= 0) & (c < side) for c in to]).all(0)
            nb = torch.where(inside, sum(c * side ** a for a, c in enumerate(to)), side ** dim)
            s = slots[nb]
            v, g = _pair_sums(p1[t], p1[s], q1[s], dim, field)
            phi.index_add_(0, t.flatten(), v.flatten())
            if field:
                e.index_add_(0, t.flatten(), g.reshape(-1, dim))
    return phi[:n], e[:n] if field else None


def _far(pos, q, levels, basis, operator, evaluate):
    """The far field level by level: `basis` [n, m] of the charges' offsets from their cell's centre in units of its
    side, `operator` [m, m] from a source cell at an offset to the target cell, `evaluate` the local sums at the charges."""
    dim, out = pos.shape[1], None
    for k in range(2, levels + 1):
        side, s = 1 << k, BOX / (1 << k)
        cell, lin = _cells(pos, k)
        w = basis((pos - (cell + 0.5) * s) / s)
        m = w.new_zeros(side ** dim, w.shape[1]).index_add_(0, lin, w * q[:, None]).view(*[side] * dim, -1)
        wide = m.new_zeros(*[side + 6] * dim, m.shape[-1])
        wide[tuple([slice(3, 3 + side)] * dim)] = m
        local = torch.zeros_like(m)
        for o in itertools.product(range(-3, 4), repeat=dim):
            if max(map(abs, o)) < 2:
                continue
            to, frm = [], []
            for v in reversed(o):   # x is the fastest axis; +3 reaches the parent's neighbours from even cells only, -3 from odd ones
                first, step = (1 if v == -3 else 0), (2 if abs(v) == 3 else 1)
                to.append(slice(first, None, step))
                frm.append(slice(3 + v + first, 3 + v + side, step))
            local[tuple(to)] += wide[tuple(frm)] @ operator(o, s)
        got = evaluate(w, local.view(side ** dim, -1)[lin], s)
        out = got if out is None else [a + b for a, b in zip(out, got)]
    return out if out is not None else [torch.zeros_like(q), torch.zeros_like(pos)]


def _log_system(xy, q, levels, field):
    """The 2D log potential (and field) to rounding: directly, or with expansions of an order at which nothing is cut."""
    n = xy.shape[0]
    if float(n) * n <= MOST_PAIRS:
        return _direct(xy, q, field)
    near = _near(xy, q, levels, field)
    if near is None:
        return None
    order = 40
    fact = torch.tensor([[(-1.0) ** (k + 1) / k * math.comb(l + k - 1, k - 1) if k else 0.0 for l in range(order + 1)]
                         for k in range(order + 1)], dtype=torch.float64, device="cuda")

    def basis(w):
        z = torch.complex(w[:, 0], w[:, 1])
        powers = [torch.ones_like(z)]
        for _ in range(order):
            powers.append(powers[-1] * z)
        return torch.stack(powers, 1)

    def operator(o, s):
        w0 = complex(o[0], o[1])
        inv = torch.tensor([w0 ** -i for i in range(2 * order + 1)], dtype=torch.complex128, device="cuda")
        i = torch.arange(order + 1, device="cuda")
        t = fact * inv[i[:, None] + i[None, :]]
        t[0, 1:] = -inv[1:order + 1] / i[1:]
        t[0, 0] = complex(np.log(-w0)) + math.log(s)
        return t

    def evaluate(w, b, s):
        phi = (w * b).sum(1).real
        if not field:
            return [phi, None]
        d = (w[:, :-1] * b[:, 1:] * torch.arange(1, order + 1, device="cuda")).sum(1) / s
        return [phi, torch.stack((-d.real, d.imag), 1)]

    phi, e = _far(xy, q, levels, basis, operator, evaluate) if field else (
        _far(xy, q, levels, basis, operator, lambda w, b, s: evaluate(w, b, s)[:1])[0], None)
    return near[0] + phi, near[1] + e if field else None


def _lagrange_system(pos, q, levels):
    """The sum that the Lagrange-node form stands for: charges at 4 nodes per axis for the cells of the interaction
    lists, the kernel itself for the adjacent cells."""
    dim = pos.shape[1]
    near = _near(pos, q, levels, False)
    if near is None:
        return None
    a = torch.tensor([-2.0, -1.0, 1.0, 2.0], dtype=torch.float64, device="cuda")
    node = torch.stack([a[torch.arange(4 ** dim, device="cuda") // 4 ** d % 4] for d in range(dim)], 1)   # x fastest

    def basis(w):
        out = None
        for d in range(dim):
            x = 5.0 * w[:, d:d + 1]
            f = torch.stack([torch.prod((x - a[a != v]) / (v - a[a != v]), 1) for v in a], 1)
            out = f if out is None else (f[:, :, None] * out[:, None, :]).flatten(1)
        return out

    def operator(o, s):
        shift = 5.0 * torch.tensor(o, dtype=torch.float64, device="cuda")
        r2 = ((node[:, None] + shift - node[None, :]) ** 2).sum(-1) * (s / 5.0) ** 2
        return 0.5 * torch.log(r2) if dim == 2 else torch.rsqrt(r2)

    return near[0] + _far(pos, q, levels, basis, operator, lambda w, b, s: [(w * b).sum(1)])[0]


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        n, levels, _ = _batch_sizes(case)
        if float((n.astype(np.float64) ** 2).sum()) > MOST_PAIRS:
            return None
        xy, q = _batch_system(case, seed)
        ends = np.concatenate(([0], np.cumsum(n)))
        return torch.cat([_direct(xy[a:b], q[a:b], False)[0] for a, b in zip(ends[:-1], ends[1:])])
    pos, q = _system(case, seed)
    if kind == "lagrange":
        return _lagrange_system(pos, q, case["levels"])
    if kind == "select":
        feats = []
        for k in range(3, 12):
            c = torch.bincount(_cells(pos, k)[1], minlength=1 << (2 * k))
            b = sum((c + 1 >= 1 << j).long() for j in range(1, 12))   # floor(log2(c + 1)), at most 11
            feats.append(torch.bincount(b, minlength=12).double() / (1 << (2 * k)))
        feats.append(torch.tensor([math.log2(case["n"]) / 22.0], dtype=torch.float64, device="cuda"))
        return {"features": torch.cat(feats), "pick": None}
    if case["family"] == "gmm" and case["n"] > 1 << 21:
        return None
    got = _log_system(pos, q, case["levels"], kind == "field")
    if got is None:
        return None
    return tuple(got) if kind == "field" else got[0] if kind != "host" else got[0].cpu()
