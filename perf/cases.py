"""The workloads that the framework's speed is judged by, through its public entry points.

A case names a particle distribution, the plan's options and the call:

  call "eval"   plan.eval(pos, q): potentials, energy and forces of one system
  call "grad"   fmm_energy(plan, pos, q) and its backward pass (autograd)
  call "batch"  FMMBatch.eval: many independent systems in one call

  dist "uniform"  uniform positions, charges +-1 (half and half)
  dist "cont"     uniform positions, charges uniform in [-1, 1], zero mean
  dist "water"    rigid triples O-H-H at 33 per unit volume, random orientation, wrapped
  dist "plummer"  clustered: a Plummer sphere of radius 0.1 in the unit box, +-1

Inputs are drawn on the device from the seed alone (the recipes of
paper_2212_13080_gb300/inputs.py).  A plan (or batch) is part of the prepared
state: a program keeps it over its time steps.  sync is the constructor's
option: True (the default) reads the device status in the call, False is what
a loop that queues its steps takes.

The energy of a single-precision plan is returned in single precision: the
library accumulates it in FP64, but its digits beyond FP32 are rounding noise
of the potentials.
"""
import math

import numpy as np
import torch

from paper_2212_13080_gb300 import FMM, FMMBatch, fmm_energy



def listed():
    def case(name, call="eval", dist="uniform", n=0, depth=3, p=4, periodic=False, continuous=False,
             precision="fp32", force_mode="adjoint", shift_free=False, sync=True):
        return dict(name=name, call=call, dist=dist, n=n, depth=depth, p=p, periodic=periodic,
                    continuous=continuous, precision=precision, force_mode=force_mode,
                    shift_free=shift_free, sync=sync)

    return [
        # the smallest call: the inner step of a small simulation that queues its steps, default precision
        case("uniform4k_fp32", n=4096, sync=False),
        # a reference calculation: the paper's 23,040 charges in 8^3 cells, in double precision
        case("uniform23k_fp64", n=23040, precision="fp64"),
        # the same system with the precomputed shift-free forms (repeated reference calculations)
        case("uniform23k_shift_free", n=23040, precision="fp64", shift_free=True),
        # a differentiable energy term: periodic water box of an ordinary simulation, forward and
        # backward through autograd, default precision, odd order, N not a multiple of a warp
        case("water67k_grad_fp32", call="grad", dist="water", n=66669, depth=4, p=5, periodic=True, continuous=True),
        # a large homogeneous system in the default precision, status read in the call
        case("uniform1m_fp32", dist="cont", n=1 << 20, depth=5, p=4, continuous=True),
        # the same on the tensor cores, steps queued
        case("uniform1m_tf32x3", dist="cont", n=1 << 20, depth=5, p=4, continuous=True, precision="tf32x3", sync=False),
        # the large periodic water box (699,050 triples), odd order
        case("water2m_tf32x3", dist="water", n=2097150, depth=6, p=5, periodic=True, continuous=True,
             precision="tf32x3", sync=False),
        # a clustered system at high order in the default precision: deep tree, most cells empty
        case("plummer1m_fp32", dist="plummer", n=1 << 20, depth=6, p=6),
        # clustered, split-BF16 far field, odd particle count
        case("plummer2m_bf16x3", dist="plummer", n=2097153, depth=6, p=6, precision="bf16x3", sync=False),
        # the largest call: 8M clustered charges, the flagship configuration
        case("plummer8m_tf32x3", dist="plummer", n=1 << 23, depth=7, p=6, precision="tf32x3", sync=False),
        # forces from the force kernels (four functionals per cell), odd particle count
        case("forcekernel300k_tf32x3", dist="cont", n=300001, depth=4, p=4, continuous=True, precision="tf32x3",
             force_mode="kernel"),
        # many small systems at once: 512 periodic boxes of 1,024 to 65,536 charges
        dict(name="batch512_tf32x3", call="batch", nsys=512, lo=1024, hi=65536, p=4, precision="tf32x3", sync=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choices(["eval", "grad", "batch"], [7, 2, 1])[0]
    if call == "batch":
        lo = _log_int(rng, 512, 4096)
        return dict(call=call, nsys=_log_int(rng, 8, 400), lo=lo, hi=lo * rng.randint(4, 16), p=rng.choice([3, 4, 4, 5]),
                    precision=rng.choice(["fp32", "tf32x3", "bf16x3"]), sync=False)
    dist = rng.choice(["uniform", "cont", "water", "plummer"])
    precision = rng.choice(["fp32", "fp32", "tf32x3", "tf32x3", "bf16x3", "tf32x1", "fp64"])
    p = rng.choice([3, 4, 4, 5, 6, 6])
    hi = {"fp64": 60000, "fp32": 1 << 20}.get(precision, 3 << 20)
    n = _log_int(rng, 2000, hi)
    if precision in ("fp64", "fp32") and n < 50000 and rng.random() < 0.15:
        p = 7  # the highest order of the paper's accuracy table; the tensor-core precisions end at 6
    if dist == "water":
        n -= n % 3
    depth = min(7, max(3, round(math.log(n / 32.0) / math.log(8.0)) + (1 if dist == "plummer" else 0)))
    continuous = dist in ("cont", "water")
    force_mode = "kernel" if call == "eval" and p <= 5 and rng.random() < 0.12 else "adjoint"
    shift_free = precision == "fp64" and dist == "uniform" and p <= 4 and depth == 3 and force_mode == "adjoint" \
        and rng.random() < 0.3
    return dict(call=call, dist=dist, n=n, depth=depth, p=p, periodic=dist == "water", continuous=continuous,
                precision=precision, force_mode=force_mode, shift_free=shift_free, sync=rng.random() < 0.5)


# ---- inputs ---------------------------------------------------------------

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _generator(seed):
    return torch.Generator(device=_device()).manual_seed(int(seed))


def _rand(g, *shape, dtype=torch.float32):
    return torch.rand(*shape, generator=g, device=_device(), dtype=dtype)


def _pm1(g, n):
    q = torch.ones(n, device=_device())
    q[n // 2:] = -1.0
    return q[torch.randperm(n, generator=g, device=_device())]


def _system(dist, n, seed):
    """pos (n, 3) float32, q (n,) float32, box (x0, y0, z0, L)."""
    g = _generator(seed)
    if dist == "uniform":
        return _rand(g, n, 3), _pm1(g, n), (0.0, 0.0, 0.0, 1.0)
    if dist == "cont":
        pos = _rand(g, n, 3)
        q = 2.0 * _rand(g, n, dtype=torch.float64) - 1.0
        return pos, (q - q.mean()).float(), (0.0, 0.0, 0.0, 1.0)
    if dist == "water":
        m = n // 3
        L = (m / 33.0) ** (1.0 / 3.0)
        O = _rand(g, m, 3, dtype=torch.float64) * L
        quat = torch.randn(m, 4, generator=g, device=_device(), dtype=torch.float64)
        w, x, y, z = (quat / quat.norm(dim=1, keepdim=True)).unbind(1)
        half = math.radians(104.52) / 2.0
        sx, cz = 0.1 * math.sin(half), 0.1 * math.cos(half)
        # the rotation's first and third columns: the H-O-H plane's axes
        ex = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y + z * w), 2 * (x * z - y * w)], 1)
        ez = torch.stack([2 * (x * z + y * w), 2 * (y * z - x * w), 1 - 2 * (x * x + y * y)], 1)
        pos = torch.stack([O, O + sx * ex + cz * ez, O - sx * ex + cz * ez], 1).reshape(-1, 3)
        pos = torch.remainder(pos, L).float()
        pos = torch.where(pos >= torch.tensor(L, dtype=torch.float32, device=pos.device), torch.zeros_like(pos), pos)
        q = torch.tensor([-0.834, 0.417, 0.417], device=_device()).repeat(m)
        return pos, q, (0.0, 0.0, 0.0, L)
    if dist == "plummer":
        parts, have = [], 0
        while have < n:
            m = int((n - have) * 1.3) + 64
            r = 0.1 / torch.sqrt(_rand(g, m, dtype=torch.float64).clamp_min(1e-12) ** (-2.0 / 3.0) - 1.0)
            d = torch.randn(m, 3, generator=g, device=_device(), dtype=torch.float64)
            x = (0.5 + r[:, None] * d / d.norm(dim=1, keepdim=True)).float()
            x = x[((x >= 0) & (x < 1)).all(1)]
            parts.append(x)
            have += x.shape[0]
        return torch.cat(parts)[:n].contiguous(), _pm1(g, n), (0.0, 0.0, 0.0, 1.0)
    raise KeyError(dist)


def _batch(case, seed):
    """Sizes log-uniform in [lo, hi], even (neutral periodic boxes), the same for every seed; depth by N."""
    rng = np.random.RandomState(5)
    counts = np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), case["nsys"])).astype(np.int64)
    counts -= counts % 2
    depths = np.clip(np.rint(np.log(counts / 32.0) / math.log(8.0)), 3, 5).astype(np.int64)
    offs = np.zeros(len(counts) + 1, np.int64)
    np.cumsum(counts, out=offs[1:])
    g = _generator(seed)
    pos = _rand(g, int(offs[-1]), 3)
    # half +1, half -1 in every system, in random order
    sysid = torch.repeat_interleave(torch.arange(len(counts), device=_device()), torch.as_tensor(counts, device=_device()))
    q = torch.where(torch.arange(int(offs[-1]), device=_device()) % 2 == 0, 1.0, -1.0)
    order = torch.argsort(sysid.double() + 0.999 * _rand(g, int(offs[-1]), dtype=torch.float64))
    return pos, q[order].contiguous(), offs, np.tile(np.array([0.0, 0.0, 0.0, 1.0]), (len(counts), 1)), depths, counts


# ---- the calls ------------------------------------------------------------

def prepare(case, seed):
    if case["call"] == "batch":
        pos, q, offs, boxes, depths, counts = _batch(case, seed)
        plan = FMMBatch(boxes, depths, case["p"], periodic=True, continuous=True, precision=case["precision"],
                        max_n=counts, sync=case["sync"])
        return dict(call="batch", plan=plan, pos=pos, q=q, offsets=offs)
    pos, q, box = _system(case["dist"], case["n"], seed)
    plan = FMM(box, case["depth"], case["p"], periodic=case["periodic"], continuous=case["continuous"],
               precision=case["precision"], force_mode=case["force_mode"], shift_free=case["shift_free"],
               max_n=case["n"], sync=case["sync"])
    if case["call"] == "grad":
        pos.requires_grad_(True)
        q.requires_grad_(True)
    return dict(call=case["call"], plan=plan, pos=pos, q=q, single=case["precision"] != "fp64")


def run(state):
    if state["call"] == "grad":
        e = fmm_energy(state["plan"], state["pos"], state["q"])
        if state["single"]:
            e = e.float()
        gpos, gq = torch.autograd.grad(e, (state["pos"], state["q"]))
        return dict(energy=e.detach(), grad_pos=gpos, grad_q=gq)
    if state["call"] == "batch":
        r = state["plan"].eval(state["pos"], state["q"], state["offsets"])
        return dict(r, energy=r["energy"].float())
    r = state["plan"].eval(state["pos"], state["q"])
    return dict(r, energy=r["energy"].float()) if state["single"] else r


# ---- what a pass cannot do without -----------------------------------------

def _cells(pos, box, depth, periodic, system=None):
    """The canonical single-precision map: cell (x, y, z) and the position in it."""
    S = 1 << depth
    u = (pos.detach() - torch.tensor(box[:3], dtype=torch.float32, device=pos.device)) / \
        torch.tensor(box[3], dtype=torch.float32, device=pos.device)
    if periodic:
        u = u - torch.floor(u)
        u = torch.where(u >= 1.0, torch.zeros_like(u), u)
    us = u * float(S)
    c = us.floor().clamp_max(S - 1)
    return c.long(), us - c


def _grid_counts(cell, S, system, nsys):
    cid = ((system * S + cell[:, 2]) * S + cell[:, 1]) * S + cell[:, 0]
    return torch.bincount(cid, minlength=nsys * S ** 3).reshape(nsys, S, S, S)


def _shifted(A, o, periodic):
    """A[s, z + oz, y + oy, x + ox, ...], zero outside the open box."""
    for axis, d in ((1, o[2]), (2, o[1]), (3, o[0])):
        if d == 0:
            continue
        S = A.shape[axis]
        if periodic:
            A = torch.roll(A, -d, axis)
        else:
            B = torch.zeros_like(A)
            m = max(0, S - abs(d))
            B.narrow(axis, max(0, -d), m).copy_(A.narrow(axis, max(0, d), m))
            A = B
    return A


def _offsets(parity):
    """The interaction list of a cell of this parity: 189 offsets."""
    rng = [range(-2 - b, 4 - b) for b in parity]
    return [(x, y, z) for z in rng[2] for y in rng[1] for x in rng[0] if max(abs(x), abs(y), abs(z)) > 1]


def _systems(case, seed):
    """[(pos, q, box, depth, system index, number of systems, particle index)] of one depth each."""
    if case["call"] != "batch":
        pos, q, box = _system(case["dist"], case["n"], seed)
        return [(pos, q, box, case["depth"], torch.zeros(len(q), dtype=torch.long, device=q.device), 1, None)], len(q), 1
    pos, q, offs, boxes, depths, counts = _batch(case, seed)
    sysid = torch.repeat_interleave(torch.arange(len(counts), device=q.device), torch.as_tensor(counts, device=q.device))
    out = []
    for d in sorted(set(depths.tolist())):
        ids = torch.as_tensor((depths == d).nonzero()[0], device=q.device)
        new = torch.full((len(counts),), -1, dtype=torch.long, device=q.device)
        new[ids] = torch.arange(len(ids), device=q.device)
        at = (new[sysid] >= 0).nonzero()[:, 0]
        out.append((pos[at], q[at], (0.0, 0.0, 0.0, 1.0), int(d), new[sysid[at]], len(ids), (at, ids)))
    return out, len(q), len(counts)


def work(case):
    """Positions and charges read once, results written once; near field: every
    unordered pair of charges in neighbouring cells once (26 flop: three
    differences, the distance, its inverse square root, potential and force of
    both); far field: the bilinear form of every interaction-list pair of cells
    that both hold charges (2 p^6 flop, times four with force kernels), and the
    weights of every charge (p^3 values in, four results out)."""
    p = case["p"]
    parts, n, nsys = _systems(case, 0)
    periodic = case["call"] == "batch" or case["periodic"]
    real = 8 if case["precision"] == "fp64" else 4
    ncomp = 4 if case.get("force_mode") == "kernel" else 1
    near = far = 0.0
    for pos, q, box, depth, system, ns, _ in parts:
        cell, _ = _cells(pos, box, depth, periodic)
        cnt = _grid_counts(cell, 1 << depth, system, ns).double()
        for x in (-1, 0, 1):
            for y in (-1, 0, 1):
                for z in (-1, 0, 1):
                    near += float((cnt * _shifted(cnt, (x, y, z), periodic)).sum())
        near -= float(len(q))
        occ = (cnt > 0).float()
        for l in range(depth, 0 if periodic else 1, -1):
            S = 1 << l
            for b in range(8):
                bx, by, bz = b & 1, (b >> 1) & 1, b >> 2
                t = torch.zeros_like(occ)
                t[:, bz::2, by::2, bx::2] = occ[:, bz::2, by::2, bx::2]
                # sum over the list of the shifted occupancy, as differences of box sums
                far += _list_pairs(t, occ, (bx, by, bz), periodic)
            occ = occ.reshape(ns, S // 2, 2, S // 2, 2, S // 2, 2).amax((2, 4, 6))
    return {"bytes": n * (16.0 + 4 * real) + nsys * 8.0,
            "flops": 13.0 * near + ncomp * far * 2.0 * p ** 6 + n * p ** 3 * 2.0 * (1 + 4)}


def _list_pairs(t, occ, parity, periodic):
    """Occupied (target, source) pairs of the interaction list: the 6^3 box less the 3^3 box around the target."""
    def box_sum(lo, hi):
        A = occ
        for axis in range(3):
            B = torch.zeros_like(A)
            for d in range(lo[axis], hi[axis] + 1):
                o = [0, 0, 0]
                o[axis] = d
                B += _shifted(A, o, periodic)
            A = B
        return A

    wide = box_sum([-2 - b for b in parity], [3 - b for b in parity])
    return float((t * (wide - box_sum([-1] * 3, [1] * 3))).double().sum())


# ---- the same results in 64 bits --------------------------------------------
#
# The method's own definitions (replacement by charges on the p-division points
# of every cell, bilinear forms over the interaction lists, direct sums over 27
# cells, split of particles near cell planes) in plain float64 torch: the
# energy as a function of positions and charges, its derivatives by autograd
# through the weights, the linear maps and the near sums written out.

F8 = torch.float64


def _lagrange(p, x):
    """Lagrange weights on the p-division points of [0, 1]: (..., p)."""
    tau = [i / (p - 1) for i in range(p)]
    cols = []
    for i in range(p):
        v = torch.ones_like(x)
        for k in range(p):
            if k != i:
                v = v * ((x - tau[k]) / (tau[i] - tau[k]))
        cols.append(v)
    return torch.stack(cols, -1)


def _split_axis(t, c, S, p, d, periodic, continuous):
    """One axis: per particle up to m entries (valid, cell, local coordinate, weight)."""
    lower = (t.detach() < d) & (torch.tensor(periodic, device=t.device) | (c > 0)) & continuous
    upper = (t.detach() > torch.tensor(1.0, dtype=torch.float32) - torch.tensor(d, dtype=torch.float32)) & \
        (torch.tensor(periodic, device=t.device) | (c < S - 1)) & continuous
    split = lower | upper
    below = torch.where(lower, c - 1, c) % S
    above = torch.where(lower, c, c + 1) % S
    sigma = torch.where(lower, t, t - 1.0) / d
    g = _lagrange(p, 0.5 * (sigma + 1.0))
    one, zero = torch.ones_like(t), torch.zeros_like(t)
    # the first entry is also the whole particle where it is not split
    out = []
    for k in range(p):
        s = -1.0 + 2.0 * k / (p - 1)
        for half in ((0, 1) if 2 * k == p - 1 else (0,)):
            w = g[..., k] * (0.5 if 2 * k == p - 1 else 1.0)
            low = 2 * k < p - 1 or (2 * k == p - 1 and half == 0)
            cell, tk = (below, 1.0 + s * d) if low else (above, s * d)
            if out:
                out.append((split, cell, one.detach() * tk, w))
            else:
                out.append((torch.ones_like(split), torch.where(split, cell, c),
                            torch.where(split, one.detach() * tk, t), torch.where(split, w, one)))
    return out


def _charges(t, cell, S, p, d, periodic, continuous):
    """The charges of all particles: (origin, cell (m, 3), local position (m, 3), weight (m,))."""
    axes = [_split_axis(t[:, a], cell[:, a], S, p, d, periodic, continuous) for a in range(3)]
    if not continuous:
        axes = [a[:1] for a in axes]
    parts = []
    for ez in axes[2]:
        for ey in axes[1]:
            for ex in axes[0]:
                at = (ex[0] & ey[0] & ez[0]).nonzero()[:, 0]
                if len(at):
                    parts.append((at, torch.stack([e[1][at] for e in (ex, ey, ez)], 1),
                                  torch.stack([e[2][at] for e in (ex, ey, ez)], 1), ex[3][at] * ey[3][at] * ez[3][at]))
    return [torch.cat([x[k] for x in parts]) for k in range(4)]


def _near(x, q, origin, cid, cell, system, S, periodic, h):
    """phi and the gradient of phi at every charge (sorted by cell), sums over the 27 cells around it."""
    n = len(q)
    start = torch.searchsorted(cid, torch.arange(int(system.max()) * S ** 3 + S ** 3 + 1, device=q.device))
    phi, gra = torch.zeros(n, dtype=F8, device=q.device), torch.zeros(n, 3, dtype=F8, device=q.device)
    every = torch.arange(n, device=q.device)
    for o in [(a, b, c) for c in (0, 1) for b in (-1, 0, 1) for a in (-1, 0, 1) if (c, b, a) >= (0, 0, 0)]:
        ov = torch.tensor(o, device=q.device)
        nb = cell + ov
        ok = torch.ones(n, dtype=torch.bool, device=q.device) if periodic else ((nb >= 0) & (nb < S)).all(1)
        nb = nb % S
        ncid = ((system * S + nb[:, 2]) * S + nb[:, 1]) * S + nb[:, 0]
        first = start[ncid]
        m = torch.where(ok, start[ncid + 1] - first, torch.zeros_like(first))
        total = torch.cumsum(m, 0)
        a = 0
        while a < n:
            base = int(total[a - 1]) if a else 0
            b = min(n, max(a + 1, int(torch.searchsorted(total, base + (1 << 25)))))
            i = torch.repeat_interleave(every[a:b], m[a:b])
            j = first[i] + torch.arange(len(i), device=q.device) - (total[i] - m[i] - base)
            if o == (0, 0, 0):
                keep = j > i
                i, j = i[keep], j[keep]
            r = (x[i] - x[j] - ov) * h
            r2 = (r * r).sum(1)
            inv = torch.where((r2 > 0) & (origin[i] != origin[j]), r2, torch.full_like(r2, math.inf)).rsqrt()
            f = r * (inv * inv * inv)[:, None]
            phi.index_add_(0, i, q[j] * inv)
            phi.index_add_(0, j, q[i] * inv)
            gra.index_add_(0, i, -q[j][:, None] * f)
            gra.index_add_(0, j, q[i][:, None] * f)
            a = b
    return phi, gra


def _nodes(p):
    i = torch.arange(p, dtype=F8, device=_device()) / (p - 1)
    z, y, x = torch.meshgrid(i, i, i, indexing="ij")
    return torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1)


def _unit_kernels(p, o, ncomp):
    """K_o[a, b] = 1/|a - (o + b)| of unit cells, and with force kernels r/|r|^3."""
    N = _nodes(p)
    r = N[:, None, :] - N[None, :, :] - torch.tensor(o, dtype=F8, device=N.device)
    inv = (r * r).sum(2).rsqrt()
    return [inv] + [r[..., a] * inv ** 3 for a in range(ncomp - 1)]


def _lattice_kernels(p, ncomp):
    """Ewald potential of the unit box less its 27 nearest images (tin foil), and minus its gradient."""
    alpha, N = 2.0, _nodes(p)
    r = (N[:, None, :] - N[None, :, :]).reshape(-1, 3).requires_grad_(ncomp > 1)
    psi = torch.full((len(r),), -math.pi / alpha ** 2, dtype=F8, device=N.device)
    for mz in range(-6, 7):
        for my in range(-6, 7):
            for mx in range(-6, 7):
                s2 = ((r + torch.tensor([mx, my, mz], dtype=F8, device=N.device)) ** 2).sum(1)
                if max(abs(mx), abs(my), abs(mz)) > 1:
                    s = s2.sqrt()
                    psi = psi + torch.erfc(alpha * s) / s
                else:
                    s = torch.where(s2 > 0, s2, torch.ones_like(s2)).sqrt()
                    psi = psi - torch.where(s2 > 0, torch.erf(alpha * s) / s, torch.full_like(s, 2 * alpha / math.sqrt(math.pi)))
    for hz in range(0, 8):
        for hy in range(-7, 8):
            for hx in range(-7, 8):
                if (hz, hy, hx) > (0, 0, 0):
                    h2 = float(hx * hx + hy * hy + hz * hz)
                    w = math.exp(-math.pi ** 2 * h2 / alpha ** 2) / (math.pi * h2)
                    if w > 1e-25:
                        psi = psi + 2 * w * torch.cos(2 * math.pi * (r @ torch.tensor([hx, hy, hz], dtype=F8, device=N.device)))
    out = [psi.detach()]
    if ncomp > 1:
        g, = torch.autograd.grad(psi.sum(), r)
        out += [-g[:, a] for a in range(3)]
    return [k.reshape(p ** 3, p ** 3) for k in out]


def _functionals(phi, l, p, periodic, ncomp):
    """L of every cell of one level from the grid charges phi (B, S, S, S, p^3), unit-box units."""
    S, B = 1 << l, phi.shape[0]
    with torch.no_grad():
        idx = torch.arange(-3, S + 3, device=phi.device)
        pad = phi
        for axis in (1, 2, 3):
            pad = pad.index_select(axis, idx % S)
            if not periodic:
                shape = [1] * 5
                shape[axis] = S + 6
                pad = pad * ((idx >= 0) & (idx < S)).to(F8).reshape(shape)
        L = [torch.zeros_like(phi) for _ in range(ncomp)]
        kernels = {}
        for b in range(8):
            bx, by, bz = b & 1, (b >> 1) & 1, b >> 2
            for o in _offsets((bx, by, bz)):
                if o not in kernels:
                    kernels[o] = _unit_kernels(p, o, ncomp)
                src = pad[:, 3 + bz + o[2]:3 + o[2] + S:2, 3 + by + o[1]:3 + o[1] + S:2, 3 + bx + o[0]:3 + o[0] + S:2]
                src = src.reshape(-1, p ** 3)
                for k in range(ncomp):
                    v = (src @ kernels[o][k].T).reshape(B, S // 2, S // 2, S // 2, -1)
                    L[k][:, bz::2, by::2, bx::2] += v * float(S) ** (1 if k == 0 else 2)
    return L


def _exact_systems(pos, q, box, depth, system, ns, p, periodic, continuous, ncomp):
    """phi, F, E per system of ns systems of one depth, in unit-box units scaled to the box."""
    S = 1 << depth
    cell, t32 = _cells(pos, box, depth, periodic)
    d = 1.0 / 256.0
    t = t32.double().requires_grad_(True)
    qv = q.detach().double().requires_grad_(True)
    origin, ccell, ct, W = _charges(t, cell, S, p, d, periodic, continuous)
    cid = ((system[origin] * S + ccell[:, 2]) * S + ccell[:, 1]) * S + ccell[:, 0]
    cid, order = torch.sort(cid, stable=True)
    origin, ccell, ct, W = origin[order], ccell[order], ct[order], W[order]
    qe = qv[origin] * W
    with torch.no_grad():
        phi_n, gra_n = _near(ct.detach(), qe.detach(), origin, cid, ccell, system[origin], S, periodic, 1.0 / S)
    # the energy's derivatives: every sum below is bilinear and symmetric, so
    # one factor is held and the other differentiated
    probe = torch.ones_like(qe).requires_grad_(True) if ncomp > 1 else None

    def grid(charge):
        g = [_lagrange(p, ct[:, a]) for a in range(3)]
        w = (g[2][:, :, None, None] * g[1][:, None, :, None] * g[0][:, None, None, :]).reshape(len(charge), -1)
        v = torch.zeros(ns * S ** 3, p ** 3, dtype=F8, device=q.device).index_add(0, cid, charge[:, None] * w)
        return v.reshape(ns, S, S, S, -1)

    def up(v, l):
        H = 1 << (l - 1)
        tau = torch.arange(p, dtype=F8, device=q.device) / (p - 1)
        G = [_lagrange(p, 0.5 * (h + tau)) for h in (0, 1)]  # (child node, parent node)
        v = v.reshape(ns, H, 2, H, 2, H, 2, p, p, p)
        v = sum(torch.einsum("nzcydxkji,iI->nzcydxkjI", v[:, :, :, :, :, :, h], G[h]) for h in (0, 1))
        v = sum(torch.einsum("nzcyxkjI,jJ->nzcyxkJI", v[:, :, :, :, h], G[h]) for h in (0, 1))
        v = sum(torch.einsum("nzyxkJI,kK->nzyxKJI", v[:, :, h], G[h]) for h in (0, 1))
        return v.reshape(ns, H, H, H, p ** 3)

    v = grid(qe)
    vp = grid(probe) if ncomp > 1 else None
    e_far = torch.zeros(ns, dtype=F8, device=q.device)
    dual = 0.0
    force = [0.0, 0.0, 0.0]
    for l in range(depth, -1, -1):
        if l >= (1 if periodic else 2):
            L = _functionals(v.detach(), l, p, periodic, ncomp)
        elif l == 0 and periodic:
            K = _lattice_kernels(p, ncomp)
            L = [v.detach() @ k.T for k in K]
        else:
            L = None
        if L is not None:
            e_far = e_far + 0.5 * (v.detach() * L[0]).reshape(ns, -1).sum(1)
            dual = dual + (v * L[0]).sum()
            for a in range(ncomp - 1):
                force[a] = force[a] + (vp * L[1 + a]).sum()
        del L
        if l == (0 if periodic else 2):
            break
        v = up(v, l)
        vp = up(vp, l) if ncomp > 1 else None
    e_near = torch.zeros(ns, dtype=F8, device=q.device).index_add(0, system[origin], 0.5 * qe.detach() * phi_n)
    surrogate = dual + (qe * phi_n).sum() + (ct * (qe.detach()[:, None] * gra_n / S)).sum()
    gq, gt = torch.autograd.grad(surrogate, (qv, t), retain_graph=ncomp > 1)
    F = -gt * S
    if ncomp > 1:  # a particle's force is the sum of the forces on its charges
        with torch.no_grad():
            f = -qe.detach()[:, None] * gra_n
        for a in range(3):
            fa, = torch.autograd.grad(force[a], probe, retain_graph=True)
            f[:, a] += qe.detach() * fa
        F = torch.zeros_like(gt).index_add(0, origin, f)
    return gq / box[3], F / box[3] ** 2, (e_far + e_near) / box[3]


def exact(case, seed):
    parts, n, nsys = _systems(case, seed)
    periodic = case["call"] == "batch" or case["periodic"]
    continuous = case["call"] == "batch" or case["continuous"]
    p, ncomp = case["p"], 4 if case.get("force_mode") == "kernel" else 1
    # dense far field in double precision at about 1 TFLOP/s: some ten seconds at most
    if sum(ns * 8.0 ** d * 1.15 * 189 * 2 * p ** 6 * ncomp for _, _, _, d, _, ns, _ in parts) > 8e12:
        return None
    dev = parts[0][1].device
    phi, F = torch.empty(n, dtype=F8, device=dev), torch.empty(n, 3, dtype=F8, device=dev)
    E = torch.empty(nsys, dtype=F8, device=dev)
    for pos, q, box, depth, system, ns, at in parts:
        f, g, e = _exact_systems(pos, q, box, depth, system, ns, p, periodic, continuous, ncomp)
        if at is None:
            phi, F, E = f, g, e
        else:
            phi[at[0]], F[at[0]], E[at[1]] = f, g, e
    if case["call"] == "grad":
        return dict(energy=E[0], grad_pos=-F, grad_q=phi)
    return dict(potential=phi, energy=E, forces=F)
