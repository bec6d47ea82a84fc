"""The work that users of this package have it do, as cases that can be timed.

A case is a dict of plain values.  ``listed()`` gives the fixed ones, ``draw``
more of the same ranges, ``prepare`` what a program holds before the call (the
density on the GPU and its plan), ``run`` one pass through the public entry
points, ``work`` the bytes and operations no implementation can do without and
``exact`` the same truncated operator evaluated in 64 bits by plain torch.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2606_13793_gb300 as fmm


def listed():
    return [
        # the smallest call: the 32^3 FP64 configuration (p = 4), as a unit
        # test, a parameter scan or an inner loop of a small box makes it;
        # latency and launches are all of it
        dict(name="fp64_32_p4", kind="solve", precision="fp64", nx=32, ny=32, nz=32, order=4, leaf=4, accel=True,
             field="blobs"),
        # a small FP32 box with the force: one field of an ensemble solved alone
        dict(name="fp32_64", kind="solve", precision="fp32", nx=64, ny=64, nz=64, order=6, leaf=4, accel=True,
             field="plummer"),
        # the solve of a caller that may not allocate (no plan), on an uneven
        # small grid
        dict(name="static_48x64x40", kind="static", precision="fp32", nx=48, ny=64, nz=40, order=6, leaf=4, accel=True,
             field="plummer"),
        # FP64 at an ordinary size: reference solutions and convergence studies
        dict(name="fp64_96", kind="solve", precision="fp64", nx=96, ny=96, nz=96, order=6, leaf=4, accel=True,
             field="plummer"),
        # the paper's own configuration: order 3, multipoles to 2, final-stage
        # M2P, leaf boxes of 2^3 cells
        dict(name="paper_fp32_128", kind="solve", precision="fp32", nx=128, ny=128, nz=128, order=3, leaf=2,
             accel=True, field="plummer", final_stage="m2p", mult_order=2),
        # tensor-core precision at a middle size with the analytic force
        dict(name="bf16x3_128_analytic", kind="solve", precision="bf16x3", nx=128, ny=128, nz=128, order=6, leaf=4,
             accel="analytic", field="plummer"),
        # a slab-like ragged grid at the highest order, potential only: extents
        # that fill no tile
        dict(name="bf16x3_ragged_p8", kind="solve", precision="bf16x3", nx=360, ny=200, nz=264, order=8, leaf=4,
             accel=False, field="lognormal"),
        # the plain FP32 production solve at 256^3
        dict(name="fp32_256", kind="solve", precision="fp32", nx=256, ny=256, nz=256, order=6, leaf=4, accel=True,
             field="lognormal"),
        # the differentiable solve at 256^3: loss 0.5 |phi - target|^2, forward
        # and backward through torch.autograd
        dict(name="fp32_256_grad", kind="grad", precision="fp32", nx=256, ny=256, nz=256, order=6, leaf=4, accel=True,
             field="lognormal"),
        # many fields of uneven sizes in one graph launch (sizes of the batch
        # workload: 64, 96, 128, 192)
        dict(name="batch_fp32_16", kind="batch", precision="fp32", fields=16, order=6, leaf=4, accel=True, sizes=2606),
        # densities that live on the host: pinned buffers in and out
        dict(name="host_bf16x3_192x3", kind="host", precision="bf16x3", nx=192, ny=192, nz=192, order=6, leaf=4,
             accel=True, fields=3, field="lognormal"),
        # the largest: the 512^3 bf16x3 headline solve with the force
        dict(name="bf16x3_512", kind="solve", precision="bf16x3", nx=512, ny=512, nz=512, order=6, leaf=4, accel=True,
             field="lognormal"),
    ]


# most cells of a drawn case, by kind of arithmetic (cost per cell differs)
_MOST = {"fp64": 96 ** 3, "fp32": 256 ** 3, "bf16x3": 512 ** 3}


def draw(rng):
    """One more case: log-uniform sizes (uneven axes, any multiple of the leaf
    side), every precision, order and leaf size the listed cases stand for."""
    kind = rng.choice(["solve"] * 6 + ["grad", "batch", "host", "static"])
    c = dict(kind=kind)
    if kind == "batch":
        c.update(precision=rng.choice(["fp32", "fp32", "bf16x3"]), fields=rng.randint(3, 20), order=rng.choice([4, 6]),
                 leaf=4, accel=rng.random() < 0.7, sizes=rng.randint(1, 10 ** 6))
        return c
    prec = "fp32" if kind == "static" else rng.choice(["fp64", "fp32", "fp32", "bf16x3", "bf16x3", "bf16x3"])
    order, leaf = rng.choice([3, 4, 5, 6, 6, 6, 7, 8]), rng.choice([4, 4, 4, 4, 2, 8])
    lo, hi = 32.0, _MOST[prec] ** (1 / 3)
    if kind == "static":
        order, leaf, hi = min(order, 6), 4, 64.0
    if kind == "host":
        hi = min(hi, 224.0)
    if kind == "grad":
        hi = min(hi, 256.0)
    if leaf == 8 or order > 6:  # costlier per cell
        hi *= 0.75
    if prec == "fp64" and (leaf == 8 or order > 6):
        hi *= 0.8
    n = math.exp(rng.uniform(math.log(lo), math.log(max(hi, lo * 1.01))))
    dims = [max(leaf * 4, int(n * rng.uniform(0.7, 1.0) / leaf) * leaf) for _ in range(3)]
    c.update(precision=prec, nx=dims[0], ny=dims[1], nz=dims[2], order=order, leaf=leaf,
             accel=True if kind == "grad" else rng.random() < 0.6, field=rng.choice(["plummer", "lognormal", "blobs"]))
    if kind == "host":
        c["fields"] = rng.randint(2, 4)
    if kind == "solve" and leaf == 4 and rng.random() < 0.15:
        c["accel"] = "analytic"
    return c


# ---------------------------------------------------------------- inputs ----


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _density(field, dims, seed, dtype):
    """[nz][ny][nx] density on the GPU, from the seed alone."""
    nx, ny, nz = dims
    dev = "cuda"
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) % (2 ** 62))
    r = np.random.default_rng(int(seed) % (2 ** 62))
    if field == "lognormal":  # exp of a Gaussian field, P(k) ~ k^-2.5, outer 10% zeroed
        white = torch.randn(nz, ny, nx, device=dev, generator=g, dtype=torch.float32)
        wk = torch.fft.rfftn(white)
        del white
        kz = torch.fft.fftfreq(nz, device=dev)[:, None, None]
        ky = torch.fft.fftfreq(ny, device=dev)[None, :, None]
        kx = torch.fft.rfftfreq(nx, device=dev)[None, None, :]
        k2 = kz * kz + ky * ky + kx * kx
        k2[0, 0, 0] = 1.0
        amp = k2.pow_(-0.625)
        amp[0, 0, 0] = 0.0
        d = torch.fft.irfftn(wk.mul_(amp), s=(nz, ny, nx))
        del wk, amp, k2
        d -= d.mean()
        d /= d.std()
        rho = torch.exp_(d - 0.5)
        for ax, n in ((2, nx), (1, ny), (0, nz)):
            pad = int(0.1 * n)
            if pad:
                rho.narrow(ax, 0, pad).zero_()
                rho.narrow(ax, n - pad, pad).zero_()
        return rho.to(dtype).contiguous()
    z = torch.arange(nz, device=dev, dtype=torch.float64)[:, None, None] + 0.5
    y = torch.arange(ny, device=dev, dtype=torch.float64)[None, :, None] + 0.5
    x = torch.arange(nx, device=dev, dtype=torch.float64)[None, None, :] + 0.5
    if field == "plummer":  # centred Plummer sphere plus 1% noise
        a = r.uniform(4.0, 20.0)
        rho0 = 3.0 / (4.0 * math.pi * a ** 3)
        r2 = (x - nx / 2) ** 2 + (y - ny / 2) ** 2 + (z - nz / 2) ** 2
        rho = rho0 * (1.0 + r2 / (a * a)) ** -2.5
        rho += 0.01 * rho0 * torch.rand(nz, ny, nx, device=dev, generator=g, dtype=torch.float64)
        return rho.to(dtype).contiguous()
    rho = torch.zeros(nz, ny, nx, device=dev, dtype=torch.float64)  # three Gaussian blobs
    for _ in range(3):
        cx, cy, cz = r.uniform(0, nx), r.uniform(0, ny), r.uniform(0, nz)
        s, m = r.uniform(2.0, 5.0), r.uniform(0.5, 2.0)
        rho += m * (2 * math.pi * s * s) ** -1.5 * torch.exp(
            -0.5 * ((x - cx) ** 2 + (y - cy) ** 2 + (z - cz) ** 2) / (s * s))
    return rho.to(dtype).contiguous()


def _dims(case):
    return case["nx"], case["ny"], case["nz"]


def _batch_dims(case):
    r = np.random.default_rng(case["sizes"])
    return [(int(n),) * 3 for n in r.choice(np.array([64, 96, 128, 192]), size=case["fields"])]


def _plan(case, dims):
    kw = {}
    if case.get("final_stage"):
        kw["final_stage"] = case["final_stage"]
    if case.get("mult_order") is not None:
        kw["mult_order"] = case["mult_order"]
    return fmm.FMMPlan(dims, order=case["order"], leaf=case["leaf"], precision=case["precision"], dx=1.0 / dims[0],
                       accel=case["accel"], **kw)


def prepare(case, seed):
    kind, dt = case["kind"], _dtype(case)
    if kind == "batch":
        dims = _batch_dims(case)
        plans = [_plan(case, d) for d in dims]
        rhos = [_density("plummer", d, seed * 1000 + i, dt) for i, d in enumerate(dims)]
        phis = [torch.empty_like(r) for r in rhos]
        accs = [r.new_empty((3,) + tuple(r.shape)) for r in rhos] if case["accel"] else None
        return dict(case=case, plans=plans, batch=fmm.BatchSolver(plans), rhos=rhos, phis=phis, accs=accs)
    dims = _dims(case)
    s = dict(case=case)
    if kind == "static":
        s["rho"] = _density(case["field"], dims, seed, dt)
        return s
    s["plan"] = _plan(case, dims)
    if kind == "host":
        shape = (dims[2], dims[1], dims[0])
        rhos = [_density(case["field"], dims, seed * 1000 + i, dt).cpu() for i in range(case["fields"])]
        s["rhos"] = [r.pin_memory() for r in rhos]
        s["phis"] = [torch.empty(shape, dtype=dt, pin_memory=True) for _ in rhos]
        s["accs"] = [torch.empty((3,) + shape, dtype=dt, pin_memory=True) for _ in rhos] if case["accel"] else None
        return s
    s["rho"] = _density(case["field"], dims, seed, dt)
    if kind == "grad":  # the target is a real potential: the solve of a second field
        s["target"] = s["plan"].solve(_density(case["field"], dims, seed * 1000 + 7, dt))
        s["rho"].requires_grad_(True)
    return s


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "batch":
        state["batch"].solve(state["rhos"], state["phis"], state["accs"])
        return dict(phi=state["phis"], accel=state["accs"])
    if kind == "static":
        dx = 1.0 / case["nx"]
        return fmm.solve_static(state["rho"], case["order"], case["leaf"], dx=dx, accel=bool(case["accel"]))
    if kind == "host":
        state["plan"].solve_host_many(state["rhos"], state["phis"], state["accs"])
        return dict(phi=state["phis"], accel=state["accs"])
    if kind == "grad":
        rho = state["rho"]
        rho.grad = None
        phi, _ = fmm.FMMSolve.apply(rho, state["plan"])
        loss = 0.5 * (phi - state["target"]).square().sum()
        loss.backward()
        return dict(phi=phi.detach(), grad=rho.grad)
    return state["plan"].solve(state["rho"], accel=bool(case["accel"]))


# ------------------------------------------------------------------ work ----


def _near_axis(n):
    return 3 * n - 2 if n > 1 else 1


def work(case):
    """Input and output bytes, and the multiply-adds of the two contractions
    (near field and M2L on the (p + 1)^2 harmonic components) once the
    reflections of the unit box have been used (8 times fewer products)."""
    grids = _batch_dims(case) if case["kind"] == "batch" else [_dims(case)] * case.get("fields", 1)
    es = 8 if case["precision"] == "fp64" else 4
    p, b = case["order"], case["leaf"]
    pairs = sum((2 * m + 1) * (p - m + 1) ** 2 for m in range(p + 1))
    total_b = total_f = 0.0
    for d in grids:
        cells = d[0] * d[1] * d[2]
        passes = 2 if case["kind"] == "grad" else 1
        ncomp = (4 if case["kind"] != "grad" else 1) if case["accel"] else 1
        total_b += es * cells * (1 + ncomp) * passes
        n = [v // b for v in d]
        near = _near_axis(n[0]) * _near_axis(n[1]) * _near_axis(n[2]) * float(b) ** 6
        far = 0.0
        while max(n) > 2:
            boxes = n[0] * n[1] * n[2]
            far += 189.0 * boxes * pairs * max(0.0, 1 - 2.0 / max(n))
            n = [(v + 1) // 2 for v in n]
        total_f += 2.0 * (near * (4 if case["accel"] == "analytic" else 1) + far) / 8.0 * passes
    return {"bytes": total_b, "flops": total_f}


# ----------------------------------------------------------------- exact ----


class _Mi:
    """Multi-indices up to order p."""

    def __init__(self, p):
        self.idx = [(a, n - a - c, c) for n in range(p + 1) for a in range(n, -1, -1) for c in range(n - a + 1)]
        self.of = {t: i for i, t in enumerate(self.idx)}
        self.n = len(self.idx)


def _taylor(u, p):
    """Taylor coefficients in t of 1 / |u + t|, u: [m, 3] float64 -> dict multi-index -> [m]."""
    r2 = (u * u).sum(1)
    out = {(0, 0, 0): 1.0 / np.sqrt(r2)}
    for n in range(1, p + 1):
        for a in range(n + 1):
            for b in range(n - a + 1):
                g = (a, b, n - a - b)
                s = np.zeros_like(r2)
                for i in range(3):
                    if g[i] >= 1:
                        h = list(g)
                        h[i] -= 1
                        s -= (2 * n - 1) * u[:, i] * out[tuple(h)]
                    if g[i] >= 2:
                        h = list(g)
                        h[i] -= 2
                        s -= (n - 1) * out[tuple(h)]
                out[g] = s / (n * r2)
    return out


def _comb(a, b):
    return float(math.comb(a[0] + b[0], a[0]) * math.comb(a[1] + b[1], a[1]) * math.comb(a[2] + b[2], a[2]))


@functools.lru_cache(maxsize=4)
def _m2l_ops(p, mo):
    """Unit-box M2L operators [n_alpha, n_beta] by target-minus-source offset."""
    mi = _Mi(p)
    offs = np.array([(x, y, z) for x in range(-3, 4) for y in range(-3, 4) for z in range(-3, 4)
                     if max(abs(x), abs(y), abs(z)) >= 2], dtype=np.float64)
    t = _taylor(offs, p)
    W = np.zeros((len(offs), mi.n, mi.n))
    for i, al in enumerate(mi.idx):
        for j, be in enumerate(mi.idx):
            if sum(al) + sum(be) <= p and sum(al) <= mo:
                W[:, i, j] = (-1.0) ** sum(al) * _comb(al, be) * -t[(al[0] + be[0], al[1] + be[1], al[2] + be[2])]
    return {tuple(int(v) for v in o): torch.from_numpy(W[k]) for k, o in enumerate(offs)}


def _shift_up(p):
    """Child -> parent (scaled), [8][alpha child, alpha parent]."""
    mi = _Mi(p)
    out = torch.zeros(8, mi.n, mi.n, dtype=torch.float64)
    for c in range(8):
        d = [0.5 if (c >> q) & 1 else -0.5 for q in range(3)]
        for j, al in enumerate(mi.idx):
            for i, be in enumerate(mi.idx):
                if all(be[q] <= al[q] for q in range(3)):
                    v = 0.5 ** sum(al)
                    for q in range(3):
                        v *= math.comb(al[q], be[q]) * d[q] ** (al[q] - be[q])
                    out[c, i, j] = v
    return out


def _shift_down(p):
    """Parent -> child (scaled), [8][beta parent, beta child]."""
    mi = _Mi(p)
    out = torch.zeros(8, mi.n, mi.n, dtype=torch.float64)
    for c in range(8):
        d = [0.5 if (c >> q) & 1 else -0.5 for q in range(3)]
        for i, ga in enumerate(mi.idx):
            for j, be in enumerate(mi.idx):
                if all(ga[q] >= be[q] for q in range(3)):
                    v = 0.5 ** (1 + sum(ga))
                    for q in range(3):
                        v *= math.comb(ga[q], be[q]) * d[q] ** (ga[q] - be[q])
                    out[c, i, j] = v
    return out


def _pad_even(t):
    """[z, y, x, k] with even extents (zeros past the end)."""
    z, y, x, _ = t.shape
    return torch.nn.functional.pad(t, (0, 0, 0, x % 2, 0, y % 2, 0, z % 2))


def _window(t, o, step, n):
    """t[o + step * i] along the three leading axes for i < n, zero outside."""
    out = t.new_zeros(tuple(n) + t.shape[3:])
    src, dst = [], []
    for q in range(3):
        i0 = max(0, -(-(-o[q]) // step)) if o[q] < 0 else 0
        i1 = min(n[q], (t.shape[q] - 1 - o[q]) // step + 1)
        if i1 <= i0:
            return out
        src.append(slice(o[q] + step * i0, o[q] + step * (i1 - 1) + 1, step))
        dst.append(slice(i0, i1))
    out[tuple(dst)] = t[tuple(src)]
    return out


def _cells(b):
    return ((torch.arange(b, dtype=torch.float64) + 0.5) / b - 0.5).cuda()


def _boxes(rho, b):
    z, y, x = rho.shape
    return rho.reshape(z // b, b, y // b, b, x // b, b).permute(0, 2, 4, 1, 3, 5)  # [Z, Y, X, z, y, x]


def _monomials(p, b):
    """[cells (z, y, x), nc] monomials at the cell centres of a unit box, and their gradients [3]."""
    mi, e = _Mi(p), _cells(b).cpu().numpy()
    z, y, x = np.meshgrid(e, e, e, indexing="ij")
    pt = [x.ravel(), y.ravel(), z.ravel()]
    V = np.stack([pt[0] ** a * pt[1] ** bb * pt[2] ** c for a, bb, c in mi.idx], 1)
    G = []
    for q in range(3):
        cols = []
        for t in mi.idx:
            v = np.full(b ** 3, float(t[q]))
            for r in range(3):
                k = t[r] - (r == q)
                v = v * (pt[r] ** k if k >= 0 else 0.0)
            cols.append(v)
        G.append(np.stack(cols, 1))
    return torch.from_numpy(V).cuda(), [torch.from_numpy(g).cuda() for g in G]


def _near_kernels(b, d):
    """[source cell, target cell] g and its three derivatives for source box offset d = (x, y, z)."""
    e = np.arange(b, dtype=np.float64)
    z, y, x = np.meshgrid(e, e, e, indexing="ij")
    pt = np.stack([x.ravel(), y.ravel(), z.ravel()], 1)
    r = pt[None, :, :] - pt[:, None, :] - b * np.array(d, dtype=np.float64)
    n = np.sqrt((r * r).sum(2))
    n0 = np.where(n == 0, 1.0, n)
    g = np.where(n == 0, -1.0, -1.0 / n0)
    return [torch.from_numpy(g).cuda()] + [torch.from_numpy(np.where(n == 0, 0.0, r[:, :, q] / n0 ** 3)).cuda()
                                            for q in range(3)]


def _stencil(phi, dx):
    """-grad(phi): 5-point central inside, 3-point one cell from an edge, one-sided at it."""
    out = []
    for ax in (2, 1, 0):
        n = phi.shape[ax]

        def at(i0, i1):
            return phi.narrow(ax, i0, i1 - i0)

        if n == 1:
            out.append(torch.zeros_like(phi))
            continue
        if n == 2:
            d = at(1, 2) - at(0, 1)
            out.append(-torch.cat([d, d], ax) / dx)
            continue
        parts = [(-3 * at(0, 1) + 4 * at(1, 2) - at(2, 3)) / 2, (at(2, 3) - at(0, 1)) / 2]
        if n > 4:
            parts.append((at(0, n - 4) - 8 * at(1, n - 3) + 8 * at(3, n - 1) - at(4, n)) / 12)
        if n > 3:
            parts.append((at(n - 1, n) - at(n - 3, n - 2)) / 2)
        parts.append((3 * at(n - 1, n) - 4 * at(n - 2, n - 1) + at(n - 3, n - 2)) / 2)
        out.append(-torch.cat(parts, ax) / dx)
    return torch.stack(out)


def _solve64(rho, case, dx, analytic):
    """phi (and the analytic acceleration) of the truncated operator, FP64 torch on the GPU."""
    p, b = case["order"], case["leaf"]
    mo = p if case.get("mult_order") is None else case["mult_order"]
    m2p = case.get("final_stage") == "m2p"
    nc = _Mi(p).n
    box = _boxes(rho.double(), b)
    nb = box.shape[:3]
    cells = box.reshape(nb + (b ** 3,))
    V, G = _monomials(p, b)
    M = [cells @ V]
    up, down = _shift_up(p).cuda(), _shift_down(p).cuda()
    while max(M[-1].shape[:3]) > 4:  # coarser levels while they hold an interaction list
        c = _pad_even(M[-1])
        M.append(sum(c[(k >> 2)::2, ((k >> 1) & 1)::2, (k & 1)::2] @ up[k] for k in range(8)))
    ops = {k: w.cuda() for k, w in _m2l_ops(p, mo).items()}
    L = None
    grad_far = None
    for lev in range(len(M) - 1, -1, -1):
        src = _pad_even(M[lev])
        npar = [v // 2 for v in src.shape[:3]]
        loc = src.new_zeros(src.shape)
        if L is not None:
            Lp = L
            for k in range(8):
                loc[(k >> 2)::2, ((k >> 1) & 1)::2, (k & 1)::2] = Lp[:npar[0], :npar[1], :npar[2]] @ down[k]
        leaf_m2p = m2p and lev == 0
        far = src.new_zeros(tuple(src.shape[:3]) + (4 if analytic else 1, b ** 3)) if leaf_m2p else None
        if max(M[lev].shape[:3]) > 2:
            for k in range(8):
                c = (k & 1, (k >> 1) & 1, k >> 2)
                acc = src.new_zeros(tuple(npar) + (nc,))
                facc = src.new_zeros(tuple(npar) + ((4 if analytic else 1) * b ** 3,)) if leaf_m2p else None
                for oz in range(-2, 4):
                    for oy in range(-2, 4):
                        for ox in range(-2, 4):  # source child position relative to the parent's first child
                            u = (c[0] - ox, c[1] - oy, c[2] - oz)
                            if max(abs(v) for v in u) < 2:
                                continue
                            s = _window(src, (oz, oy, ox), 2, npar)
                            if leaf_m2p:
                                facc += s @ _m2p_op(p, mo, b, u, analytic)
                            else:
                                acc += s @ ops[u]
                sl = (slice(c[2], None, 2), slice(c[1], None, 2), slice(c[0], None, 2))
                if leaf_m2p:
                    far[sl] = facc.reshape(tuple(npar) + (-1, b ** 3))
                else:
                    loc[sl] += acc
        L = loc
    L = L[:nb[0], :nb[1], :nb[2]]
    out = [(L @ V.T) / b]
    if analytic:
        out += [(L @ g.T) / (b * b) for g in G]
    if m2p:
        far = far[:nb[0], :nb[1], :nb[2]]
        for i in range(len(out)):
            out[i] = out[i] + far[..., i, :] / (b if i == 0 else b * b)
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx_ in (-1, 0, 1):
                s = _window(cells, (dz, dy, dx_), 1, nb)
                ks = _near_kernels(b, (dx_, dy, dz))
                for i in range(len(out)):
                    out[i] += s @ ks[i]
                del s

    def grid(t):
        return t.reshape(nb + (b, b, b)).permute(0, 3, 1, 4, 2, 5).reshape(rho.shape).contiguous()

    phi = grid(out[0]) * (dx * dx)
    if analytic:
        return phi, torch.stack([grid(t) * -dx for t in out[1:]])
    return phi, None


@functools.lru_cache(maxsize=512)
def _m2p_op(p, mo, b, u, analytic):
    """[alpha, comps * cells]: leaf multipoles of a box at offset u to the target's cells (box units)."""
    mi, e = _Mi(p), _cells(b).cpu().numpy()
    z, y, x = np.meshgrid(e, e, e, indexing="ij")
    pts = np.stack([x.ravel(), y.ravel(), z.ravel()], 1) + np.array(u, dtype=np.float64)
    t = _taylor(pts, p + 1)
    W = np.zeros((mi.n, 4 if analytic else 1, b ** 3))
    for i, al in enumerate(mi.idx):
        if sum(al) > mo:
            continue
        W[i, 0] = (-1.0) ** sum(al) * -t[al]
        if analytic:
            for q in range(3):
                h = list(al)
                h[q] += 1
                W[i, 1 + q] = (-1.0) ** sum(al) * (al[q] + 1) * -t[tuple(h)]
    return torch.from_numpy(W.reshape(mi.n, -1)).cuda()


def exact(case, seed):
    kind, dt = case["kind"], _dtype(case)
    cells = sum(d[0] * d[1] * d[2] for d in (_batch_dims(case) if kind == "batch" else [_dims(case)]))
    cost = cells * (case["order"] + 1) ** 6 / case["leaf"] ** 3
    if cost > 3e11 or cells > 140e6:  # over about 20 seconds in 64 bits
        return None

    def one(rho, dims):
        dx = 1.0 / dims[0]
        analytic = case["accel"] == "analytic"
        phi, acc = _solve64(rho, case, dx, analytic)
        if case["accel"] and not analytic:
            acc = _stencil(phi, dx)
        return phi, acc

    if kind == "batch":
        dims = _batch_dims(case)
        got = [one(_density("plummer", d, seed * 1000 + i, dt), d) for i, d in enumerate(dims)]
        return dict(phi=[g[0] for g in got], accel=[g[1] for g in got] if case["accel"] else None)
    dims = _dims(case)
    if kind == "host":
        got = [one(_density(case["field"], dims, seed * 1000 + i, dt), dims) for i in range(case["fields"])]
        return dict(phi=[g[0] for g in got], accel=[g[1] for g in got] if case["accel"] else None)
    rho = _density(case["field"], dims, seed, dt)
    if kind == "grad":
        dx = 1.0 / dims[0]
        phi, _ = _solve64(rho, case, dx, False)
        target, _ = _solve64(_density(case["field"], dims, seed * 1000 + 7, dt), case, dx, False)
        grad, _ = _solve64(phi - target, case, dx, False)  # the operator is symmetric
        return dict(phi=phi, grad=grad)
    phi, acc = one(rho, dims)
    return (phi, acc) if case["accel"] else phi
