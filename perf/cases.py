"""What a user of the patch library runs, as measurable cases.

Every case is one call (or one engine step made of several calls) through the
package's public binding (paper_2302_09005_gb300.fv, .learned), on inputs of
the library's own workloads: i.i.d. random Euler states, periodic / outflow /
wall patch meshes, uneven 3^3/5^3/7^3 batches, a 3:1 refined mesh, the paper's
2D p = 17 offload, the learned correction's shear layer and its training.

  listed()             the named cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  inputs on the GPU, handles, plans
  run(state)           one pass; returns every output
  work(case)           bytes and operations a pass cannot do without
  exact(case, seed)    the same outputs in 64 bits with plain torch
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2302_09005_gb300 import fv, learned

GAMMA = 1.4
CFL = 0.4
# an upper bound of |u| + c of the random states below (|u| <= 0.5,
# c <= sqrt(1.4 * 1.5 / 0.5)): explicit time steps are taken from it
LAM_BOUND = 2.6
MAX_CELLS = 262144 * 125  # the largest mesh below


# --------------------------------------------------------------------------
# The cases
# --------------------------------------------------------------------------
def listed():
    return [
        # one small task of the engine: 64 patches of 3x3, the smallest batch
        # the paper's kernels are called with; launch latency counts
        {"name": "update_2d_fp64_p3_n64", "op": "update", "d": 2, "prec": "fp64", "lo": 3,
         "hi": 3, "n": 64, "lam": False, "plan": False},
        # an AMR task batch straight from the engine: ragged sizes, FP32, the
        # per-patch wave speeds asked for, no plan made beforehand
        {"name": "update_3d_fp32_ragged_n20011", "op": "update", "d": 3, "prec": "fp32",
         "lo": 2, "hi": 8, "n": 20011, "lam": True, "plan": False},
        # the paper's own benchmark shape (2D, p = 17), patches in host memory,
        # copies included, advanced in place
        {"name": "offload_2d_fp64_p17_n8192", "op": "host", "d": 2, "prec": "fp64", "p": 17,
         "n": 8192},
        # the plain method at scale: a time step of a 320^3 periodic domain
        # with the primitive carry (the benchmark's step)
        {"name": "step_3d_fp64_p5_64x64x64", "op": "step", "d": 3, "prec": "fp64", "p": 5,
         "gx": 64, "gy": 64, "gz": 64, "boundary": 0, "carry": True, "plan": False},
        # the same domain in FP32, planned once
        {"name": "step_3d_fp32_p5_64x64x64", "op": "step", "d": 3, "prec": "fp32", "p": 5,
         "gx": 64, "gy": 64, "gz": 64, "boundary": 0, "carry": False, "plan": True},
        # a small simulation: 64^2 cells in 8x8 patches, 50 steps in one
        # captured graph; the gaps between tiny kernels count
        {"name": "run_2d_fp64_p8_8x8_50steps", "op": "run", "d": 2, "prec": "fp64", "p": 8,
         "gx": 8, "gy": 8, "gz": 1, "boundary": 0, "steps": 50, "plan": False},
        # uneven batching: 200,000 patches of 3^3 / 5^3 / 7^3, 20 steps a graph
        {"name": "run_3d_fp64_uneven_n200000_20steps", "op": "uneven", "prec": "fp64",
         "n": 200000, "steps": 20},
        # the precision workload: 4095^2 cells in 5x5 patches, FP32
        {"name": "run_2d_fp32_p5_819x819_20steps", "op": "run", "d": 2, "prec": "fp32", "p": 5,
         "gx": 819, "gy": 819, "gz": 1, "boundary": 0, "steps": 20, "plan": True},
        # an engine that keeps its steps apart and logs conservation: halo
        # fill, CFL reduce, update with the device time step, per-patch sums;
        # odd mesh, outflow boundaries
        {"name": "engine_3d_fp64_p6_21x19x23", "op": "engine", "d": 3, "prec": "fp64", "p": 6,
         "gx": 21, "gy": 19, "gz": 23, "boundary": -1},
        # a refined mesh (22,933 patches on two levels): inter-level halos and
        # the update with a cell size and CFL step per patch
        {"name": "amr_3d_fp64_p5_base3", "op": "amr", "d": 3, "prec": "fp64", "p": 5, "base": 3,
         "block": 5},
        # one learned step of the 1024^2 shear layer (correction network on
        # the tensor cores, halo fill, corrected update)
        {"name": "learned_2d_fp64_p8_1024", "op": "learned", "prec": "fp64", "p": 8, "N": 1024},
        # training of the correction: 20 Adam steps of 32,768 samples
        {"name": "train_b32768_20steps", "op": "train", "batch": 32768, "nb": 10, "steps": 20},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mesh(rng, d, p, max_cells, min_patches=8):
    """A patch grid of d axes, nearly square, of log-uniform total size."""
    n = _logint(rng, min_patches, max(min_patches + 1, max_cells // p ** d))
    g = []
    for k in range(d):
        w = n ** (1.0 / (d - k))
        v = max(1, int(round(w * rng.uniform(0.8, 1.25)))) if k + 1 < d else max(1, int(round(w)))
        g.append(v)
        n = max(1.0, n / v)
    while g[0] * (g[1] if d > 1 else 1) * (g[2] if d > 2 else 1) * p ** d > max_cells:
        k = max(range(d), key=lambda m: g[m])
        g[k] -= 1
    return g + [1] * (3 - d)


def draw(rng):
    op = rng.choice(["update", "update", "update", "host", "step", "step", "run", "run",
                     "uneven", "engine", "amr", "learned", "train"])
    prec = rng.choice(["fp64", "fp32"])
    d = rng.choice([2, 3])
    p = rng.randint(2, 17) if d == 2 else rng.randint(2, 8)
    if op == "update":
        ragged = rng.random() < 0.4
        lo = rng.randint(1, max(1, p - 1)) if ragged else p
        n = _logint(rng, 16, min(400000, 8_000_000 // p ** d))
        return {"op": op, "d": d, "prec": prec, "lo": lo, "hi": p, "n": n,
                "lam": rng.random() < 0.5, "plan": rng.random() < 0.5}
    if op == "host":
        n = _logint(rng, 16, min(100000, 8_000_000 // (p + 2) ** d))
        return {"op": op, "d": d, "prec": prec, "p": p, "n": n}
    if op == "step":
        g = _mesh(rng, d, p, MAX_CELLS // 4)
        carry = prec == "fp64" and rng.random() < 0.7
        return {"op": op, "d": d, "prec": prec, "p": p, "gx": g[0], "gy": g[1], "gz": g[2],
                "boundary": rng.choice([0, 0, -1, -2]), "carry": carry,
                "plan": rng.random() < 0.6}
    if op == "run":
        g = _mesh(rng, d, p, 4_000_000)
        return {"op": op, "d": d, "prec": prec, "p": p, "gx": g[0], "gy": g[1], "gz": g[2],
                "boundary": rng.choice([0, 0, -1, -2]), "steps": rng.randint(2, 50),
                "plan": rng.random() < 0.6}
    if op == "uneven":
        return {"op": op, "prec": prec, "n": _logint(rng, 500, 150000),
                "steps": rng.randint(2, 20)}
    if op == "engine":
        g = _mesh(rng, d, p, 8_000_000)
        return {"op": op, "d": d, "prec": prec, "p": p, "gx": g[0], "gy": g[1], "gz": g[2],
                "boundary": rng.choice([0, -1, -2])}
    if op == "amr":
        p = rng.randint(3, 6)
        base = rng.choice([1, 2]) if d == 3 else rng.choice([2, 3, 4])
        return {"op": op, "d": d, "prec": prec, "p": p, "base": base,
                "block": rng.randint(1, 3 ** base - 2)}
    if op == "learned":
        p = rng.randint(3, 16)
        return {"op": op, "prec": prec, "p": p, "N": p * rng.randint(max(2, 64 // p), 1024 // p)}
    return {"op": op, "batch": _logint(rng, 100, 32768), "nb": rng.randint(1, 10),
            "steps": rng.randint(1, 20)}


# --------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------
def _dtype(case):
    return torch.float64 if case["prec"] == "fp64" else torch.float32


def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1000003 + salt)
    return g


def _states(g, n, d):
    """n random states: rho ~ U[0.5, 1.5], u_k ~ U[-0.5, 0.5], p ~ U[0.5, 1.5]."""
    r = torch.rand((n, d + 2), generator=g, device="cuda", dtype=torch.float64)
    q = torch.empty_like(r)
    rho = 0.5 + r[:, 0]
    u = r[:, 1:1 + d] - 0.5
    q[:, 0] = rho
    q[:, 1:1 + d] = rho[:, None] * u
    q[:, d + 1] = (0.5 + r[:, d + 1]) / (GAMMA - 1) + 0.5 * rho * (u * u).sum(1)
    return q


def _box(p, d):
    return (p + 2) ** d * (d + 2)


def _layout(sizes, d):
    """Offsets of consecutive patches, each rounded up to 4 elements."""
    lens = (sizes.astype(np.int64) + 2) ** d * (d + 2)
    lens = (lens + 3) // 4 * 4
    off = np.zeros(len(sizes), dtype=np.int64)
    off[1:] = np.cumsum(lens[:-1])
    return off, int(lens.sum())


def _chunks(n, per):
    step = max(1, 4_000_000 // max(1, per))
    for a in range(0, n, step):
        yield a, min(n, a + step)


def _classes(sizes):
    for p in sorted(set(sizes.tolist())):
        yield p, np.nonzero(sizes == p)[0]


def _index(off, cells):
    """Flat element indices (n, cells) of patches at device offsets."""
    return off[:, None] + torch.arange(cells, device="cuda")[None, :]


def _fill(q, off, sizes, d, seed):
    """Random states in every cell of every patch (halos included)."""
    g = _gen(seed)
    toff = torch.from_numpy(off).cuda()
    s = d + 2
    for p, idx in _classes(sizes):
        L = _box(p, d)
        for a, b in _chunks(len(idx), L // s):
            sel = toff[torch.from_numpy(idx[a:b]).cuda()]
            q[_index(sel, L)] = _states(g, (b - a) * (L // s), d).view(b - a, L).to(q.dtype)


def _sizes(case, seed):
    op = case["op"]
    if op == "uneven":
        n = case["n"]
        n5, n7 = int(round(0.3 * n)), int(round(0.2 * n))
        v = np.concatenate([np.full(n - n5 - n7, 3), np.full(n5, 5), np.full(n7, 7)])
        np.random.default_rng(seed).shuffle(v)
        return v.astype(np.int32), 3
    if op == "update":
        # the same sizes for every seed, in another order
        v = np.random.default_rng(case["n"]).integers(case["lo"], case["hi"] + 1, case["n"])
        np.random.default_rng(seed).shuffle(v)
        return v.astype(np.int32), case["d"]
    if op == "amr":
        return np.full(len(_tree(case)[0]), case["p"], dtype=np.int32), case["d"]
    n = case["n"] if op == "host" else case["gx"] * case["gy"] * case["gz"]
    return np.full(n, case["p"], dtype=np.int32), case["d"]


def _neighbours(case):
    """-x, +x, -y, +y(, -z, +z) neighbours of a patch grid, x fastest; the
    patches of an uneven batch are periodic on their own."""
    if case["op"] == "uneven":
        return np.repeat(np.arange(case["n"], dtype=np.int32)[:, None], 6, axis=1)
    d = case["d"]
    shape = (case["gx"], case["gy"], case["gz"])[:d]
    n = int(np.prod(shape))
    i = np.arange(n)
    out = np.empty((n, 2 * d), dtype=np.int32)
    stride = 1
    for k in range(d):
        c = i // stride % shape[k]
        for side, e in ((0, -1), (1, 1)):
            w = (c + e) % shape[k]
            nb = i + (w - c) * stride
            if case["boundary"]:
                nb = np.where((c + e >= 0) & (c + e < shape[k]), nb, case["boundary"])
            out[:, 2 * k + side] = nb
        stride *= shape[k]
    return out


def _tree(case):
    """Level and coordinates of a two-level 3:1 tree: every cell of level
    `base`, a central block of them refined."""
    d, base, m = case["d"], case["base"], case["block"]
    nb = 3 ** base
    lo = (nb - m) // 2
    ax = np.meshgrid(*[np.arange(nb)] * d, indexing="ij")
    c = np.stack([a.reshape(-1) for a in reversed(ax)], axis=1)
    fine = np.all((c >= lo) & (c < lo + m), axis=1)
    ch = np.stack([a.reshape(-1) for a in np.meshgrid(*[np.arange(3)] * d, indexing="ij")], 1)
    kids = (3 * c[fine][:, None, :] + ch[None, :, ::-1]).reshape(-1, d)
    coord = np.concatenate([c[~fine], kids]).astype(np.int32)
    level = np.concatenate([np.full((~fine).sum(), base), np.full(len(kids), base + 1)])
    return level.astype(np.int32), coord


def _dx(case):
    if case["op"] in ("update", "host", "uneven"):
        return 1.0 / 64
    return 1.0 / (case["gx"] * case["p"])


def _dt(case, d):
    return CFL * _dx(case) / (d * LAM_BOUND)


def _shear(N, seed):
    """Shear layer: rho = 2, u = -0.5 in the middle band, else rho = 1,
    u = 0.5; p = 2.5; v = sum of four sines of amplitude 0.01 at most."""
    g = _gen(seed, 7)
    x = (torch.arange(N, device="cuda", dtype=torch.float64) + 0.5) / N
    a = torch.rand(4, generator=g, device="cuda", dtype=torch.float64)
    ph = 2 * math.pi * torch.rand(4, generator=g, device="cuda", dtype=torch.float64)
    v = sum(a[k] * torch.sin(2 * math.pi * (k + 1) * x + ph[k]) for k in range(4))
    v = v * (0.01 / v.abs().max())
    band = ((x - 0.5).abs() < 0.25)[:, None].expand(N, N)
    rho = torch.where(band, 2.0, 1.0).double()
    u = torch.where(band, -0.5, 0.5).double()
    v = v[None, :].expand(N, N)
    return torch.stack([rho, rho * u, rho * v,
                        2.5 / (GAMMA - 1) + 0.5 * rho * (u * u + v * v)], dim=-1)


def _network(seed):
    """Parameters of the 16-64-64-4 network, drawn like its initialisation
    with small biases (FP64)."""
    g = _gen(seed, 11)
    parts = []
    for rows, cols, scale in ((64, 16, 1.0), (64, 64, 1.0), (4, 64, 0.1)):
        w = torch.randn((rows, cols), generator=g, device="cuda", dtype=torch.float64)
        parts.append((scale / math.sqrt(cols)) * w.reshape(-1))
        parts.append(0.05 * torch.randn(rows, generator=g, device="cuda", dtype=torch.float64))
    return torch.cat(parts).float()


def _norm(case):
    """Normalisation of a shear layer's stencils (rho, j_n, j_t, E)."""
    mu = torch.tensor([1.5, 0.0, 0.0, 6.4] * 4)
    sd = torch.tensor([0.5, 0.5, 0.5, 0.2] * 4)
    sdy = torch.full((4,), 1e-4)
    return torch.cat([mu, sd, sdy]).float().cuda()


def _samples(case, seed):
    """Training pairs: normalised stencils and targets that depend on them."""
    g = _gen(seed, 13)
    n = case["batch"] * case["nb"]
    x = torch.randn((n, 16), generator=g, device="cuda")
    w = torch.randn((16, 4), generator=g, device="cuda") / 4
    t = torch.tanh(x @ w) + 0.1 * torch.randn((n, 4), generator=g, device="cuda")
    return x, t


_STREAM = []


def _stream():
    """The one stream of the program, which all its handles work on."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


class _State:
    """What a program keeps between calls: buffers, handle, plan, stream."""

    def __init__(self, case):
        self.case = case
        self.stream = _stream()


def prepare(case, seed):
    op = case["op"]
    st = _State(case)
    if op == "train":
        st.x, st.t = _samples(case, seed)
        st.params = _network(seed)
        st.losses = torch.zeros(case["steps"], device="cuda")
        torch.cuda.current_stream().synchronize()
        st.trainer = fv.MlpTrainer(case["batch"], st.stream)
        st.done = 0
        return st
    prec = fv.FV_FP64 if case["prec"] == "fp64" else fv.FV_FP32
    if op == "learned":
        N, p = case["N"], case["p"]
        st.params, st.norm = _network(seed), _norm(case)
        st.mesh = learned.Mesh2D(N, p, prec, st.stream, U=_shear(N, seed).cpu().numpy())
        st.corr = torch.zeros(st.mesh.n * fv.fv_corr_stride(st.mesh.b.h), device="cuda")
        st.dt = CFL / N / (2 * 2.5)
        torch.cuda.current_stream().synchronize()
        return st
    sizes, d = _sizes(case, seed)
    off, total = _layout(sizes, d)
    q = torch.zeros(total, dtype=_dtype(case), device="cuda")
    _fill(q, off, sizes, d, seed)
    pmax = int(sizes.max())
    st.n = len(sizes)
    st.dx, st.dt = (_dx(case), _dt(case, d)) if op != "amr" else (0.0, 0.0)
    torch.cuda.current_stream().synchronize()
    st.b = fv.Batch(d, precision=prec, max_patch_size=pmax, stream=st.stream)
    if op == "host":
        st.q = torch.empty(total, dtype=q.dtype, pin_memory=True)
        st.q.copy_(q)
        st.off, st.sizes = off, sizes
        return st
    st.q, st.out = q, torch.zeros_like(q)
    st.off, st.sizes = torch.from_numpy(off).cuda(), torch.from_numpy(sizes).cuda()
    if op in ("run", "uneven", "step", "engine"):
        st.nbr = torch.from_numpy(_neighbours(case)).cuda()
    if op == "update" and case["lam"] or op in ("engine", "amr"):
        st.lam = torch.zeros(st.n, dtype=torch.float64, device="cuda")
    if op == "engine":
        st.sums = torch.zeros((st.n, d + 2), dtype=torch.float64, device="cuda")
        st.totals = torch.zeros(d + 2, dtype=torch.float64, device="cuda")
        st.dt_dev = torch.zeros(1, dtype=torch.float64, device="cuda")
    if op == "amr":
        level, coord = _tree(case)
        st.plan = fv.AmrPlan(st.b.h, level, coord, off, case["p"], 0)
        st.dxp = torch.from_numpy(3.0 ** -level / case["p"]).cuda()
        st.dtp = torch.zeros(st.n, dtype=torch.float64, device="cuda")
    torch.cuda.current_stream().synchronize()
    if case.get("plan") or op == "uneven":
        fv.fv_batch_plan(st.b.h, st.sizes, st.n)
        fv.fv_batch_set_schedule(st.b.h, fv.FV_SCHED_CLASSES)
    if op == "step":
        # the simulation is under way: the CFL maximum is on the device and,
        # with the carry, one step has left its primitives
        st.b.halo_fill(st.q, st.off, st.sizes, st.nbr)
        st.b.max_eigenvalue(st.q, st.off, st.sizes, CFL, st.dx)
        st.prim = None
        if case["carry"]:
            m = st.n * st.b.prim_stride()
            st.prim = [torch.zeros(m, dtype=q.dtype, device="cuda") for _ in range(2)]
            torch.cuda.current_stream().synchronize()
            st.b.time_step_prim(st.q, st.out, None, st.prim[0], st.off, st.sizes, st.nbr, st.dx,
                                CFL)
            st.q, st.out = st.out, st.q
    return st


# --------------------------------------------------------------------------
# One pass
# --------------------------------------------------------------------------
def run(st):
    case, op = st.case, st.case["op"]
    if op == "update":
        st.b.update(st.q, st.out, st.off, st.sizes, st.dx, st.dt,
                    lambda_patch=st.lam if case["lam"] else None)
        return [st.out, st.lam] if case["lam"] else [st.out]
    if op == "host":
        fv.fv_patch_update_host(st.b.h, st.q, st.q, st.off, st.sizes, st.n, st.dx, st.dt)
        return [st.q]
    if op == "step":
        if st.prim is not None:
            st.b.time_step_prim(st.q, st.out, st.prim[0], st.prim[1], st.off, st.sizes, st.nbr,
                                st.dx, CFL)
            st.prim.reverse()
        else:
            st.b.time_step(st.q, st.out, st.off, st.sizes, st.nbr, st.dx, CFL)
        st.q, st.out = st.out, st.q
        return [st.q] if st.prim is None else [st.q, st.prim[0]]
    if op in ("run", "uneven"):
        st.b.run_steps(st.q, st.out, st.off, st.sizes, st.nbr, st.dx, CFL, case["steps"],
                       use_graph=True)
        return [st.q if case["steps"] % 2 == 0 else st.out]
    if op == "engine":
        st.b.halo_fill(st.q, st.off, st.sizes, st.nbr)
        st.b.max_eigenvalue(st.q, st.off, st.sizes, CFL, st.dx, per_patch=st.lam,
                            dt_out=st.dt_dev)
        st.b.update(st.q, st.out, st.off, st.sizes, st.dx, -1.0)
        fv.fv_patch_sums(st.b.h, st.out, st.off, st.sizes, st.n, st.sums, st.totals)
        return [st.q, st.out, st.lam, st.dt_dev, st.sums, st.totals]
    if op == "amr":
        st.plan.fill(st.q)
        fv.fv_patch_update_local(st.b.h, st.q, st.out, st.off, st.sizes, st.n, st.dxp, st.dtp,
                                 CFL, st.lam)
        return [st.q, st.out, st.dtp, st.lam]
    if op == "learned":
        st.mesh.step_learned(st.dt, st.params, st.norm, st.corr)
        return [st.mesh.x, st.corr]
    st.trainer.train_steps(st.params, st.x, st.t, case["batch"], st.done + 1, case["steps"],
                           1e-3, st.losses)
    st.done += case["steps"]
    return [st.params, st.losses]


# --------------------------------------------------------------------------
# Work
# --------------------------------------------------------------------------
def _flops(d, cells, faces, prim_cells):
    """Operations of Eq. 2-5: fluxes of the faces, updates of the cells,
    primitives (two operations an FMA)."""
    return faces * (10 + 6 * d) + cells * (2 * d + 1) * (d + 2) + prim_cells * (14 + 5 * d)


def work(case):
    op = case["op"]
    if op == "train":
        B, s = case["batch"], case["steps"]
        return {"bytes": float(s * (B * 80 + 5508 * 4 * 6)), "flops": float(s * B * 6 * 5376)}
    es = 8 if case["prec"] == "fp64" else 4
    if op == "learned":
        cells, p = case["N"] ** 2, case["p"]
        corr = (cells // p ** 2) * 8 * (p + 1) * p * 4
        return {"bytes": float(2 * cells * 4 * es + corr),
                "flops": float(2 * cells * 2 * 5376 + _flops(2, cells, 2 * cells, cells))}
    sizes, d = _sizes(case, 0)
    s = d + 2
    z = sizes.astype(np.float64)
    n, cells = len(z), float((z ** d).sum())
    halo = float((2 * d * z ** (d - 1)).sum())
    faces = float((d * (z + 1) * z ** (d - 1)).sum())
    state = cells * s * es
    if op in ("step", "run", "uneven"):
        steps = case.get("steps", 1)
        b = 2 * state + (12 + 8 * d) * n
        if case.get("carry"):
            b += 2 * cells * (d + 3) * es
        return {"bytes": steps * b, "flops": steps * _flops(d, cells, faces, cells)}
    b = 2 * state + halo * s * es + 12 * n
    f = _flops(d, cells, faces, cells + halo)
    if op == "update" and case["lam"]:
        b += 8 * n
    if op in ("engine", "amr"):
        b += halo * s * es + (8 + 8 * d + 8 * s) * n
    return {"bytes": float(b), "flops": float(f)}


# --------------------------------------------------------------------------
# The same in 64 bits with plain torch
# --------------------------------------------------------------------------
def _prims(Q):
    d = Q.shape[-1] - 2
    rho = Q[..., 0]
    u = [Q[..., 1 + k] / rho for k in range(d)]
    p = (GAMMA - 1) * (Q[..., d + 1] - 0.5 * sum(Q[..., 1 + k] * u[k] for k in range(d)))
    return u, p, torch.sqrt(GAMMA * p / rho)


def _flux(Q, k):
    """f^k (Eq. 2) and |u_k| + c."""
    d = Q.shape[-1] - 2
    u, p, c = _prims(Q)
    f = Q * u[k][..., None]
    f[..., 1 + k] += p
    f[..., d + 1] += p * u[k]
    return f, u[k].abs() + c


def _rusanov(Q, dx, dt, corr=None):
    """New interior of patches Q (n, [p + 2] * d, s), axis d - k is direction
    k; the largest a of every patch's faces.  dx, dt: numbers or (n,)."""
    d = Q.shape[-1] - 2
    n = Q.shape[0]
    lam = torch.zeros(n, dtype=Q.dtype, device=Q.device)
    parts = []
    for k in range(d):
        ax = d - k
        B = Q
        for m in range(1, d + 1):
            if m != ax:
                B = B.narrow(m, 1, B.shape[m] - 2)
        f, w = _flux(B, k)
        e = B.shape[ax] - 1
        L, R = (lambda t: t.narrow(ax, 0, e)), (lambda t: t.narrow(ax, 1, e))
        a = torch.maximum(L(w), R(w))
        lam = torch.maximum(lam, a.reshape(n, -1).amax(1))
        F = 0.5 * (L(f) + R(f) - a[..., None] * (R(B) - L(B)))
        if corr is not None:
            F = F + corr[k]
        parts.append(F.narrow(ax, 1, e - 1) - F.narrow(ax, 0, e - 1))
    I = Q
    for m in range(1, d + 1):
        I = I.narrow(m, 1, I.shape[m] - 2)
    r = (dt(lam) if callable(dt) else dt) / dx
    if torch.is_tensor(r) and r.dim() == 1:
        r = r.view([n] + [1] * (d + 1))
    return I - r * sum(parts), lam


def _inner(Q):
    d = Q.shape[-1] - 2
    for m in range(1, d + 1):
        Q = Q.narrow(m, 1, Q.shape[m] - 2)
    return Q


def _halos(Q, nbr):
    """Fill the face halos in place (neighbour, -1 outflow, -2 wall)."""
    d = Q.shape[-1] - 2
    p = Q.shape[1] - 2
    own = torch.arange(len(Q), device="cuda")
    for k in range(d):
        ax = d - k
        T = Q
        for m in range(1, d + 1):
            if m != ax:
                T = T.narrow(m, 1, p)
        for side in (0, 1):
            nb = nbr[:, 2 * k + side].long()
            far = T.select(ax, 1 if side else p)[torch.where(nb >= 0, nb, own)]
            near = T.select(ax, p if side else 1).clone()
            wall = near.clone()
            wall[..., 1 + k] *= -1
            shape = [-1] + [1] * (far.dim() - 1)
            v = torch.where((nb >= 0).view(shape), far,
                            torch.where((nb == -2).view(shape), wall, near))
            T.select(ax, p + 1 if side else 0).copy_(v)


def _max_speed(Q):
    out = 0.0
    for a, b in _chunks(len(Q), Q[0].numel()):
        u, _, c = _prims(_inner(Q[a:b]))
        out = max(out, max((x.abs() + c).max().item() for x in u))
    return out


def _step(Q, dx, dt):
    new = torch.empty_like(_inner(Q))
    lam = torch.zeros(len(Q), dtype=torch.float64, device="cuda")
    for a, b in _chunks(len(Q), Q[0].numel()):
        x = dx if not torch.is_tensor(dx) else dx[a:b]
        t = dt if not callable(dt) else (lambda w, x=x: dt(w, x))
        new[a:b], lam[a:b] = _rusanov(Q[a:b], x, t)
    return new, lam


def _prim_block(Q, case, stride):
    """Carried primitives of the interior: (u_1..u_d, p, c, E + p) by
    component, x fastest, in blocks of `stride` elements."""
    d = Q.shape[-1] - 2
    I = _inner(Q)
    u, p, c = _prims(I)
    comp = u + [p, c, I[..., d + 1] + p]
    out = torch.zeros((len(Q), stride), dtype=torch.float64, device="cuda")
    flat = torch.stack([v.reshape(len(Q), -1) for v in comp], 1).reshape(len(Q), -1)
    out[:, :flat.shape[1]] = flat
    return out.reshape(-1)


def exact(case, seed):
    op = case["op"]
    if op == "train":
        return _exact_train(case, seed)
    if op == "learned":
        return _exact_learned(case, seed)
    sizes, d = _sizes(case, seed)
    s = d + 2
    off, total = _layout(sizes, d)
    q = torch.zeros(total, dtype=_dtype(case), device="cuda")
    _fill(q, off, sizes, d, seed)
    q = q.double()
    out = q.clone() if op == "host" else torch.zeros_like(q)
    toff = torch.from_numpy(off).cuda()
    groups = []  # (indices of the patches, element indices, patches)
    for p, idx in _classes(sizes):
        sel = torch.from_numpy(idx).cuda()
        ei = _index(toff[sel], _box(p, d))
        groups.append((sel, ei, q[ei].view([len(idx)] + [p + 2] * d + [s])))

    def put(buf, ei, Q):
        buf[ei] = Q.reshape(len(Q), -1)

    if op in ("update", "host"):
        lam = torch.zeros(len(sizes), dtype=torch.float64, device="cuda")
        for sel, ei, Q in groups:
            box = out[ei].view(Q.shape)
            new, l = _step(Q, _dx(case), _dt(case, d))
            _inner(box).copy_(new)
            put(out, ei, box)
            lam[sel] = l
        if op == "host":
            return [out.cpu()]
        return [out, lam] if case["lam"] else [out]
    if op == "amr":
        return _exact_amr(case, groups[0][2], groups[0][1], q, out)
    if op == "uneven":  # every patch is periodic on its own
        nbrs = [torch.arange(len(Q), device="cuda")[:, None].expand(-1, 6) for _, _, Q in groups]
    else:
        nbrs = [torch.from_numpy(_neighbours(case)).cuda()]
    dx = _dx(case)
    for (_, _, Q), nb in zip(groups, nbrs):
        _halos(Q, nb)
    if op == "engine":
        sel, ei, Q = groups[0]
        lam = _step(Q, dx, 0.0)[1]
        dt = CFL * dx / (d * lam.max().item())
        new, _ = _step(Q, dx, dt)
        put(q, ei, Q)
        box = torch.zeros_like(Q)
        _inner(box).copy_(new)
        put(out, ei, box)
        sums = new.reshape(len(new), -1, s).sum(1)
        return [q, out, lam, torch.tensor([dt], dtype=torch.float64), sums, sums.sum(0)]
    # time steps, ping-pong between the two buffers; halos are gathered from
    # the neighbours, those in the buffers stay as they were
    bufs = [[Q for _, _, Q in groups], [torch.zeros_like(Q) for _, _, Q in groups]]
    nsteps = case["steps"] if op != "step" else (2 if case["carry"] else 1)
    for k in range(nsteps):
        src, dst = bufs[k % 2], bufs[1 - k % 2]
        dt = CFL * dx / (d * max(_max_speed(Q) for Q in src))
        for Q, D, nb in zip(src, dst, nbrs):
            H = Q.clone()
            _halos(H, nb)
            _inner(D).copy_(_step(H, dx, dt)[0])
    last = bufs[nsteps % 2]
    res = torch.zeros_like(q)
    for (_, ei, _), Q in zip(groups, last):
        put(res, ei, Q)
    if case.get("carry"):
        stride = ((d + 3) * case["p"] ** d + 1) // 2 * 2
        return [res, _prim_block(last[0], case, stride)]
    return [res]


def _exact_amr(case, Q, ei, q, out):
    d, p, base = case["d"], case["p"], case["base"]
    level, coord = _tree(case)
    lev = torch.from_numpy(level).cuda()
    co = torch.from_numpy(coord).long().cuda()
    s = d + 2
    nc = 3 ** base * p  # cells per axis of the coarse level

    def cells(sel, lo, hi, m):
        """Linear indices, in a grid of m cells per axis, of the cells with
        local coordinates lo..hi-1 of the selected patches."""
        lin = 0
        for k in reversed(range(d)):
            g = (co[sel][:, k:k + 1] * p + torch.arange(lo, hi, device="cuda")) % m
            lin = lin * m + g.view([len(sel)] + [1] * (d - 1 - k) + [hi - lo] + [1] * k)
        return lin

    ic = torch.nonzero(lev == base).flatten()
    jf = torch.nonzero(lev == base + 1).flatten()
    C = torch.zeros((nc ** d, s), dtype=torch.float64, device="cuda")
    C[cells(ic, 0, p, nc)] = _inner(Q[ic])
    F = C.view([nc] * d + [s])
    for m in range(d):
        F = F.repeat_interleave(3, dim=m)
    F = F.reshape(-1, s)
    F[cells(jf, 0, p, 3 * nc)] = _inner(Q[jf])
    M = F.view([v for _ in range(d) for v in (nc, 3)] + [s])
    C = M.mean(dim=[2 * m + 1 for m in range(d)]).reshape(-1, s)
    H = Q.clone()
    H[ic] = C[cells(ic, -1, p + 1, nc)]
    H[jf] = F[cells(jf, -1, p + 1, 3 * nc)]
    for k in range(d):  # face halos only: edges and corners stay
        ax = d - k
        A, B = Q, H
        for m in range(1, d + 1):
            if m != ax:
                A, B = A.narrow(m, 1, p), B.narrow(m, 1, p)
        for e in (0, p + 1):
            A.select(ax, e).copy_(B.select(ax, e))
    dx = torch.from_numpy(3.0 ** -level / p).cuda()
    new, lam = _step(Q, dx, lambda w, x: CFL * x / (d * w))
    q[ei] = Q.reshape(len(Q), -1)
    box = torch.zeros_like(Q)
    _inner(box).copy_(new)
    out[ei] = box.reshape(len(Q), -1)
    return [q, out, CFL * dx / (d * lam), lam]


def _split(theta):
    shapes = ((64, 16), (64,), (64, 64), (64,), (4, 64), (4,))
    parts, i = [], 0
    for sh in shapes:
        n = int(np.prod(sh))
        parts.append(theta[i:i + n].view(sh))
        i += n
    return parts


def _mlp(theta, x):
    w1, b1, w2, b2, w3, b3 = _split(theta)
    h = torch.nn.functional.gelu(x @ w1.T + b1)
    h = torch.nn.functional.gelu(h @ w2.T + b2)
    return h @ w3.T + b3


def _exact_train(case, seed):
    x, t = (v.double() for v in _samples(case, seed))
    th = _network(seed).double()
    m, v = torch.zeros_like(th), torch.zeros_like(th)
    B, losses = case["batch"], []
    for k in range(1, case["steps"] + 1):
        r0 = (k - 1) % case["nb"] * B
        th = th.detach().requires_grad_(True)
        loss = ((_mlp(th, x[r0:r0 + B]) - t[r0:r0 + B]) ** 2).mean()
        g, = torch.autograd.grad(loss, th)
        losses.append(loss.detach())
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        th = th.detach() - 1e-3 * (m / (1 - 0.9 ** k)) / ((v / (1 - 0.999 ** k)).sqrt() + 1e-8)
    return [th, torch.stack(losses)]


def _exact_learned(case, seed):
    N, p = case["N"], case["p"]
    U = _shear(N, seed).to(_dtype(case)).double()
    theta, norm = _network(seed).double(), _norm(case).double()
    mu, sd, sdy = norm[:16], norm[16:32], norm[32:]
    dt, dx = CFL / N / (2 * 2.5), 1.0 / N
    g = N // p
    corr = torch.zeros((g, g, 2, 4, p + 1, p), dtype=torch.float64, device="cuda")
    new = U.clone()
    for k in (0, 1):
        ax = 1 - k
        swap = [0, 1, 2, 3] if k == 0 else [0, 2, 1, 3]
        V = U[..., swap]
        X = torch.cat([V.roll(sh, ax) for sh in (2, 1, 0, -1)], -1)
        C = torch.cat([_mlp(theta, (c - mu) / sd) for c in X.reshape(-1, 16).split(1 << 18)])
        C = (C.view(N, N, 4) * sdy)[..., swap]  # on the face below each cell
        f, w = _flux(U, k)
        a = torch.maximum(w, w.roll(1, ax))
        F = 0.5 * (f + f.roll(1, ax) - a[..., None] * (U - U.roll(1, ax))) + C
        new -= dt / dx * (F.roll(-1, ax) - F)
        # per patch: faces b = 0..p along k, transverse index fastest
        i = (torch.arange(g, device="cuda")[:, None] * p
             + torch.arange(p + 1, device="cuda")[None, :]) % N
        if k == 0:  # C[y, x]: (b, t, a, face, v) -> (b, a, v, face, t)
            corr[:, :, 0] = C[:, i].view(g, p, g, p + 1, 4).permute(0, 2, 4, 3, 1)
        else:
            corr[:, :, 1] = C[i].view(g, p + 1, g, p, 4).permute(0, 2, 4, 1, 3)
    box = torch.zeros((g * g, p + 2, p + 2, 4), dtype=torch.float64, device="cuda")
    box[:, 1:-1, 1:-1] = new.view(g, p, g, p, 4).permute(0, 2, 1, 3, 4).reshape(g * g, p, p, 4)
    es = 8 if case["prec"] == "fp64" else 4
    L = (p + 2) ** 2 * 4
    stride = -(-L // (32 // es)) * (32 // es)
    out = torch.zeros((g * g, stride), dtype=torch.float64, device="cuda")
    out[:, :L] = box.reshape(g * g, L)
    return [out.reshape(-1), corr.reshape(-1)]
