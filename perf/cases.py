"""The work that programs built on this library have it do, as cases for timing and comparison.

A case is a dict of plain values.  ``listed()`` names twelve of them, ``draw(rng)`` gives more of
the same ranges, ``prepare(case, seed)`` makes a program's inputs on the GPU (matrices, plans,
dense batches), ``run(state)`` takes one pass through the public entry points, ``work(case)``
says what the pass cannot do without and ``exact(case, seed)`` gives the result in 64 bits with
plain torch where that has a fixed layout and takes a few seconds at most.

The matrices are water boxes at 1 g/cc like the repository's workloads: atom blocks (O, H, H per
molecule; 13/5, 23/7 or 4/1 functions), a block wherever two atoms are closer than 8 A, entries
falling off as exp(-0.3 r^2).  "decay" adds 2 to the diagonal; "gapped" replaces the
intra-molecular part by one with 4 levels near -1 and the rest near +1 and scales the coupling so
that every eigenvalue stays 0.25 away from mu = 0 (4 occupied states per molecule).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2003_03868_gb300 as gb

R_CUT, DECAY, BOX_32 = 8.0, 0.3, 9.86
PRECS = {"fp64": gb.DBCSR_FP64, "mixed": gb.DBCSR_MIXED, "bf16x3": gb.DBCSR_BF16X3, "tf32": gb.DBCSR_TF32,
         "tf32x3": gb.DBCSR_TF32X3}


def listed():
    return [
        # the scalars of one SCF step on a small box: Tr(P H), Tr(P) and a spectral bound, each
        # read back by the host; the smallest calls
        {"name": "scalars-32h2o", "kind": "scalars", "n_mol": 32, "o": 13, "h": 5},
        # one product of a small system (N = 736), pattern unknown beforehand
        {"name": "mult-32h2o", "kind": "multiply", "n_mol": 32, "o": 13, "h": 5, "matrix": "decay", "eps": 1e-6,
         "prec": "fp64"},
        # the same size in a loop with a fixed pattern: new values into the planned product
        {"name": "plan-32h2o", "kind": "plan", "n_mol": 32, "o": 13, "h": 5, "eps": 1e-6, "prec": "fp64"},
        # an update C <- 1.5 C - 0.5 A B of a general basis: every block edge from 1 to 32 occurs
        {"name": "ragged-update", "kind": "ragged", "nblk": 160, "density": 0.25, "eps": 1e-3, "prec": "fp64"},
        # the first product of the sign method on 1,024 waters (N = 23,552)
        {"name": "mult-1024h2o", "kind": "multiply", "n_mol": 1024, "o": 13, "h": 5, "matrix": "gapped", "eps": 1e-7,
         "prec": "fp64"},
        # a low-precision product with a large basis (split BF16 on the tensor cores)
        {"name": "mult-bf16x3-512h2o", "kind": "multiply", "n_mol": 512, "o": 23, "h": 7, "matrix": "gapped",
         "eps": 1e-6, "prec": "bf16x3"},
        # density matrix in FP64 throughout, tight filter: the reference run of a study
        {"name": "sign-fp64-512h2o", "kind": "sign", "n_mol": 512, "o": 13, "h": 5, "eps": 1e-7, "tol": 1e-9,
         "prec": "fp64", "order": 2},
        # production density matrix: precision ladder, large basis (N = 75,776), the largest
        {"name": "sign-mixed-2048h2o", "kind": "sign", "n_mol": 2048, "o": 23, "h": 7, "eps": 1e-6, "tol": 1e-8,
         "prec": "mixed", "order": 2},
        # many small systems of uneven sizes solved as one batch
        {"name": "batch-12-small", "kind": "batch", "n_sys": 12, "lo": 20, "hi": 100, "eps": 1e-6, "tol": 1e-9,
         "prec": "mixed"},
        # canonical density matrix without a chemical potential (single-product steps)
        {"name": "purify-tc2-256h2o", "kind": "purify", "n_mol": 256, "o": 13, "h": 5, "eps": 1e-7, "tol": 1e-9,
         "method": "tc2"},
        # the submatrix method with a minimal basis: dense batches on the TF32 tensor cores
        {"name": "submatrix-192h2o", "kind": "submatrix", "n_mol": 192, "o": 4, "h": 1, "tol": 1e-5},
        # batched dense product close to FP32 arithmetic, the size of those submatrices
        {"name": "dense-tf32x3-400", "kind": "dense", "nb": 400, "n": 400, "prec": "tf32x3"},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["scalars", "multiply", "multiply", "plan", "ragged", "sign", "sign", "batch", "purify",
                       "submatrix", "dense"])
    o, h = rng.choice([(13, 5), (23, 7), (13, 7), (23, 5)])
    eps = 10.0 ** rng.uniform(-7.0, -5.0)
    if kind == "scalars":
        return {"kind": kind, "n_mol": log(8, 256), "o": o, "h": h}
    if kind == "multiply":
        return {"kind": kind, "n_mol": log(9, 700), "o": o, "h": h, "matrix": rng.choice(["decay", "gapped"]),
                "eps": rng.choice([eps, eps, 0.0]) if o == 13 else eps, "prec": rng.choice(["fp64", "fp64", "bf16x3"])}
    if kind == "plan":
        return {"kind": kind, "n_mol": log(8, 120), "o": o, "h": h, "eps": eps,
                "prec": rng.choice(["fp64", "fp64", "bf16x3"])}
    if kind == "ragged":
        return {"kind": kind, "nblk": rng.randint(20, 240), "density": rng.uniform(0.05, 0.5),
                "eps": rng.choice([0.0, 1e-3, 1e-1]), "prec": "fp64"}
    if kind == "sign":
        return {"kind": kind, "n_mol": log(16, 300), "o": o, "h": h, "eps": eps, "tol": 1e-8,
                "prec": rng.choice(["fp64", "mixed"]), "order": rng.choice([2, 2, 3, 5])}
    if kind == "batch":
        return {"kind": kind, "n_sys": rng.randint(2, 16), "lo": 10, "hi": rng.randint(30, 100), "eps": eps,
                "tol": 1e-9, "prec": rng.choice(["fp64", "mixed"])}
    if kind == "purify":
        return {"kind": kind, "n_mol": log(16, 300), "o": o, "h": h, "eps": eps, "tol": 1e-9,
                "method": rng.choice(["tc2", "trs4"])}
    if kind == "submatrix":
        return {"kind": kind, "n_mol": log(24, 220), "o": 4, "h": 1, "tol": 1e-5}
    prec = rng.choice(["tf32", "tf32x3", "fp64"])
    return {"kind": kind, "nb": log(4, 400) if prec != "fp64" else log(2, 60), "n": rng.randint(60, 500), "prec": prec}


# ------------------------------------------------------------------ inputs
def _rng(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + salt) % (1 << 62))
    return g


def _u(g, *shape):
    return torch.rand(*shape, dtype=torch.float64, device="cuda", generator=g)


class _Blocks:
    """Block-CSR arrays: row pointers and columns on the host, values on the GPU."""

    def __init__(self, bs, rows, cols, data):
        self.bs = np.ascontiguousarray(bs, dtype=np.int32)
        self.rows = np.ascontiguousarray(rows, dtype=np.int32)
        self.cols = np.ascontiguousarray(cols, dtype=np.int32)
        self.rp = np.zeros(len(self.bs) + 1, dtype=np.int64)
        np.cumsum(np.bincount(self.rows, minlength=len(self.bs)), out=self.rp[1:])
        self.data = data

    def matrix(self):
        torch.cuda.current_stream().synchronize()
        return gb.Matrix.from_blocks(self.bs, self.rp, self.cols, None, on_device=True, data_ptr=self.data.data_ptr())

    def dense(self):
        return _dense(self.bs, self.rows, self.cols, self.data)


def _offsets(bs, rows, cols):
    area = bs[rows].astype(np.int64) * bs[cols].astype(np.int64)
    off = np.zeros(len(area) + 1, dtype=np.int64)
    np.cumsum(area, out=off[1:])
    return off


def _classes(bs, rows, cols):
    """(m, n, block indices) for every block shape that occurs."""
    key = bs[rows].astype(np.int64) * 64 + bs[cols]
    order = np.argsort(key, kind="stable")
    ks, first = np.unique(key[order], return_index=True)
    for k, sel in zip(ks, np.split(order, first[1:])):
        yield int(k) // 64, int(k) % 64, sel


def _dense(bs, rows, cols, data):
    start = np.zeros(len(bs) + 1, dtype=np.int64)
    np.cumsum(bs, out=start[1:])
    n = int(start[-1])
    off = _offsets(bs, rows, cols)
    out = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    for m, k, sel in _classes(bs, rows, cols):
        i = torch.from_numpy(start[rows[sel]]).cuda()[:, None, None] + torch.arange(m, device="cuda")[None, :, None]
        j = torch.from_numpy(start[cols[sel]]).cuda()[:, None, None] + torch.arange(k, device="cuda")[None, None, :]
        o = torch.from_numpy(off[sel]).cuda()[:, None] + torch.arange(m * k, device="cuda")[None, :]
        out[i, j] = data[o].reshape(-1, m, k)
    return out


def _water(n_mol, basis, seed, matrix):
    """A water box's matrix ("decay", "gapped")."""
    g = _rng(seed, 1)
    box = BOX_32 * (n_mol / 32.0) ** (1.0 / 3.0)
    # molecules on randomly chosen, jittered cells of a cubic grid, numbered in random order
    grid = int(math.ceil(n_mol ** (1.0 / 3.0) - 1e-9))
    site = torch.argsort(_u(g, grid ** 3))[:n_mol]
    cell = torch.stack([site // (grid * grid), (site // grid) % grid, site % grid], 1).double()
    oxy = (cell + 0.5 + 0.24 * (_u(g, n_mol, 3) - 0.5)) * (box / grid)
    # rigid water, two orthonormal random directions
    e1 = torch.randn(n_mol, 3, dtype=torch.float64, device="cuda", generator=g)
    e1 = e1 / e1.norm(dim=1, keepdim=True)
    e2 = torch.randn(n_mol, 3, dtype=torch.float64, device="cuda", generator=g)
    e2 = e2 - (e2 * e1).sum(1, keepdim=True) * e1
    e2 = e2 / e2.norm(dim=1, keepdim=True)
    half = math.radians(104.52) / 2
    pos = torch.stack([oxy, oxy + 0.9572 * (math.sin(half) * e1 + math.cos(half) * e2),
                       oxy + 0.9572 * (-math.sin(half) * e1 + math.cos(half) * e2)], 1).reshape(-1, 3)
    na = 3 * n_mol
    r2 = torch.zeros(na, na, dtype=torch.float64, device="cuda")
    for ax in range(3):
        d = pos[:, None, ax] - pos[None, :, ax]
        d -= box * torch.round(d / box)
        r2 += d * d
    near = r2 < R_CUT * R_CUT
    near.fill_diagonal_(True)
    rows_t, cols_t = near.nonzero(as_tuple=True)
    fac = torch.exp(-DECAY * r2[rows_t, cols_t])
    del r2, near, d
    key = rows_t * na + cols_t
    twin = torch.searchsorted(key, cols_t * na + rows_t)
    bs = np.tile(np.array([basis[0], basis[1], basis[1]], dtype=np.int32), n_mol)
    rows, cols = rows_t.cpu().numpy(), cols_t.cpu().numpy()
    off = _offsets(bs, rows, cols)
    off_t = torch.from_numpy(off).cuda()
    data = torch.empty(int(off[-1]), dtype=torch.float64, device="cuda")
    rowsum = torch.zeros(na, 32, dtype=torch.float64, device="cuda")
    for m, n, sel_np in _classes(bs, rows, cols):
        sel = torch.from_numpy(sel_np).cuda()
        sel = sel[rows_t[sel] <= cols_t[sel]]
        for part in torch.split(sel, max(1, (1 << 25) // (m * n))):
            v = (2.0 * _u(g, len(part), m, n) - 1.0) * fac[part][:, None, None]
            diag = rows_t[part] == cols_t[part]
            if m == n:
                v = torch.where(diag[:, None, None], 0.5 * (v + v.transpose(1, 2)), v)
                if matrix == "decay":
                    v = v + diag.double()[:, None, None] * 2.0 * torch.eye(m, dtype=torch.float64, device="cuda")
            e = torch.arange(m * n, device="cuda")
            data[(off_t[part][:, None] + e).reshape(-1)] = v.reshape(-1)
            data[(off_t[twin[part]][:, None] + e).reshape(-1)] = v.transpose(1, 2).reshape(-1)
            inter = (rows_t[part] // 3 != cols_t[part] // 3).double()[:, None]
            rowsum[:, :m].index_add_(0, rows_t[part], v.abs().sum(2) * inter)
            rowsum[:, :n].index_add_(0, cols_t[part], v.abs().sum(1) * inter)
    if matrix == "gapped":
        gmax = float(rowsum.max())
        if gmax > 0:
            data *= float(np.float32(0.5 / gmax))             # rounded: the sums above vary in the last bit
        # intra-molecular part: 4 levels near -1, the others near +1, in random orthogonal bases
        d = basis[0] + 2 * basis[1]
        level = torch.cat([-1.0 + 0.25 * torch.linspace(-1, 1, 4, dtype=torch.float64),
                           1.0 + 0.25 * torch.linspace(-1, 1, max(d - 4, 1), dtype=torch.float64)[:d - 4]]).cuda()
        mol = torch.diag_embed(level.expand(n_mol, d).contiguous())
        for _ in range(3):
            w = torch.randn(n_mol, d, 1, dtype=torch.float64, device="cuda", generator=g)
            q = torch.eye(d, dtype=torch.float64, device="cuda") - 2.0 * w @ w.transpose(1, 2) / (w * w).sum(1, True)
            mol = q @ mol @ q
        mol = 0.5 * (mol + mol.transpose(1, 2))
        loc = [0, basis[0], basis[0] + basis[1], d]
        for a in range(3):
            for b in range(3):
                i = torch.arange(n_mol, device="cuda")
                at = torch.searchsorted(key, (3 * i + a) * na + 3 * i + b)
                blk = mol[:, loc[a]:loc[a + 1], loc[b]:loc[b + 1]].reshape(n_mol, -1)
                e = torch.arange(blk.shape[1], device="cuda")
                data[(off_t[at][:, None] + e).reshape(-1)] = blk.reshape(-1)
    return _Blocks(bs, rows, cols, data)


def _ragged_sizes(nblk):
    """Every block edge from 1 to 32, shuffled."""
    return np.random.default_rng(nblk).permutation(np.arange(nblk) % 32 + 1).astype(np.int32)


def _ragged(nblk, density, seed, salt):
    """Blocks present at random, the diagonal kept."""
    r = np.random.default_rng([int(seed), salt])
    bs = _ragged_sizes(nblk)
    present = r.random((nblk, nblk)) < density
    np.fill_diagonal(present, True)
    rows, cols = np.nonzero(present)
    n = int(_offsets(bs, rows, cols)[-1])
    # block norms over several orders of magnitude, as a filtered matrix has them
    scale = torch.from_numpy(10.0 ** r.uniform(-4.0, 0.0, len(rows))).cuda()
    area = torch.from_numpy(np.diff(_offsets(bs, rows, cols))).cuda()
    data = (2.0 * _u(_rng(seed, salt), n) - 1.0) * torch.repeat_interleave(scale, area)
    return _Blocks(bs, rows, cols, data)


def _batch_sizes(case):
    """(molecules, O block, H block) of every system of a batch: log-uniform sizes, mixed bases."""
    r = np.random.default_rng([case["n_sys"], case["lo"], case["hi"]])
    return [(int(round(math.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]))))), int(r.choice([13, 23])),
             int(r.choice([5, 7]))) for _ in range(case["n_sys"])]


def _dense_inputs(case, seed):
    g = _rng(seed, 5)
    nb, n = case["nb"], case["n"]
    dt = torch.float64 if case["prec"] == "fp64" else torch.float32
    # matrices like the submatrices: a strong diagonal and small couplings
    A = ((_u(g, nb, n, n) - 0.5) * (2.0 / math.sqrt(n)) + torch.eye(n, dtype=torch.float64, device="cuda")).to(dt)
    B = ((_u(g, nb, n, n) - 0.5) * (2.0 / math.sqrt(n)) + torch.eye(n, dtype=torch.float64, device="cuda")).to(dt)
    return A, B


def prepare(case, seed):
    k = case["kind"]
    s = {"case": case}
    if k == "dense":
        s["A"], s["B"] = _dense_inputs(case, seed)
        s["C"] = torch.empty_like(s["A"])
    elif k == "ragged":
        s["A"], s["B"], s["C0"] = (_ragged(case["nblk"], case["density"], seed, t).matrix() for t in (1, 2, 3))
        s["out"] = _buffers(case["nblk"], *_room(case))
    elif k == "batch":
        sizes = _batch_sizes(case)
        s["H"] = [_water(n, (o, h), seed * 100 + i, "gapped").matrix() for i, (n, o, h) in enumerate(sizes)]
        s["out"] = [_buffers(3 * n, *_room(case, n, o, h)) for n, o, h in sizes]
    else:
        b = _water(case["n_mol"], (case["o"], case["h"]), seed,
                   case.get("matrix", "decay" if k == "plan" else "gapped"))
        s["H"] = b.matrix()
        if k == "scalars":
            p = _water(case["n_mol"], (case["o"], case["h"]), seed + 500009, "gapped")
            s["P"] = p.matrix()
        else:
            s["out"] = _buffers(3 * case["n_mol"], *_room(case, case["n_mol"], case["o"], case["h"]))
        if k == "plan":
            s["C"] = gb.Matrix(b.bs)
            s["plan"] = gb.Plan(1.0, s["H"], s["H"], s["C"], case["eps"], PRECS[case["prec"]])
            s["values"] = b.data
            torch.cuda.current_stream().synchronize()
    return s


# ------------------------------------------------------------------ one pass
def _room(case, n_mol=0, o=0, h=0):
    """Room for the blocks and values of a result: the same for every input of the case."""
    if case["kind"] == "ragged":
        n = int(_ragged_sizes(case["nblk"]).sum())
        return case["nblk"] ** 2, n * n
    nblk, n = 3 * n_mol, n_mol * (o + 2 * h)
    eps = case.get("eps", 1.0)
    if case["kind"] == "submatrix":
        reach = 1.0                                           # the pattern of H
    elif eps == 0.0 or case["kind"] == "plan":
        reach = 9.0                                           # every pair within 16 A
    else:
        reach = max(0.7, 0.95 + 0.55 * math.log10(1e-6 / eps)) * (2.0 if case.get("matrix") == "decay" else 1.0)
    blocks = min(nblk * nblk, int(nblk * 240 * reach))
    return blocks, min(n * n, int(1.05 * blocks * ((o + 2 * h) / 3.0) ** 2) + 1024)


def _buffers(nblk, blocks, values):
    """Pinned host buffers that a program keeps for a result of at most this size."""
    return {"rp": torch.zeros(nblk + 1, dtype=torch.int64).pin_memory(),
            "col": torch.zeros(blocks, dtype=torch.int32).pin_memory(),
            "data": torch.zeros(values, dtype=torch.float64, pin_memory=True)}


def _out(M, b):
    """The matrix in the program's host buffers (whole buffers; the matrix fills their front)."""
    M.export_to(b["rp"].data_ptr(), b["col"].data_ptr(), b["col"].numel(), b["data"].data_ptr(), b["data"].numel())
    return b


def run(s):
    c = s["case"]
    k = c["kind"]
    if k == "scalars":
        return {"e_band": gb.trace_product(s["P"], s["H"]), "trace": gb.trace(s["P"]),
                "bound": gb.gershgorin(s["H"], 0.0)}
    if k == "multiply":
        C = gb.Matrix(s["H"].blk_size)
        gb.multiply(1.0, s["H"], s["H"], 0.0, C, c["eps"], PRECS[c["prec"]], stats=False)
        return _out(C, s["out"])
    if k == "plan":
        s["H"].put_values(s["values"].data_ptr())
        s["plan"].execute()
        return _out(s["C"], s["out"])
    if k == "ragged":
        C = s["C0"].copy()
        gb.multiply(-0.5, s["A"], s["B"], 1.5, C, c["eps"], PRECS[c["prec"]], stats=False)
        return _out(C, s["out"])
    if k == "sign":
        r = gb.sign_iterate(s["H"], 0.0, c["eps"], c["tol"], prec=PRECS[c["prec"]], order=c["order"])
    elif k == "purify":
        r = gb.purify(s["H"], 4 * c["n_mol"], c["eps"], c["tol"], method=c["method"])
    elif k == "submatrix":
        r = gb.submatrix_sign(s["H"], 0.0, c["tol"], prec=gb.DBCSR_MIXED)
    elif k == "batch":
        Ps, reps, _ = gb.sign_iterate_batched(s["H"], [0.0] * len(s["H"]), c["eps"], c["tol"], prec=PRECS[c["prec"]])
        return {"P": [_out(P, b) for P, b in zip(Ps, s["out"])],
                "e_band": np.array([x.e_band for x in reps]), "steps": np.array([x.iterations for x in reps])}
    elif k == "dense":
        gb.dense_multiply(PRECS[c["prec"]], c["nb"], c["n"], 1.0, s["A"].data_ptr(), s["B"].data_ptr(), 0.0,
                          s["C"].data_ptr())
        return {"C": s["C"]}
    return {"P": _out(r.P, s["out"]), "e_band": float(r.report.e_band), "steps": int(r.report.iterations)}


# ------------------------------------------------------------------ what it cannot do without
def _water_size(n_mol, o, h):
    """(blocks, elements, mean block edge, neighbours per atom) of a water box's matrix."""
    near = min(3.0 * n_mol, 215.0)              # atoms within 8 A at 1 g/cc
    blocks = 3.0 * n_mol * near
    edge = (o + 2.0 * h) / 3.0
    return blocks, blocks * edge * edge, edge, near


def work(case):
    """Inputs read once, outputs written once; the flops of the block products that reach the
    filter (for a filtered product of two 8 A matrices about 0.44 of the pattern's), once per
    product of an iteration, a symmetric one counted half."""
    k = case["kind"]
    if k == "dense":
        e = 8 if case["prec"] == "fp64" else 4
        nb, n = case["nb"], case["n"]
        return {"bytes": 3.0 * e * nb * n * n, "flops": 2.0 * nb * n ** 3}
    if k == "ragged":
        n, d = case["nblk"], case["density"]
        return {"bytes": 8.0 * n * n * 16.5 ** 2 * (3 * d + 1), "flops": 2.0 * d * d * (n * 16.5) ** 3}
    if k == "batch":
        mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        one = work({"kind": "sign", "n_mol": mean, "o": 18, "h": 6, "order": 2, "prec": case["prec"],
                    "eps": case["eps"]})
        return {"bytes": case["n_sys"] * one["bytes"], "flops": case["n_sys"] * one["flops"]}
    blocks, el, edge, near = _water_size(case["n_mol"], case["o"], case["h"])
    if k == "scalars":
        return {"bytes": 24.0 * el, "flops": 4.0 * el}
    filtered = 1.0 if case.get("eps", 1.0) == 0.0 or near < 215 else 0.44
    product = 2.0 * filtered * blocks * near * edge ** 3
    if k in ("multiply", "plan"):
        return {"bytes": 16.0 * el, "flops": product}
    if k == "submatrix":
        n = near * edge
        return {"bytes": 16.0 * el, "flops": 3.0 * case["n_mol"] * 20 * 2 * 2.0 * n ** 3}
    products = {"tc2": 19, "trs4": 18}[case["method"]] if k == "purify" else 20
    return {"bytes": 16.0 * el, "flops": products * 0.5 * product}


# ------------------------------------------------------------------ 64 bits
def _blocked(bs, D, keep, room):
    """Blocks (I, J) with keep[I, J] of the dense D as block-CSR arrays, in buffers of that room."""
    rows, cols = np.nonzero(keep)
    start = np.zeros(len(bs) + 1, dtype=np.int64)
    np.cumsum(bs, out=start[1:])
    off = _offsets(bs, rows, cols)
    data = torch.zeros(room[1], dtype=torch.float64, device=D.device)
    for m, n, sel in _classes(bs, rows, cols):
        i = torch.from_numpy(start[rows[sel]]).cuda()[:, None, None] + torch.arange(m, device="cuda")[None, :, None]
        j = torch.from_numpy(start[cols[sel]]).cuda()[:, None, None] + torch.arange(n, device="cuda")[None, None, :]
        o = torch.from_numpy(off[sel]).cuda()[:, None] + torch.arange(m * n, device="cuda")[None, :]
        data[o.reshape(-1)] = D[i, j].reshape(-1)
    rp = np.zeros(len(bs) + 1, dtype=np.int64)
    np.cumsum(np.bincount(rows, minlength=len(bs)), out=rp[1:])
    col = np.zeros(room[0], dtype=np.int32)
    col[:len(cols)] = cols
    return {"rp": rp, "col": col, "data": data}


def _block_norms(bs, D):
    of = torch.from_numpy(np.repeat(np.arange(len(bs)), bs)).cuda()
    s = torch.zeros(len(bs), D.shape[1], dtype=torch.float64, device="cuda").index_add_(0, of, D * D)
    return torch.zeros(len(bs), len(bs), dtype=torch.float64, device="cuda").index_add_(1, of, s).sqrt().cpu().numpy()


def _pattern(b):
    p = np.zeros((len(b.bs), len(b.bs)), dtype=bool)
    p[b.rows, b.cols] = True
    return p


def exact(case, seed):
    k = case["kind"]
    if k == "dense":
        A, B = _dense_inputs(case, seed)
        return {"C": torch.matmul(A.double(), B.double())}
    if k == "ragged":
        a, b, c = (_ragged(case["nblk"], case["density"], seed, t) for t in (1, 2, 3))
        D = 1.5 * c.dense() - 0.5 * torch.matmul(a.dense(), b.dense())
        cand = (_pattern(a).astype(np.float32) @ _pattern(b).astype(np.float32) > 0) | _pattern(c)
        keep = cand & ((_block_norms(a.bs, D) >= case["eps"]) | np.eye(len(a.bs), dtype=bool))
        return _blocked(a.bs, D, keep, _room(case))
    if k == "scalars":
        h = _water(case["n_mol"], (case["o"], case["h"]), seed, "gapped").dense()
        p = _water(case["n_mol"], (case["o"], case["h"]), seed + 500009, "gapped").dense()
        return {"e_band": float((p * h.T).sum()), "trace": float(p.trace()), "bound": float(h.abs().sum(1).max())}
    if k in ("multiply", "plan") and case["n_mol"] * (case["o"] + 2 * case["h"]) <= 8000:
        a = _water(case["n_mol"], (case["o"], case["h"]), seed, case.get("matrix", "decay"))
        d = a.dense()
        D = torch.matmul(d, d)
        cand = _pattern(a).astype(np.float32) @ _pattern(a).astype(np.float32) > 0
        eye = np.eye(len(a.bs), dtype=bool)
        room = _room(case, case["n_mol"], case["o"], case["h"])
        if k == "multiply":
            return _blocked(a.bs, D, cand & ((_block_norms(a.bs, D) >= case["eps"]) | eye), room)
        # a planned product keeps every block that may reach the filter; smaller ones become zero
        nrm = _block_norms(a.bs, d)
        bound = nrm @ nrm
        if np.any((bound > 0.9 * case["eps"]) & (bound < 1.1 * case["eps"])):
            return None
        small = torch.from_numpy((_block_norms(a.bs, D) < case["eps"]) & ~eye).cuda()
        of = torch.from_numpy(np.repeat(np.arange(len(a.bs)), a.bs)).cuda()
        D = torch.where(small[of][:, of], torch.zeros((), dtype=torch.float64, device="cuda"), D)
        return _blocked(a.bs, D, cand & ((bound >= case["eps"]) | eye), room)
    # a density matrix has the pattern that the iteration's filter leaves
    return None
