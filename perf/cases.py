"""What users of the framework have it do, as cases that can be timed and compared.

A linear-scaling solve spends its time in masked block products (FP64, split-BF16 and
emulated FP64, on uniform and on mixed bases), in the drivers that string them together
(Hotelling inversion, LNV steps), in traces over large patterns, and, with the learned start,
in training a small network and applying it to a cell.  Each case is one of these through the
binding's public calls.  Sizes are the ones of the repository's own tests and benchmark:
diamond silicon cells (a = 10.26 bohr) of 64 to 4096 atoms with 4 or 9 orbitals per atom,
ranges 10/12 (sp) and 14/16 bohr (SZP), and the four mixed-species cells of the batched
benchmark.

`exact` is plain torch in 64 bits: dense masked products, a dense LNV iteration, the network
written out; it shares with `prepare` only the inputs.
"""
import math

import numpy as np
import torch

from paper_2205_08941_gb300 import cq
from paper_2205_08941_gb300 import inputs as I

DEV = "cuda:0"
F64 = torch.float64
PREC = {"fp64": cq.CQ_FP64, "split": cq.CQ_SPLIT_BF16X3, "emu": cq.CQ_FP64_EMU}
# lattice, density (atoms per cubic angstrom) and r_L of the batched benchmark's cells
BATCH = [((3, 3, 3), 0.05, 14.0), ((4, 3, 3), 0.03, 16.0), ((4, 4, 3), 0.06, 12.0),
         ((4, 4, 4), 0.045, 15.0)]
# operand and result patterns of the three products of an LNV evaluation, as multiples of
# (r_S, r_L): X = L.S, U = S.X, R = U.X kept on P_L
PRODUCTS = {"LSX": ((0, 1), (1, 0), (1, 1)), "SXU": ((1, 0), (1, 1), (2, 1)),
            "UXL": ((2, 1), (1, 1), (0, 1))}
N_IN, N_OUT, DIMS = 64, 81, (64, 256, 256, 256, 81)


def _product(name, cells, norb, prod, prec):
    return {"name": name, "kind": "product", "cells": cells, "norb": norb, "prod": prod,
            "prec": prec}


def listed():
    return [
        # the smallest call: one product of a 64-atom sp cell, as the quick tests and every
        # small molecule-sized system run it; latency counts
        _product("product fp64 si64 L.S", "2x2x2", 4, "LSX", "fp64"),
        # the batched benchmark's four mixed-species cells (5/9/13 orbitals), FP64
        _product("product fp64 batch S.X", "batch4", 0, "SXU", "fp64"),
        # one of the two long products of a mixed-precision step on the 512-atom SZP cell
        _product("product split si512 S.X", "4x4x4", 9, "SXU", "split"),
        # the product that dominates the step of the 4096-atom SZP benchmark cell
        _product("product split si4096 U.X", "8x8x8", 9, "UXL", "split"),
        # the same kind of product on the batched mixed-species cells
        _product("product split batch U.X", "batch4", 0, "UXL", "split"),
        # FP64-accurate products on the tensor cores (emulated), 512-atom SZP cell
        _product("product emu si512 U.X", "4x4x4", 9, "UXL", "emu"),
        # overlap inversion of a 216-atom SZP cell: the start and the first Hotelling steps
        {"name": "hotelling si216", "kind": "hotelling", "cells": "3x3x3", "norb": 9, "steps": 3},
        # a whole call: LNV object and two mixed-precision steps on the 512-atom SZP cell
        {"name": "lnv split si512", "kind": "lnv", "cells": "4x4x4", "norb": 9, "prec": "split",
         "steps": 2},
        # a whole call on the 64-atom sp cell in FP64: many short launches and host reads
        {"name": "lnv fp64 si64", "kind": "lnv", "cells": "2x2x2", "norb": 4, "prec": "fp64",
         "steps": 4},
        # training the learned start: minibatches of the benchmark's size
        {"name": "learned train 4096", "kind": "train", "rows": 4096, "batches": 8},
        # applying it: descriptors, network and rotation of every pair of a 1728-atom cell
        {"name": "learned apply si1728", "kind": "apply", "cells": "6x6x6", "norb": 9},
        # Tr(XY) and <X, Y> over the 30-bohr pattern of the 4096-atom cell: memory-bound
        {"name": "traces si4096", "kind": "trace", "cells": "8x8x8", "norb": 9},
    ]


def _cells_up_to(rng, lo, hi):
    """A box of nx x ny x nz conventional cells whose atom count is spread over [lo, hi] by
    its logarithm (anisotropic boxes among them)."""
    target = math.exp(rng.uniform(math.log(lo), math.log(hi))) / 8.0
    while True:
        n = [max(1, min(8, round(target ** (1 / 3.0) * math.exp(rng.uniform(-0.4, 0.4)))))
             for _ in range(3)]
        if lo <= 8 * n[0] * n[1] * n[2] <= hi and min(n) >= 2:
            return "x".join(str(v) for v in n)


def draw(rng):
    kind = rng.choice(["product", "product", "product", "hotelling", "lnv", "train", "apply",
                       "trace"])
    norb = rng.choice([4, 9, 9])
    if kind == "product":
        prec = rng.choice(["fp64", "split", "split", "emu"])
        prod = rng.choice(["LSX", "SXU", "UXL"])
        if prec != "emu" and rng.random() < 0.25:
            # a batch of 2 to 4 mixed-species cells drawn like the benchmark's
            n = rng.randint(2, 4)
            cells = "mixed:" + ";".join(
                "%s,%.4f,%.2f" % (_cells_up_to(rng, 64, 512), rng.uniform(0.03, 0.06),
                                  rng.uniform(12.0, 16.0)) for _ in range(n))
            return {"kind": kind, "cells": cells, "norb": 0, "prod": prod, "prec": prec}
        hi = {"fp64": 512, "emu": 512, "split": 1728}[prec]
        return {"kind": kind, "cells": _cells_up_to(rng, 64, hi), "norb": norb, "prod": prod,
                "prec": prec}
    if kind == "hotelling":
        return {"kind": kind, "cells": _cells_up_to(rng, 64, 320), "norb": norb,
                "steps": rng.randint(1, 4)}
    if kind == "lnv":
        prec = rng.choice(["fp64", "split", "split", "emu"])
        return {"kind": kind, "cells": _cells_up_to(rng, 64, 512 if prec == "split" else 128),
                "norb": norb, "prec": prec, "steps": rng.randint(1, 3)}
    if kind == "train":
        return {"kind": kind, "rows": int(math.exp(rng.uniform(math.log(64), math.log(8192)))),
                "batches": rng.randint(1, 8)}
    return {"kind": kind, "cells": _cells_up_to(rng, 64, 1728 if kind == "apply" else 4096),
            "norb": norb}


# ------------------------------------------------------------------ inputs (both sides)

def _geometry(case):
    """The cells of a case: [(inputs.Cell, r_S, r_L)].  The atoms are the case's own; a seed
    gives other values on the same patterns, as successive iterates and models do."""
    if case["cells"].startswith(("batch", "mixed")):
        if case["cells"] == "batch4":
            spec = BATCH
        else:
            spec = []
            for part in case["cells"][6:].split(";"):
                n, dens, rl = part.split(",")
                spec.append((tuple(int(v) for v in n.split("x")), float(dens), float(rl)))
        return [(I.mixed_cell(n, dens, 0.1, 3 + k), rl - 2.0, rl)
                for k, (n, dens, rl) in enumerate(spec)]
    n = tuple(int(v) for v in case["cells"].split("x"))
    rs, rl = (10.0, 12.0) if case["norb"] == 4 else (14.0, 16.0)
    return [(I.diamond_cell(n, a=10.26, sigma=0.1, seed=2, norb=case["norb"]), rs, rl)]


def _range(mult, rs, rl):
    return mult[0] * rs + mult[1] * rl


class _Blocks:
    """Blocks of a range-cutoff pattern in the layout of include/cq.h: pairs (i, j) with
    minimum-image distance below the range (and i == j), by row then column, each block
    row-major and padded to an even length."""

    def __init__(self, cells, mult):
        ii, jj, dd, nbs, base = [], [], [], [], 0
        for cell, rs, rl in cells:
            r = _range(mult, rs, rl)
            pos = torch.tensor(cell.pos, device=DEV)
            box = torch.tensor(cell.box, device=DEV)
            n = pos.shape[0]
            for s in range(0, n, 512):
                d = pos[None, :, :] - pos[s:s + 512, None, :]
                d = d - box * torch.round(d / box)
                d2 = (d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2]
                keep = d2 < r * r
                rows = torch.arange(s, min(n, s + 512), device=DEV)
                keep[rows - s, rows] = True
                i, j = torch.nonzero(keep, as_tuple=True)
                ii.append(i + s + base)
                jj.append(j + base)
                dd.append(torch.sqrt(d2[i, j]))
            nbs.append(torch.tensor(cell.nb.astype(np.int64), device=DEV))
            base += n
        self.i, self.j, self.dist = torch.cat(ii), torch.cat(jj), torch.cat(dd)
        self.nb = torch.cat(nbs)
        self.n_orb = int(self.nb.sum())
        size = self.nb[self.i] * self.nb[self.j]
        self.uniform = int(self.nb[0]) if bool((self.nb == self.nb[0]).all()) else 0
        self.pad = (size + 1) // 2 * 2
        self.off = torch.zeros(size.shape[0] + 1, dtype=torch.int64, device=DEV)
        torch.cumsum(self.pad, 0, out=self.off[1:])
        self.n_values = int(self.off[-1])
        self.size = size

    def random(self, seed, decay=4.0):
        """N(0, 1) exp(-r / decay) values: the decay of the solver's matrices."""
        gen = torch.Generator(device=DEV)
        gen.manual_seed(seed)
        v = torch.randn(self.n_values, dtype=F64, device=DEV, generator=gen)
        w = torch.exp(-self.dist / decay)
        if self.uniform:
            u = v.view(-1, int(self.pad[0]))
            u *= w[:, None]
            u[:, self.uniform * self.uniform:] = 0.0
            return v
        v *= torch.repeat_interleave(w, self.pad)
        v[(self.off[:-1] + self.size)[self.pad != self.size]] = 0.0
        return v

    def places(self, start=0, end=None):
        """(value index, scalar row, scalar column) of every value of blocks start..end."""
        orb = torch.cumsum(self.nb, 0) - self.nb
        end = self.i.shape[0] if end is None else end
        i, j, size = self.i[start:end], self.j[start:end], self.size[start:end]
        blk = torch.repeat_interleave(torch.arange(i.shape[0], device=DEV), size)
        first = torch.cumsum(size, 0) - size
        e = torch.arange(blk.shape[0], device=DEV) - first[blk]
        nj = self.nb[j][blk]
        return (self.off[start:end][blk] + e, orb[i][blk] + e // nj, orb[j][blk] + e % nj)

    def dense(self, values):
        m = torch.zeros(self.n_orb * self.n_orb, dtype=F64, device=DEV)
        step = 1 << 20
        for s in range(0, self.i.shape[0], step):
            at, r, c = self.places(s, min(self.i.shape[0], s + step))
            m[r * self.n_orb + c] = values[at]
        return m.view(self.n_orb, self.n_orb)

    def values(self, m):
        out = torch.zeros(self.n_values, dtype=F64, device=DEV)
        at, r, c = self.places()
        out[at] = m[r, c]
        return out

    def masked(self, m):
        out = torch.zeros_like(m)
        _, r, c = self.places()
        out[r, c] = m[r, c]
        return out

    def from_pairs(self, pb):
        """Values of an inputs.PairBlocks list whose pairs are those of this pattern."""
        out = torch.zeros(self.n_values, dtype=F64, device=DEV)
        at, _, _ = self.places()
        out[at] = torch.tensor(pb.values, device=DEV)
        return out


def _patterns(ctx, cells, *mults):
    pos, nb, start, boxes = I.concat_cells([c[0] for c in cells])
    pos_d = torch.tensor(pos, device=DEV)
    nb_d = torch.tensor(nb, dtype=torch.int32, device=DEV)
    out = []
    for m in mults:
        r = [_range(m, rs, rl) for _, rs, rl in cells]
        out.append(ctx.pattern(pos_d, boxes[0], nb_d, r[0]) if len(cells) == 1 else
                   ctx.pattern_batch(pos_d, start, boxes, nb_d, r))
    return out


def _overlap_hamiltonian(cells, seed):
    """S and H of the two-centre model, its bond integrals scaled by up to 3 % each, and the
    number of electrons (4 per atom)."""
    cell, rs, _ = cells[0]
    model, rng = I.silicon_model(rs), np.random.default_rng(seed)
    for par in (model.v, model.s):
        for key in par:
            par[key] *= rng.uniform(0.97, 1.03)
    S, H = I.overlap_hamiltonian(cell, model)
    b = _Blocks(cells, (1, 0))
    return b, b.from_pairs(S), b.from_pairs(H), 4.0 * cell.n_atoms


def _pm_start(cells, seed):
    """S, H and the Palser-Manolopoulos start L0, from dense algebra in plain torch."""
    bS, S, H, ne = _overlap_hamiltonian(cells, seed)
    bL = _Blocks(cells, (0, 1))
    s, h = bS.dense(S), bS.dense(H)
    t = torch.linalg.inv(s)
    t = 0.5 * (t + t.T)
    th = t @ h
    n, occ = bS.n_orb, ne / 2.0
    mu = torch.trace(th) / n
    diag = torch.diagonal(th)
    rad = th.abs().sum(1) - diag.abs()
    lam = torch.minimum(occ / ((diag + rad).max() - mu), (n - occ) / (mu - (diag - rad).min()))
    l0 = (lam / n) * (mu * t - th @ t) + (occ / n) * t
    return bS, S, H, bL, bL.values(0.5 * (l0 + l0.T)), ne


def _weights(seed):
    """Network weights and biases (layer by layer, row-major in x out) at the scale of a
    He-style start, and per-column scales of the network's outputs."""
    rng = np.random.default_rng(seed)
    w = [rng.normal(0.0, math.sqrt(2.0 / DIMS[l]), DIMS[l] * DIMS[l + 1]) for l in range(4)]
    b = [rng.normal(0.0, 0.02, DIMS[l + 1]) for l in range(4)]
    return (np.concatenate(w).astype(np.float32), np.concatenate(b).astype(np.float32))


def _scales(seed):
    rng = np.random.default_rng(seed)
    f = lambda x: x.astype(np.float32)
    return (f(rng.uniform(0.0, 1.0, N_IN)), f(rng.uniform(0.5, 2.0, N_IN)),
            f(rng.normal(0.0, 0.05, N_OUT)), f(np.exp(rng.normal(-3.0, 0.5, N_OUT))))


def _samples(case, seed):
    """Minibatches of descriptors (bounded, correlated like the radial sums) and targets."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    rows, mix = case["rows"], torch.randn(16, N_IN, device=DEV, generator=gen) * 0.25
    out = []
    for _ in range(case["batches"]):
        z = torch.randn(rows, 16, device=DEV, generator=gen)
        d = (z @ mix).tanh() + 0.1 * torch.randn(rows, N_IN, device=DEV, generator=gen)
        t = 0.05 * torch.randn(rows, N_OUT, device=DEV, generator=gen) + 0.02 * d[:, :1]
        out.append((d.contiguous(), t.contiguous()))
    return out


# ------------------------------------------------------------------ prepare and run

def prepare(case, seed):
    kind = case["kind"]
    ctx = cq.Context(0)
    if kind == "train":
        g = cq.Guess(ctx, seed=1)
        g.set_params(*_weights(seed))
        sc = _scales(seed + 1)
        g.set_scale(*sc)
        return {"kind": kind, "ctx": ctx, "guess": g, "batches": _samples(case, seed), "lr": 2e-3}
    cells = _geometry(case)
    if kind == "product":
        mults = PRODUCTS[case["prod"]]
        pA, pB, pC = _patterns(ctx, cells, *mults)
        A = _Blocks(cells, mults[0]).random(2 * seed + 1)
        B = _Blocks(cells, mults[1]).random(2 * seed + 2)
        assert A.shape[0] == pA.n_values and B.shape[0] == pB.n_values
        return {"kind": kind, "ctx": ctx, "pA": pA, "A": A, "pB": pB, "B": B, "pC": pC,
                "C": ctx.zeros(pC), "prec": PREC[case["prec"]]}
    if kind == "trace":
        (pX,) = _patterns(ctx, cells, (1, 1))
        b = _Blocks(cells, (1, 1))
        assert b.n_values == pX.n_values
        return {"kind": kind, "ctx": ctx, "pX": pX, "X": b.random(2 * seed + 1),
                "Y": b.random(2 * seed + 2)}
    if kind == "apply":
        (pL,) = _patterns(ctx, cells, (0, 1))
        g = cq.Guess(ctx, seed=1)
        g.set_params(*_weights(seed))
        g.set_scale(*_scales(seed + 1))
        return {"kind": kind, "ctx": ctx, "guess": g, "pL": pL, "L": ctx.zeros(pL)}
    pS, pL = _patterns(ctx, cells, (1, 0), (0, 1))
    if kind == "hotelling":
        _, S, _, _ = _overlap_hamiltonian(cells, seed)
        return {"kind": kind, "ctx": ctx, "pS": pS, "S": S, "pT": pL, "T": ctx.zeros(pL),
                "steps": case["steps"]}
    _, S, H, _, L0, ne = _pm_start(cells, seed)
    return {"kind": kind, "ctx": ctx, "pS": pS, "S": S, "H": H, "pL": pL, "L0": L0,
            "L": ctx.zeros(pL), "ne": ne, "prec": PREC[case["prec"]], "steps": case["steps"]}


def run(state):
    s, ctx = state, state["ctx"]
    if s["kind"] == "product":
        return ctx.bsmm(1.0, s["pA"], s["A"], s["pB"], s["B"], 0.0, s["pC"], s["C"], s["prec"])
    if s["kind"] == "trace":
        return {"trace": ctx.trace_prod(s["pX"], s["X"], s["pX"], s["Y"]),
                "dot": ctx.dot(s["pX"], s["X"], s["Y"])}
    if s["kind"] == "apply":
        return s["guess"].apply(s["pL"], s["L"])
    if s["kind"] == "train":
        g = s["guess"]
        for d, t in s["batches"]:
            g.train_step(d, t, s["lr"], loss=False)
        sq, rows = g.loss_sum(reset=True)
        w, b = g.params()
        return {"loss": sq / (rows * N_OUT), "weights": w, "biases": b}
    if s["kind"] == "hotelling":
        ctx.hotelling_init(s["pS"], s["S"], s["pT"], s["T"])
        resid = [ctx.hotelling_step(s["pS"], s["S"], s["pT"], s["T"]) for _ in range(s["steps"])]
        return {"T": s["T"], "resid": resid}
    s["L"].copy_(s["L0"])
    lnv = ctx.lnv(s["pS"], s["S"], s["H"], s["pL"], s["L"], s["ne"], s["prec"])
    reps = [lnv.step() for _ in range(s["steps"])]
    lnv.close()
    return {"L": s["L"], "steps": [[r[k] for k in ("energy", "n_elec", "mu", "gnorm", "alpha")]
                                   for r in reps]}


# ------------------------------------------------------------------ work

def _triplets(cells, mults):
    """Useful flops of a masked product: sum of 2 n_i n_k n_j over its (i, k, j)."""
    total = 0.0
    for c in cells:
        m = []
        for mult in mults:
            b = _Blocks([c], mult)
            a = torch.zeros(b.nb.shape[0], b.nb.shape[0], dtype=F64, device=DEV)
            a[b.i, b.j] = 1.0
            m.append(a)
        nb = b.nb.to(F64)
        k = (m[0] * nb[None, :]) @ m[1]
        total += 2.0 * float((m[2] * k * nb[:, None] * nb[None, :]).sum())
    return total


def work(case):
    """Bytes: each input array read once and each result written once.  Flops: the useful
    flops of the products (2 n_i n_k n_j per triplet), of the network's layers, or one
    multiply-add per value."""
    kind = case["kind"]
    n_w = sum(DIMS[l] * DIMS[l + 1] for l in range(4))
    if kind == "train":
        rows = case["rows"] * case["batches"]
        return {"bytes": 4.0 * rows * (N_IN + N_OUT) + 8.0 * n_w, "flops": 6.0 * rows * n_w}
    cells = _geometry(case)
    size = lambda mult: 8.0 * float(_Blocks(cells, mult).size.sum())
    if kind == "product":
        mults = PRODUCTS[case["prod"]]
        return {"bytes": sum(size(m) for m in mults), "flops": _triplets(cells, mults)}
    if kind == "trace":  # the two calls each read both matrices
        return {"bytes": 4.0 * size((1, 1)), "flops": 4.0 * size((1, 1)) / 8.0}
    if kind == "apply":
        b = _Blocks(cells, (0, 1))
        pairs = float((b.i <= b.j).sum())
        return {"bytes": 24.0 * b.nb.shape[0] + 4.0 * n_w + size((0, 1)), "flops": 2.0 * pairs * n_w}
    if kind == "hotelling":
        f = _triplets(cells, ((1, 0), (0, 1), (1, 1))) + _triplets(cells, ((0, 1), (1, 1), (0, 1)))
        return {"bytes": case["steps"] * (size((1, 0)) + 2 * size((0, 1))), "flops": case["steps"] * f}
    x, u, r = (_triplets(cells, PRODUCTS[p]) for p in ("LSX", "SXU", "UXL"))
    # the object's first evaluation, then per step two trial points and an evaluation
    evaluation, trial = 2 * x + 2 * u + 3 * r, 2 * x + u + 2 * r
    return {"bytes": (1 + case["steps"]) * (2 * size((1, 0)) + 2 * size((0, 1))),
            "flops": evaluation + case["steps"] * (2 * trial + evaluation)}


# ------------------------------------------------------------------ exact results

def _exact_product(case, seed):
    cells = _geometry(case)
    mults = PRODUCTS[case["prod"]]
    bA, bB, bC = (_Blocks(cells, m) for m in mults)
    A, B = bA.dense(bA.random(2 * seed + 1)), bB.dense(bB.random(2 * seed + 2))
    if bA.n_orb <= 6000:
        return bC.values(A @ B)
    # large cells: strips of eight consecutive atoms (one conventional cell), only the
    # columns that the strip's blocks of C hold
    out = torch.zeros(bC.n_values, dtype=F64, device=DEV)
    n = bC.nb.shape[0]
    ends = torch.searchsorted(bC.i, torch.arange(n + 1, device=DEV)).tolist()
    for s in range(0, n, 8):
        at, r, c = bC.places(ends[s], ends[min(n, s + 8)])
        cols, where = torch.unique(c, return_inverse=True)
        r0, r1 = int(r.min()), int(r.max()) + 1
        out[at] = (A[r0:r1] @ B[:, cols])[r - r0, where]
    return out


def _exact_hotelling(case, seed):
    cells = _geometry(case)
    bS, S, _, _ = _overlap_hamiltonian(cells, seed)
    bT, bV = _Blocks(cells, (0, 1)), _Blocks(cells, (1, 1))
    s = bS.dense(S)
    one = torch.eye(bS.n_orb, dtype=F64, device=DEV)
    t = one / s.abs().sum(1).max()
    resid = []
    for _ in range(case["steps"]):
        v = bV.masked(s @ t)
        resid.append(float(torch.linalg.norm(v - one)))
        t = 2.0 * t - bT.masked(t @ v)
    return {"T": bT.values(t), "resid": resid}


def _exact_lnv(case, seed):
    """The LNV iteration of include/cq.h on dense matrices (masked to the patterns)."""
    cells = _geometry(case)
    bS, S, H, bL, L0, ne = _pm_start(cells, seed)
    bX, bU = _Blocks(cells, (1, 1)), _Blocks(cells, (2, 1))
    s, h, l = bS.dense(S), bS.dense(H), bL.dense(L0)
    n_l = float(bL.size.sum())
    mX, mU, mL = (b.masked(torch.ones(b.n_orb, b.n_orb, dtype=F64, device=DEV)) for b in (bX, bU, bL))
    tr = lambda a, b: float((a * b.T).sum())
    dot = lambda a, b: float((a * b).sum())

    def number(l):
        x = mX * (l @ s)
        u = mU * (s @ x)
        r3 = mL * (u @ x)
        return x, u, 2.0 * (3.0 * tr(x, x) - 2.0 * tr(l, r3)), 12.0 * (mL * u - r3)

    def energy(l, x, u):
        y = mX * (l @ h)
        r1 = mL * (u @ y)
        return y, r1, 2.0 * (3.0 * tr(x, y) - 2.0 * tr(l, r1))

    tol = 1e-9 if case["prec"] == "split" else 1e-10

    def corrected(l):
        x, u, n, gn = number(l)
        for _ in range(5):
            if abs(n - ne) <= tol * ne:
                break
            l = l + ((ne - n) / dot(gn, gn)) * gn
            x, u, n, gn = number(l)
        y, r1, e = energy(l, x, u)
        z = mU * (s @ y)
        r2 = mL * (z @ x)
        ge = 2.0 * (3.0 * (mL * (z + z.T)) - 2.0 * (r1 + r1.T + r2))
        return l, e, n, ge, gn

    def cubic(f0, g, a1, f1, a2, f2):
        r1, r2 = f1 - f0 - g * a1, f2 - f0 - g * a2
        det = a1 * a1 * a2 * a2 * (a2 - a1)
        return (r1 * a2 ** 3 - r2 * a1 ** 3) / det, (a1 * a1 * r2 - a2 * a2 * r1) / det

    l, e, n, ge, gn = corrected(l)
    out, g_prev, d_prev, a_prev = [], None, None, None
    for _ in range(case["steps"]):
        mu = dot(ge, gn) / dot(gn, gn)
        g = ge - mu * gn
        d = -g
        if g_prev is not None:
            d = d + max(0.0, dot(g, g - g_prev) / dot(g_prev, g_prev)) * d_prev
        d = d - (dot(d, gn) / dot(gn, gn)) * gn
        if dot(g, d) >= 0.0:
            d = -g
        a1 = a_prev if a_prev is not None else 0.1 * math.sqrt(n_l) / math.sqrt(dot(g, g))
        a2 = 2.0 * a1
        trial = []
        for a in (a1, a2):
            x, u, nt, _ = number(l + a * d)
            trial.append((energy(l + a * d, x, u)[2], nt))
        ge_d, gn_d = dot(ge, d), dot(gn, d)
        e2, e3 = cubic(e, ge_d, a1, trial[0][0], a2, trial[1][0])
        n2, n3 = cubic(n, gn_d, a1, trial[0][1], a2, trial[1][1])
        w1, w2, w3 = ge_d - mu * gn_d, e2 - mu * n2, e3 - mu * n3
        disc = 4.0 * w2 * w2 - 12.0 * w3 * w1
        den = 2.0 * w2 + math.sqrt(disc) if disc >= 0.0 else 0.0
        alpha = -2.0 * w1 / den if den > 0.0 else -1.0
        if alpha <= 0.0:
            alpha = min(2.0 * a2, 0.01 * math.sqrt(n_l / dot(d, d)))
        l, e, n, ge, gn = corrected(l + alpha * d)
        g_prev, d_prev, a_prev = g, d, alpha
        mu = dot(ge, gn) / dot(gn, gn)
        g = ge - mu * gn
        out.append([e, n, mu, math.sqrt(dot(g, g) / n_l), alpha])
    return {"L": bL.values(l), "steps": out}


def _layers(w, b):
    W, B, ow, ob = [], [], 0, 0
    for l in range(4):
        W.append(w[ow:ow + DIMS[l] * DIMS[l + 1]].view(DIMS[l], DIMS[l + 1]))
        B.append(b[ob:ob + DIMS[l + 1]])
        ow += DIMS[l] * DIMS[l + 1]
        ob += DIMS[l + 1]
    return W, B


def _network(x, W, B):
    for l in range(4):
        x = x @ W[l] + B[l]
        if l < 3:
            x = x * torch.sigmoid(x)
    return x


def _exact_train(case, seed):
    t64 = lambda a: torch.tensor(np.asarray(a, dtype=np.float64), device=DEV)
    w, b = (t64(v) for v in _weights(seed))
    im, isc, om, osc = (t64(v) for v in _scales(seed + 1))
    mom = [[torch.zeros_like(v), torch.zeros_like(v)] for v in (w, b)]
    sq = 0.0
    for k, (d, t) in enumerate(_samples(case, seed), 1):
        w.requires_grad_(True)
        b.requires_grad_(True)
        y = _network((d.to(F64) - im) / isc, *_layers(w, b))
        err = y - (t.to(F64) - om) / osc
        loss = (err * err).mean()
        grads = torch.autograd.grad(loss, (w, b))
        sq += float(loss.detach()) * err.numel()
        w, b = w.detach(), b.detach()
        new = []
        for v, gr, m in zip((w, b), grads, mom):
            m[0] = 0.9 * m[0] + 0.1 * gr
            m[1] = 0.999 * m[1] + 0.001 * gr * gr
            new.append(v - 2e-3 * (m[0] / (1 - 0.9 ** k)) / (torch.sqrt(m[1] / (1 - 0.999 ** k)) + 1e-8))
        w, b = new
    rows = case["rows"] * case["batches"]
    return {"loss": sq / (rows * N_OUT), "weights": w, "biases": b}


def _d_forms():
    q = np.zeros((5, 3, 3))
    h = 1.0 / math.sqrt(2.0)
    for a, (r, c) in enumerate(((0, 1), (1, 2), (2, 0))):
        q[a, r, c] = q[a, c, r] = h
    q[3] = np.diag([h, -h, 0.0])
    q[4] = np.diag([-1.0, -1.0, 2.0]) / math.sqrt(6.0)
    return torch.tensor(q, device=DEV)


def _exact_apply(case, seed):
    cells = _geometry(case)
    cell = cells[0][0]
    bL = _Blocks(cells, (0, 1))
    n, nb = cell.n_atoms, case["norb"]
    pos, box = torch.tensor(cell.pos, device=DEV), torch.tensor(cell.box, device=DEV)
    t64 = lambda a: torch.tensor(np.asarray(a, dtype=np.float64), device=DEV)
    W, B = _layers(*(t64(v) for v in _weights(seed)))
    im, isc, om, osc = (t64(v) for v in _scales(seed + 1))
    counts = torch.bincount(bL.i, minlength=n)
    first = torch.cumsum(counts, 0) - counts
    width = int(counts.max())
    Q = _d_forms()
    out = torch.zeros(bL.i.shape[0], int(bL.pad[0]), dtype=F64, device=DEV)
    key = bL.i * n + bL.j
    sel = torch.nonzero(bL.i <= bL.j).flatten()
    arange = torch.arange(width, device=DEV)
    unit = lambda v: v / torch.linalg.norm(v, dim=-1, keepdim=True)
    for c in range(0, sel.shape[0], 8192):
        blk = sel[c:c + 8192]
        i, j = bL.i[blk], bL.j[blk]
        at = (first[i][:, None] + arange).clamp(max=bL.j.shape[0] - 1)
        k = bL.j[at]
        there = (arange < counts[i][:, None]) & (k != i[:, None])
        d = pos[k] - pos[i][:, None]
        d = d - box * torch.round(d / box)
        dij = pos[j] - pos[i]
        dij = dij - box * torch.round(dij / box)
        on = i == j
        r2 = (d * d).sum(-1).masked_fill(~there, math.inf)
        near = d[torch.arange(len(blk), device=DEV), r2.argmin(1)]
        e3 = unit(torch.where(on[:, None], near, dij))
        m = 0.5 * dij
        there = there & (k != j[:, None])
        w = d - m[:, None]
        perp = w - (w * e3[:, None]).sum(-1, keepdim=True) * e3[:, None]
        off = torch.linalg.norm(perp, dim=-1) >= 1e-6
        w2 = (w * w).sum(-1)
        e1 = unit(perp[torch.arange(len(blk), device=DEV),
                       w2.masked_fill(~(there & off), math.inf).argmin(1)])
        e2 = torch.linalg.cross(e3, e1)
        R = torch.stack([e1, e2, e3], 1)
        rho = torch.sqrt(w2)
        use = there & (rho < 8.0) & (rho >= 1e-6)
        x, y, z = ((w @ R.transpose(1, 2)) / rho.clamp(min=1e-6)[..., None]).unbind(-1)
        ang = torch.stack([torch.ones_like(x), z, x, y, 0.5 * (3 * z * z - 1), x * z, y * z,
                           0.5 * (x * x - y * y), x * y], -1)
        cut = torch.where(use, 0.5 * (1.0 + torch.cos(math.pi * rho / 8.0)), 0.0)
        g6 = torch.arange(6, device=DEV, dtype=F64)
        rad = torch.exp(-0.5 * ((rho[..., None] - 1.6 * g6) / 1.2) ** 2) * cut[..., None]
        g10 = torch.arange(10, device=DEV, dtype=F64)
        rij = torch.linalg.norm(dij, dim=-1, keepdim=True)
        desc = torch.cat([torch.exp(-0.5 * ((rij - 1.6 * g10) / 1.6) ** 2),
                          torch.einsum("pkn,pka->pna", rad, ang).reshape(len(blk), 54)], 1)
        loc = (_network((desc - im) / isc, W, B) * osc + om).view(-1, 9, 9)
        D = torch.zeros(len(blk), 9, 9, dtype=F64, device=DEV)
        D[:, 0, 0] = 1.0
        D[:, 1:4, 1:4] = R
        D[:, 4:, 4:] = torch.einsum("pji,ajk,pkl,bil->pab", R, Q, R, Q)
        D, loc = D[:, :nb, :nb], loc[:, :nb, :nb]
        v = D.transpose(1, 2) @ loc @ D
        # an on-site block is its own mirror: its lower triangle stands for both
        v[on] = torch.tril(v[on]) + torch.tril(v[on], -1).transpose(1, 2)
        out[blk, :nb * nb] = v.reshape(-1, nb * nb)
        mirror = torch.searchsorted(key, j * n + i)
        out[mirror, :nb * nb] = v.transpose(1, 2).reshape(-1, nb * nb)
    return out.view(-1)


def _exact_trace(case, seed):
    cells = _geometry(case)
    b = _Blocks(cells, (1, 1))
    nb, p = b.uniform, int(b.pad[0])
    X = b.random(2 * seed + 1).view(-1, p)[:, :nb * nb]
    Y = b.random(2 * seed + 2).view(-1, p)[:, :nb * nb]
    key = b.i * b.nb.shape[0] + b.j
    mirror = torch.searchsorted(key, b.j * b.nb.shape[0] + b.i)
    YT = Y[mirror].view(-1, nb, nb).transpose(1, 2).reshape(-1, nb * nb)
    return {"trace": float((X * YT).sum()), "dot": float((X * Y).sum())}


def exact(case, seed):
    kind = case["kind"]
    return {"product": _exact_product, "hotelling": _exact_hotelling, "lnv": _exact_lnv,
            "train": _exact_train, "apply": _exact_apply, "trace": _exact_trace}[kind](case, seed)
