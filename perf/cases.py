"""Performance cases of the library, through its public entry points.

The cases are the calls that programs make: single block-sparse products and
sums, the batched leaf routine, and whole factorizations (refinement in FP64
and with the mixed-precision schedule, localized, batched) with the adjoint as
the backward direction.  Inputs are the seeded Gaussian-overlap matrices of
``synth`` (1D chains and 3D clusters) or dense blocks of N(0,1) values; a
program keeps one library context for many matrices, and so does this file.
"""
from __future__ import annotations

import math
from functools import lru_cache

import numpy as np
import torch

from paper_1901_07993_gb300 import ifac, synth

PREC = {"fp64": ifac.FP64, "tf32": ifac.TF32, "bf16": ifac.BF16, "split": ifac.FP64_SPLIT}


def listed():
    return [
        # a small FP64 product with a ragged last block: one step of a small
        # factorization, where launches and read-backs count
        dict(name="product_fp64_chain1000", kind="product", geom="chain", n=1000, bs=32, prec="fp64",
             tA=False, tB=False, tau=1e-10),
        # Z^T X of a 3D cluster in FP64: many blocks per row, bound by the FP64 pipe
        dict(name="product_fp64_cluster2048_t", kind="product", geom="cluster", n=2048, bs=32, prec="fp64",
             tA=True, tB=False, tau=1e-10),
        # the dense BF16 product of the benchmark's kernel probe
        dict(name="product_bf16_dense8192", kind="product", geom="dense", n=8192, bs=64, prec="bf16",
             tA=False, tB=False, tau=0.0),
        # the upper-triangle Z^T (S Z) of an FP64-accurate residual on a chain
        dict(name="symproduct_split_chain65536", kind="symproduct", geom="chain", n=65536, bs=64, prec="split",
             tA=True, tB=False, tau=1e-12),
        # Z + M of a refinement sweep: the memory-bound sums
        dict(name="sum_chain65536", kind="sum", geom="chain", n=65536, bs=64, alpha=1.0, beta=-0.375, gamma=1.0),
        # the leaves of one localized factorization, 512 rows each
        dict(name="leaf_512x8", kind="leaf", nl=512, count=8),
        # refinement from a scaled identity in FP64 on the 4096-row chain
        dict(name="refine_fp64_chain4096", kind="refine", geom="chain", n=4096, bs=32, prec="fp64", tau=1e-10,
             target=1e-10, m=2, slices=7),
        # the benchmark's default workload: TF32 sweeps, split FP64-accurate delta
        dict(name="refine_tf32_chain262144", kind="refine", geom="chain", n=262144, bs=64, prec="tf32", tau=1e-12,
             target=1e-10, m=2, slices=7),
        # the same schedule on a 3D cluster, whose factor is block-dense
        dict(name="refine_tf32_cluster4096", kind="refine", geom="cluster", n=4096, bs=64, prec="tf32", tau=1e-14,
             target=1e-10, m=2, slices=8),
        # localized inverse factorization of the 4096-row chain, 512-row leaves
        dict(name="localized_fp64_chain4096", kind="localized", geom="chain", n=4096, bs=32, tau=1e-10,
             target=1e-10, leaf=512),
        # the gradient of a loss through six sweeps (forward recording and reverse pass)
        dict(name="adjoint_fp64_chain16384", kind="adjoint", n=16384, bs=32, K=6, tau=1e-10),
        # several independent matrices of different sizes refined together
        dict(name="batched_tf32_8x512_2048", kind="batched", count=8, nmin=512, nmax=2048, bs=64, prec="tf32",
             tau=1e-12, target=1e-10, slices=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["product", "product", "symproduct", "sum", "leaf", "refine", "refine", "localized", "adjoint",
                       "batched"])
    if kind == "product":
        geom = rng.choice(["chain", "cluster", "dense"])
        prec = rng.choice(["fp64", "tf32", "bf16", "split"])
        bs = rng.choice([16, 32, 64] if prec == "fp64" else [32, 64, 128])
        hi = {"chain": 65536, "cluster": 2048, "dense": 1024 if prec == "fp64" else 8192}[geom]
        if geom == "dense" and prec == "split":
            hi = 4096
        return dict(kind=kind, geom=geom, n=_log_int(rng, 300, hi), bs=bs, prec=prec, tA=rng.random() < 0.5,
                    tB=rng.random() < 0.25, tau=0.0 if geom == "dense" else rng.choice([1e-12, 1e-10, 1e-5]))
    if kind == "symproduct":
        return dict(kind=kind, geom="chain", n=_log_int(rng, 1000, 65536), bs=64,
                    prec=rng.choice(["tf32", "bf16", "split"]), tA=True, tB=False, tau=rng.choice([1e-12, 1e-10]))
    if kind == "sum":
        geom = rng.choice(["chain", "chain", "cluster"])
        return dict(kind=kind, geom=geom, n=_log_int(rng, 500, 65536 if geom == "chain" else 4096),
                    bs=rng.choice([16, 32, 64, 128]), alpha=1.0, beta=rng.choice([1.0, -1.0, -0.375]),
                    gamma=rng.choice([0.0, 1.0]))
    if kind == "leaf":
        return dict(kind=kind, nl=_log_int(rng, 32, 512), count=rng.randint(1, 16))
    if kind == "refine":
        if rng.random() < 0.4:
            return dict(kind=kind, geom="chain", n=_log_int(rng, 500, 8192), bs=rng.choice([16, 32, 64]),
                        prec="fp64", tau=rng.choice([1e-10, 1e-8]), target=1e-10, m=rng.choice([2, 4]), slices=7)
        if rng.random() < 0.5:
            bs = rng.choice([32, 64, 64, 128])
            return dict(kind=kind, geom="chain", n=_log_int(rng, 2000, 262144 if bs == 64 else 98304), bs=bs,
                        prec=rng.choice(["tf32", "bf16"]), tau=1e-12, target=1e-10, m=2, slices=7)
        return dict(kind=kind, geom="cluster", n=_log_int(rng, 700, 3000), bs=64, prec="tf32", tau=1e-14,
                    target=1e-10, m=2, slices=8)
    if kind == "localized":
        return dict(kind=kind, geom="chain", n=_log_int(rng, 500, 8192), bs=32, tau=1e-10, target=1e-10,
                    leaf=rng.choice([128, 256, 512]))
    if kind == "adjoint":
        return dict(kind=kind, n=_log_int(rng, 500, 16384), bs=32, K=rng.randint(2, 6), tau=1e-10)
    return dict(kind=kind, count=rng.randint(2, 8), nmin=512, nmax=rng.choice([1024, 1500, 2048]), bs=64,
                prec=rng.choice(["tf32", "bf16"]), tau=1e-12, target=1e-10, slices=8)


# ---------------------------------------------------------------- inputs

_contexts = {}


def _context(slices=7):
    """One library context for each slice count, as a program keeps it."""
    if slices not in _contexts:
        ctx = ifac.Context()
        ctx.set_split_slices(slices)
        _contexts[slices] = ctx
    return _contexts[slices]


@lru_cache(maxsize=64)
def _geometry(geom, n, bs, which):
    return synth.chain(n, seed=which) if geom == "chain" else synth.cluster(n, bs, seed=which)


def _overlap(geom, n, bs, seed, which=0):
    """The overlap matrix of one molecule at a geometry step: the centres moved by 1e-5 bohr, so that every
    value is another one while the block patterns stay those of the molecule."""
    g = _geometry(geom, n, bs, which)
    step = 1e-5 * np.random.default_rng(seed).standard_normal(g.xyz.shape)
    return synth.overlap_bsr(synth.Geometry(g.xyz + step, g.alpha), bs)


def _dense(n, bs, seed):
    """Every block stored, entries N(0,1); padding rows and columns are those of the identity."""
    nb = -(-n // bs)
    g = torch.Generator(device="cuda").manual_seed(seed)
    d = torch.zeros(nb * bs, nb * bs, dtype=torch.float64, device="cuda")
    d[:n, :n] = torch.randn(n, n, generator=g, dtype=torch.float64, device="cuda")
    d.diagonal()[n:] = 1.0
    val = d.view(nb, bs, nb, bs).transpose(1, 2).reshape(nb * nb, bs, bs).contiguous()
    rp = torch.arange(nb + 1, dtype=torch.int32, device="cuda") * nb
    ci = torch.arange(nb, dtype=torch.int32, device="cuda").repeat(nb)
    return ifac.BorrowedBSR(n, bs, rp, ci, val)


def _operands(case, seed):
    """Two matrices of about one pattern: the overlaps of two geometry steps (the second stands in for Z or X)."""
    if case["geom"] == "dense":
        return _dense(case["n"], case["bs"], 2 * seed), _dense(case["n"], case["bs"], 2 * seed + 1)
    ctx = _context()
    return tuple(ifac.upload(ctx, _overlap(case["geom"], case["n"], case["bs"], 2 * seed + k)) for k in (0, 1))


def _leaves(case, seed):
    """Diagonal parts of chain overlaps, dense."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    c, nl = case["count"], case["nl"]
    x = torch.cumsum(1.4 + 0.2 * (torch.rand(c, nl, generator=g, dtype=torch.float64, device="cuda") - 0.5), dim=1)
    a = torch.tensor(synth.EXPONENTS, dtype=torch.float64, device="cuda").repeat(-(-nl // 3))[:nl]
    s, p = a[:, None] + a[None, :], a[:, None] * a[None, :]
    return (2 * p.sqrt() / s) ** 1.5 * torch.exp(-p / s * (x[:, :, None] - x[:, None, :]) ** 2)


def _member_sizes(case):
    r = np.random.default_rng(3)
    return np.exp(r.uniform(math.log(case["nmin"]), math.log(case["nmax"]), size=case["count"])).astype(int).tolist()


def prepare(case, seed):
    kind = case["kind"]
    ctx = _context(case.get("slices", 7))
    st = dict(case=case, ctx=ctx)
    if kind in ("product", "symproduct", "sum"):
        st["A"], st["B"] = _operands(case, seed)
    elif kind == "leaf":
        st["S"] = _leaves(case, seed)
    elif kind == "batched":
        st["S"] = [ifac.upload(ctx, _overlap("cluster" if j % 2 else "chain", n, case["bs"], 1000 * seed + j, which=j))
                   for j, n in enumerate(_member_sizes(case))]
        st["opts"] = ifac.opts(prec=PREC[case["prec"]], max_iter=100)
    elif kind == "adjoint":
        h = _overlap("chain", case["n"], case["bs"], seed)
        st["S"], st["F"] = ifac.upload(ctx, h), ifac.upload(ctx, synth.fock_like(h, seed=seed + 5))
    else:
        st["S"] = ifac.upload(ctx, _overlap(case["geom"], case["n"], case["bs"], seed))
        st["opts"] = (ifac.opts(leaf_size=case["leaf"]) if kind == "localized" else
                      ifac.opts(m=case["m"], prec=PREC[case["prec"]]))
    return st


# ---------------------------------------------------------------- one pass

def _out(M):
    rp, ci, val = ifac.device_tensors(M)
    return dict(row_ptr=rp, col_idx=ci, val=val)


def run(st):
    c, ctx = st["case"], st["ctx"]
    kind = c["kind"]
    if kind == "product":
        return _out(ifac.bsr_gemm_trunc(ctx, st["A"], c["tA"], st["B"], c["tB"], 1.0, c["tau"], PREC[c["prec"]]))
    if kind == "symproduct":
        return _out(ifac.bsr_gemm_sym_trunc(ctx, st["A"], c["tA"], st["B"], c["tB"], 1.0, c["tau"], PREC[c["prec"]]))
    if kind == "sum":
        return _out(ifac.bsr_add(ctx, c["alpha"], st["A"], c["beta"], st["B"], c["gamma"]))
    if kind == "leaf":
        Z, info, _ = ifac.leaf_invchol_batched(ctx, st["S"])
        return dict(Z=Z, info=info)
    if kind == "refine":
        Z, rep = ifac.inv_factor_refine(ctx, st["S"], c["tau"], c["target"], st["opts"])
        return dict(_out(Z), sweeps=rep.sweeps)
    if kind == "localized":
        Z, rep = ifac.inv_factor_localized(ctx, st["S"], c["tau"], c["target"], st["opts"])
        return dict(_out(Z), sweeps=rep.sweeps)
    if kind == "adjoint":
        L, G = ifac.inv_factor_refine_adjoint(ctx, st["S"], st["F"], c["K"], c["tau"])
        return dict(_out(G), loss=L)
    Zs, reps, _ = ifac.inv_factor_refine_batched(ctx, st["S"], c["tau"], c["target"], st["opts"])
    return [_out(Z) for Z in Zs]


# ---------------------------------------------------------------- the work of one pass

def _pattern(case):
    """(block rows, stored blocks, block pairs of A B) with the case's geometry."""
    n, bs = case["n"], case["bs"]
    nb = -(-n // bs)
    if case["geom"] == "dense":
        return nb, nb * nb, nb ** 3
    if case["geom"] == "chain":  # overlaps reach about 14 centres: three blocks a row
        return nb, max(1, 3 * nb - 2), max(1, 9 * nb - 10)
    S = _overlap("cluster", n, bs, 0)
    per = np.diff(S.row_ptr).astype(np.float64)
    return nb, S.nnzb, float((per ** 2).sum())


def _factor_work(geom, n, bs, products):
    """S read and Z written once; the block pairs of the truncated products."""
    nb = -(-n // bs)
    if geom == "chain":  # S, the iterates and delta hold about three blocks a row, a product eight pairs
        return 8.0 * bs * bs * 6 * nb, 2.0 * bs ** 3 * 8 * nb * products
    # block-dense factors; the symmetric products form one triangle
    return 16.0 * (nb * bs) ** 2, 0.62 * 2.0 * float(nb * bs) ** 3 * products


def work(case):
    kind = case["kind"]
    if kind == "leaf":
        nl, c = case["nl"], case["count"]
        return dict(bytes=16.0 * c * nl * nl, flops=2.0 / 3.0 * c * nl ** 3)
    if kind == "batched":
        w = [_factor_work("cluster" if j % 2 else "chain", n, case["bs"], 40) for j, n in
             enumerate(_member_sizes(case))]
        return dict(bytes=sum(x for x, _ in w), flops=sum(y for _, y in w))
    if kind == "adjoint":  # four products a sweep in the recording run, eight in the reverse pass
        b, f = _factor_work("chain", case["n"], case["bs"], 12 * case["K"])
        return dict(bytes=b * 1.5, flops=f)
    if kind == "localized":  # the leaves, and products of the coupling blocks between them
        b, f = _factor_work("chain", case["n"], case["bs"], 1.5)
        return dict(bytes=b, flops=f + 2.0 / 3.0 * case["n"] * float(min(case["leaf"], case["n"])) ** 2)
    if kind == "refine":  # products of five sweeps in FP64; of eleven with the mixed schedule on clusters
        b, f = _factor_work(case["geom"], case["n"], case["bs"],
                            46 if case["geom"] == "cluster" else 22 if case["prec"] == "fp64" else 34)
        return dict(bytes=b, flops=f)
    nb, nnzb, pairs = _pattern(case)
    blk = float(case["bs"]) ** 2
    if kind == "sum":
        return dict(bytes=24.0 * blk * nnzb, flops=3.0 * blk * nnzb)
    return dict(bytes=24.0 * blk * nnzb, flops=2.0 * blk * case["bs"] * pairs * (0.5 if kind == "symproduct" else 1.0))


# ---------------------------------------------------------------- the same in 64 bits

class _Full:
    """A block-sparse matrix as a full one with the mask of its stored blocks."""

    def __init__(self, val, mask, bs):
        self.val, self.mask, self.bs = val, mask, bs

    def t(self):
        return _Full(self.val.T, self.mask.T, self.bs)

    def mm(self, other, tau, alpha=1.0):
        v = alpha * (self.val @ other.val)
        return _Full(v, (self.mask.double() @ other.mask.double()) > 0, self.bs).trunc(tau)

    def norms(self):
        nb = self.mask.shape[0]
        return self.val.reshape(nb, self.bs, nb, self.bs).square().sum(dim=(1, 3)).sqrt()

    def only(self, mask):
        return _Full(self.val * mask.repeat_interleave(self.bs, 0).repeat_interleave(self.bs, 1), mask, self.bs)

    def trunc(self, tau):
        return self.only(self.mask & ~(self.norms() < tau)) if tau > 0 else self

    def plus(self, a, other=None, b=0.0, diag=0.0):
        v, m = a * self.val, self.mask
        if other is not None:
            v, m = v + b * other.val, m | other.mask
        if diag:
            v = v + diag * torch.eye(v.shape[0], dtype=v.dtype, device=v.device)
            m = m | torch.eye(m.shape[0], dtype=torch.bool, device=m.device)
        return _Full(v, m, self.bs)

    def out(self):
        nb, bs = self.mask.shape[0], self.bs
        rows, cols = torch.nonzero(self.mask, as_tuple=True)
        rp = torch.zeros(nb + 1, dtype=torch.int32, device="cuda")
        rp[1:] = torch.cumsum(self.mask.sum(1), 0).int()
        return dict(row_ptr=rp, col_idx=cols.int(),
                    val=self.val.detach().reshape(nb, bs, nb, bs).transpose(1, 2)[rows, cols].contiguous())


def _full(M):
    """The full matrix of a device matrix or of borrowed tensors."""
    rp, ci, val = ifac.device_tensors(M) if isinstance(M, ifac.DeviceBSR) else M.keep
    nb, bs = rp.numel() - 1, val.shape[1]
    rows = torch.repeat_interleave(torch.arange(nb, device="cuda"), (rp[1:] - rp[:-1]).long())
    v = torch.zeros(nb, nb, bs, bs, dtype=torch.float64, device="cuda")
    v[rows, ci.long()] = val
    mask = torch.zeros(nb, nb, dtype=torch.bool, device="cuda")
    mask[rows, ci.long()] = True
    return _Full(v.transpose(1, 2).reshape(nb * bs, nb * bs), mask, bs)


def _start_scale(S):
    return 1.0 / math.sqrt(float(S.val.abs().sum(dim=1).max()))


def _b(k):
    return 1.0 if k == 0 else _b(k - 1) * (2 * k - 1) / (2 * k)


def _refine(S, tau, target, m):
    """Refinement from a scaled identity with truncated products and the automatic stop rule."""
    S = S.trunc(tau)
    eye = torch.eye(S.mask.shape[0], dtype=torch.bool, device="cuda")
    Z = _Full(_start_scale(S) * torch.eye(S.val.shape[0], dtype=torch.float64, device="cuda"), eye, S.bs)
    prev, sweeps = math.inf, 0
    while True:
        D = Z.t().mm(S.mm(Z, tau), tau).plus(-1.0, diag=1.0)
        e = float(torch.linalg.norm(D.val))
        if e <= target or e > prev ** (m + 1):
            return Z, sweeps
        power, P = D, D.plus(_b(1))
        for k in range(2, m + 1):
            power = power.mm(D, tau)
            P = P.plus(1.0, power, _b(k))
        Z = Z.plus(1.0, Z.mm(P, tau), 1.0)
        prev, sweeps = e, sweeps + 1


def _adjoint(S, F, K, tau):
    """(loss, gradient on S's blocks) of K sweeps, each product on its recorded blocks."""
    G = S.val.clone().requires_grad_(True)
    T = _Full(G, S.mask, S.bs).only(S.trunc(tau).mask)
    eye = torch.eye(S.mask.shape[0], dtype=torch.bool, device="cuda")
    Z = _Full(_start_scale(S.trunc(tau)) * torch.eye(G.shape[0], dtype=torch.float64, device="cuda"), eye, S.bs)
    for _ in range(K):
        D = Z.t().mm(T.mm(Z, tau), tau).plus(-1.0, diag=1.0)
        P = D.plus(0.5, D.mm(D, tau), 0.375)
        Z = Z.plus(1.0, Z.mm(P, tau), 1.0)
    L = (Z.val * (F.val @ Z.val)).sum()
    L.backward()
    return float(L.detach()), _Full(G.grad, S.mask, S.bs).only(S.mask)


def exact(case, seed):
    kind = case["kind"]
    if kind == "leaf":
        S = _leaves(case, seed)
        L = torch.linalg.cholesky(S)
        eye = torch.eye(case["nl"], dtype=torch.float64, device="cuda").expand_as(S)
        return dict(Z=torch.linalg.solve_triangular(L, eye, upper=False).mT.contiguous(), info=None)
    # as full matrices, at sizes where that takes seconds; the mixed schedule's
    # factor is S^-1/2 times a nearly orthogonal matrix that its roundings make
    limit = 8192 if kind in ("product", "symproduct", "sum") else 4096
    if kind in ("localized", "batched") or case["n"] > limit or case.get("prec") in ("tf32", "bf16") and kind == "refine":
        return None
    st = prepare(case, seed)
    if kind == "adjoint":
        L, G = _adjoint(_full(st["S"]), _full(st["F"]), case["K"], case["tau"])
        return dict(G.out(), loss=L)
    if kind == "refine":
        Z, sweeps = _refine(_full(st["S"]), case["tau"], case["target"], case["m"])
        return dict(Z.out(), sweeps=sweeps)
    A, B = _full(st["A"]), _full(st["B"])
    if kind == "sum":
        return A.plus(case["alpha"], B, case["beta"], case["gamma"]).out()
    A, B = A.t() if case["tA"] else A, B.t() if case["tB"] else B
    if kind == "product":
        return A.mm(B, case["tau"]).out()
    # the upper block triangle, truncated, and its mirror image
    C = A.mm(B, 0.0)
    U = C.only(C.mask.triu()).trunc(case["tau"])
    strict = U.only(U.mask.triu(1))
    return U.plus(1.0, strict.t(), 1.0).out()
