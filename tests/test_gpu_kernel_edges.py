"""Kernels at the sizes and values where they can go wrong: tile edges,
remainders, few long and many short block rows, values of very different
magnitude, matrices that start off a 16-byte boundary."""
import numpy as np
import pytest

import oracle
from paper_1901_07993_gb300 import synth

pytestmark = pytest.mark.gpu
FP64, TF32, BF16, FP64_SPLIT = 0, 1, 2, 3


@pytest.fixture(scope="module")
def ctx():
    import torch
    from paper_1901_07993_gb300 import build as libbuild
    from paper_1901_07993_gb300 import ifac
    assert torch.cuda.is_available()
    libbuild.build()
    return ifac.Context()


def full(h):
    D = np.zeros((h.nb * h.bs, h.nb * h.bs))
    for I in range(h.nb):
        for q in range(h.row_ptr[I], h.row_ptr[I + 1]):
            J = h.col_idx[q]
            D[I * h.bs:(I + 1) * h.bs, J * h.bs:(J + 1) * h.bs] = h.val[q]
    return D


def borrowed(h, shift):
    """h in torch tensors whose values start `shift` doubles past an allocation."""
    import torch
    from paper_1901_07993_gb300 import ifac
    buf = torch.zeros(h.val.size + shift, dtype=torch.float64, device="cuda")
    val = buf[shift:].view(h.nnzb, h.bs, h.bs)
    val.copy_(torch.from_numpy(np.ascontiguousarray(h.val)))
    return ifac.BorrowedBSR(h.n, h.bs, torch.from_numpy(h.row_ptr).cuda(), torch.from_numpy(h.col_idx).cuda(), val)


@pytest.mark.parametrize("bs,nb,density,tA,tB,shift", [(64, 3, 1.0, False, False, 0), (64, 11, 1.0, True, False, 1),
                                                       (32, 30, 0.8, False, True, 1), (128, 4, 1.0, True, True, 0),
                                                       (64, 40, 0.05, False, False, 1)])
def test_split_row_scales(ctx, bs, nb, density, tA, tB, shift):
    """Scales of rows and columns whose magnitudes span 2^-300 .. 2^300, each
    beginning with entries 2^-180 below its largest; block rows in several
    parts (few long ones) and in one; values off a 16-byte boundary.  Bound:
    K 2^-(7 s - 5) max|a_i.| max|b_.j| + 2 K 2^-53 (|A||B|)_ij with s = 7."""
    from paper_1901_07993_gb300 import ifac
    rng = np.random.default_rng(5)
    A = synth.random_bsr(nb, bs, density, seed=81)
    B = synth.random_bsr(nb, bs, density, seed=82)
    r = np.exp2(rng.integers(-300, 300, nb * bs).astype(float)).reshape(nb, bs)
    for M, t in ((A, tA), (B, not tB)):
        rows = np.repeat(np.arange(nb), np.diff(M.row_ptr))
        for q in range(M.nnzb):
            v = M.val[q].T if t else M.val[q]
            v[:, :3] *= 2.0 ** -180
            v *= r[M.col_idx[q] if t else rows[q]][:, None]
    got = ifac.bsr_gemm_trunc(ctx, borrowed(A, shift), tA, borrowed(B, shift), tB, 1.0, 0.0, FP64_SPLIT).download()
    ref = oracle.gemm(A, B, tA, tB, 1.0, 0.0)
    assert np.array_equal(got.row_ptr, ref.row_ptr) and np.array_equal(got.col_idx, ref.col_idx)
    Ad, Bd = (full(A).T if tA else full(A)), (full(B).T if tB else full(B))
    K = nb * bs
    lim = (K * 2.0 ** -44 * np.outer(np.abs(Ad).max(axis=1), np.abs(Bd).max(axis=0))
           + 2 * K * 2.0 ** -53 * (np.abs(Ad) @ np.abs(Bd)))
    assert np.all(np.abs(full(got) - full(ref)) <= lim)


@pytest.mark.parametrize("nl,count", [(1, 1), (32, 3), (33, 2), (64, 1), (95, 20), (160, 40), (320, 13), (480, 9),
                                      (1024, 1)])
def test_leaf_cluster_sizes(ctx, nl, count):
    """Leaves of one to 32 tiles in clusters of one to 16 CTAs (the counts run
    through the rule's cluster sizes), ragged sizes among them: against numpy's
    inverse Cholesky factor (condition number about 4: 64 nl 2^-53 relative),
    triangular, and a bad pivot reported where it is."""
    import torch
    from paper_1901_07993_gb300 import ifac
    rng = np.random.default_rng(nl)
    G = rng.standard_normal((count, nl, nl)) / np.sqrt(nl)
    S = np.eye(nl) + 0.25 * np.matmul(G, G.transpose(0, 2, 1))
    Z, info, rc = ifac.leaf_invchol_batched(ctx, torch.from_numpy(S).cuda())
    Z = Z.cpu().numpy()
    ref = np.linalg.inv(np.linalg.cholesky(S)).transpose(0, 2, 1)
    assert rc == 0 and not info.any().item()
    assert np.array_equal(Z, np.triu(Z))
    err = np.linalg.norm(Z - ref, axis=(1, 2)) / np.linalg.norm(ref, axis=(1, 2))
    assert err.max() <= 64 * nl * 2.0 ** -53
    # the last matrix gets a negative pivot at row p; the others are unaffected
    p = (2 * nl) // 3
    S[-1, p, p] = -1.0
    Z2, info, rc = ifac.leaf_invchol_batched(ctx, torch.from_numpy(S).cuda())
    assert rc == ifac.ERR_NOT_SPD and info[-1].item() == p + 1 and not info[:-1].any().item()
    assert np.array_equal(Z2.cpu().numpy()[:-1], Z[:-1])


@pytest.mark.parametrize("bs,nb,ns,kind", [(64, 3, 8, "normal"), (64, 7, 8, "normal"), (64, 23, 8, "ones"),
                                           (64, 40, 8, "ones"), (64, 65, 8, "ones"), (64, 9, 3, "normal"),
                                           (64, 15, 5, "normal"), (32, 30, 6, "ones"), (128, 4, 8, "normal"),
                                           (64, 65, 7, "ones")])
def test_split_class_sums(bs, nb, ns, kind):
    """The weight classes in the 64-bit sums: one and several windows, odd and
    even slice counts, and units that fall between two classes or below
    several of them (entries of one magnitude: |sum| up to K, so the unit
    2^-f grows with K).  Bound: K 2^-(7 s - 5) r_i c_j for the slices, half a
    unit 2^-f for each window (at least three blocks of 64, or their share)
    and K 2^-53 (|A||B|)_ij; f >= min(56, 62 - ceil(log2(1.125 K + 2)), 7 (s + 1))."""
    from paper_1901_07993_gb300 import ifac
    ctx = ifac.Context()
    ctx.set_split_slices(ns)
    rng = np.random.default_rng(7)
    A, B = synth.random_bsr(nb, bs, 1.0, seed=91), synth.random_bsr(nb, bs, 1.0, seed=92)
    if kind == "ones":
        for M in (A, B):
            M.val[:] = np.where(rng.random(M.val.shape) < 0.5, 1.0, 1.0 - 2.0 ** -9) - 2.0 ** -40 * rng.random(M.val.shape)
    got = ifac.bsr_gemm_trunc(ctx, ifac.upload(ctx, A), False, ifac.upload(ctx, B), False, 1.0, 0.0,
                              FP64_SPLIT).download()
    Ad, Bd = full(A), full(B)
    ref, K = Ad @ Bd, nb * bs
    f = min(56, 62 - int(np.ceil(np.log2(1.125 * K + 2))), 7 * (ns + 1))
    r, c = np.abs(Ad).max(axis=1), np.abs(Bd).max(axis=0)
    windows = -(-K // 192)
    lim = ((K * 2.0 ** -(7 * ns - 5) + windows * 4 * 2.0 ** -f) * np.outer(r, c)
           + 2 * K * 2.0 ** -53 * (np.abs(Ad) @ np.abs(Bd)))
    assert np.all(np.abs(full(got) - ref) <= lim)
    norms = np.sqrt((got.val ** 2).sum(axis=(1, 2)))
    dev = ifac.bsr_gemm_trunc(ctx, ifac.upload(ctx, A), False, ifac.upload(ctx, B), False, 1.0, 0.0, FP64_SPLIT)
    assert abs(ifac.bsr_fro(ctx, dev) - np.sqrt((norms ** 2).sum())) <= 1e-12 * np.sqrt((norms ** 2).sum())


@pytest.mark.parametrize("bs,nb,density,shift", [(64, 1, 1.0, 0), (64, 40, 0.9, 1), (32, 70, 0.6, 0), (32, 5, 0.3, 3),
                                                 (128, 3, 0.7, 2), (16, 33, 0.5, 1), (5, 9, 0.4, 0), (6, 9, 0.4, 1),
                                                 (16, 1100, 0.9, 0)])
def test_sum_edges(ctx, bs, nb, density, shift):
    """Sums equal to the oracle's, value for value: long and short rows, block sizes of
    each kernel shape, values off a 32-byte boundary, missing blocks, zeros,
    subnormals, infinities and values whose squares leave FP32's range.  The
    norms within 2^-40."""
    from paper_1901_07993_gb300 import ifac
    A = synth.random_bsr(nb, bs, density, seed=61)
    B = synth.random_bsr(nb, bs, density, seed=62, empty_rows=min(1, nb - 1))
    rng = np.random.default_rng(3)
    special = np.array([0.0, -0.0, 5e-324, -1e-310, 1e-200, 1e30, -1e150, np.inf])
    for M in (A, B):
        M.val[: M.nnzb // 3] = special[rng.integers(0, len(special) - 1, M.val[: M.nnzb // 3].shape)]
    dA, dB = borrowed(A, shift), borrowed(B, shift)
    for alpha, beta, gamma in ((1.0, -0.375, 1.0), (-1.0, 1.0, 0.0), (0.5, 2.0, -3.0)):
        ref = oracle.add(alpha, A, beta, B, gamma)
        dev = ifac.bsr_add(ctx, alpha, dA, beta, dB, gamma)
        got = dev.download()
        assert np.array_equal(got.row_ptr, ref.row_ptr) and np.array_equal(got.col_idx, ref.col_idx)
        assert np.array_equal(got.val, ref.val)  # (the library's leading 0 + x is x: -0 stays -0)
        f = np.sqrt((np.asarray(ref.val) ** 2).sum())
        assert abs(ifac.bsr_fro(ctx, dev) - f) <= 1e-12 * f
    A.val[0, 0, 0] = np.inf
    got = ifac.bsr_add(ctx, 1.0, borrowed(A, shift), 0.0, None, 0.0)
    assert np.isinf(ifac.bsr_fro(ctx, got)) and np.array_equal(got.download().val, A.val)


def _pattern_ref(A, B, tA, tB, upper):
    """Stored blocks of op(A) op(B) before truncation."""
    ma, mb = np.zeros((A.nb, A.nb), int), np.zeros((A.nb, A.nb), int)
    for m, h in ((ma, A), (mb, B)):
        m[np.repeat(np.arange(h.nb), np.diff(h.row_ptr)), h.col_idx] = 1
    m = (ma.T if tA else ma) @ (mb.T if tB else mb) > 0
    return np.triu(m) if upper else m


@pytest.mark.parametrize("nb,density", [(1, 1.0), (31, 0.1), (33, 0.9), (64, 1.0), (255, 0.02), (512, 0.006),
                                        (512, 0.2), (513, 0.006), (1100, 0.002), (1500, 0.0003)])
@pytest.mark.parametrize("tA,tB", [(False, False), (True, False), (False, True), (True, True)])
def test_patterns(ctx, nb, density, tA, tB):
    """Patterns of products and sums on both sides of the one-CTA limits (block
    rows, stored blocks, expected result), empty rows included, against
    numpy's: every block once, rows sorted, and the values of a product and of
    a truncation in the right place."""
    from paper_1901_07993_gb300 import ifac
    A = synth.random_bsr(nb, 16, density, seed=nb, empty_rows=nb // 7)
    B = synth.random_bsr(nb, 16, density, seed=nb + 1, empty_rows=nb // 9)
    if A.nnzb == 0 or B.nnzb == 0:
        pytest.skip("an operand without blocks")
    dA, dB = ifac.upload(ctx, A), ifac.upload(ctx, B)
    ref = _pattern_ref(A, B, tA, tB, False)
    for tau in (0.0, 60.0):
        got = ifac.bsr_gemm_trunc(ctx, dA, tA, dB, tB, 1.0, tau).download()
        want = oracle.gemm(A, B, tA, tB, 1.0, tau)
        if tau == 0.0:
            assert np.array_equal(got.row_ptr, np.concatenate([[0], np.cumsum(ref.sum(axis=1))]))
            assert np.array_equal(got.col_idx, np.nonzero(ref)[1])
        assert np.array_equal(got.row_ptr, want.row_ptr) and np.array_equal(got.col_idx, want.col_idx)
        assert got.nnzb == 0 or np.abs(got.val - want.val).max() <= 1e-12 * np.abs(want.val).max()
    s, ws = ifac.bsr_add(ctx, 1.0, dA, 2.0, dB, 0.5).download(), oracle.add(1.0, A, 2.0, B, 0.5)
    assert np.array_equal(s.row_ptr, ws.row_ptr) and np.array_equal(s.col_idx, ws.col_idx)
    assert np.array_equal(s.val, ws.val)
    t, wt = ifac.bsr_truncate(ctx, dA, 16.0).download(), oracle.truncate(A, 16.0)
    assert np.array_equal(t.row_ptr, wt.row_ptr) and np.array_equal(t.col_idx, wt.col_idx)
    assert np.array_equal(t.val, wt.val)


@pytest.mark.parametrize("bs,nb,density", [(64, 5, 1.0), (64, 40, 0.4), (64, 64, 1.0), (64, 130, 0.05), (64, 300, 0.012),
                                           (32, 100, 0.3), (32, 520, 0.004), (128, 20, 0.6), (64, 1500, 0.0012)])
@pytest.mark.parametrize("prec", [TF32, BF16])
def test_tile_plans(ctx, bs, nb, density, prec):
    """Tile lists and plans of every kind (one CTA or several, records in one
    pass or counted first, tiles from C's blocks, both tile shapes at bs 64):
    small integers, so that every product is exact."""
    from paper_1901_07993_gb300 import ifac
    rng = np.random.default_rng(nb)
    A = synth.random_bsr(nb, bs, density, seed=nb)
    B = synth.random_bsr(nb, bs, density, seed=nb + 1, empty_rows=1)
    A.val[:] = rng.integers(-1, 2, A.val.shape)
    B.val[:] = rng.integers(-1, 2, B.val.shape)
    dA, dB = ifac.upload(ctx, A), ifac.upload(ctx, B)
    for tA in (False, True):
        want = oracle.gemm(A, B, tA, False, 1.0, 0.0)
        got = ifac.bsr_gemm_trunc(ctx, dA, tA, dB, False, 1.0, 0.0, prec).download()
        assert np.array_equal(got.row_ptr, want.row_ptr) and np.array_equal(got.col_idx, want.col_idx)
        assert np.array_equal(got.val, want.val)
        if bs == 64:
            up = ifac.bsr_gemm_sym_trunc(ctx, dA, True, dA, False, 1.0, 0.0, prec).download()
            ref = oracle.gemm(A, A, True, False, 1.0, 0.0)
            assert np.array_equal(up.col_idx, ref.col_idx) and np.array_equal(up.val, ref.val)


@pytest.mark.parametrize("bs,nb,density", [(32, 1, 1.0), (32, 50, 1.0), (32, 52, 1.0), (64, 3, 0.7), (64, 51, 0.9),
                                           (64, 53, 1.0), (16, 40, 0.5)])
@pytest.mark.parametrize("tA,tB", [(False, False), (True, False), (False, True), (True, True)])
def test_fp64_product_block_counts(ctx, bs, nb, density, tA, tB):
    """FP64 products on both sides of the limit on output blocks at which a
    block stops being split over four CTAs (2584 blocks on 152 SMs): values
    within 2 K 2^-53 (|A||B|)_ij, norms within 1e-13, pairs counted once."""
    from paper_1901_07993_gb300 import ifac
    A = synth.random_bsr(nb, bs, density, seed=71)
    B = synth.random_bsr(nb, bs, density, seed=72)
    if A.nnzb == 0 or B.nnzb == 0:
        pytest.skip("an operand without blocks")
    dev = ifac.bsr_gemm_trunc(ctx, borrowed(A, 1), tA, borrowed(B, 1), tB, -0.75, 0.0)
    got, ref = dev.download(), oracle.gemm(A, B, tA, tB, -0.75, 0.0)
    assert np.array_equal(got.row_ptr, ref.row_ptr) and np.array_equal(got.col_idx, ref.col_idx)
    Ad, Bd = (full(A).T if tA else full(A)), (full(B).T if tB else full(B))
    lim = 2 * nb * bs * 2.0 ** -53 * (np.abs(Ad) @ np.abs(Bd))
    assert np.all(np.abs(full(got) - full(ref)) <= lim + 1e-300)
    norms = np.sqrt((np.asarray(ref.val) ** 2).sum(axis=(1, 2)))
    tau = float(np.median(norms)) * (1 + 1e-9)
    cut = ifac.bsr_gemm_trunc(ctx, borrowed(A, 1), tA, borrowed(B, 1), tB, -0.75, tau)
    assert cut.nnzb == int((norms >= tau).sum())
    assert abs(ifac.bsr_fro(ctx, dev) - np.sqrt((norms ** 2).sum())) <= 1e-13 * np.sqrt((norms ** 2).sum())


@pytest.mark.parametrize("bs", [32, 64, 128])
@pytest.mark.parametrize("tA,tB,shift", [(False, False, 0), (True, False, 1), (False, True, 0), (True, True, 2)])
@pytest.mark.parametrize("ns", [3, 5, 8])
def test_split_banded_operands(bs, tA, tB, shift, ns):
    """Operands of many short block rows (scales and slices in one kernel) with
    empty rows and values off a 32-byte boundary, magnitudes over 2^+-40 with
    zeros and exact powers of two among them (ties of the digits): the bound of
    the row-scale test for s slices."""
    from paper_1901_07993_gb300 import ifac
    ctx = ifac.Context()
    ctx.set_split_slices(ns)
    nb = 330
    rng = np.random.default_rng(11)

    def banded(seed):
        mask = np.abs(np.subtract.outer(np.arange(nb), np.arange(nb))) <= 1
        mask[rng.choice(nb, 5, replace=False)] = False
        rows, cols = np.nonzero(mask)
        v = rng.standard_normal((len(rows), bs, bs)) * np.exp2(rng.integers(-40, 41, (len(rows), 1, 1)))
        v[::3] = np.exp2(rng.integers(-12, 13, v[::3].shape)) * rng.integers(-1, 2, v[::3].shape)
        rp = np.concatenate([[0], np.cumsum(mask.sum(axis=1))]).astype(np.int32)
        return synth.HostBSR(nb * bs, bs, rp, cols.astype(np.int32), v)

    A, B = banded(1), banded(2)
    got = ifac.bsr_gemm_trunc(ctx, borrowed(A, shift), tA, borrowed(B, shift), tB, 1.0, 0.0, FP64_SPLIT).download()
    ref = oracle.gemm(A, B, tA, tB, 1.0, 0.0)
    assert np.array_equal(got.row_ptr, ref.row_ptr) and np.array_equal(got.col_idx, ref.col_idx)

    def maxima(M, t):  # largest magnitude of every scalar row of op(M), by block row
        out = np.zeros((nb, bs))
        rows = np.repeat(np.arange(nb), np.diff(M.row_ptr))
        for q in range(M.nnzb):
            v = np.abs(M.val[q].T if t else M.val[q]).max(axis=1)
            I = M.col_idx[q] if t else rows[q]
            out[I] = np.maximum(out[I], v)
        return out

    r, c = maxima(A, tA), maxima(B, not tB)
    absA = synth.HostBSR(A.n, bs, A.row_ptr, A.col_idx, np.abs(A.val))
    absB = synth.HostBSR(B.n, bs, B.row_ptr, B.col_idx, np.abs(B.val))
    aref = oracle.gemm(absA, absB, tA, tB, 1.0, 0.0)
    K = 3 * bs
    rows = np.repeat(np.arange(nb), np.diff(ref.row_ptr))
    lim = (K * 2.0 ** -(7 * ns - 5) * r[rows][:, :, None] * c[ref.col_idx][:, None, :]
           + 2 * K * 2.0 ** -53 * np.asarray(aref.val))
    assert np.all(np.abs(got.val - ref.val) <= lim)


@pytest.mark.parametrize("nb,density", [(34, 1.0), (35, 1.0), (36, 0.9), (37, 1.0), (39, 0.7), (70, 0.6), (131, 0.3)])
@pytest.mark.parametrize("prec", [TF32, BF16])
def test_wide_tiles(ctx, nb, density, prec):
    """Dense low-precision products around the block count from which a CTA
    takes 256 x 256 elements (1216 blocks of C), with every remainder of the
    block rows modulo four: small integers, so that values, norms and the
    truncation at a median norm are exact; full and upper-triangle products."""
    from paper_1901_07993_gb300 import ifac
    rng = np.random.default_rng(nb)
    A = synth.random_bsr(nb, 64, density, seed=nb, n=nb * 64 - 5)
    B = synth.random_bsr(nb, 64, density, seed=nb + 1, n=nb * 64 - 5)
    A.val[:] = rng.integers(-2, 3, A.val.shape)
    B.val[:] = rng.integers(-2, 3, B.val.shape)
    dA, dB = ifac.upload(ctx, A), ifac.upload(ctx, B)
    for tA, tB in ((False, False), (True, False), (False, True)):
        want = oracle.gemm(A, B, tA, tB, -0.5, 0.0)
        dev = ifac.bsr_gemm_trunc(ctx, dA, tA, dB, tB, -0.5, 0.0, prec)
        got = dev.download()
        assert np.array_equal(got.row_ptr, want.row_ptr) and np.array_equal(got.col_idx, want.col_idx)
        assert np.array_equal(got.val, want.val)
        norms = np.sqrt((np.asarray(want.val) ** 2).sum(axis=(1, 2)))
        total = np.sqrt((norms ** 2).sum())
        assert abs(ifac.bsr_fro(ctx, dev) - total) <= 1e-11 * total
        tau = float(np.median(norms)) * (1 + 1e-9)
        assert ifac.bsr_gemm_trunc(ctx, dA, tA, dB, tB, -0.5, tau, prec).nnzb == int((norms >= tau).sum())
    up, ref = ifac.bsr_gemm_sym_trunc(ctx, dA, True, dA, False, 1.0, 0.0, prec).download(), oracle.gemm(A, A, True)
    assert np.array_equal(up.col_idx, ref.col_idx) and np.array_equal(up.val, ref.val)
