"""Calls that once went wrong: each test names what it guards."""
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


@pytest.mark.parametrize("bs", [32, 64])
def test_split_block_norms(ctx, bs):
    """Norms of FP64 output blocks that a cluster of four CTAs forms (their sums
    of squares meet in one CTA): products of one block pair each, whose CTAs
    end soonest; the same norms every time, within 1e-13 of the values'."""
    from paper_1901_07993_gb300 import ifac
    nb = 500
    v = np.random.default_rng(1).standard_normal((nb, bs, bs))
    A = synth.HostBSR(nb * bs, bs, np.arange(nb + 1, dtype=np.int32), np.arange(nb, dtype=np.int32), v)
    dA = ifac.upload(ctx, A)
    first = None
    for _ in range(20):
        C = ifac.bsr_gemm_trunc(ctx, dA, False, dA, True, 1.0, 0.0)
        fro = ifac.bsr_fro(ctx, C)
        val = C.download().val
        want = np.sqrt((val ** 2).sum())
        assert abs(fro - want) <= 1e-13 * want
        first = fro if first is None else first
        assert fro == first


def test_adjoint_blocks_without_pairs(ctx):
    """Masked products whose output blocks have no block pair (an F of one
    block): L and the gradient as the oracle's."""
    from paper_1901_07993_gb300 import ifac
    K, tau = 3, 1e-10
    S = synth.chain_overlap(512, 32, seed=0)
    F = synth.HostBSR(S.n, 32, np.concatenate([[0], np.ones(S.nb)]).astype(np.int32), np.zeros(1, np.int32),
                      np.random.default_rng(2).standard_normal((1, 32, 32)))
    c = 1.0 / np.sqrt(oracle.gershgorin(oracle.truncate(S, tau)))
    tape, Fo = oracle.Tape(S, c, K, tau), oracle.Mat(F.n, F.bs, F.row_ptr, F.col_idx, F.val)
    L_ref, blocks = tape.loss(Fo), tape.adjoint(Fo).blocks()
    L, G = ifac.inv_factor_refine_adjoint(ctx, ifac.upload(ctx, S), ifac.upload(ctx, F), K, tau)
    assert abs(L - L_ref) <= 1e-12 * abs(L_ref)
    g = G.download()
    rows = np.repeat(np.arange(S.nb), np.diff(S.row_ptr))
    want = np.array([blocks.get((int(i), int(j)), np.zeros((32, 32))) for i, j in zip(rows, S.col_idx)])
    assert np.linalg.norm(g.val - want) <= 1e-10 * np.linalg.norm(want)


def _first_product(nb, bs, per_row, q):
    """(in a process of its own) S S of a banded matrix as the first call"""
    import torch
    from paper_1901_07993_gb300 import ifac
    w = per_row // 2
    rows, cols = np.nonzero(np.abs(np.subtract.outer(np.arange(nb), np.arange(nb))) <= w)
    rp = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=nb))]).astype(np.int32)
    A = synth.HostBSR(nb * bs, bs, rp, cols.astype(np.int32), np.random.default_rng(3).standard_normal((len(rows), bs, bs)))
    try:
        torch.cuda.init()
        c = ifac.Context()
        dA = ifac.upload(c, A)
        got = ifac.bsr_gemm_trunc(c, dA, False, dA, False, 1.0, 0.0).download()
        ref = oracle.gemm(A, A, False, False, 1.0, 0.0)
        same = np.array_equal(got.row_ptr, ref.row_ptr) and np.array_equal(got.col_idx, ref.col_idx)
        q.put("ok" if same and np.abs(got.val - ref.val).max() <= 1e-12 * np.abs(ref.val).max() else "wrong result")
    except Exception as e:  # reported by the parent
        q.put(f"{type(e).__name__}: {e}")


@pytest.mark.parametrize("nb,per_row", [(395, 3), (396, 3), (397, 3), (372, 5)])
def test_first_product_of_a_process(nb, per_row):
    """The first product of a process, its pattern formed by one CTA whose shared
    memory (4 (2 nb (ceil(nb / 32) | 1) + 2 (nb + 1) + nnzb) bytes, 49,088 and
    49,104 among the cases) lies around the 48 KB that a kernel has without
    asking, its 128 static bytes included."""
    import multiprocessing as mp
    m = mp.get_context("spawn")
    q = m.Queue()
    p = m.Process(target=_first_product, args=(nb, 16, per_row, q))
    p.start()
    try:
        assert q.get(timeout=180) == "ok"
    finally:
        p.join(30)


@pytest.mark.parametrize("bs", [32, 64, 128])
@pytest.mark.parametrize("v", [2.0 ** 19, 2.0 ** 20, 1.5 * 2.0 ** 26, 1.875 * 2.0 ** 27, 2.0 ** 28, 2.0 ** 40])
def test_norms_of_large_values(ctx, bs, v):
    """Block norms of blocks filled with one magnitude: the FP32 sums of squares
    of a whole warp (up to 2^11 values) stay in range or the values are squared
    in FP64.  Sums, products in every precision by the identity (exact), narrow
    tiles, tiles of CTA pairs and of 256 x 256 elements: norms within 2^-36."""
    from paper_1901_07993_gb300 import ifac
    sign = np.random.default_rng(4).integers(0, 2, (40 * 40, bs, bs)) * 2.0 - 1.0

    def full_bsr(nb):
        rp = (np.arange(nb + 1) * nb).astype(np.int32)
        return synth.HostBSR(nb * bs, bs, rp, np.tile(np.arange(nb), nb).astype(np.int32), v * sign[:nb * nb])

    def eye(nb, filled):  # the identity, stored on every block or on the diagonal
        if filled:
            val = np.zeros((nb * nb, bs, bs))
            val[::nb + 1] = np.eye(bs)
            return synth.HostBSR(nb * bs, bs, (np.arange(nb + 1) * nb).astype(np.int32),
                                 np.tile(np.arange(nb), nb).astype(np.int32), val)
        return synth.HostBSR(nb * bs, bs, np.arange(nb + 1, dtype=np.int32), np.arange(nb, dtype=np.int32),
                             np.tile(np.eye(bs), (nb, 1, 1)))

    def check(M, nb):
        want = v * nb * bs
        assert abs(ifac.bsr_fro(ctx, M) - want) <= 2.0 ** -36 * want

    for nb in (2, 36) if bs == 64 else (2,):
        V = ifac.upload(ctx, full_bsr(nb))
        check(ifac.bsr_add(ctx, 1.0, V, 0.0, None, 0.0), nb)
        check(ifac.bsr_add(ctx, 0.5, V, 0.5, V, 0.0), nb)
        for prec in (TF32, BF16, FP64_SPLIT):
            check(ifac.bsr_gemm_trunc(ctx, ifac.upload(ctx, eye(nb, False)), False, V, False, 1.0, 0.0, prec), nb)
    check(ifac.bsr_gemm_trunc(ctx, ifac.upload(ctx, eye(2, False)), False, ifac.upload(ctx, full_bsr(2)), False, 1.0, 0.0)
          if bs < 128 else ifac.bsr_add(ctx, 1.0, ifac.upload(ctx, full_bsr(2)), 0.0, None, 0.0), 2)
    if bs != 64:
        return
    for nb in (20, 36):  # pairs, 256 x 256
        V, E = ifac.upload(ctx, full_bsr(nb)), ifac.upload(ctx, eye(nb, True))
        for prec in (TF32, BF16):
            check(ifac.bsr_gemm_trunc(ctx, E, False, V, False, 1.0, 0.0, prec), nb)
    U = ifac.upload(ctx, full_bsr(2))
    for prec in (FP64, TF32, BF16, FP64_SPLIT):
        check(ifac.bsr_gemm_sym_trunc(ctx, ifac.upload(ctx, eye(2, False)), False, U, False, 1.0, 0.0, prec), 2)


@pytest.mark.parametrize("bs,nb", [(64, 400), (32, 700)])
@pytest.mark.parametrize("tA,tB", [(False, False), (True, False), (False, True), (True, True)])
def test_split_operand_with_one_long_row(ctx, bs, nb, tA, tB):
    """Split products of an operand with one full block row among short ones:
    values within K 2^-(7 s - 5) r_i c_j + 2 K 2^-53 (|A||B|)_ij (K scalar
    terms, s = 7), and no more than six times the time of the same number of
    blocks in short rows (one CTA for every block of the long row: 20 times and
    more)."""
    import time

    import torch
    from paper_1901_07993_gb300 import ifac
    band = np.abs(np.subtract.outer(np.arange(nb), np.arange(nb)))
    long_row = band <= 1
    long_row[nb // 2] = True

    def make(mask, seed):
        rows, cols = np.nonzero(mask)
        rp = np.concatenate([[0], np.cumsum(mask.sum(axis=1))]).astype(np.int32)
        v = np.random.default_rng(seed).standard_normal((len(rows), bs, bs))
        return synth.HostBSR(nb * bs, bs, rp, cols.astype(np.int32), v)

    A, B, even = make(long_row, 1), make(band <= 1, 2), make(band <= 1, 3)
    dA, dB, dE = ifac.upload(ctx, A), ifac.upload(ctx, B), ifac.upload(ctx, even)
    prod = lambda X: ifac.bsr_gemm_trunc(ctx, X, tA, dB, tB, 1.0, 0.0, FP64_SPLIT)
    got, ref = prod(dA).download(), oracle.gemm(A, B, tA, tB, 1.0, 0.0)
    assert np.array_equal(got.row_ptr, ref.row_ptr) and np.array_equal(got.col_idx, ref.col_idx)
    K = nb * bs
    mx = [np.abs(M.val).max() for M in (A, B)]
    assert np.abs(got.val - ref.val).max() <= (K * 2.0 ** -44 + 2 * K * 2.0 ** -53 * K) * mx[0] * mx[1]

    def best(X):
        t = []
        for _ in range(6):
            torch.cuda.synchronize()
            a = time.perf_counter()
            prod(X)
            torch.cuda.synchronize()
            t.append(time.perf_counter() - a)
        return min(t)

    assert best(dA) <= 6 * best(dE)


def test_split_fixed_point_bits():
    """The fixed-point sums keep f = 62 - ceil(log2(1.125 b + 2)) bits, b the
    product of the largest scaled row and column 2-norms, each widened by 0.0125
    sqrt(K) and rounded up by no more than 1e-4.  Here 1.125 b + 2 = 128 (1 -
    1e-4) for norms rounded up by 1e-4, so f = 55: the entries (sums that cancel
    to v 2^-28, v an odd multiple of 2^-27) are multiples of 2^-55 and come out
    exactly; one bit less and each is off by 2^-55."""
    from paper_1901_07993_gb300 import ifac
    ctx = ifac.Context()
    ctx.set_split_slices(8)
    nb, bs = 3, 64
    K = nb * bs
    rk = 0.0125 * np.sqrt(K)
    v = (np.sqrt((128 * (1 - 1e-4) - 2) / 1.125) - rk) / (np.sqrt(K) * 1.0001)
    v = (round(v * 2 ** 27) | 1) / 2.0 ** 27
    j = np.arange(K)
    Ad = np.full((K, K), v)
    Bd = np.where((j[:, None] + j[None, :]) % 2 == 1, v, -v)
    Bd[j, j] += 2.0 ** -28
    rp, ci = (np.arange(nb + 1) * nb).astype(np.int32), np.tile(np.arange(nb), nb).astype(np.int32)
    blocks = lambda D: D.reshape(nb, bs, nb, bs).transpose(0, 2, 1, 3).reshape(nb * nb, bs, bs).copy()
    A, B = (ifac.upload(ctx, synth.HostBSR(K, bs, rp, ci, blocks(D))) for D in (Ad, Bd))
    for X, tX, Y, tY in ((A, False, B, False), (A, True, B, False), (A, False, B, True)):
        got = ifac.bsr_gemm_trunc(ctx, X, tX, Y, tY, 1.0, 0.0, FP64_SPLIT).download()
        assert np.array_equal(got.val, np.full((nb * nb, bs, bs), v * 2.0 ** -28))


@pytest.mark.parametrize("bs,nb", [(32, 2), (64, 700), (128, 40)])
def test_split_norm_bounds_hold(bs, nb):
    """The bounds of rows with many values are bounds: all-equal rows, long
    enough that FP32 sums of their squares round the same way again and again,
    and rows whose largest value comes last; no overflow of the fixed-point sums
    and values within the slices' bound."""
    from paper_1901_07993_gb300 import ifac
    ctx = ifac.Context()
    rng = np.random.default_rng(9)
    rows = np.concatenate([np.zeros(nb, int), np.arange(1, nb)])  # block row 0 full, the others one block
    cols = np.concatenate([np.arange(nb), np.zeros(nb - 1, int)])
    order = np.lexsort((cols, rows))
    rows, cols = rows[order], cols[order]
    rp = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=nb))]).astype(np.int32)
    val = np.full((len(rows), bs, bs), 1.0 - 2.0 ** -24)
    val[rows > 0] = rng.standard_normal((int((rows > 0).sum()), bs, bs)) * np.exp2(np.linspace(-60, 0, bs))
    A = synth.HostBSR(nb * bs, bs, rp, cols.astype(np.int32), val)
    dA = ifac.upload(ctx, A)
    got, ref = ifac.bsr_gemm_trunc(ctx, dA, False, dA, True, 1.0, 0.0, FP64_SPLIT).download(), oracle.gemm(A, A, False, True)
    K = nb * bs
    top = np.abs(A.val).max()
    assert np.abs(got.val - ref.val).max() <= (K * 2.0 ** -44 + 2 * K * 2.0 ** -53 * K) * top ** 2


def _inverse_cholesky(S, dtype, tile=32):
    """Z = L^-T by tiles in dtype: pivots by root and division, panels by
    substitution, a tile's product subtracted whole; W = L^-1 alike."""
    n = S.shape[0]
    A, W = S.astype(dtype), np.zeros((n, n), dtype)
    for k in range(0, n, tile):
        e = min(k + tile, n)
        for j in range(k, e):
            A[j, j] = np.sqrt(A[j, j])
            A[j + 1:, j] /= A[j, j]
            for i in range(j + 1, e):
                A[i:, i] -= A[i:, j] * A[i, j]
        if e < n:
            A[e:, e:] -= np.tril(A[e:, k:e] @ A[e:, k:e].T)
    L = np.tril(A)
    for k in range(0, n, tile):
        e = min(k + tile, n)
        for i in range(k, e):  # the tile's own inverse
            W[i, k:i] = -(L[i, k:i] @ W[k:i, k:i]) / L[i, i]
            W[i, i] = 1 / L[i, i]
        rhs = np.zeros((e - k, k), dtype)
        for m in range(0, k, tile):
            rhs -= L[k:e, m:m + tile] @ W[m:m + tile, :k]
        W[k:e, :k] = W[k:e, k:e] @ rhs
    return W.T


LEAVES = [("cluster", 0), ("cluster", 1), ("cluster", 2), ("chain", 0), ("spd", 2), ("spd", 5), ("points", 18),
          ("points", 10), ("points", 15)]


def _leaf_matrix(kind, k):
    if kind == "cluster":
        return synth.cluster_overlap(512, 32, seed=k).to_dense()[:256, :256]
    if kind == "chain":
        return synth.chain_overlap(512, 32, seed=k).to_dense()[:256, :256]
    r = np.random.default_rng(100 + k)
    n = 256
    if kind == "spd":  # condition 10^k
        Q, _ = np.linalg.qr(r.standard_normal((n, n)))
        S = (Q * np.logspace(0, -k, n)) @ Q.T
        return (S + S.T) / 2
    x = np.sort(r.uniform(0, 1, n) * n * r.uniform(0.45, 0.9))  # condition 8.6e5, 2.7e10, 3.8e10
    return np.exp(-(x[:, None] - x[None]) ** 2) + 10 ** r.uniform(-10.5, -5) * np.eye(n)


@pytest.mark.parametrize("kind,k", LEAVES)
def test_leaf_accuracy(ctx, kind, k):
    """Leaf factors of well and badly conditioned matrices: no more than twice
    as far from the factor in extended precision as the plain tiled algorithm in
    FP64 (with tiles of 16, 32 or 64, whichever is farthest)."""
    import torch
    from paper_1901_07993_gb300 import ifac
    S = _leaf_matrix(kind, k)
    exact = _inverse_cholesky(S, np.longdouble)
    dist = lambda Z: float(np.linalg.norm((Z - exact).astype(float)) / np.linalg.norm(exact.astype(float)))
    plain = max(dist(_inverse_cholesky(S, np.float64, tile)) for tile in (16, 32, 64))
    for count in (1, 20):  # clusters of different sizes
        Z, info, rc = ifac.leaf_invchol_batched(ctx, torch.from_numpy(np.ascontiguousarray(np.tile(S, (count, 1, 1)))).cuda())
        assert rc == 0
        Z = Z.cpu().numpy()
        assert np.array_equal(Z[0], Z[-1])
        assert dist(Z[0]) <= 2 * plain


def test_streams_with_work_ahead():
    """Counts that kernels write for the host: right with work of the caller's
    queued ahead on the stream, and when the context moves to another stream
    between calls (small and large patterns, truncation, plans)."""
    import torch
    from paper_1901_07993_gb300 import ifac
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    ctx = ifac.Context(stream=streams[0].cuda_stream)
    mats = [synth.random_bsr(nb, 32, d, seed=nb) for nb, d in ((40, 0.3), (700, 0.004))]
    refs = [(oracle.gemm(M, M, True, False, 1.0, 30.0), oracle.add(1.0, M, 2.0, M, 1.0)) for M in mats]
    for i in range(6):
        st = streams[i % 2]
        ctx.set_stream(st.cuda_stream)
        M, (prod, total) = mats[(i // 2) % 2], refs[(i // 2) % 2]
        dM = ifac.upload(ctx, M)
        with torch.cuda.stream(st):
            torch.cuda._sleep(100_000_000)  # about 50 ms
        got = ifac.bsr_gemm_trunc(ctx, dM, True, dM, False, 1.0, 30.0, FP64_SPLIT if i % 3 == 2 else FP64).download()
        assert np.array_equal(got.row_ptr, prod.row_ptr) and np.array_equal(got.col_idx, prod.col_idx)
        assert np.abs(got.val - prod.val).max() <= 1e-11 * np.abs(prod.val).max()
        s = ifac.bsr_add(ctx, 1.0, dM, 2.0, dM, 1.0).download()
        assert np.array_equal(s.col_idx, total.col_idx) and np.array_equal(s.val, total.val)


def _on_device(nb, bs, rows, cols, val):
    import torch
    from paper_1901_07993_gb300 import ifac
    rp = torch.from_numpy(np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=nb))]).astype(np.int32)).cuda()
    return ifac.BorrowedBSR(nb * bs, bs, rp, torch.from_numpy(cols.astype(np.int32)).cuda(), val)


@pytest.mark.parametrize("prec", [TF32, FP64_SPLIT])
def test_scan_of_many_counts(ctx, prec):
    """Tile lists and plans of more than 2^18 blocks and tiles, whose scans go
    through the chunks' sums: the identity times a band of small integers is
    that band."""
    import torch
    from paper_1901_07993_gb300 import ifac
    nb, bs, w = 30000, 32, 4
    rows = np.repeat(np.arange(nb), 2 * w + 1)
    cols = (np.arange(nb)[:, None] + np.arange(-w, w + 1)[None]).ravel()
    ok = (cols >= 0) & (cols < nb)
    rows, cols = rows[ok], cols[ok]
    assert len(rows) > 1 << 18
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    val = torch.randint(-3, 4, (len(rows), bs, bs), device="cuda", generator=g).double()
    eye = torch.eye(bs, dtype=torch.float64, device="cuda").expand(nb, bs, bs).contiguous()
    E, A = _on_device(nb, bs, np.arange(nb), np.arange(nb), eye), _on_device(nb, bs, rows, cols, val)
    C = ifac.bsr_gemm_trunc(ctx, E, False, A, False, 1.0, 0.0, prec)
    rp, ci, v = ifac.device_tensors(C)
    assert torch.equal(rp, A.keep[0]) and torch.equal(ci, A.keep[1]) and torch.equal(v, val)


@pytest.mark.parametrize("bs", [32, 64, 128])
@pytest.mark.parametrize("prec", [TF32, BF16, FP64_SPLIT])
def test_plans_counted_first(ctx, bs, prec):
    """Tile plans whose records are counted before they are written (more than
    2^25 words if every tile had all K steps), their tile lists scanned by
    several CTAs: small integers, so that every product is exact."""
    from paper_1901_07993_gb300 import ifac
    nb = 4400 if bs == 128 else 2600
    rng = np.random.default_rng(nb)
    A = synth.random_bsr(nb, bs, 2.0 / nb, seed=1, empty_rows=3)
    B = synth.random_bsr(nb, bs, 2.0 / nb, seed=2)
    A.val[:] = rng.integers(-1, 2, A.val.shape)
    B.val[:] = rng.integers(-1, 2, B.val.shape)
    dA, dB = ifac.upload(ctx, A), ifac.upload(ctx, B)
    for tA in (False, True):
        want = oracle.gemm(A, B, tA, False, 1.0, 0.0)
        assert want.nnzb > 8192 and want.nnzb * nb * {32: 6, 64: 3, 128: 2}[bs] > 1 << 25
        got = ifac.bsr_gemm_trunc(ctx, dA, tA, dB, False, 1.0, 0.0, prec).download()
        assert np.array_equal(got.row_ptr, want.row_ptr) and np.array_equal(got.col_idx, want.col_idx)
        assert np.array_equal(got.val, want.val)


@pytest.mark.parametrize("prec", [TF32, BF16])
def test_wide_plan_counted_first(ctx, prec):
    """The same for tiles of 256 x 256: full operands of 410 block rows against
    FP32 products of the same small integers (exact: |sums| < 2^24)."""
    import torch
    from paper_1901_07993_gb300 import ifac
    nb, bs = 410, 64
    n = nb * bs
    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    D = [torch.randint(-1, 2, (n, n), device="cuda", generator=g).float() for _ in range(2)]
    rows, cols = np.repeat(np.arange(nb), nb), np.tile(np.arange(nb), nb)
    block = lambda X: X.view(nb, bs, nb, bs).transpose(1, 2).reshape(nb * nb, bs, bs)
    dA, dB = (_on_device(nb, bs, rows, cols, block(X).double().contiguous()) for X in D)
    C = ifac.bsr_gemm_trunc(ctx, dA, False, dB, False, 1.0, 0.0, prec)
    assert not torch.backends.cuda.matmul.allow_tf32
    want = block(D[0] @ D[1])
    assert C.nnzb == nb * nb and torch.equal(ifac.device_tensors(C)[2], want.double())


class TrackingAllocator:
    """torch's caching allocator behind the library's allocator interface:
    bytes held now and at most."""

    def __init__(self):
        self.live, self.now, self.peak = {}, 0, 0

    def alloc(self, nbytes, stream):
        import torch
        p = torch.cuda.caching_allocator_alloc(nbytes, stream=int(stream))
        self.live[p] = nbytes
        self.now += nbytes
        self.peak = max(self.peak, self.now)
        return p

    def free(self, ptr, stream):
        import torch
        self.now -= self.live.pop(ptr)
        torch.cuda.caching_allocator_delete(ptr)


@pytest.mark.parametrize("bs,nb,prec", [(16, 400, FP64), (32, 900, TF32), (64, 700, BF16), (64, 700, FP64_SPLIT)])
@pytest.mark.parametrize("tau", [0.0, 1e3])
def test_memory_of_a_callers_allocator(bs, nb, prec, tau):
    """From a caller's allocator a product takes what its result, its copies and
    slices of the operands, and lists of a few words for each block need (here
    1 KB for each block row beside nb^2 words twice and three bitmaps), and the
    lists of results, of sums and truncations too, are at most 64 KB too long."""
    import torch
    from paper_1901_07993_gb300 import ifac
    mem = TrackingAllocator()
    ctx = ifac.Context(allocator=(mem.alloc, mem.free))
    rows, cols = np.nonzero(np.abs(np.subtract.outer(np.arange(nb), np.arange(nb))) <= 1)
    rp = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=nb))]).astype(np.int32)
    val = np.random.default_rng(1).standard_normal((len(rows), bs, bs)) * np.where(rows == cols, 100.0, 0.01)[:, None, None]
    A = synth.HostBSR(nb * bs, bs, rp, cols.astype(np.int32), val)
    dA = ifac.upload(ctx, A)
    exact = lambda n: 4 * (nb + 1) + max(n, 1) * (4 + 8 + 8 * bs * bs)
    base = mem.now
    assert base == exact(A.nnzb)
    full = 5 * nb - 6
    copies = {FP64: 0, TF32: 4, BF16: 2, FP64_SPLIT: 14}[prec] * 2 * (A.nnzb + 1) * bs * bs
    room = exact(full) + copies + 8 * nb * nb + 3 * nb * (nb + 31) // 8 + 1024 * nb + (exact(full) if tau else 0)
    fits = lambda held, need: need <= held <= need + 2 * 65536
    mem.peak = mem.now
    C = ifac.bsr_gemm_trunc(ctx, dA, False, dA, False, 1.0, tau, prec)
    held = mem.now
    assert fits(held - base, exact(C.nnzb)) and (C.nnzb == full) == (tau == 0.0)
    assert mem.peak - base <= room, (mem.peak - base, room)
    want = oracle.gemm(A, A, False, False, 1.0, tau)
    got = C.download()
    assert np.array_equal(got.col_idx, want.col_idx) and np.abs(got.val - want.val).max() <= 4e-3 * np.abs(want.val).max()
    S = ifac.bsr_add(ctx, 1.0, C, 1.0, dA, 0.0)
    assert fits(mem.now - held, exact(S.nnzb))
    held = mem.now
    T = ifac.bsr_truncate(ctx, dA, 5.0 * bs)
    assert T.nnzb == nb and fits(mem.now - held, exact(nb))
    del C, S, T, dA
    torch.cuda.synchronize()
    assert not mem.live


def test_pattern_longer_than_expected(ctx):
    """A product whose operands' rows do not meet evenly (a full column times a
    full row): more blocks than the averages promise, whole all the same."""
    from paper_1901_07993_gb300 import ifac
    for nb in (30, 200, 500):
        col, row = np.zeros((nb, nb), bool), np.zeros((nb, nb), bool)
        col[:, nb // 3] = True
        row[nb // 3] = True
        M = []
        for k, mask in enumerate((col, row)):
            r, c = np.nonzero(mask)
            rp = np.concatenate([[0], np.cumsum(mask.sum(axis=1))]).astype(np.int32)
            M.append(synth.HostBSR(nb * 16, 16, rp, c.astype(np.int32), np.random.default_rng(k).standard_normal((nb, 16, 16))))
        dA, dB = ifac.upload(ctx, M[0]), ifac.upload(ctx, M[1])
        for A, B, hA, hB, t in ((dA, dB, M[0], M[1], False), (dB, dA, M[1], M[0], True)):
            got, want = ifac.bsr_gemm_trunc(ctx, A, t, B, t, 1.0, 0.0).download(), oracle.gemm(hA, hB, t, t, 1.0, 0.0)
            assert got.nnzb == nb * nb and np.array_equal(got.col_idx, want.col_idx)
            assert np.abs(got.val - want.val).max() <= 1e-12 * np.abs(want.val).max()


SPECIAL = np.array([np.inf, -np.inf, np.nan, 1e300, -1e39, 3e38, 2.0 ** -126, 2.0 ** -127, 5e-324, -0.0])


def _with_specials(nb, bs, seed):
    """Full matrix of small values with one special value in some columns."""
    rng = np.random.default_rng(seed)
    val = rng.standard_normal((nb * nb, bs, bs))
    for c in range(0, bs, 3):
        val[rng.integers(nb * nb), rng.integers(bs), c] = SPECIAL[rng.integers(len(SPECIAL))]
    rp, ci = (np.arange(nb + 1) * nb).astype(np.int32), np.tile(np.arange(nb), nb).astype(np.int32)
    return synth.HostBSR(nb * bs, bs, rp, ci, val)


@pytest.mark.filterwarnings("ignore:invalid value", "ignore:overflow")
@pytest.mark.parametrize("bs", [5, 16, 32, 64, 128])
def test_sums_of_infinities_and_nan(ctx, bs):
    """Sums with infinities and NaN among the operands equal numpy's, value for
    value; the norms of their blocks are infinite or NaN, and a truncation
    drops the others only."""
    from paper_1901_07993_gb300 import ifac
    nb = 3
    A, B = _with_specials(nb, bs, 1), _with_specials(nb, bs, 2)
    dA, dB = ifac.upload(ctx, A), ifac.upload(ctx, B)
    for alpha, beta in ((1.0, -1.0), (-0.375, 2.0), (3.0, 0.7)):
        want = alpha * A.val + beta * B.val
        dev = ifac.bsr_add(ctx, alpha, dA, beta, dB, 0.0)
        np.testing.assert_array_equal(dev.download().val, want)
        norms = np.sqrt((want ** 2).sum(axis=(1, 2)))
        fro = ifac.bsr_fro(ctx, dev)
        total = np.sqrt((norms ** 2).sum())
        assert np.isnan(fro) == np.isnan(total) and (np.isnan(total) or fro == total)
        tau = 4.0 * bs  # above every ordinary block, below infinity
        assert ifac.bsr_truncate(ctx, dev, tau).nnzb == int((~(norms < tau)).sum())


@pytest.mark.filterwarnings("ignore:invalid value", "ignore:overflow")
@pytest.mark.parametrize("bs", [32, 64, 128])
@pytest.mark.parametrize("prec", [TF32, BF16])
@pytest.mark.parametrize("tB", [False, True])
def test_low_precision_copies_of_special_values(ctx, bs, prec, tB):
    """The identity times a matrix with infinities, NaN, values past FP32's range
    and subnormals: the rounded value in its place, and 0 times infinity or NaN
    elsewhere in its column."""
    from paper_1901_07993_gb300 import ifac
    nb = 2
    n = nb * bs
    A = _with_specials(nb, bs, 3)
    eye = synth.HostBSR(n, bs, A.row_ptr, A.col_idx, np.stack([np.eye(bs) * (i == j) for i in range(nb) for j in range(nb)]))
    if prec == TF32:  # FP32, then ten fraction bits, ties away
        f = A.val.astype(np.float32)
        low = ((f.view(np.uint32) + np.uint32(0x1000)) & np.uint32(0xffffe000)).view(np.float32)
    else:  # seven fraction bits of the FP64 value, ties to even
        f = A.val
        u = f.view(np.uint64)
        u = (u + np.uint64((1 << 44) - 1) + ((u >> np.uint64(45)) & np.uint64(1))) & ~np.uint64((1 << 45) - 1)
        low = u.view(np.float64).astype(np.float32)
    low = np.where(np.isfinite(f), low, f).astype(float)
    low = np.where(np.abs(A.val) < 2.0 ** -126, 0.0, low)
    D = low.reshape(nb, nb, bs, bs).transpose(0, 2, 1, 3).reshape(n, n)
    M = D.T if tB else D
    bad = ~np.isfinite(M)
    want = np.where(np.isfinite(M), M, 0.0)
    cols = bad.any(axis=0)
    want[:, cols] = np.nan
    want[bad & (bad.sum(axis=0) == 1)[None, :]] = M[bad & (bad.sum(axis=0) == 1)[None, :]]
    got = ifac.bsr_gemm_trunc(ctx, ifac.upload(ctx, eye), False, ifac.upload(ctx, A), tB, 1.0, 0.0, prec).download()
    G = got.val.reshape(nb, nb, bs, bs).transpose(0, 2, 1, 3).reshape(n, n)
    np.testing.assert_array_equal(G, want)


@pytest.mark.filterwarnings("ignore:invalid value", "ignore:overflow")
def test_symmetric_completion_of_infinities_and_nan(ctx):
    """Symmetric products whose values hold infinities and NaN: the upper
    blocks are the product's, the lower ones their transposes."""
    from paper_1901_07993_gb300 import ifac
    nb, bs = 3, 64
    A = _with_specials(nb, bs, 5)
    dA = ifac.upload(ctx, A)
    full = ifac.bsr_gemm_trunc(ctx, dA, True, dA, False, -0.5, 0.0).download()
    got = ifac.bsr_gemm_sym_trunc(ctx, dA, True, dA, False, -0.5, 0.0).download()
    assert not np.isfinite(full.val).all() and np.isfinite(full.val).any()
    for i in range(nb):
        for j in range(nb):
            block = full.val[i * nb + j] if j >= i else full.val[j * nb + i].T
            np.testing.assert_array_equal(got.val[i * nb + j], block)
