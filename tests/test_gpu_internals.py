"""Single kernels of the library against an independent computation, through the test hooks."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2310_03921_gb300 import build, gap
    build.build()
    return gap


@pytest.mark.parametrize("n_gp", [1, 2, 4, 8])
@pytest.mark.parametrize("n", [1, 1023, 1025, 8192, 8193, 20000, 67583])
def test_rows_of_every_gp(G, n, n_gp):
    """Row lists, ranks and counts exactly the host's: one block (up to 8192 atoms) and a block per 1024, atoms without
    a GP among them, species in runs and mixed."""
    rng = np.random.default_rng(10 * n + n_gp)
    mixed = rng.integers(0, n_gp + 1, n)  # species n_gp has no GP
    runs = np.sort(mixed)[::-1]
    for z in (mixed, runs):
        rows, counts, gp, rank = G.test_gp_rows(z, n_gp)
        assert np.array_equal(gp, np.where(z < n_gp, z, -1))
        want_rank = np.full(n, -1)
        for s in range(n_gp):
            atoms = np.flatnonzero(z == s)
            want_rank[atoms] = np.arange(atoms.size)
            assert counts[s] == atoms.size
            assert np.array_equal(rows[s, :atoms.size], atoms) and np.all(rows[s, atoms.size:] == -1)
        assert np.array_equal(rank, want_rank)


def test_rows_of_a_one_species_model(G):
    for n in (7, 9001):
        rows, counts, gp, rank = G.test_gp_rows(np.full(n, 5), 1, one=True)
        assert counts[0] == n and np.all(gp == 0)
        assert np.array_equal(rows[0], np.arange(n)) and np.array_equal(rank, np.arange(n))


@pytest.mark.parametrize("blocks", [0, 1, 2, 3, 4, 5, 31, 32])
def test_wait_expiry_in_the_middle_of_a_product(G, blocks):
    """A CTA whose waits run out after some blocks of K waits for the copies and MMAs it has issued and ends in an error
    status; the product after it is exact."""
    rng = np.random.default_rng(3)
    A = rng.integers(-8, 9, size=(500, 256)).astype(np.float32)
    B = rng.integers(-8, 9, size=(700, 256)).astype(np.float32)
    st, code = G.test_tc_expiry(blocks)
    assert (st, code) == (0, 0) if blocks == 32 else (st == -4 and code), (st, code)
    assert np.array_equal(G.test_bf16_gemm(A, B), A @ B.T)


def _pairs(counts, seed, span=3.0):
    """Random pair derivatives and vectors of atoms with that many pairs, magnitudes over 10^(+-span), the last pair of
    every atom nearly cancelling its first."""
    rng = np.random.default_rng(seed)
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    P = off[-1]
    f = (rng.normal(size=(P, 3)) * 10.0 ** rng.uniform(-span, span, (P, 1))).astype(np.float32)
    v = rng.normal(size=(P, 4)).astype(np.float32)
    for a, b in zip(off[:-1], off[1:]):
        if b - a > 1:
            f[b - 1], v[b - 1] = -f[a], v[a] * np.float32(1 + 2.0 ** -20)
    return off, rng.permutation(P).astype(np.int32), v, f


def _gather_exact(off, rev, v, f):
    """Sums in exact integer arithmetic by math.fsum of the exact FP64 products, and the sums of magnitudes."""
    import math
    n = off.size - 1
    f, v = f.astype(np.float64), v.astype(np.float64)  # products of two FP32 numbers are exact in FP64
    F, Fa, W, Wa = np.zeros((n, 3)), np.zeros((n, 3)), np.zeros((n, 9)), np.zeros((n, 9))
    for j in range(n):
        p = np.arange(off[j], off[j + 1])
        for a in range(3):
            t = np.concatenate([f[p, a], -f[rev[p], a]])
            F[j, a], Fa[j, a] = math.fsum(t), np.abs(t).sum()
            for b in range(3):
                t = -f[p, a] * v[p, b]
                W[j, 3 * a + b], Wa[j, 3 * a + b] = math.fsum(t), np.abs(t).sum()
    return F, Fa, W, Wa


PAIR_COUNTS = [[1], [3], [8], [0, 9, 0, 40], list(range(35)), [29] * 50, [500, 3, 120]]


@pytest.mark.parametrize("counts", PAIR_COUNTS, ids=len)
def test_pair_sums_of_fp32_terms(G, counts):
    """Compensated sums with exact products: of n pairs the second word collects up to 4 n roundings of 2^-24 of the
    terms and rounds as often itself, at most (4 n)^2 2^-48 of them (sums of FP32-rounded products are off by 2^-25)."""
    off, rev, v, f = _pairs(counts, len(counts))
    F, W = G.test_gather(off, rev, v, f)
    Fx, Fa, Wx, Wa = _gather_exact(off, rev, v, f)
    bound = (4.0 * np.array(counts)[:, None]) ** 2 * 2.0 ** -48
    assert np.all(np.abs(F - Fx) <= bound * Fa)
    assert np.all(np.abs(W - Wx) <= bound * Wa)
    if max(counts) > 1:
        print("largest error over the terms' magnitudes: F %.2e W %.2e" % (
            (np.abs(F - Fx)[Fa > 0] / Fa[Fa > 0]).max(), (np.abs(W - Wx)[Wa > 0] / Wa[Wa > 0]).max()))


@pytest.mark.parametrize("counts", PAIR_COUNTS, ids=len)
def test_pair_sums_hold_no_less_than_fp64(G, counts):
    """Three words per sum: the last one rounds at most (4 n)^3 2^-72 of the terms' magnitudes, the result once and its
    lower words once, 2^-52 of it."""
    off, rev, v, f = _pairs(counts, 7 + len(counts))
    F, W = G.test_gather(off, rev, v, f)
    Fx, Fa, Wx, Wa = _gather_exact(off, rev, v, f)
    tail = (4.0 * np.array(counts)[:, None]) ** 3 * 2.0 ** -72
    assert np.all(np.abs(F - Fx) <= 2.0 ** -52 * np.abs(Fx) + tail * Fa)
    assert np.all(np.abs(W - Wx) <= 2.0 ** -52 * np.abs(Wx) + tail * Wa)


def test_pair_sums_beyond_fp32(G):
    """Sums that leave FP32's range, infinite terms and NaN: as the FP64 sums."""
    off, rev, v, f = _pairs([4, 12, 3, 20, 0, 7], 3)
    rev = np.arange(off[-1], dtype=np.int32)  # a pair's force against itself: F = 0 for finite terms
    f[off[0]:off[1]] = 3e38
    f[off[1]] = np.inf
    f[off[3] + 9, 1] = np.nan
    F, W = G.test_gather(off, rev, v, f)
    f64, v64 = f.astype(np.float64), v.astype(np.float64)
    with np.errstate(invalid="ignore"):
        for j in range(6):
            p = slice(off[j], off[j + 1])
            t = f64[p, :, None] * v64[p, None, :3]
            Wx, Wa, Fx = -t.sum(0).reshape(9), np.abs(t).sum(0).reshape(9), (f64[p] - f64[rev[p]]).sum(0)
            ok = np.isfinite(Wx)
            assert np.array_equal(np.isnan(W[j]), np.isnan(Wx))
            assert np.array_equal(W[j][np.isinf(Wx)], Wx[np.isinf(Wx)])
            assert np.all(np.abs(W[j] - Wx)[ok] <= 1e-13 * Wa[ok])
            assert np.array_equal(F[j], Fx, equal_nan=True)


@pytest.mark.parametrize("K,nsplit", [(16, 2), (256, 2), (320, 2), (48, 3)])
@pytest.mark.parametrize("counts", [[48], [0, 70, 1, 16, 15, 17, 0], [400, 33, 5], [31] * 40], ids=["one", "ragged", "long", "many"])
def test_knm_target_sums(G, counts, K, nsplit):
    """A target's sum over its triples: FP32 over at most sixteen of them, FP64 beyond.  Every J . X is a product of
    small whole numbers, exact on the tensor cores.  A target's first triple is 2^26 times the others and its own tile
    holds nothing else of the target, so that tile is exact, the others are off by sixteen roundings of 2^-24 of their
    terms at most and the FP64 sum by 2^-50 of the whole; a longer FP32 sum would lose the small terms altogether."""
    rng = np.random.default_rng(K + len(counts))
    T, M, R = sum(counts), 130, 37
    src = rng.integers(0, R, T)
    J = rng.integers(1, 4, (3 * T, K)).astype(np.float32) * (rng.random((3 * T, K)) < 8 / K)
    X = rng.integers(1, 4, (M, K)).astype(np.float32)
    W = rng.uniform(0.5, 1.5, (R, M)).astype(np.float32)
    W[0] = 1.0
    J = J.reshape(T, 3, K)
    off = np.concatenate([[0], np.cumsum(counts)])
    for a, c in zip(off, counts):
        if c:
            src[a] = 0
            J[a] *= 2.0 ** 26
            J[a + 1:a + min(c, 16)] = 0.0
    out = G.test_knm_rows(counts, src, J.reshape(3 * T, K), X, W, nsplit)
    P = (J.astype(np.float64) @ X.T.astype(np.float64)) * W[src].astype(np.float64)[:, None, :]
    for j, (a, c) in enumerate(zip(off, counts)):
        exact, rest = P[a:a + c].sum(0), P[a + 1:a + c].sum(0)
        bound = 16 * 2.0 ** -24 * rest + 2.0 ** -50 * np.abs(exact)
        assert np.all(np.abs(out[3 * j:3 * j + 3] - exact) <= bound), j


def test_pair_root_and_quotient(G):
    """Correctly rounded but for one result in 2^32 (the error before the last rounding is 2^-33 of the last place), so
    at most one of these three million may be the neighbouring number."""
    rng = np.random.default_rng(5)
    n = 1 << 20
    r2 = np.concatenate([rng.uniform(1e-6, 30.0, n), np.ldexp(rng.uniform(1, 2, n), rng.integers(-110, 110, n)),
                         30.25 * (1 - np.ldexp(1.0, -rng.integers(1, 53, 1000))),  # at a cutoff
                         1e-30 * rng.uniform(0.1, 10, 1000), np.ldexp(rng.integers(1, 1 << 52, 1000).astype(float), -30)])
    r = np.sqrt(r2[rng.permutation(r2.size)])
    a = r2 * np.where(rng.random(r2.size) < 0.5, -1.0, 1.0)
    root, _ = G.test_fp64_pair(r2, r)
    _, quot = G.test_fp64_pair(a, r)
    for got, ref in ((root, np.sqrt(r2)), (quot, a / r)):
        off = got != ref
        assert off.sum() <= 1 and np.all(np.abs(got - ref) <= np.spacing(np.abs(ref)))


def test_pair_root_and_quotient_of_other_arguments(G):
    a = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1e-320, 1e308, -1.0, 5e-324, 1e-200, 1.0, 1.0, 0.0, 1.0])
    b = np.array([2.0, 3.0, 2.0, 2.0, 2.0, 2.0, 1e-10, 2.0, 3.0, 1e200, 0.0, np.inf, 0.0, np.nan])
    with np.errstate(all="ignore"):
        root, quot = G.test_fp64_pair(a, b)
        assert np.array_equal(root, np.sqrt(a), equal_nan=True)
        assert np.array_equal(quot, a / b, equal_nan=True)
