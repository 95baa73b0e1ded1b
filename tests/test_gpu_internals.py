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
