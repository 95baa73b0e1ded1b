"""GPU parity at the edges of the kernels' tiles: few atoms, few sparse points,
isolated atoms, remainders of the block sizes (tolerances of the parity tests)."""
import numpy as np
import pytest

import oracle as O
from paper_2310_03921_gb300 import synth as S
from _models import oracle_model

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2310_03921_gb300 import build, gap
    build.build()
    return gap


def _cluster(k):
    """The first k atoms of a displaced diamond cell, without periodicity (the last one moved out of reach)."""
    s = S.displaced_diamond(0, 7, (2, 2, 2), 0.1)
    pos = s.pos[:k].copy()
    if k > 1:
        pos[-1] += 40.0
    return S.Structure(pos, s.species[:k], s.cell, np.zeros(3, np.int32))


@pytest.mark.parametrize("M", [1, 7, 9, 65])
@pytest.mark.parametrize("atoms", [1, 7, 9, 64])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-6), ("fp32", 1e-4), ("bf16x3", 1e-4)])
def test_contraction_edges(G, atoms, M, prec, tol):
    soap_o, model_o, sparse, alpha = oracle_model(0, M, n_cells=1 if M <= 64 else 2)
    w = S.workload(0)
    s = _cluster(atoms)
    E, le, F, V = O.predict(soap_o, model_o, s)
    model = G.Model(G.Soap.from_spec(w.soap), sparse, alpha, w.delta, w.zeta)
    out = model.predict(G.Batch.from_synth(S.make_batch([s]), device="cuda"), precision=prec)
    assert np.abs(out["local_e"].cpu().numpy() - le).max() <= tol
    assert np.abs(out["forces"].cpu().numpy() - F).max() <= tol
    assert abs(float(out["energy"][0]) - E) <= tol * atoms
    assert np.abs(out["virial"][0].cpu().numpy() - V).max() <= 10 * tol * max(1.0, np.abs(V).max())


@pytest.mark.parametrize("prec,rel", [("bf16x3", 5e-5), ("bf16x6", 2e-5)])
@pytest.mark.parametrize("M", [1, 127, 129])
def test_knm_edges_one_species(G, M, prec, rel):
    """Force rows at the edges of the point tiles and of the groups of 16 triples: an isolated atom, few and many
    triples per target, D = 105 and 252."""
    for index, cells in ((0, [_cluster(9), S.displaced_diamond(0, 3, (2, 2, 2), 0.1), _cluster(1)]),
                         (1, [S.displaced_diamond(1, 3, (1, 1, 2), 0.1), _cluster(17)])):
        soap_o, model_o, sparse, alpha = oracle_model(index, M, n_cells=1 if M <= 64 else 3)
        w = S.workload(index)
        ref = np.concatenate([O.knm(soap_o, model_o, c) for c in cells])
        model = G.Model(G.Soap.from_spec(w.soap), sparse, alpha, w.delta, w.zeta)
        K = model.assemble_knm(G.Batch.from_synth(S.make_batch(cells), device="cuda"), precision=prec).cpu().numpy()
        assert np.abs(K - ref).max() <= rel * np.abs(ref).max()


@pytest.mark.parametrize("prec,rel", [("bf16x3", 5e-5), ("bf16x6", 2e-5)])
def test_knm_edges_four_species(G, prec, rel):
    """Four GPs in one launch, targets without a source of some species (their columns are zero)."""
    soap_o, model_o, sparse, alpha = oracle_model(3, 33, n_max=4, l_max=3, n_cells=1)
    w = S.workload(3)
    lone = S.Structure(np.zeros((1, 3)), np.array([2], np.int32), np.eye(3) * 30.0, np.zeros(3, np.int32))
    cells = [S.random_packing(3, 5, 8, 0.05, 1.8, n_species=2), lone, S.random_packing(3, 6, 40, 0.05, 1.8, n_species=4)]
    ref = np.concatenate([O.knm(soap_o, model_o, c) for c in cells])
    soap = G.Soap(4, 3, w.soap.rc, w.soap.sigma, w.soap.d, w.soap.central_weight, 4, 4, w.soap.mix_w)
    model = G.Model(soap, sparse, alpha, w.delta, w.zeta)
    K = model.assemble_knm(G.Batch.from_synth(S.make_batch(cells), device="cuda"), precision=prec).cpu().numpy()
    assert np.abs(K - ref).max() <= rel * np.abs(ref).max()
    assert np.all(K[ref == 0.0] == 0.0)


@pytest.mark.parametrize("n", [1, 7, 8, 9, 31, 33, 63, 64, 65, 96, 129])
def test_factor_and_inverse_edges(G, n):
    """Cholesky factor and inverse at the edges of the 8-row panels and 64-row blocks: backward error of the factor
    within 64 n u of the diagonal's scale, R X = I to 1e-10 (the tolerances of the solve's own tests)."""
    rng = np.random.default_rng(n)
    A = rng.normal(size=(n + 40, n)) * 10.0 ** rng.uniform(-2, 2, n)
    Gm = A.T @ A
    R, X = G.test_chol_inv(Gm)
    d = np.sqrt(np.diag(Gm))
    assert (np.abs(R.T @ R - Gm) / np.outer(d, d)).max() <= 64 * n * 2.0 ** -53
    assert np.abs(R @ X - np.eye(n)).max() <= 1e-10
    assert np.all(np.tril(R, -1) == 0.0) and np.all(np.tril(X, -1) == 0.0)


def test_factor_of_an_indefinite_matrix_is_an_error(G):
    for n in (9, 64, 100):
        Gm = np.eye(n)
        Gm[n - 2, n - 2] = -1.0
        with pytest.raises(G.GapError):
            G.test_chol_inv(Gm)


def test_batches_denser_than_any_before(G):
    """A call may size its pair arrays from earlier calls: denser batches, of more and of fewer atoms, give what a
    fresh model gives, and so does a sparse one after them."""
    _, _, sparse, alpha = oracle_model(0, 30, n_cells=1)
    w = S.workload(0)

    def model():
        soap = G.Soap.from_spec(w.soap)
        return soap, G.Model(soap, sparse, alpha, w.delta, w.zeta)

    cells = [_cluster(9), S.displaced_diamond(0, 3, (2, 2, 2), 0.1), S.displaced_diamond(0, 4, (1, 1, 1), 0.1)]
    squeezed = S.displaced_diamond(0, 5, (2, 2, 2), 0.05, a=4.2)
    cells += [squeezed, _cluster(1), _cluster(9), squeezed]
    soap, kept = model()
    for s in cells:
        b = G.Batch.from_synth(S.make_batch([s]), device="cuda")
        fsoap, fresh = model()
        for prec in ("fp64", "bf16x3"):
            got, ref = kept.predict(b, prec), fresh.predict(b, prec)
            for k in ref:
                assert np.array_equal(got[k].cpu().numpy(), ref[k].cpu().numpy()), (k, s.n)
            assert np.array_equal(soap.descriptor(b, prec).cpu().numpy(), fsoap.descriptor(b, prec).cpu().numpy())
        assert soap.descriptor_sizes(b) == fsoap.descriptor_sizes(b)


@pytest.mark.parametrize("prec", ["bf16x3", "bf16x6"])
@pytest.mark.parametrize("atoms,M", [(1, 257), (64, 600), (9, 513)])
def test_gradient_product_split_over_points(G, atoms, M, prec):
    """Few atoms and many sparse points: the gradient product's sum over the points runs in parts."""
    soap_o, model_o, sparse, alpha = oracle_model(1, M, n_cells=3)
    w = S.workload(1)
    s = _cluster(atoms)
    E, le, F, V = O.predict(soap_o, model_o, s)
    model = G.Model(G.Soap.from_spec(w.soap), sparse, alpha, w.delta, w.zeta)
    out = model.predict(G.Batch.from_synth(S.make_batch([s]), device="cuda"), precision=prec)
    assert np.abs(out["local_e"].cpu().numpy() - le).max() <= 1e-4
    assert np.abs(out["forces"].cpu().numpy() - F).max() <= 1e-4
    assert np.abs(out["virial"][0].cpu().numpy() - V).max() <= 1e-3 * max(1.0, np.abs(V).max())


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16x3"])
def test_wrong_species_of_a_one_species_model(G, prec):
    """The host takes n rows for a one-species model: a wrong species on the device leaves no row unset, the call ends
    in an error and the next one is right."""
    soap_o, model_o, sparse, alpha = oracle_model(0, 30, n_cells=1)
    w = S.workload(0)
    model = G.Model(G.Soap.from_spec(w.soap), sparse, alpha, w.delta, w.zeta)
    s = _cluster(64)
    E, le, F, V = O.predict(soap_o, model_o, s)
    bad = S.make_batch([s])
    bad.species[:] = 5
    for call in (model.predict, model.assemble_knm):
        with pytest.raises(G.GapError, match="species"):
            call(G.Batch.from_synth(bad, device="cuda"), precision=prec)
    out = model.predict(G.Batch.from_synth(S.make_batch([s]), device="cuda"), precision=prec)
    assert np.abs(out["local_e"].cpu().numpy() - le).max() <= 1e-4


@pytest.mark.parametrize("zeta", [1, 2, 3, 5])
@pytest.mark.parametrize("prec", ["bf16x3", "bf16x6"])
def test_tensor_core_powers(G, zeta, prec):
    """Powers other than 4 take the general epilogue of the energy products: energies, forces and K_NM rows, at a
    ragged number of rows and of points."""
    soap_o, model_o, sparse, alpha = oracle_model(0, 130, n_cells=3)
    w = S.workload(0)
    mo = O.Model(sparse, alpha, w.delta, zeta)
    s = _cluster(33)
    E, le, F, V = O.predict(soap_o, mo, s)
    ref = O.knm(soap_o, mo, s)
    model = G.Model(G.Soap.from_spec(w.soap), sparse, alpha, w.delta, zeta)
    batch = G.Batch.from_synth(S.make_batch([s]), device="cuda")
    out = model.predict(batch, precision=prec)
    assert np.abs(out["local_e"].cpu().numpy() - le).max() <= 1e-4
    assert np.abs(out["forces"].cpu().numpy() - F).max() <= 1e-4
    K = model.assemble_knm(batch, precision=prec).cpu().numpy()
    assert np.abs(K - ref).max() <= (5e-5 if prec == "bf16x3" else 2e-5) * np.abs(ref).max()
