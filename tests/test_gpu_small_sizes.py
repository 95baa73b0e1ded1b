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
