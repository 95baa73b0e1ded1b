"""Calls that size their pair arrays from earlier calls on the same handle."""
import numpy as np
import pytest

from paper_2310_03921_gb300 import synth as S
from _models import oracle_model

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2310_03921_gb300 import build, gap
    build.build()
    return gap


@pytest.fixture
def handles(G):
    _, _, sparse, alpha = oracle_model(0, 30, n_cells=1)
    w = S.workload(0)
    soap = G.Soap.from_spec(w.soap)
    return soap, G.Model(soap, sparse, alpha, w.delta, w.zeta)


def _batch(G, s):
    return G.Batch.from_synth(S.make_batch([s]), device="cuda")


def test_a_denser_batch_leaves_no_error_message(G, handles):
    """The call runs again with room for every pair and succeeds: the last error stays the caller's."""
    soap, model = handles
    wide, dense = S.displaced_diamond(0, 3, (2, 2, 2), 0.05, a=6.5), S.displaced_diamond(0, 5, (2, 2, 2), 0.05, a=4.2)
    for call in (model.predict, soap.descriptor):
        call(_batch(G, wide), "fp64")
        with pytest.raises(G.GapError):
            G.test_tc_force_variant(4)
        message = G.lib().gap_last_error()
        call(_batch(G, dense), "fp64")
        assert G.lib().gap_last_error() == message
