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


def test_room_ahead_that_cannot_be_had(G, handles):
    """After a dense cell, 4000 atoms without a pair would get room for 195 thousand: where memory has no place for it
    the call still succeeds, with room for its own pairs."""
    soap, model = handles
    dense = S.displaced_diamond(0, 5, (2, 2, 2), 0.05, a=4.2)
    pos = 20.0 * np.stack(np.meshgrid(*[np.arange(16.0)] * 3, indexing="ij"), -1).reshape(-1, 3)[:4000]
    gas = S.Structure(pos, np.zeros(4000, np.int32), np.eye(3) * 320.0, np.ones(3, np.int32))
    for call, prec in ((soap.descriptor, "fp64"), (model.predict, "fp64")):
        call(_batch(G, dense), prec)
        G.test_fail_alloc_above(6500000)  # their FP64 vectors, 7.8 MB with the slack, do not fit; all that goes by atoms does
        try:
            got = call(_batch(G, gas), prec)
        finally:
            G.test_fail_alloc_above(-1)
        assert b"cudaMalloc" not in G.lib().gap_last_error()
        p = got["local_e"] if isinstance(got, dict) else got
        assert np.allclose(p.cpu().numpy()[1:], p.cpu().numpy()[0], atol=1e-12)


def test_gp_rows_are_a_stage_of_their_own(G, handles):
    """One interval per call, beside the neighbours' two (the inputs before the rows, the lists after them)."""
    _, model = handles
    b = _batch(G, S.displaced_diamond(0, 3, (2, 2, 2), 0.05))
    G.profile_enable(True)
    try:
        for _ in range(3):
            model.predict(b, "fp64")
        stages = G.profile_read()
    finally:
        G.profile_enable(False)
    assert stages["gp_rows"][1] == 3 and stages["gp_rows"][0] > 0.0
    assert stages["neighbours"][1] == 6 and stages["neighbours"][0] > 0.0


def test_variance_of_atoms_of_no_gp(G, handles):
    """Atoms whose species word names no GP have no local energy, and so no variance, in a one-species model too."""
    import torch
    soap, model = handles
    w = S.workload(0)
    cells = [S.displaced_diamond(0, 600 + c, (1, 1, 2), 0.15) for c in range(4)]
    K = model.assemble_knm(G.Batch.from_synth(S.make_batch(cells), device="cuda"), precision="fp64")
    model.set_posterior(K, torch.full((K.shape[0],), 0.1, dtype=torch.float64, device="cuda"))
    good = S.displaced_diamond(0, 700, (2, 2, 2), 0.1)
    bad = S.Structure(good.pos, np.full(good.n, 3, np.int32), good.cell, good.pbc)
    ref = model.predict_variance(_batch(G, good)).cpu().numpy()
    got = model.predict_variance(G.Batch.from_synth(S.make_batch([good, bad]), device="cuda")).cpu().numpy()
    assert ref.max() > 0 and np.allclose(got[:good.n], ref, atol=1e-10 * w.delta ** 2)
    assert np.all(got[good.n:] == 0.0)


@pytest.mark.parametrize("n", [3, 100000])
def test_batches_of_many_configurations(G, handles, n):
    """Isolated atoms, each a configuration of its own: beyond about 80 thousand the cells' geometry is not pinned.  All
    energies are the first one's, a batch of one's."""
    soap, model = handles
    cell = np.repeat(12.0 * np.eye(3)[None], n, 0)
    pos = np.random.default_rng(1).uniform(0.0, 12.0, (n, 3))
    import torch
    dev = lambda a, t: torch.as_tensor(a, dtype=t, device="cuda")  # noqa: E731
    b = G.Batch(dev(pos, torch.float64), dev(np.zeros(n), torch.int32), cell, np.ones((n, 3), np.int32),
                np.arange(n + 1, dtype=np.int32))
    one = G.Batch(dev(pos[:1], torch.float64), dev(np.zeros(1), torch.int32), cell[:1], np.ones((1, 3), np.int32),
                  np.array([0, 1], np.int32))
    for _ in range(2):
        out = model.predict(b, "bf16x3")
        E = out["energy"].cpu().numpy()
        ref = float(model.predict(one, "bf16x3")["energy"][0])
        assert E.shape == (n,) and np.abs(E - ref).max() <= 1e-5 * max(1.0, abs(ref))
        assert float(out["forces"].abs().max()) <= 1e-6
