"""The tile autotuner's classes."""
import numpy as np
import pytest

from paper_2310_03921_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2310_03921_gb300 import build, gap
    build.build()
    return gap


@pytest.mark.parametrize("alone_first", [True, False])
def test_energies_alone_are_a_class_of_their_own(G, alone_first):
    """An energies-only prediction and one with forces each tune the kernel-energy product (one stores W, the other does
    not), in either order.  1100 or 1400 points: column counts that no other test tunes."""
    w = S.workload(0)
    M = 1100 if alone_first else 1400
    rng = np.random.default_rng(M)
    X = 1.0 + 0.2 * rng.normal(size=(M, 105))
    X /= np.linalg.norm(X, axis=1, keepdims=True)
    model = G.Model(G.Soap.from_spec(w.soap), [X], [0.1 * rng.normal(size=M)], w.delta, w.zeta)
    b = G.Batch.from_synth(S.make_batch([S.displaced_diamond(0, 3, (3, 3, 3), 0.1)]), device="cuda")
    kernel = lambda: sum(e["epilogue"] == "kernel" for e in G.tile_tuning())  # noqa: E731
    calls = [dict(forces=False, virial=False), {}]
    n, energy = [kernel()], []
    for kw in calls if alone_first else calls[::-1]:
        energy.append(float(model.predict(b, "bf16x3", **kw)["energy"][0]))
        n.append(kernel())
    assert n == [n[0], n[0] + 1, n[0] + 2]
    assert abs(energy[0] - energy[1]) <= 1e-4 * b.n_atoms
    for kw in calls:  # tuned: the same tile from now on
        e = [float(model.predict(b, "bf16x3", **kw)["energy"][0]) for _ in range(2)]
        assert e[0] == e[1]
    assert kernel() == n[2]
