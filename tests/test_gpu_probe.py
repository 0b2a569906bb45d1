"""The single-error analysis of streaming circuits, one sweep of tile passes with the
measurements inside (fidelity on the circuit's own passes, or on passes of its own where
those are not register-blocked; outcome probability on the doubled state): every
location's value against the FP64 oracle, over tile sizes and odd qubit counts."""
import numpy as np
import pytest

from oracle import exhaustive as ox
from workloads import circuits as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tile,flags", [(14, 8, 0), (14, 10, 0), (15, 11, 0), (14, 12, 0), (15, 13, 0), (15, 14, 0),
                                          (15, 13, 16)])
@pytest.mark.parametrize("kind", ["fidelity", "outcome"])
def test_streaming_single_errors(kind, n, tile, flags):
    from paper_2301_07264_gb300 import arso
    circ = C.random_circuit(n, 40, 100 + n + tile)
    circ.criterion = C.Criterion(kind, target=5, threshold=0.5, aggregate="mean")
    cc = arso.compile_circuit(n, circ.gates, tile_qubits=tile, flags=flags)
    P, per = arso.exhaustive(cc, circ.criterion)
    again = arso.exhaustive(cc, circ.criterion)[1]
    a = ox.analyse(circ)
    want = np.concatenate([a["per_location"][e] for e in ("X", "Z", "Y")])
    assert np.max(np.abs(per - want)) < 1e-5
    assert np.max(np.abs(P[1:] - [a["P_e"][e] for e in ("X", "Z", "Y")])) < 1e-5
    assert np.array_equal(per, again)
