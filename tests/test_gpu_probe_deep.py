"""Single-error analysis of a circuit whose gates share one tile: its one pass is cut between
phases, so that the sums fit their buffer. One-qubit rotations only, so every value is known in
closed form."""
import numpy as np
import pytest

from workloads import circuits as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["fidelity", "outcome"])
def test_deep_pass(kind):
    from paper_2301_07264_gb300 import arso
    n, act, G = 20, 12, 20004
    rng = np.random.default_rng(1)
    ang = rng.uniform(-3, 3, G)
    for q in range(act):  # every qubit ends at 0.3, so that outcome 0 is likely
        ang[G - act + q] = 0.3 - ang[q:G - act:act].sum()
    gates = [W.Gate("RY", (k % act,), (float(ang[k]),)) for k in range(G)]
    after = np.stack([np.cumsum(ang[q::act]) for q in range(act)], 1).reshape(-1)  # angle after gate k
    if kind == "fidelity":
        want = np.concatenate([np.sin(after) ** 2, np.cos(after) ** 2, np.zeros(G)])
    else:
        rest = 0.3 - after  # <0| RY(rest) P RY(after) |0>, and the other qubits' cos^2(0.15)
        c, s, rc, rs = np.cos(after / 2), np.sin(after / 2), np.cos(rest / 2), np.sin(rest / 2)
        others = np.cos(0.15) ** (2 * (act - 1))
        want = np.concatenate([(rc * s - rs * c) ** 2, (rc * c + rs * s) ** 2, (rc * s + rs * c) ** 2]) * others
    cc = arso.compile_circuit(n, gates)
    _, per = arso.exhaustive(cc, W.Criterion(kind, target=0, threshold=0.5, aggregate="mean"))
    # 20,004 gates of at most 6e-8 each as a random walk: 8.5e-6; a factor of ten, twice for the square
    assert np.max(np.abs(per - want)) < 2e-4
