"""Small angles in the register program: errors on qubits whose pending phase is small, where
the float cosine of the phase is exactly 1 although the phase is not, against the FP64 oracle."""
import numpy as np
import pytest

from oracle import statevector
from workloads import circuits as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _phases(n, angle):
    """Small phases of every kind pending on the qubits (RZ, P, one left by a fused run), then a
    rotation of each qubit that mixes the halves an X or Y error exchanges."""
    rng = np.random.default_rng(1)
    g = [W.Gate("H", (q,)) for q in range(n)]
    for k in range(3):
        for q in range(n):
            g.append(W.Gate("RZ" if q % 2 else "P", (q,), (angle * (1 + k),)))
        for q in range(0, n - 1, 2):
            g += [W.Gate("CX", (q, q + 1)), W.Gate("RZ", (q + 1,), (angle,)), W.Gate("CX", (q, q + 1))]
        g += [W.Gate("U", (q,), matrix=W.haar_su2(rng)) for q in range(n)]
    return W.Circuit(n, g)


# 2-norm: some 150 FP32 gates of at most 6e-8 each, added as a random walk or fully in step, stay
# below 1e-5; a correction left out at a phase of 1e-4 is off by 1e-4 and more
@pytest.mark.parametrize("angle", [1e-7, 1e-5, 5e-5, 1e-4, 2e-4, 1e-3])
@pytest.mark.parametrize("n,tile", [(10, 0), (14, 10), (14, 12), (15, 13)])
def test_errors_on_small_phases(n, tile, angle):
    from paper_2301_07264_gb300 import arso
    circ = _phases(n, angle)
    cc = arso.compile_circuit(n, circ.gates, tile_qubits=tile)
    rng = np.random.default_rng(2)
    lists = [[(l, 1 + 2 * (l % 2)) for l in sorted(set(int(v) for v in rng.integers(0, circ.L, 12)))] for _ in range(4)]
    errs = arso.error_list_from_host(cc, lists)
    out = torch.empty((len(lists), 1 << n), dtype=torch.complex64, device="cuda")
    arso.trajectory_states(cc, errs, 0, len(lists), out)
    got = out.cpu().numpy()
    for k, ev in enumerate(lists):
        assert np.linalg.norm(got[k] - statevector.simulate(circ, ev)) < 2e-5, ev


# one rotation's own amplitude, far below what the rest of the state rounds to
@pytest.mark.parametrize("n,tile", [(10, 0), (14, 12)])
@pytest.mark.parametrize("fused,angle", [(False, 1e-6), (False, 1e-9), (False, 1e-12), (False, 1e-14),
                                         (True, 1e-6), (True, 1e-9), (True, 1e-12)])
def test_tiny_rotations_keep_their_amplitude(n, tile, fused, angle):
    from paper_2301_07264_gb300 import arso
    g = [W.Gate("RX", (1,), (angle,))]
    if fused:  # between CX gates that a run would take it with
        g = [W.Gate("CX", (0, 1))] + g + [W.Gate("CX", (0, 1)), W.Gate("CX", (1, 0))]
    cc = arso.compile_circuit(n, g, tile_qubits=tile)
    out = torch.empty(1 << n, dtype=torch.complex64, device="cuda")
    arso.reference_state(cc, out)
    got = complex(out[3 if fused else 2].item())
    assert abs(got / (-1j * np.sin(angle / 2)) - 1) < 1e-6, got
