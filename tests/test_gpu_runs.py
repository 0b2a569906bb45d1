"""Fused runs of the register program (Toffoli networks, CX conjugations of rotations, H
pairs around them): the fused form, and the gates one by one in a trajectory with an error
inside the run, both against the FP64 oracle amplitude by amplitude."""
import numpy as np
import pytest

from oracle import statevector
from workloads import circuits as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _circuit(n, seed):
    rng = np.random.default_rng(seed)
    g = [W.Gate("H", (q,)) for q in range(n)] + [W.Gate("U", (q,), matrix=W.haar_su2(rng)) for q in range(n)]
    for k in range(14):
        a, b, c = (int(v) for v in rng.permutation(n)[:3])
        if k % 5 == 4:
            a, b, c = (0, a, b) if a and b else (a, b, c)  # the lanes of the packed registers
        kind = k % 7
        if kind in (0, 1):
            g += W.toffoli_clifford_t(a, b, c)
        elif kind == 2:  # CCZ: H around a Toffoli
            g += [W.Gate("H", (c,))] + W.toffoli_clifford_t(a, b, c) + [W.Gate("H", (c,))]
        elif kind == 3:  # a ZZ rotation
            g += [W.Gate("CX", (a, b)), W.Gate("RZ", (b,), (0.3 + k,)), W.Gate("CX", (a, b))]
        elif kind == 4:  # flips under conditions with a constant, and phases pending on the target
            g += [W.Gate("Z", (c,)), W.Gate("X", (a,))] + W.toffoli_clifford_t(a, b, c) + [W.Gate("X", (a,)), W.Gate("CX", (b, c))]
        elif kind == 5:
            g += [W.Gate("T", (c,)), W.Gate("RZ", (a,), (0.9,))] + W.toffoli_clifford_t(a, b, c)
        else:
            g += [W.Gate("S", (c,)), W.Gate("CX", (a, c)), W.Gate("CX", (b, c)), W.Gate("CX", (a, c))]
        if k % 3 == 2:
            g.append(W.Gate("RY", (c,), (0.5 + k,)))
    return W.Circuit(n, g)


@pytest.mark.parametrize("n,tile", [(10, 0), (13, 0), (14, 10), (14, 12), (15, 13), (15, 14)])
def test_fused_runs(n, tile):
    from paper_2301_07264_gb300 import arso
    circ = _circuit(n, n + tile)
    cc = arso.compile_circuit(n, circ.gates, tile_qubits=tile)
    rng = np.random.default_rng(3)
    lists = [[]] + [[(int(l), 1 + k % 3)] for k, l in enumerate(np.linspace(0, circ.L - 1, 36).astype(int))]
    for _ in range(8):
        locs = sorted(set(int(v) for v in rng.integers(0, circ.L, 5)))
        lists.append([(l, int(rng.integers(1, 4))) for l in locs])
    errs = arso.error_list_from_host(cc, lists)
    out = torch.empty((len(lists), 1 << n), dtype=torch.complex64, device="cuda")
    arso.trajectory_states(cc, errs, 0, len(lists), out)
    got = out.cpu().numpy()
    for k, ev in enumerate(lists):
        assert np.max(np.abs(got[k] - statevector.simulate(circ, ev))) < 1e-5, ev
