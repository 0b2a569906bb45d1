"""The register program's frame forms of one-qubit gates (arso register-blocked
kernels): cases where a form ends or changes - the rescaling of a long run of dense
gates, matrices that are diagonal, antidiagonal, near a right angle or not unitary,
phases pending at CX targets, SWAP and two-qubit matrices - with errors after every
gate, amplitude by amplitude against the FP64 oracle."""
import numpy as np
import pytest

from oracle import sampling, statevector
from workloads import circuits as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _gate(name, *q, params=(), matrix=None):
    return W.Gate(name, q, tuple(params), None if matrix is None else np.asarray(matrix, dtype=complex))


def _rx_run(n):  # 320 dense gates: the stored state outgrows the true one by 2^40 several times
    rng = np.random.default_rng(1)
    g = []
    for k in range(320):
        g.append(_gate("RX", k % n, params=(float(rng.uniform(1.2, 1.9)),)))
        if k % 29 == 28:
            g.append(_gate("CX", k % n, (k + 1) % n))
    return g


def _special(n):
    rng = np.random.default_rng(2)
    e = np.exp(1j * 0.3)
    mats = [[[e, 0], [0, np.conj(e)]], [[0, e], [1j, 0]], [[1, 0], [0, 1]], [[0, 1], [1, 0]],
            [[0.9, 0.2], [0.1j, 1.05]], [[np.cos(1e-8), -np.sin(1e-8)], [np.sin(1e-8), np.cos(1e-8)]]]
    g = [_gate("H", q) for q in range(n)]
    for k in range(60):
        q, r = (int(v) for v in rng.permutation(n)[:2])
        kind = k % 6
        if kind < 2:
            g.append(_gate("U", q, matrix=mats[int(rng.integers(len(mats)))]))
        g.append(_gate(("T", "S", "RZ", "Z", "TDG", "P")[kind], q, params=(0.7 + k,)))
        g.append(_gate(("CX", "CX", "SWAP", "CP", "CZ", "U2")[kind], r, q, params=(0.4,),
                       matrix=W.haar_u4(rng) if kind == 5 else None))
        g.append(_gate(("H", "Y", "X", "RY", "U", "H")[kind], r, params=(np.pi / 2,),
                       matrix=W.haar_su2(rng) if kind == 4 else None))
    return g


@pytest.mark.parametrize("n,tile", [(10, 0), (13, 0), (14, 10), (14, 11), (15, 12), (15, 13), (15, 14)])
@pytest.mark.parametrize("make", [_rx_run, _special])
def test_frame_forms(make, n, tile):
    from paper_2301_07264_gb300 import arso
    circ = W.Circuit(n, make(n))
    cc = arso.compile_circuit(n, circ.gates, tile_qubits=tile)
    T, p = 3, 0.1
    errs = arso.sample_errors(cc, p, p, p, 7, 0, T)
    lists = sampling.sample(7, 0, T, circ.L, p, p, p)
    out = torch.empty((T, 1 << n), dtype=torch.complex64, device="cuda")
    arso.trajectory_states(cc, errs, 0, T, out)
    got = out.cpu().numpy()
    for t in range(T):
        want = statevector.simulate(circ, lists[t])
        assert np.max(np.abs(got[t] - want)) < 1e-5 * max(1.0, np.max(np.abs(want)))
