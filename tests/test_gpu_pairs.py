"""CZ and dense two-qubit gates on every ordered pair of a tile's qubits (register bits, thread
bits, bits outside the first tile, tile bit 0 on its own path) with Pauli errors between them,
amplitude by amplitude against the FP64 oracle."""
import itertools

import numpy as np
import pytest

from oracle import sampling, statevector
from workloads import circuits as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tile", [(10, 0), (12, 0), (13, 0), (14, 10), (14, 12), (14, 13), (15, 14)])
@pytest.mark.parametrize("name", ["CZ", "U2"])
def test_every_pair(name, n, tile):
    from paper_2301_07264_gb300 import arso
    rng = np.random.default_rng(5)
    pairs = list(itertools.permutations(range(n), 2)) if name == "U2" else list(itertools.combinations(range(n), 2))
    rng.shuffle(pairs)
    gates = [W.Gate("U", (q,), matrix=W.haar_su2(rng)) for q in range(n)]
    for i, (a, b) in enumerate(pairs):
        gates.append(W.Gate(name, (int(a), int(b)), matrix=W.haar_u4(rng) if name == "U2" else None))
        if i % 11 == 10:
            gates.append(W.Gate("H", (int(b),)))
    circ = W.Circuit(n, gates)
    cc = arso.compile_circuit(n, circ.gates, tile_qubits=tile)
    T, p = 3, 0.05
    errs = arso.sample_errors(cc, p, p, p, 11, 0, T)
    lists = sampling.sample(11, 0, T, circ.L, p, p, p)
    out = torch.empty((T, 1 << n), dtype=torch.complex64, device="cuda")
    arso.trajectory_states(cc, errs, 0, T, out)
    got = out.cpu().numpy()
    for t in range(T):  # up to 220 gates of at most 4 * 2^-24 of the norm each, adding like random signs: 3.5e-6
        want = statevector.simulate(circ, lists[t])
        assert np.linalg.norm(got[t] - want) < 1e-5
