"""One-qubit matrices without a frame form (unitary only up to the rounding of each 32-bit entry),
in passes full of them and in ones that hold a few, against the FP64 oracle."""
import numpy as np
import pytest

from oracle import sampling, statevector
from workloads import circuits as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tile", [(10, 0), (14, 10), (14, 13), (15, 13), (15, 14)])
@pytest.mark.parametrize("every", [1, 2, 40])
def test_full_matrices(n, tile, every):
    from paper_2301_07264_gb300 import arso
    rng = np.random.default_rng(n + every)
    g = []
    for k in range(120):
        q = int(rng.integers(n))
        m = (W.haar_su2(rng) * np.exp(1j * rng.uniform(0, 6))).astype(np.complex64).astype(complex)
        g.append(W.Gate("U", (q,), matrix=m) if k % every == 0 else W.Gate("RX", (q,), (0.1 + k,)))
        if k % 5 == 4:
            g.append(W.Gate("CX", (q, (q + 1) % n)))
    circ = W.Circuit(n, g)
    cc = arso.compile_circuit(n, circ.gates, tile_qubits=tile)
    T, p = 3, 0.05
    errs = arso.sample_errors(cc, p, p, p, 5, 0, T)
    lists = sampling.sample(5, 0, T, circ.L, p, p, p)
    out = torch.empty((T, 1 << n), dtype=torch.complex64, device="cuda")
    arso.trajectory_states(cc, errs, 0, T, out)
    got = out.cpu().numpy()
    for t in range(T):
        assert np.max(np.abs(got[t] - statevector.simulate(circ, lists[t]))) < 1e-5
