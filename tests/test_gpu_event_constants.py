"""Constants that error events bring into a trajectory (the frame phase after an X or Y error,
the scale of a fused run) keep the norm, however many events there are."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_many_events_keep_the_norm():
    from paper_2301_07264_gb300 import arso
    from workloads import circuits as W
    # T gates leave odd powers of e^{i pi/4} as frame phases: the same rounded constant in every
    # event. Some 70 events a trajectory; their mean stays within one rounding of a scalar
    # (without compensation -8.6e-7, with a factor that rounds back -1.2e-7)
    r = np.random.default_rng(2)
    gates = []
    for _ in range(3000):
        a, b = (int(v) for v in r.permutation(16)[:2])
        name = ("H", "T", "S", "CX", "X", "TDG")[int(r.integers(6))]
        gates.append(W.Gate(name, (a, b) if name == "CX" else (a,)))
    cc = arso.compile_circuit(16, gates)
    errs = arso.sample_errors(cc, 0.02 / 3, 0.02 / 3, 0.02 / 3, 3, 0, 64)
    psi = torch.empty((64, 1 << 16), dtype=torch.complex64, device="cuda")
    torch.cuda.synchronize()
    arso.trajectory_states(cc, errs, 0, 64, psi)
    norm = psi.to(torch.complex128).abs().square().sum(1).sqrt()
    assert abs(float(norm.mean()) - 1.0) < 2.0 ** -24
