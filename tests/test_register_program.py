"""The register programs that the host writes for the complex64 kernels, run on the CPU in FP64
with the constants they hold (program_emulator.cpp): what the gates become, and how far the
constants alone take a trajectory from the FP64 one."""
import os
import subprocess

import numpy as np
import pytest

from paper_2301_07264_gb300 import arso, build
from workloads import circuits as W

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def emulate(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("emulator") / "program_emulator")
    cuda = build._cuda_home()
    flags = [f for f in build.CXX_FLAGS if f not in ("-fPIC", "-Wall")]
    subprocess.run(["g++", *flags, "-w", "-I", os.path.join(cuda, "include"), "-I", build.INCLUDE, "-o", exe,
                    os.path.join(HERE, "program_emulator.cpp")], check=True)

    def run(circ, tile=0, seed=0, events=0):
        lines = [f"{circ.n} {tile} {seed} {events}"]
        for g in circ.gates:
            m = [] if g.matrix is None else [v for z in np.asarray(g.matrix, complex).reshape(-1) for v in (z.real, z.imag)]
            q = list(g.qubits) + [0]
            lines.append(" ".join(map(repr, [arso.GATE_KIND[g.name], q[0], q[1], float(g.params[0]) if g.params else 0.0,
                                             len(m), *map(float, m)])))
        r = subprocess.run([exe], input="\n".join(lines), capture_output=True, text=True, check=True)
        w = r.stdout.split()
        return {w[i]: float(w[i + 1]) for i in range(0, len(w), 2)}

    return run


def _rounded(circ):
    """The circuit with its matrices in complex64."""
    return W.Circuit(circ.n, [W.Gate(g.name, g.qubits, g.params, None if g.matrix is None else
                                     np.asarray(g.matrix).astype(np.complex64).astype(complex)) for g in circ.gates])


@pytest.mark.parametrize("n,tile", [(10, 0), (14, 12)])
def test_matrices_given_in_32_bits_take_the_frame_form(emulate, n, tile):
    # [[a, b], [-conj b, conj a]] is unitary up to a scale whatever the rounding of a and b, so
    # none needs a full matrix; the scale stays in the result
    circ = _rounded(W.brickwork(n, 10, 3))
    r = emulate(circ, tile, 1, 6)
    assert r["dense"] == 0
    assert r["error"] < 2e-6  # 100 constants of at most 6e-8, as a random walk with a factor of three


def _clifford_t(n, G, seed):
    r = np.random.default_rng(seed)
    out = []
    for _ in range(G):
        a, b = (int(v) for v in r.permutation(n)[:2])
        name = ("H", "T", "S", "CX", "X", "TDG")[int(r.integers(6))]
        out.append(W.Gate(name, (a, b) if name == "CX" else (a,)))
    return W.Circuit(n, out)


@pytest.mark.parametrize("circ,tile", [(W.cuccaro_adder(7, 100, 77), 13), (W.cuccaro_adder(7, 100, 77), 10),
                                       (_clifford_t(14, 600, 1), 10), (_clifford_t(12, 600, 1), 0)])
@pytest.mark.parametrize("events", [0, 5, 30])
def test_constants_do_not_add_up(emulate, circ, tile, events):
    # the scalar of a frame, the phase after an error and the scale of a run are rounded constants
    # that all amplitudes share; however many there are, the norm is off by one rounding of the
    # scalar (2^-24), not by one a pass and an event
    assert abs(emulate(circ, tile, 3, events)["norm"]) < 2.0 ** -24
