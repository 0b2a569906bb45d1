"""The library's memory pool: error lists made on one stream and run on another, several
threads at once, and memory given back with the last handle."""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

from workloads import circuits as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _scores(arso, cc, circ, seed, sample_stream, run_stream, T=200, p=3e-3):
    errs = arso.sample_errors(cc, p, p, p, seed, 0, T, sample_stream)
    out = np.zeros(T)
    arso.run_trajectories(cc, errs, circ.criterion, out, None, run_stream)
    return out


def test_streams_and_threads_share_the_pool():
    from paper_2301_07264_gb300 import arso
    circs = [C.brickwork(14, 6, 1), C.qft_basis(11, 99), C.qaoa_maxcut(8, 3), C.quantum_volume(10, 2)]
    for c in circs:
        if c.criterion.kind == "binning":
            c.criterion = C.Criterion("binning", basis_set=tuple(range(0, 1 << c.n, 3)))
    ccs = [arso.compile_circuit(c.n, c.gates) for c in circs]
    want = [[_scores(arso, cc, c, s, None, None) for s in range(6)] for cc, c in zip(ccs, circs)]
    got = [[None] * 6 for _ in circs]

    def work(k):
        a, b = torch.cuda.Stream(), torch.cuda.Stream()
        for s in range(6):
            got[k][s] = _scores(arso, ccs[k], circs[k], s, a, b)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(circs))]
    [t.start() for t in threads]
    [t.join() for t in threads]
    for w, g in zip(want, got):
        for x, y in zip(w, g):
            assert np.array_equal(x, y)


CHILD = """
import gc
import numpy as np, torch
from paper_2301_07264_gb300 import arso
from workloads import circuits as C
torch.cuda.synchronize()
free0 = torch.cuda.mem_get_info()[0]
circ = C.brickwork(22, 4, 1)
cc = arso.compile_circuit(circ.n, circ.gates)
errs = arso.sample_errors(cc, 1e-2, 1e-2, 1e-2, 0, 0, 40)
arso.run_trajectories(cc, errs, circ.criterion, np.zeros(40))  # 32 MiB a state: over 1 GiB of working states
used = free0 - torch.cuda.mem_get_info()[0]
del cc, errs
gc.collect()
left = free0 - torch.cuda.mem_get_info()[0]
assert used > 1 << 30, used
assert left < (256 << 20) + (64 << 20), left
"""


def test_memory_goes_back_with_the_last_handle():
    # in a process of its own: no other test's handles keep memory mapped
    subprocess.run([sys.executable, "-c", CHILD], check=True, timeout=300,
                   cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
