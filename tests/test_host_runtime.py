"""The library's host side against a runtime without a GPU (fake_cuda.cpp): what is waited for
before memory is read or freed."""
import ctypes as C

import numpy as np
import pytest

from paper_2301_07264_gb300 import arso
from workloads import circuits as W

import fake_cuda  # noqa: E402  (beside this file)


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    return fake_cuda.load(tmp_path_factory.mktemp("fake"))


@pytest.fixture
def lib(library):
    library.fake_fail_at(-1)
    library.fake_fail_launch_at(-1)
    library.fake_device(0)
    library.fake_reset_counts()
    return library


def ok(lib, status):
    assert status == arso.OK, lib.arso_last_error().decode()


def compiled(lib, circ, tile=0, flags=0):
    arr, keep = arso._gates_array(circ.gates)
    h = C.c_void_p()
    o = arso.CompileOpts(0, tile, 0, 0, 0, flags)
    ok(lib, lib.arso_compile_circuit(circ.n, arr, len(circ.gates), C.byref(o), C.byref(h)))
    return h


def sampled(lib, cc, stream, n=8):
    e = C.c_void_p()
    ok(lib, lib.arso_sample_errors(cc, 0.01, 0.01, 0.01, 1, 0, n, stream, C.byref(e)))
    return e


# resident, streaming on 13- and 12-qubit tiles, tensor phases
CIRCUITS = [(W.brickwork(11, 6, 1), 0, 0), (W.brickwork(14, 6, 1), 0, 0), (W.qaoa_maxcut(14, 1), 12, 0),
            (W.brickwork(14, 6, 1), 12, arso.OPT_TENSOR_PHASES)]


@pytest.mark.parametrize("k", range(len(CIRCUITS)))
@pytest.mark.parametrize("kind", ["fidelity", "outcome"])
def test_uploads_are_done_before_kernels_of_other_streams(lib, k, kind):
    # a copy from pageable memory returns before it has reached the device, and a stream that
    # does not wait for the legacy stream would read what was there
    st = lib.fake_stream(0)
    crit = arso.make_criterion(W.Criterion(kind, target=1, threshold=0.5))
    cc = compiled(lib, *CIRCUITS[k])
    e = sampled(lib, cc, st)
    score = (C.c_double * 8)()
    ok(lib, lib.arso_run_trajectories(cc, e, C.byref(crit), st, score, None))
    P = (C.c_double * 4)()
    ok(lib, lib.arso_exhaustive(cc, C.byref(crit), st, P, None))
    lib.arso_error_list_free(e)
    lib.arso_circuit_free(cc)
    assert lib.fake_launches(b"kernel") > 0
    assert lib.fake_violation(0) == 0


def test_autotune_leaves_no_handle_counted(lib):
    # with the last handle the pools' memory goes back, whether or not one was made by autotune
    arr, keep = arso._gates_array(CIRCUITS[1][0].gates)
    crit, best, ms, n = arso.make_criterion(W.Criterion("fidelity")), arso.CompileOpts(), (C.c_double * 16)(), C.c_uint32()
    ok(lib, lib.arso_autotune(14, arr, len(CIRCUITS[1][0].gates), C.byref(crit), C.c_double(1e-3), C.c_uint64(4),
                              C.c_uint64(0), None, lib.fake_stream(0), C.byref(best), ms, C.byref(n)))
    assert n.value > 1
    before = lib.fake_trims()
    lib.arso_circuit_free(compiled(lib, *CIRCUITS[0]))
    assert lib.fake_trims() == before + 2  # both pools


@pytest.mark.parametrize("kind", ["fidelity", "outcome"])
def test_exhaustive_scratch_is_bounded_on_one_deep_pass(lib, kind):
    # 20,000 one-qubit gates on the qubits of one tile: the sums of one pass would take a
    # gigabyte (twice that for two states), the state itself 8 MiB
    n = 20
    gates = [W.Gate("RY", (k % 12,), (0.1 + k,)) for k in range(20000)]
    cc = compiled(lib, W.Circuit(n, gates))
    crit = arso.make_criterion(W.Criterion(kind, target=1, threshold=0.5))
    P = (C.c_double * 4)()
    lib.fake_reset_counts()
    ok(lib, lib.arso_exhaustive(cc, C.byref(crit), lib.fake_stream(0), P, None))
    lib.arso_circuit_free(cc)
    assert lib.fake_launches(b"probe_kernel") >= 2
    assert lib.fake_largest() <= 256 << 20


def test_a_failed_call_does_not_fail_the_next(lib):
    stream = lib.fake_stream(0)
    cc = compiled(lib, *CIRCUITS[1])
    for k in range(4):
        lib.fake_fail_at(k)
        e = C.c_void_p()
        assert lib.arso_sample_errors(cc, 0.01, 0.01, 0.01, 1, 0, 8, stream, C.byref(e)) == arso.ENOMEM
        lib.fake_fail_at(-1)
        lib.arso_error_list_free(sampled(lib, cc, stream))
    lib.arso_circuit_free(cc)


def _calls(lib, stream):
    """The calls that hold an error list or a criterion's table, each as (name, call)."""
    circs = {k: compiled(lib, *CIRCUITS[k]) for k in (0, 1)}
    lists = {k: sampled(lib, cc, stream) for k, cc in circs.items()}
    crit = arso.make_criterion(W.Criterion("binning", basis_set=(0, 3), threshold=0.5))
    score, P, res = (C.c_double * 8)(), (C.c_double * 4)(), arso.Result()
    out = []
    for k, cc in circs.items():
        e = lists[k]
        ptr = lambda *v: C.cast((C.c_void_p * len(v))(*v), C.c_void_p)  # noqa: E731
        out += [("sample", lambda cc=cc: _sample(lib, cc, stream)),
                ("trajectories", lambda cc=cc, e=e: lib.arso_run_trajectories(cc, e, C.byref(crit), stream, score, None)),
                ("batch", lambda cc=cc, e=e: lib.arso_run_batch(C.c_size_t(1), ptr(cc), ptr(e), C.byref(crit),
                                                                C.c_void_p(stream), ptr(C.addressof(score)), None)),
                ("exhaustive", lambda cc=cc: lib.arso_exhaustive(cc, C.byref(crit), stream, P, None)),
                ("success", lambda cc=cc: lib.arso_success_prob(cc, C.byref(crit), 1e-3, 1, 8, 0, stream, C.byref(res)))]
    return out, circs, lists


def _sample(lib, cc, stream):
    e = C.c_void_p()
    st = lib.arso_sample_errors(cc, 0.01, 0.01, 0.01, 1, 0, 8, stream, C.byref(e))
    if st == arso.OK:
        lib.arso_error_list_free(e)
    return st


@pytest.mark.parametrize("what", ["allocation", "launch"])
def test_failing_calls_wait_before_lists_are_freed(lib, what):
    # every allocation, then every launch of every call fails once: memory that kernels in
    # flight may read is freed only after they have been waited for, by the call itself or,
    # its own list, by the caller
    stream = lib.fake_stream(0)
    fail, tried = (lib.fake_fail_at, lib.fake_allocs) if what == "allocation" else (lib.fake_fail_launch_at, lib.fake_tried)
    failed = 0
    for i in range(10):
        for k in range(60):
            calls, circs, lists = _calls(lib, stream)
            lib.fake_reset_counts()
            fail(k)
            status = calls[i][1]()
            done = tried() <= k
            fail(-1)
            for e in lists.values():
                lib.arso_error_list_free(e)
            for cc in circs.values():
                lib.arso_circuit_free(cc)
            assert lib.fake_violation(1) == 0, (calls[i][0], k)
            failed += status != arso.OK
            if done:
                assert status == arso.OK
                break
    assert failed > 40


def test_memory_is_freed_in_its_own_context(lib):
    # handles and lists of device 0 freed while device 1 is current, then of a context that a
    # reset of its device has ended; calls on the new context work
    for reset in (False, True):
        st = lib.fake_stream(0)
        cc = compiled(lib, *CIRCUITS[1])
        e = sampled(lib, cc, st)
        lib.fake_reset_counts()
        if reset:
            lib.fake_device_reset(0)
        else:
            lib.fake_device(1)
        live = lib.fake_live()
        lib.arso_error_list_free(e)
        lib.arso_circuit_free(cc)
        assert lib.fake_current() == (0 if reset else 1)
        assert (lib.fake_live() == live) == reset  # what a reset took is not freed again
        lib.fake_device(0)
        cc = compiled(lib, *CIRCUITS[1])
        e = sampled(lib, cc, lib.fake_stream(0))
        lib.arso_error_list_free(e)
        lib.arso_circuit_free(cc)
        assert [lib.fake_violation(k) for k in (1, 2, 3)] == [0, 0, 0]


def test_shared_memory_is_allowed_on_every_device(lib):
    crit = arso.make_criterion(W.Criterion("fidelity", threshold=0.5))
    score = (C.c_double * 8)()
    outs = (C.c_void_p * 1)(C.addressof(score))
    for dev in (0, 1, 0):
        lib.fake_device(dev)
        st = lib.fake_stream(dev)
        for k in range(len(CIRCUITS)):
            cc = compiled(lib, *CIRCUITS[k])
            e = sampled(lib, cc, st)
            ok(lib, lib.arso_run_trajectories(cc, e, C.byref(crit), st, score, None))
            ok(lib, lib.arso_run_batch(C.c_size_t(1), (C.c_void_p * 1)(cc.value), (C.c_void_p * 1)(e.value), C.byref(crit),
                                       C.c_void_p(st), outs, None))
            lib.arso_error_list_free(e)
            lib.arso_circuit_free(cc)
    assert [lib.fake_violation(k) for k in (2, 3, 4)] == [0, 0, 0]


def test_full_matrices_take_the_wide_pass_kernel(lib):
    # matrices that are unitary only up to their 32-bit rounding, entry by entry, have no frame
    # form; a long run of rotations holds one full matrix in 80 gates, to restore the scale
    rng = np.random.default_rng(1)
    full = [W.Gate("U", (k % 12,), matrix=(W.haar_su2(rng) * np.exp(1j * k)).astype(np.complex64).astype(complex))
            for k in range(200)]
    crit = arso.make_criterion(W.Criterion("fidelity", threshold=0.5))
    score = (C.c_double * 8)()
    for gates, wide in ((full, True), ([W.Gate("RX", (k % 12,), (1.0 + k,)) for k in range(200)], False)):
        cc = compiled(lib, W.Circuit(15, gates))
        st = lib.fake_stream(0)
        e = sampled(lib, cc, st)
        lib.fake_reset_counts()
        ok(lib, lib.arso_run_trajectories(cc, e, C.byref(crit), st, score, None))
        lib.arso_error_list_free(e)
        lib.arso_circuit_free(cc)
        assert (lib.fake_launches(b"pass_rb_kernelILi256ELi2E") > 0) == wide
        assert (lib.fake_launches(b"pass_rb_kernelILi256ELi3E") > 0) != wide
