"""The host side of the library (plans, copies, error reports) on a CUDA runtime
that runs on the host (fake_device.cpp): aaqaoa_host.cu compiled as C++ and
linked with it. The fake runs queued work only when the host synchronises, so
what a queued operation still needs then has to be there."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2410_22247_gb300 import _native as N
from paper_2410_22247_gb300 import build as B
from paper_2410_22247_gb300 import workloads as W

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I",
                           os.path.join(cuda, "include"), "-I", B.INCLUDE, "-I", B.CSRC, "-o", out,
                           os.path.join(HERE, "fake_device.cpp"), "-x", "c++",
                           os.path.join(B.CSRC, "aaqaoa_host.cu")])
    lib = ctypes.CDLL(out)
    for name, res, args in N._PROTOS:
        if hasattr(lib, name):
            getattr(lib, name).restype = res
            getattr(lib, name).argtypes = args
    return lib


def _p(a):
    return a.ctypes.data_as(ctypes.POINTER(ctypes.c_int32))


class FakePlan:
    """A plan of the fake library on a buffer of host memory (its own, or `buffer`)."""

    def __init__(self, lib, graph, p, batch=1, grad=True, buffer=None):
        n, e = graph
        self.lib, self.p, self.m = lib, p, len(e)
        e = np.ascontiguousarray(e, dtype=np.int32).reshape(-1)
        self.h = ctypes.c_void_p()
        assert lib.aaqaoa_prepare(n, self.m, _p(e), 0, None, None, None, p, 0, None, ctypes.byref(self.h)) == 0
        self.back(batch, grad, buffer)

    def back(self, batch, grad, buffer=None):
        size = ctypes.c_size_t()
        assert self.lib.aaqaoa_workspace_bytes(self.h, batch, int(grad), ctypes.byref(size)) == 0
        self.buffer = np.zeros(size.value + 256, dtype=np.uint8) if buffer is None else buffer
        at = (self.buffer.ctypes.data + 255) & ~255
        assert self.buffer.nbytes >= size.value + 256
        assert self.lib.aaqaoa_set_workspace(self.h, ctypes.c_void_p(at), size.value, batch, int(grad)) == 0

    @classmethod
    def unbacked(cls, lib, graph, p):
        """A plan without a workspace (schedules only)."""
        self = cls.__new__(cls)
        n, e = graph
        self.lib, self.p, self.m, self.h = lib, p, len(e), ctypes.c_void_p()
        e = np.ascontiguousarray(e, dtype=np.int32).reshape(-1)
        assert lib.aaqaoa_prepare(n, self.m, _p(e), 0, None, None, None, p, 0, None, ctypes.byref(self.h)) == 0
        return self

    def value(self, g, b):
        return 1000.0 * self.m + np.sum(g) + 2.0 * np.sum(b)

    def expect(self, g, b):
        out = np.zeros(1)
        rc = self.lib.aaqaoa_expect(self.h, g.ctypes.data, b.ctypes.data, 0, 0, out.ctypes.data)
        return rc, out[0]

    def expect_batch(self, g, b):
        out = np.zeros(len(g))
        rc = self.lib.aaqaoa_expect_batch(self.h, len(g), g.ctypes.data, b.ctypes.data, 0, out.ctypes.data)
        return rc, out

    def grad(self, g, b):
        out, dg, db = np.zeros(1), np.zeros(self.p), np.zeros(self.p)
        rc = self.lib.aaqaoa_grad(self.h, g.ctypes.data, b.ctypes.data, 0, out.ctypes.data, dg.ctypes.data,
                                  db.ctypes.data)
        return rc, out[0]

    def expect_device(self, g, b, out):
        return self.lib.aaqaoa_expect_device(self.h, 1, g.ctypes.data, b.ctypes.data, 0, out.ctypes.data)

    def close(self):
        self.lib.aaqaoa_destroy(self.h)


@pytest.mark.parametrize("n", [10, 14, 18])
def test_plans_may_take_turns_on_one_workspace(lib, n):
    """A MaxCut plan keeps nothing in its workspace from one call to the next:
    plans used one after the other may have the same one."""
    a = FakePlan(lib, W.complete_graph(n), 2)
    b = FakePlan(lib, W.cycle_graph(n), 2, buffer=a.buffer)
    x, y = np.array([0.3, 0.2]), np.array([0.1, 0.4])
    for pl in (a, b, a):
        rc, E = pl.expect(x, y)
        assert rc == 0 and abs(E - pl.value(x, y)) < 1e-9
    a.close()
    b.close()


@pytest.mark.parametrize("n,batch", [(10, 4), (14, 4), (18, 4), (22, 1), (22, 3), (22, 300)])
def test_copies_read_living_memory(lib, n, batch):
    """The angles of a call, and what a plan puts into its workspace, may be read
    by the device as late as the call's own synchronisation."""
    before = lib.fake_changed_sources()
    pl = FakePlan(lib, W.cycle_graph(n), 2, batch=min(batch, 4), grad=False)
    rng = np.random.default_rng(n)
    g, b = rng.uniform(0, 3, (batch, 2)), rng.uniform(0, 1, (batch, 2))
    rc, E = pl.expect_batch(g, b) if batch > 1 else pl.expect(g[0], b[0])
    assert rc == 0
    assert np.allclose(E, [pl.value(g[k], b[k]) for k in range(batch)], rtol=0, atol=1e-9)
    assert lib.fake_changed_sources() == before
    pl.close()


TIMEOUT = -5


def test_a_team_that_gives_up_is_reported(lib):
    """The expired wait of a team (n = 18): host calls return TIMEOUT and the plan
    recovers; device calls leave NaN until the error has been fetched."""
    pl = FakePlan(lib, W.cycle_graph(18), 2)
    x, y = np.array([0.3, 0.2]), np.array([0.1, 0.4])
    for call in (pl.expect, pl.grad):
        assert lib.aaqaoa_inject_fault(pl.h, N.AAQAOA_FAULT_DROP_ARRIVAL) == 0
        assert call(x, y)[0] == TIMEOUT
        rc, E = call(x, y)
        assert rc == 0 and abs(E - pl.value(x, y)) < 1e-9
    out = np.zeros(1)
    assert lib.aaqaoa_inject_fault(pl.h, N.AAQAOA_FAULT_DROP_ARRIVAL) == 0
    for _ in range(2):
        out[0] = 7.0
        assert pl.expect_device(x, y, out) == 0
        lib.cudaStreamSynchronize(None)
        assert np.isnan(out[0])
    assert lib.aaqaoa_sync(pl.h) == TIMEOUT
    assert pl.expect_device(x, y, out) == 0 and lib.aaqaoa_sync(pl.h) == 0
    assert abs(out[0] - pl.value(x, y)) < 1e-9
    pl.close()


def test_angles_that_are_no_numbers_give_no_number(lib):
    for n in (10, 18):
        pl = FakePlan(lib, W.cycle_graph(n), 1)
        rc, E = pl.expect(np.array([np.nan]), np.array([0.1]))
        assert rc == 0 and np.isnan(E)
        pl.close()


def test_drop_arrival_needs_a_team(lib):
    for n in (4, 10, 16, 22):
        pl = FakePlan(lib, W.cycle_graph(n), 1)
        assert lib.aaqaoa_inject_fault(pl.h, N.AAQAOA_FAULT_DROP_ARRIVAL) == -6
        pl.close()


@pytest.mark.parametrize("n", [4, 10, 14, 18, 22])
def test_an_unreported_timeout_reaches_the_next_host_call(lib, n):
    """A device call's expired wait is reported by whichever call waits next, a
    one-point energy or gradient among them; the one after that is right."""
    pl = FakePlan(lib, W.cycle_graph(n), 2)
    x, y = np.array([0.3, 0.2]), np.array([0.1, 0.4])
    for call in (pl.expect, pl.grad):
        assert lib.aaqaoa_inject_fault(pl.h, N.AAQAOA_FAULT_UNREPORTED) == 0
        assert call(x, y)[0] == TIMEOUT
        rc, E = call(x, y)
        assert rc == 0 and (n == 4 or abs(E - pl.value(x, y)) < 1e-9)
    pl.close()


def test_host_calls_without_a_pinned_row(lib):
    """Plans beyond the 64 that hold a pinned row copy their results back."""
    x, y = np.array([0.3]), np.array([0.1])
    plans = [FakePlan(lib, W.cycle_graph(6 + k % 4), 1, grad=False) for k in range(70)]
    for pl in plans:
        rc, E = pl.expect(x, y)
        assert rc == 0 and abs(E - pl.value(x, y)) < 1e-9
    for pl in plans[64:]:
        assert lib.aaqaoa_inject_fault(pl.h, N.AAQAOA_FAULT_UNREPORTED) == 0
        assert pl.expect(x, y)[0] == TIMEOUT
    for pl in plans:
        pl.close()


def test_the_pinned_rows_leave_captures_of_other_threads_alone(lib):
    """The block of pinned rows is made in the relaxed capture mode (any other
    would end a global-mode capture in another thread), which is then put back."""
    pl = FakePlan(lib, W.cycle_graph(10), 1)
    mode = lib.fake_capture_mode()
    rc, _ = pl.expect(np.array([0.3]), np.array([0.1]))
    assert rc == 0 and lib.fake_unsafe_allocations() == 0 and lib.fake_capture_mode() == mode == 0
    pl.close()


@pytest.mark.parametrize("n", [10, 14, 18])
def test_device_results_over_their_angles(lib, n):
    """A result row that overlaps the angles is written only when they have been read."""
    for at in range(0, 6):
        buf = np.zeros(12)
        buf[2:4], buf[4:6] = [0.3, 0.2], [0.1, 0.4]
        pl = FakePlan(lib, W.cycle_graph(n), 2)
        g, b = buf[2:4], buf[4:6]
        want = pl.value(g, b)
        out = buf[at:at + 5]
        assert lib.aaqaoa_grad_device(pl.h, g.ctypes.data, b.ctypes.data, 0, out.ctypes.data) == 0
        assert lib.aaqaoa_sync(pl.h) == 0
        assert abs(out[0] - want) < 1e-9 and np.allclose(out[1:], [0.3, 0.2, 0.1, 0.4])
        pl.close()


def _schedules(pl):
    out = []
    for mode in (0, 1, 2):
        rows, cnt = np.zeros((64, 5), dtype=np.int32), ctypes.c_int()
        assert pl.lib.aaqaoa_get_schedule(pl.h, mode, _p(rows), 64, ctypes.byref(cnt)) == 0
        out.append(rows[:cnt.value].tolist())
    return out


@pytest.mark.parametrize("n", [14, 18, 20, 22, 24, 27, 30])
def test_a_tuned_plan_set_again_changes_nothing(lib, n):
    """set_pass_plan(*autotune()) leaves the calls as they were: one launch up to 20
    qubits, the gradient's own forward passes above; so does the default written
    out above 20 qubits. Other plans run as written."""
    pl = FakePlan(lib, W.cycle_graph(n), 2) if n < 26 else FakePlan.unbacked(lib, W.cycle_graph(n), 2)
    x, y = np.array([0.3, 0.2]), np.array([0.1, 0.4])

    def launches():
        if n > 20:
            return 0
        before = lib.fake_circuit_launches()
        assert pl.expect(x, y)[0] == 0
        return lib.fake_circuit_launches() - before

    plan4 = np.zeros(4, dtype=np.int32)
    if n < 26:
        before = _schedules(pl)
        assert lib.aaqaoa_set_pass_plan(pl.h, 9, 0, 0, 0) in (0, -1)  # (what it was before does not matter)
        assert lib.aaqaoa_autotune(pl.h, _p(plan4)) == 0
        tuned = _schedules(pl)
        assert launches() == (1 if n <= 20 else 0)
        assert lib.aaqaoa_set_pass_plan(pl.h, *[int(v) for v in plan4]) == 0
        assert _schedules(pl) == tuned and launches() == (1 if n <= 20 else 0)
        assert lib.aaqaoa_set_pass_plan(pl.h, 0, 0, 0, 0) == 0
        assert _schedules(pl) == before
    else:
        before = _schedules(pl)
    other = FakePlan.unbacked(lib, W.cycle_graph(n), 2)
    assert lib.aaqaoa_get_pass_plan(other.h, _p(plan4)) == 0
    assert lib.aaqaoa_set_pass_plan(other.h, *[int(v) for v in plan4]) == 0
    if n > 20:
        assert _schedules(other) == before
    if n in (18, 20):
        assert lib.aaqaoa_set_pass_plan(pl.h, 9, 2, 8, 2) == 0 and launches() == 0
    other.close()
    pl.close()


@pytest.mark.parametrize("n,fields", [(22, None), (22, True), (18, None)])
def test_launch_records_tell_halves_from_whole_states(lib, n, fields):
    """Passes of a MaxCut plan move half of the bytes that their records count
    (bit 4 of the flags); those of an Ising plan, with the whole state, all."""
    x, y = np.array([0.3, 0.2]), np.array([0.1, 0.4])
    e = np.ascontiguousarray(W.cycle_graph(n)[1], dtype=np.int32).reshape(-1)
    if fields:
        pl = FakePlan.unbacked(lib, W.cycle_graph(n), 2)
        lib.aaqaoa_destroy(pl.h)
        F = lambda a: a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))
        w, h = np.ones(len(e) // 2), np.ones(n)
        pl.h = ctypes.c_void_p()
        assert lib.aaqaoa_prepare_ising(n, len(e) // 2, _p(e), F(w), F(h), 0, None, None, None, 0, None, None, None, 2,
                                        0, None, ctypes.byref(pl.h)) == 0
        pl.back(1, False)
    else:
        pl = FakePlan(lib, W.cycle_graph(n), 2, grad=False)
        assert lib.aaqaoa_set_pass_plan(pl.h, 9, 2 if n > 18 else 1, 0, 0) == 0
    assert lib.aaqaoa_profile_enable(pl.h, 1) == 0
    assert pl.expect(x, y)[0] == 0
    cnt, flags, by = ctypes.c_int(), np.zeros(32, dtype=np.int32), np.zeros(32)
    assert lib.aaqaoa_profile_launches(pl.h, 32, ctypes.byref(cnt), None, _p(flags), None,
                                       by.ctypes.data_as(ctypes.POINTER(ctypes.c_double))) == 0
    states = by[:cnt.value] > 0
    assert states.sum() >= 2
    assert ((flags[:cnt.value] & 16 != 0) == (states & (not fields))).all()
    pl.close()


@pytest.mark.parametrize("n,flags", [(13, 0), (12, 1), (5, 0)])
def test_a_batch_of_small_graphs_stores_no_states(lib, n, flags):
    """Graphs that run in one CTA or cluster need their functions, angles and results
    in a batch's workspace, and no statevector each."""
    G = 400
    e = np.ascontiguousarray(W.cycle_graph(n)[1], dtype=np.int32).reshape(-1)
    desc = (N.GraphDesc * G)(*[N.GraphDesc(n, len(e) // 2, _p(e), 0, None, None, None) for _ in range(G)])
    h, size = ctypes.c_void_p(), ctypes.c_size_t()
    assert lib.aaqaoa_prepare_multi(G, desc, 2, flags, None, ctypes.byref(h)) == 0
    assert lib.aaqaoa_multi_workspace_bytes(h, ctypes.byref(size)) == 0
    assert size.value < G * (12 << 10) + (1 << 20)
    lib.aaqaoa_destroy_multi(h)


@pytest.mark.parametrize("n", [10, 14, 18])
def test_a_launch_without_a_result_is_an_error(lib, n):
    """A one-point host call whose pinned row stays unwritten does not return the row
    of the call before."""
    pl = FakePlan(lib, W.cycle_graph(n), 1)
    x, y = np.array([0.3]), np.array([0.1])
    assert pl.expect(x, y)[0] == 0
    for call in (pl.expect, pl.grad):
        lib.fake_lose_next_launch()
        assert call(x, y)[0] == -4
        rc, E = call(x, y)
        assert rc == 0 and abs(E - pl.value(x, y)) < 1e-9
    pl.close()
