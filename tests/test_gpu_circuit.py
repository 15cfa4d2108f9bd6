"""Whole circuits in one launch, and the flip-symmetric half of the passes, at
the sizes where their shapes change: one CTA up to a team of 128, odd and even
numbers of stored index bits, the first and last sizes of a register stage,
more points than CTAs at once, phase tables that do not fit, pair passes over
one qubit and over the most. Oracle: the plain FP64 statevector code;
tolerances as in test_gpu_parity (complex128 1e-10, complex64 1e-5, gradients
on the energy's scale).
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2410_22247_gb300 import workloads as W
from paper_2410_22247_gb300 import orbits as ORB

pytestmark = pytest.mark.gpu

TOL = {"c64": 1e-5, "c128": 1e-10}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _plan(n, e, p, prec, **kw):
    from paper_2410_22247_gb300.api import Plan
    return Plan(n, e, p, orbits=ORB.edge_orbits(n, e, weights=kw.get("weights")), precision=prec, **kw)


def _check(got, ref, prec):
    E, dg, db = got
    Er, dgr, dbr = ref
    scale = max(abs(Er), 1.0)
    assert abs(E - Er) <= TOL[prec] * scale
    assert np.max(np.abs(np.concatenate([dg - dgr, db - dbr]))) <= TOL[prec] * scale


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("n", [4, 5, 6, 8, 9, 11, 12, 13, 14, 15, 16, 17, 18, 19, 20])
def test_one_launch_matches_oracle(n, prec):
    n, e = W.prufer_tree(n, 300 + n)
    g, b = W.random_angles(2, 40 + n)  # both rotation forms occur over the sizes
    pl = _plan(n, e, 2, prec)
    _check(pl.grad(g, b, "red"), O.energy_grad(n, e, g, b), prec)
    if n >= 5:
        assert pl.launch_count() == 1
    if n <= 13:
        assert np.max(np.abs(pl.statevector(g, b) - O.qaoa_state(n, e, g, b))) <= TOL[prec]
    assert abs(pl.expect(g, b, "red") - O.energy(n, e, g, b)) <= TOL[prec] * max(n / 2, 1)


@pytest.mark.parametrize("n,B,prec", [(9, 700, "c64"), (13, 3, "c64"), (13, 320, "c128"), (14, 40, "c64"),
                                      (15, 5, "c128"), (16, 20, "c64"), (18, 3, "c64")])
def test_points_share_a_launch(n, B, prec):
    n, e = W.circulant_graph(n, (1, 3))
    a = [W.random_angles(2, 900 + k) for k in range(B)]
    gs, bs = np.array([x[0] for x in a]), np.array([x[1] for x in a])
    pl = _plan(n, e, 2, prec, batch=B)
    E, dg, db = pl.grad_batch(gs, bs, "red")
    assert pl.launch_count() == 1
    assert np.array_equal(pl.grad_batch(gs, bs, "red")[0], E)
    for k in {0, 1, B // 2, B - 1}:
        _check((E[k], dg[k], db[k]), O.energy_grad(n, e, gs[k], bs[k]), prec)


@pytest.mark.parametrize("prec", ["c64", "c128"])
def test_tables_larger_than_shared_memory(prec):
    n, e = W.star_graph(12)
    w = [51] * 11  # 562 table entries per layer, two tables, 24 layers
    g, b = W.random_angles(24, 5)
    pl = _plan(n, e, 24, prec, weights=w)
    got = pl.grad(g, b, "red")
    assert pl.launch_count() == 1
    # 24 layers with cut values up to 561: errors on the scale of the norm
    # bounds, max O for the energy and 2 max O max C for a gradient component
    ref = O.energy_grad_w(n, e, w, g, b)
    assert abs(got[0] - ref[0]) <= TOL[prec] * 561
    assert np.max(np.abs(np.concatenate([got[1] - ref[1], got[2] - ref[2]]))) <= TOL[prec] * 2 * 561 ** 2


@pytest.mark.parametrize("n,plan,prec", [(14, (13, 1, 12, 1), "c64"), (14, (9, 1, 8, 1), "c64"),
                                         (15, (13, 2, 12, 2), "c64"), (18, (9, 1, 12, 1), "c64"),
                                         (13, (12, 1, 11, 1), "c128"), (14, (8, 1, 7, 1), "c128"),
                                         (17, (8, 1, 11, 1), "c128")])
def test_pair_passes_match_oracle(n, plan, prec):
    n, e = W.prufer_tree(n, 70 + n)
    pl = _plan(n, e, 2, prec)
    pl.set_pass_plan(*plan)
    for seed in (3, 4):
        g, b = W.random_angles(2, seed)
        _check(pl.grad(g, b, "red"), O.energy_grad(n, e, g, b), prec)
        assert pl.launch_count() > 1
        psi = O.qaoa_state(n, e, g, b)
        assert np.max(np.abs(pl.statevector(g, b) - psi)) <= TOL[prec]
    pl.set_pass_plan()
    _check(pl.grad(g, b, "red"), O.energy_grad(n, e, g, b), prec)


@pytest.mark.parametrize("plan", [(9, 2, 10, 2), (12, 2, 12, 2), (8, 2, 8, 2)])
def test_ising_turnaround_over_odd_and_even_groups(plan):
    """The turnaround's group has 5, 4 and 6 qubits; in the last layer of the
    second angles |sin beta| > |cos beta| (the cot form, whose butterfly and
    inverse change the sign once per qubit)."""
    n, e = W.prufer_tree(20, 8)
    w, h = W.ising_couplings(n, e, 9)
    from paper_2410_22247_gb300.api import Plan
    pl = Plan(n, e, 2, precision="c64", with_grad=True, couplings=w, fields=h)
    pl.set_pass_plan(*plan)
    adj = pl.schedule(True)
    assert adj[0][2] == adj[0][3], "no turnaround"
    scale = float(np.sum(np.abs(w)) + np.sum(np.abs(h)))
    for beta in ([0.4, 0.3], [0.4, 1.2]):
        E, dg, db = pl.grad([0.5, 0.8], beta, "full")
        Er, dgr, dbr = O.ising_energy_grad(n, O.ising(e, w, h), np.array([0.5, 0.8]), np.array(beta))
        assert abs(E - Er) <= 1e-5 * scale
        assert np.max(np.abs(np.concatenate([dg - dgr, db - dbr]))) <= 1e-5 * scale


@pytest.mark.parametrize("n,prec", [(5, "c64"), (10, "c128"), (13, "c64"), (16, "c64"), (20, "c64"), (20, "c128")])
def test_plans_take_turns_on_one_workspace(n, prec):
    """Two plans used one after the other on one buffer: a call depends on nothing
    that another plan's set-up or call left there, to the last bit."""
    import ctypes

    from paper_2410_22247_gb300 import _native as N
    a = [W.random_angles(2, 60 + k) for k in range(3)]
    gs, bs = np.array([x[0] for x in a]), np.array([x[1] for x in a])

    def results(pl):
        one, many = pl.grad(gs[0], bs[0], "red"), pl.grad_batch(gs, bs, "red")
        return np.concatenate([np.ravel(x) for x in one + many])

    plans = [_plan(*graph, 2, prec, batch=3) for graph in (W.cycle_graph(n), W.star_graph(n))]
    alone = [results(pl) for pl in plans]
    assert not np.array_equal(alone[0], alone[1])
    buf = plans[0].workspace
    N.check(N.aaqaoa_set_workspace(plans[1].handle, ctypes.c_void_p(buf.data_ptr()), buf.numel(), 3, 1),
            "set_workspace")
    for k in (0, 1, 0, 1):
        assert np.array_equal(results(plans[k]), alone[k])


@pytest.mark.parametrize("n,prec", [(18, "c64"), (20, "c64"), (19, "c128")])
def test_expired_wait_of_a_team_is_reported_and_the_plan_recovers(n, prec):
    """One CTA of a team never arrives (a bounded wait of about a second): host calls
    raise, device calls leave NaN instead of the previous results until the error
    has been fetched, and the next call is right again."""
    import torch

    from paper_2410_22247_gb300 import _native as N
    n, e = W.prufer_tree(n, 7)
    g, b = W.random_angles(2, 9)
    pl = _plan(n, e, 2, prec)
    ref = O.energy_grad(n, e, g, b)
    _check(pl.grad(g, b, "red"), ref, prec)
    assert pl.launch_count() == 1
    N.check(N.aaqaoa_inject_fault(pl.handle, N.AAQAOA_FAULT_DROP_ARRIVAL), "inject")
    with pytest.raises(N.AAQAOAError, match="TIMEOUT"):
        pl.grad(g, b, "red")
    _check(pl.grad(g, b, "red"), ref, prec)
    dg = torch.tensor(g, dtype=torch.float64, device="cuda")
    db = torch.tensor(b, dtype=torch.float64, device="cuda")
    out = torch.empty(5, dtype=torch.float64, device="cuda")
    pl.grad_device(dg, db, out, "red")
    N.check(N.aaqaoa_inject_fault(pl.handle, N.AAQAOA_FAULT_DROP_ARRIVAL), "inject")
    for _ in range(2):
        pl.grad_device(dg, db, out, "red")
        assert torch.isnan(out).all()
    with pytest.raises(N.AAQAOAError, match="TIMEOUT"):
        pl.sync()
    pl.grad_device(dg, db, out, "red")
    pl.sync()
    row = out.cpu().numpy()
    _check((row[0], row[1:3], row[3:]), ref, prec)


@pytest.mark.parametrize("n", [5, 10, 16])
def test_no_team_to_drop_an_arrival_from(n):
    from paper_2410_22247_gb300 import _native as N
    pl = _plan(*W.cycle_graph(n), 1, "c64")
    assert N.aaqaoa_inject_fault(pl.handle, N.AAQAOA_FAULT_DROP_ARRIVAL) == -6


@pytest.mark.parametrize("n,prec", [(4, "c64"), (8, "c64"), (10, "c128"), (16, "c64"), (20, "c64"), (22, "c64")])
def test_unreported_timeout_reaches_the_next_host_call(n, prec):
    """The error flag of an earlier device call, through every form of a one-point
    host call: one CTA, a cluster, a team, the passes."""
    from paper_2410_22247_gb300 import _native as N
    n, e = W.cycle_graph(n)
    g, b = W.random_angles(1, 3)
    pl = _plan(n, e, 1, prec)
    for call in (lambda: pl.expect(g, b, "red"), lambda: pl.grad(g, b, "red")[0]):
        want = call()
        N.check(N.aaqaoa_inject_fault(pl.handle, N.AAQAOA_FAULT_UNREPORTED), "inject")
        with pytest.raises(N.AAQAOAError, match="TIMEOUT"):
            call()
        assert call() == want


@pytest.mark.parametrize("n,prec", [(4, "c64"), (10, "c64"), (12, "c128"), (16, "c64"), (18, "c64"), (20, "c128"),
                                    (22, "c64")])
def test_device_calls_replay_from_a_captured_graph(n, prec):
    """A gradient call captured into the caller's CUDA graph reads the angles of the
    replay: one CTA, a cluster, a team (a cooperative launch), the passes."""
    import torch
    from paper_2410_22247_gb300.api import Plan
    n, e = W.cycle_graph(n)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        pl = Plan(n, e, 2, orbits=ORB.edge_orbits(n, e), precision=prec, stream=st)
        dg = torch.zeros(2, dtype=torch.float64, device="cuda")
        db = torch.zeros(2, dtype=torch.float64, device="cuda")
        out = torch.zeros(5, dtype=torch.float64, device="cuda")
        pl.grad_device(dg, db, out, "red")
        pl.sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        pl.grad_device(dg, db, out, "red")
    for seed in (2, 3):
        g, b = W.random_angles(2, seed)
        dg.copy_(torch.tensor(g))
        db.copy_(torch.tensor(b))
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        pl.sync()
        row = out.cpu().numpy()
        _check((row[0], row[1:3], row[3:]), O.energy_grad(n, e, g, b), prec)
