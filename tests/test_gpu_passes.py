"""The tiled passes at 14 to 20 qubits, where MaxCut energies and gradients take the
whole-circuit launch by default: the default pass plan, written out, makes them
run the passes. Single points and batches, many layers, isolated vertices and
the phase's edge angles against the oracle; tolerances as in test_gpu_parity.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2410_22247_gb300 import orbits as ORB
from paper_2410_22247_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"c64": 1e-5, "c128": 1e-10}

GRAPHS = {
    "reg14": lambda: W.random_regular(14, 3, 3),
    "prufer15": lambda: W.prufer_tree(15, 5),
    "reg16": lambda: W.random_regular(16, 3, 1),
    "isolated18": lambda: (18, W.prufer_tree(12, 8)[1]),
    "prufer18": lambda: W.prufer_tree(18, 6),
    "cycle20": lambda: W.cycle_graph(20),
}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _check(got, ref, prec):
    E, dg, db = got
    Er, dgr, dbr = ref
    floor = (1.0 if prec == "c64" else 1e-3) * max(abs(Er), 1.0)
    g, r = np.concatenate([dg, db]), np.concatenate([dgr, dbr])
    assert abs(E - Er) <= TOL[prec] * max(abs(Er), 1.0)
    assert np.all(np.abs(g - r) <= TOL[prec] * np.maximum(np.abs(r), floor))


def _passes(graph, p, prec, batch=1):
    from paper_2410_22247_gb300.api import Plan
    n, e = graph
    pl = Plan(n, e, p, orbits=ORB.edge_orbits(n, e), precision=prec, batch=batch, with_grad=True)
    pl.set_pass_plan(*pl.pass_plan())
    return pl


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_points_and_batches(name, prec):
    n, e = GRAPHS[name]()
    p, B = 3, 5
    rng = W.rng(40 + n)
    gs, bs = rng.uniform(0, np.pi, (B, p)), rng.uniform(-np.pi / 2, np.pi / 2, (B, p))
    pl = _passes((n, e), p, prec, batch=3)
    E, dg, db = pl.grad_batch(gs, bs, "red")
    assert pl.launch_count() > 1
    Eb = pl.expect_batch(gs, bs, "full")
    for k in range(B):
        ref = O.energy_grad(n, e, gs[k], bs[k])
        _check((E[k], dg[k], db[k]), ref, prec)
        assert abs(Eb[k] - ref[0]) <= TOL[prec] * max(abs(ref[0]), 1.0)
    _check(pl.grad(gs[0], bs[0], "red"), O.energy_grad(n, e, gs[0], bs[0]), prec)
    assert pl.launch_count() > 1


@pytest.mark.parametrize("prec", ["c64", "c128"])
def test_many_layers(prec):
    n, e = W.prufer_tree(16, 4)
    g, b = W.random_angles(12, 41)
    pl = _passes((n, e), 12, prec)
    _check(pl.grad(g, b, "red"), O.energy_grad(n, e, g, b), prec)
    assert pl.launch_count() > 1


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("g,b", [([0.0, 0.7], [0.3, 0.0]), ([0.9, 1.3], [np.pi / 4, -np.pi / 4]),
                                 ([2 * np.pi, -0.4], [np.pi / 2, 1e-9]), ([40.0, -17.3], [2.3, -1.9])])
def test_edge_angles(g, b, prec):
    n, e = W.random_regular(16, 3, 1)
    pl = _passes((n, e), 2, prec)
    _check(pl.grad(g, b, "red"), O.energy_grad(n, e, g, b), prec)
    psi, ref = pl.statevector(g, b), O.qaoa_state(n, e, g, b)
    assert np.max(np.abs(psi - ref)) <= TOL[prec] * np.max(np.abs(ref))
