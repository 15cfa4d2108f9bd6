"""The calls whose time is measured: listed and drawn cases of the framework's work.

Each case is one call that a user's program makes through the public Python
entry points (``Plan``, ``MultiPlan``, ``energy``): energies, adjoint
gradients, batches of angles, uneven batches of graphs, per-edge correlations
and samples, for MaxCut and Ising objectives in complex64 and complex128.
``prepare`` builds what such a program holds before the call (graph, edge
orbits, plan with its workspace, angles), ``run`` is the call, ``exact`` gives
the same values from a plain 64-bit statevector simulation in torch.

Amplitudes are complex64 or complex128; the values a call returns carry the
precision of its amplitudes and are handed on in it (float32 or float64). A
gradient call's results are one row, (E, dE/dgamma, dE/dbeta), as an optimiser
takes them.
"""
import math

import numpy as np
import torch

from paper_2410_22247_gb300 import orbits as ORB
from paper_2410_22247_gb300 import workloads as W
from paper_2410_22247_gb300.api import MultiPlan, Plan, energy


def listed():
    return [
        # one step of an optimiser loop on a small graph: the smallest call, latency counts
        {"name": "grad_petersen10_p2_c64", "call": "grad", "graph": "petersen", "n": 10, "p": 2, "precision": "c64"},
        # the 16 x 16 angle grid of a small dense graph, FP64 throughout
        {"name": "grid_complete12_p1_c128", "call": "grid", "graph": "complete", "n": 12, "p": 1,
         "precision": "c128", "side": 16},
        # a training step through torch.autograd on a mid-size graph: several short launches
        {"name": "autograd_regular16_p3_c64", "call": "autograd", "graph": "regular3", "n": 16, "p": 3,
         "precision": "c64"},
        # multi-start optimisation: the gradients of 16 points in one call
        {"name": "gradbatch_prufer22_p2_c64", "call": "grad_batch", "graph": "prufer", "n": 22, "p": 2,
         "precision": "c64", "points": 16},
        # a random tree's gradient in complex128 (the FP64 form of the same path)
        {"name": "grad_prufer24_p3_c128", "call": "grad", "graph": "prufer", "n": 24, "p": 3, "precision": "c128"},
        # an Ising objective with real couplings and fields
        {"name": "ising_grad_regular26_p2_c64", "call": "ising_grad", "graph": "regular3", "n": 26, "p": 2,
         "precision": "c64"},
        # <ZZ> of every edge: the check of the orbits behind H_red, per-edge analysis
        {"name": "edgezz_regular28_p2_c64", "call": "edge_zz", "graph": "regular3", "n": 28, "p": 2,
         "precision": "c64"},
        # the headline evaluation: energy and gradient at n = 30 from angles on the device
        {"name": "grad_star30_p2_c64", "call": "grad_device", "graph": "star", "n": 30, "p": 2, "precision": "c64"},
        # the energy of a large tree with H_red (an odd number of qubits)
        {"name": "energy_heap31_p1_c64", "call": "energy", "graph": "heap", "n": 31, "p": 1, "precision": "c64"},
        # a 64 x 64 energy landscape of one graph in one call
        {"name": "landscape_star20_p1_c64", "call": "grid", "graph": "star", "n": 20, "p": 1, "precision": "c64",
         "side": 64},
        # many small instances of different size in one call
        {"name": "uneven256_n12to22_p2_c64", "call": "uneven", "count": 256, "lo": 12, "hi": 22, "p": 2,
         "precision": "c64"},
        # the pipeline's end: bitstrings drawn from the final state
        {"name": "sample_prufer20_p2_c128", "call": "sample", "graph": "prufer", "n": 20, "p": 2,
         "precision": "c128", "shots": 4096},
    ]


def draw(rng):
    call = rng.choice(["grad", "grad", "grad_device", "energy", "energy", "autograd", "grid", "grad_batch",
                       "ising_grad", "edge_zz", "uneven", "sample"])
    precision = rng.choice(["c64", "c64", "c128"])
    big = precision == "c128"  # FP64 arithmetic costs more: smaller states for the same time
    p = rng.choice([1, 1, 2, 2, 3, 4])
    if call == "uneven":
        lo = rng.randint(6, 14)
        return {"call": call, "count": int(round(math.exp(rng.uniform(math.log(8), math.log(320))))), "lo": lo,
                "hi": lo + rng.randint(4, 8 if not big else 5), "p": min(p, 2), "precision": precision}
    if call == "grid":
        n = rng.randint(8, 20 if not big else 16)
        return {"call": call, "graph": rng.choice(["star", "prufer", "cycle", "heap"]), "n": n, "p": 1,
                "precision": precision, "side": rng.randint(5, 64 if n < 20 else 48)}
    if call == "sample":
        return {"call": call, "graph": rng.choice(["prufer", "cycle", "star"]), "n": rng.randint(9, 22), "p": min(p, 2),
                "precision": "c128", "shots": int(round(math.exp(rng.uniform(math.log(64), math.log(16384)))))}
    if call == "ising_grad":
        return {"call": call, "graph": rng.choice(["prufer", "cycle", "star"]), "n": rng.randint(8, 27 if not big else 22),
                "p": min(p, 2), "precision": precision}
    if call == "grad_batch":
        n = rng.randint(8, 22 if not big else 19)
        return {"call": call, "graph": rng.choice(["prufer", "heap", "cycle"]), "n": n, "p": min(p, 3),
                "precision": precision, "points": rng.randint(2, 24)}
    top = {"grad": 28, "grad_device": 28, "energy": 30, "autograd": 24, "edge_zz": 28}[call] - (5 if big else 0)
    n = rng.randint(6, top)
    graph = rng.choice(["prufer", "star", "cycle", "heap", "complete"] if n <= 16 else ["prufer", "star", "cycle", "heap"])
    return {"call": call, "graph": graph, "n": n, "p": p, "precision": precision}


# ---------------------------------------------------------------- inputs
def graph_of(case, seed):
    n = case["n"]
    name = case["graph"]
    if name == "petersen":
        return W.generalized_petersen(5, 2)
    if name == "complete":
        return W.complete_graph(n)
    if name == "star":
        return W.star_graph(n)
    if name == "cycle":
        return W.cycle_graph(n)
    if name == "heap":
        return W.heap_binary_tree(n)
    if name == "prufer":
        return W.prufer_tree(n, 17 + seed)
    if name == "regular3":
        return W.random_regular(n, 3, 23 + seed)
    raise ValueError(name)


def angles_of(case, seed):
    """Rows of (gamma, beta) of the case's points: random, or a grid whose
    offset inside a cell is random."""
    p = case["p"]
    if case["call"] == "grid":
        k = case["side"]
        og, ob = np.random.Generator(np.random.PCG64(1000 + seed)).uniform(0.0, 1.0, 2)
        g = (np.arange(k) + og) * (math.pi / k)
        b = (np.arange(k) + ob) * (math.pi / 2 / k)
        G, B = np.meshgrid(g, b, indexing="ij")
        return G.reshape(-1, 1).copy(), B.reshape(-1, 1).copy()
    points = case.get("points", case.get("count", 1))
    rows = [W.random_angles(p, 1000 * (seed + 1) + k) for k in range(points)]
    return np.array([r[0] for r in rows]), np.array([r[1] for r in rows])


def prepare(case, seed):
    call, p, precision = case["call"], case["p"], case["precision"]
    g, b = angles_of(case, seed)
    s = {"call": call, "real": np.float64 if precision == "c128" else np.float32, "g": g, "b": b}
    if call == "uneven":
        graphs = [(n, e, ORB.edge_orbits_native(n, e))
                  for _, n, e in W.mixed_graph_batch(case["count"], case["lo"], case["hi"], 7 + seed)]
        s["plan"] = MultiPlan(graphs, p, precision=precision)
        return s
    n, e = graph_of(case, seed)
    if call == "ising_grad":
        w, h = W.ising_couplings(n, e, 31 + seed)
        s["plan"] = Plan(n, e, p, precision=precision, with_grad=True, couplings=w, fields=h)
        s["g"], s["b"] = g[0], b[0]
        return s
    grads = call in ("grad", "grad_device", "autograd", "grad_batch")
    batch = len(g) if call in ("grid", "grad_batch") else 1
    s["plan"] = Plan(n, e, p, orbits=ORB.edge_orbits_native(n, e), precision=precision, batch=batch, with_grad=grads)
    if batch == 1 and call not in ("grid", "grad_batch"):
        s["g"], s["b"] = g[0], b[0]
    if call == "grad_device":
        s["dg"] = torch.tensor(s["g"], dtype=torch.float64, device="cuda")
        s["db"] = torch.tensor(s["b"], dtype=torch.float64, device="cuda")
        s["out"] = torch.empty(1 + 2 * p, dtype=torch.float64, device="cuda")
    elif call == "autograd":
        s["dg"] = torch.tensor(s["g"], dtype=torch.float64, device="cuda", requires_grad=True)
        s["db"] = torch.tensor(s["b"], dtype=torch.float64, device="cuda", requires_grad=True)
    elif call == "sample":
        s["u"] = np.random.Generator(np.random.PCG64(77 + seed)).uniform(0.0, 1.0, case["shots"])
    return s


# ---------------------------------------------------------------- the call
def run(s):
    plan, real, call = s["plan"], s["real"], s["call"]
    if call in ("grad", "ising_grad"):
        E, dg, db = plan.grad(s["g"], s["b"], "red" if call == "grad" else "full")
        return np.concatenate([[E], dg, db]).astype(real)
    if call == "grad_device":
        plan.grad_device(s["dg"], s["db"], s["out"], "red")
        return s["out"].to(torch.float64 if real is np.float64 else torch.float32)
    if call == "autograd":
        g, b = s["dg"], s["db"]
        g.grad = b.grad = None
        E = energy(g, b, plan, "red")
        E.backward()
        row = torch.cat([E.detach().reshape(1), g.grad, b.grad])
        return row if real is np.float64 else row.float()
    if call == "energy":
        return real(plan.expect(s["g"], s["b"], "red"))
    if call == "grid":
        return plan.expect_batch(s["g"], s["b"], "red").astype(real)
    if call == "grad_batch":
        E, dg, db = plan.grad_batch(s["g"], s["b"], "red")
        return np.concatenate([E[:, None], dg, db], axis=1).astype(real)
    if call == "uneven":
        return plan.expect(s["g"], s["b"], "red").astype(real)
    if call == "edge_zz":
        return plan.edge_zz(s["g"], s["b"]).astype(real)
    if call == "sample":
        x, cut = plan.sample(s["g"], s["b"], s["u"])
        return x.astype(np.int64), cut
    raise ValueError(call)


# ---------------------------------------------------------------- its work
def work(case):
    """Bytes: the angles and results, and for states beyond the on-chip memory
    (64 MB) one write of the state and one read and write of every vector a
    layer transforms: (2p + 1) S for an energy, (6p + 1) S for a gradient. S is
    the part of the state that is independent: half of it for MaxCut
    objectives, whose states do not change when all bits flip. Operations: per
    amplitude and layer two multiply-adds per qubit and a complex factor."""
    p, amp = case["p"], 16 if case["precision"] == "c128" else 8
    call = case["call"]
    if call == "uneven":
        sizes = [n for _, n, _ in W.mixed_graph_batch(case["count"], case["lo"], case["hi"], 7)]
        rows, points = len(sizes), 1
    else:
        sizes = [case["n"]]
        points = rows = case["side"] ** 2 if call == "grid" else case.get("points", 1)
    grad = call in ("grad", "grad_device", "autograd", "grad_batch", "ising_grad")
    bytes_, flops = 8.0 * rows * (2 * p + (1 + 2 * p if grad else 1)), 0.0
    for n in sizes:
        amps = float(2 ** n if call == "ising_grad" else 2 ** (n - 1)) * points
        if amps * amp > 64e6:
            bytes_ += (6 * p + 1 if grad else 2 * p + 1) * amps * amp
        flops += amps * p * (4 * n + 6) * (1 if not grad else 4)
    if call == "sample":
        bytes_ += 8.0 * case["shots"] + 12.0 * case["shots"]
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------- 64 bits
def _diagonal(n, edges, w, h, dev):
    """C(x) = sum_e w_e [x_u != x_v] + sum_i h_i x_i for all x."""
    x = torch.arange(2 ** n, device=dev)
    c = torch.zeros(2 ** n, dtype=torch.float64, device=dev)
    for (u, v), we in zip(edges.tolist(), w):
        c += float(we) * (((x >> u) ^ (x >> v)) & 1)
    if h is not None:
        for i in range(n):
            c += float(h[i]) * ((x >> i) & 1)
    return c


def _mix(psi, n, betas, sign=1.0):
    """exp(-i sign beta X) on every qubit of each row of psi [rows, 2^n], in place."""
    rows = psi.shape[0]
    c = torch.tensor(np.cos(betas), dtype=torch.float64, device=psi.device).view(rows, 1, 1)
    s = torch.tensor(np.sin(betas) * sign, dtype=torch.float64, device=psi.device).view(rows, 1, 1) * -1j
    for q in range(n):
        v = psi.view(rows, 2 ** (n - q - 1), 2, 2 ** q)
        a, b = v[:, :, 0], v[:, :, 1]
        t = a.clone()
        a.mul_(c).addcmul_(b, s)
        b.mul_(c).addcmul_(t, s)
        del t


def _phase(psi, C, gammas, sign=1.0):
    for r, g in enumerate(gammas):
        step = 1 << 26
        for k in range(0, psi.shape[1], step):
            a = C[k:k + step] * (-sign * float(g))
            psi[r, k:k + step] *= torch.polar(torch.ones_like(a), a)


def _state(n, C, g, b):
    psi = torch.full((len(g), 2 ** n), 2.0 ** (-n / 2), dtype=torch.complex128, device=C.device)
    for l in range(g.shape[1]):
        _phase(psi, C, g[:, l])
        _mix(psi, n, b[:, l])
    return psi


def _density(psi, r):
    return psi[r].real ** 2 + psi[r].imag ** 2


def _grad_row(n, C, g, b):
    """E, dE/dgamma, dE/dbeta of one point by the adjoint recursion."""
    p = len(g)
    phi = _state(n, C, g[None], b[None])
    E = float((_density(phi, 0) * C).sum())
    lam = phi * C
    dg, db = np.zeros(p), np.zeros(p)
    for l in range(p - 1, -1, -1):
        acc = 0.0
        for q in range(n):
            f = phi.view(2 ** (n - q - 1), 2, 2 ** q)
            m = lam.view(2 ** (n - q - 1), 2, 2 ** q)
            for a in (0, 1):
                u, v = m[:, a], f[:, 1 - a]
                acc += float((u.real * v.imag).sum() - (u.imag * v.real).sum())
        db[l] = 2.0 * acc
        _mix(phi, n, b[None, l], -1.0)
        _mix(lam, n, b[None, l], -1.0)
        dg[l] = 2.0 * float(((lam.real * phi.imag - lam.imag * phi.real) * C).sum())
        _phase(phi, C, g[None, l], -1.0)
        _phase(lam, C, g[None, l], -1.0)
    return np.concatenate([[E], dg, db])


def _energies(n, C, g, b):
    """Energies of the rows of (g, b), a few rows at a time."""
    rows = max(1, min(len(g), (1 << 27) >> n))
    out = np.zeros(len(g))
    for k in range(0, len(g), rows):
        psi = _state(n, C, g[k:k + rows], b[k:k + rows])
        for r in range(psi.shape[0]):
            out[k + r] = float((_density(psi, r) * C).sum())
    return out


def exact(case, seed):
    call = case["call"]
    if call == "sample":
        return None  # whole numbers
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    g, b = angles_of(case, seed)
    if call == "uneven":
        out = []
        for i, (_, n, e) in enumerate(W.mixed_graph_batch(case["count"], case["lo"], case["hi"], 7 + seed)):
            out.append(_energies(n, _diagonal(n, e, np.ones(len(e)), None, dev), g[i:i + 1], b[i:i + 1])[0])
        return np.array(out)
    n, e = graph_of(case, seed)
    w, h = W.ising_couplings(n, e, 31 + seed) if call == "ising_grad" else (np.ones(len(e)), None)
    C = _diagonal(n, e, w, h, dev)
    if call in ("grad", "ising_grad", "grad_device", "autograd"):
        return _grad_row(n, C, g[0], b[0])
    if call == "energy":
        return np.float64(_energies(n, C, g, b)[0])
    if call == "grid":
        return _energies(n, C, g, b)
    if call == "grad_batch":
        return np.stack([_grad_row(n, C, g[k], b[k]) for k in range(len(g))])
    d = _density(_state(n, C, g, b), 0)  # edge_zz
    x = torch.arange(2 ** n, device=dev)
    return np.array([float((d * (1 - 2 * (((x >> u) ^ (x >> v)) & 1))).sum()) for u, v in e.tolist()])
