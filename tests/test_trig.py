"""The sine and cosine behind every phase table and mixer angle (aaqaoa_trig.h),
on the host against mpmath and on the device against the host, over quadrant
edges, negative and large angles and the switch to the library's function.

Tolerance, from the rounding steps: the reduced argument is off by half an ulp
(2^-54), the polynomial part of either value (at most 0.31) by two relative
roundings, the result by half an ulp (2^-54): below 2^-52 in all."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2410_22247_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
SWITCH = 1e9 * np.pi / 2  # |x| from which the library's function is called


def _angles():
    rng = np.random.default_rng(5)
    k = np.concatenate([np.arange(-40, 41), rng.integers(-10 ** 9, 10 ** 9, 200)]).astype(np.float64)
    edges = np.concatenate([k * (np.pi / 4), k * (np.pi / 2)])
    near = [edges, np.nextafter(edges, np.inf), np.nextafter(edges, -np.inf), edges + 1e-9, edges - 1e-5]
    spread = [rng.uniform(-s, s, 400) for s in (1e-8, 1.0, 4.0, 120.0, 1e4, 1e6, 1e9, SWITCH)]
    switch = SWITCH * (1 + np.array([-1e-9, -1e-12, -2e-16, 0, 2e-16, 1e-12, 1e-9, 1e-3]))
    x = np.concatenate(near + spread + [switch, -switch, [0.0, -0.0, 5e-324, 1e300]])
    return np.ascontiguousarray(x)


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("trig") / "libtrig.so")
    subprocess.check_call([B.nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-shared", "-o", out, os.path.join(HERE, "trig_probe.cu")])
    return ctypes.CDLL(out)


def _host(probe, x):
    z = np.zeros((len(x), 2))
    probe.probe_host(ctypes.c_void_p(x.ctypes.data), ctypes.c_void_p(z.ctypes.data), len(x))
    return z


def test_host_form_matches_mpmath(probe):
    mp = pytest.importorskip("mpmath")
    x = _angles()
    with mp.workprec(200):
        err = [max(abs(mp.mpf(float(c)) - mp.cos(mp.mpf(float(a)))), abs(mp.mpf(float(s)) - mp.sin(mp.mpf(float(a)))))
               for a, (c, s) in zip(x, _host(probe, x))]
    assert max(err) <= 2.0 ** -52, (float(max(err)), x[int(np.argmax([float(e) for e in err]))])


def test_host_form_of_no_number(probe):
    assert np.isnan(_host(probe, np.array([np.nan, np.inf, -np.inf]))).all()


@pytest.mark.parametrize("real", ["float", "double"])
def test_dropped_factor_and_its_powers(probe, real):
    """f = 1 / sqrt(1 + t^2) for the rounded t, and f^k, k <= 34. Double: f^k right to
    one rounding (2^-53 relative; f in two parts, products with their errors: the
    rest is below 2^-90). Float: t is off by three roundings to float, 3 2^-24,
    and f to second order in that, below 2^-45."""
    mp = pytest.importorskip("mpmath")
    n = 34
    rng = np.random.default_rng(11)
    angles = np.concatenate([rng.uniform(-np.pi, np.pi, 300), [0.0, np.pi / 4, -np.pi / 4, 1e-9, np.pi / 2, 3.0]])
    worst = 0.0
    with mp.workprec(250):
        for a in angles:
            u, v = float(np.sin(a)), float(np.cos(a))
            if abs(u) > abs(v):
                u, v = -v, u
            t, f = ctypes.c_double(), np.zeros(2)
            sq, ch = np.zeros(n + 1), np.zeros(n + 1)
            P = lambda x: ctypes.c_void_p(x.ctypes.data)
            probe.probe_mix(ctypes.c_double(u), ctypes.c_double(v), int(real == "float"), n, ctypes.byref(t), P(f),
                            P(sq), P(ch))
            exact = (1 if v > 0 else -1) / mp.sqrt(1 + mp.mpf(t.value) ** 2)
            for k in range(n + 1):
                for x in (sq[k], ch[k]):
                    err = float(abs(mp.mpf(float(x)) / exact ** k - 1))
                    worst = max(worst, err / (2.0 ** -53 * (1 + 1e-6) if real == "double"
                                              else k * 2.0 ** -45 + 2.0 ** -53))
    assert worst <= 1.0


@pytest.mark.gpu
def test_device_form_is_the_host_form(probe):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    x = _angles()
    dx = torch.tensor(x, device="cuda")
    dz = torch.empty(len(x), 2, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert probe.probe_device(ctypes.c_void_p(dx.data_ptr()), ctypes.c_void_p(dz.data_ptr()), len(x)) == 0
    z, h = dz.cpu().numpy(), _host(probe, x)
    own = np.abs(x) < SWITCH * (1 - 1e-8)
    assert np.array_equal(z[own], h[own])  # the same operations
    assert np.max(np.abs(z - h)) <= 2.0 ** -52 + 2.0 ** -52  # the library's functions: two ulp each at most
