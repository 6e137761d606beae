"""The L-BFGS direction's inner products, memories of several groups of pairs, and the
line search's scalar arithmetic, each against 64 bits, through a small library that
compiles the solver's kernels beside the test."""
import ctypes as C
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

import paper_2412_14973_gb300 as T
from paper_2412_14973_gb300 import build as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    T.lib()
    here = os.path.dirname(os.path.abspath(__file__))
    out = str(tmp_path_factory.mktemp("probe") / "libprobe_vec.so")
    libdir = os.path.dirname(T.tlr_mdd.lib_path()) if hasattr(T, "tlr_mdd") else os.path.join(B.PKG, "lib")
    r = subprocess.run([B._nvcc(), *B.ARCH, *B.FLAGS, "-shared", "-cudart", "static", os.path.join(here, "_probe_vec.cu"),
                        "-o", out, "-L" + libdir, "-ltlr_mdd", "-Xlinker", "-rpath", "-Xlinker", libdir, "-Xlinker",
                        "-Bsymbolic"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = C.CDLL(out)
    vp = C.c_void_p
    L.probe_scalar.argtypes = [vp, vp, vp, C.c_int]
    L.probe_argmin.argtypes = [vp, vp, vp, C.c_int]
    L.probe_direction.argtypes = [C.c_longlong, C.c_int, C.c_int, C.c_int] + [vp] * 9
    return L


def _pairs(n2, k, rng):
    """k pairs with <s, y> > 0 and a gradient."""
    s = rng.standard_normal((k, n2)).astype(np.float32)
    y = (s * (0.5 + rng.random((1, n2))) + 0.1 * rng.standard_normal((k, n2))).astype(np.float32)
    return s, y, rng.standard_normal(n2).astype(np.float32)


def _two_loop(s, y, g):
    s, y, q = s.astype(float), y.astype(float), g.astype(float).copy()
    a = []
    for i in range(len(s) - 1, -1, -1):
        a.append(s[i] @ q / (s[i] @ y[i]))
        q -= a[-1] * y[i]
    q *= (s[-1] @ y[-1]) / (y[-1] @ y[-1])
    for i, ai in zip(range(len(s)), reversed(a)):
        q += (ai - y[i] @ q / (s[i] @ y[i])) * s[i]
    return -q


@pytest.mark.parametrize("n2,m,k", [(2, 3, 1), (1030, 10, 10), (45056, 10, 10), (77824, 3, 3), (77826, 11, 11),
                                    (5000, 20, 20), (40002, 32, 32), (300000, 25, 25)])
def test_direction_and_its_products(probe, n2, m, k):
    import torch
    rng = np.random.default_rng(n2 + k)
    s, y, g = _pairs(n2, k, rng)
    ring = m + 1
    dv = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
    S, Y = torch.zeros(ring, n2, device="cuda"), torch.zeros(ring, n2, device="cuda")
    SY = torch.zeros(ring * ring, dtype=torch.float64, device="cuda")
    YY = torch.zeros_like(SY)
    x, v, gd, d = dv(g), dv(0 * g), dv(g), torch.zeros(n2, device="cuda")
    sums = np.zeros(5 * k + 1)
    slot0 = m - 1                        # the ring wraps
    for i in range(k):
        slot = (slot0 + i) % ring
        S[slot], Y[slot] = dv(s[i]), dv(y[i])
        rc = probe.probe_direction(n2, m, i + 1, slot, *[t.data_ptr() for t in (x, v, gd, d, S, Y, SY, YY)],
                                   sums.ctypes.data)
        assert rc == 0
    got = d.cpu().numpy().astype(float)
    want = _two_loop(s, y, g)
    assert np.linalg.norm(got - want) <= 2e-5 * np.linalg.norm(want)
    if n2 <= 77824:
        # every product rounded to FP32, their sum in 64 bits
        for j in range(k):
            sj, yj, sn, yn = s[k - 1 - j], y[k - 1 - j], s[-1], y[-1]
            for t, (a, b) in enumerate([(sj, g), (yj, g), (sj, yn), (sn, yj), (yj, yn)]):
                p = (a * b).astype(float)
                assert abs(sums[5 * j + t] - p.sum()) <= 1e-13 * np.abs(p).sum(), (j, t)
        p = (g * g).astype(float)
        assert abs(sums[5 * k] - p.sum()) <= 1e-13 * p.sum()


def test_reciprocals_and_cube_roots(probe):
    import torch
    rng = np.random.default_rng(5)
    x = np.concatenate([rng.standard_normal(3000) * 10.0 ** rng.uniform(-29, 29, 3000),
                        rng.standard_normal(500) * 10.0 ** rng.uniform(-200, 200, 500), [1.0, -8.0, 27.0, 1e30, 1e-30]])
    xd = torch.from_numpy(x).cuda()
    r, c = torch.empty_like(xd), torch.empty_like(xd)
    assert probe.probe_scalar(xd.data_ptr(), r.data_ptr(), c.data_ptr(), len(x)) == 0
    r, c = r.cpu().numpy(), c.cpu().numpy()
    # within an ulp: |x r - 1| <= 2^-52, and the root's cube on either side of x an ulp off
    assert all(abs(Fraction(float(a)) * Fraction(float(b)) - 1) <= Fraction(1, 2 ** 52) for a, b in zip(x, r))
    for a, b in zip(x, c):
        lo, hi = sorted(Fraction(float(np.nextafter(b, t))) ** 3 for t in (-np.inf, np.inf))
        assert lo <= Fraction(float(a)) <= hi


def test_the_quartics_minimiser(probe):
    import torch
    rng = np.random.default_rng(6)
    n = 2000
    c = rng.standard_normal((n, 5))
    c[:, 4] = np.abs(c[:, 4]) * 10.0 ** rng.uniform(-6, 3, n)
    c[:, 1] = -np.abs(c[:, 1])
    c[::10, 3] = 0.0
    c[1::50, 4] = 0.0
    c[1::50, 3] = np.abs(c[1::50, 3])
    c[2::50, 3:] = 0.0                   # a parabola
    c[2::50, 2] = np.abs(c[2::50, 2])
    cd = torch.from_numpy(c).cuda()
    a, ok = torch.zeros(n, dtype=torch.float64, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda")
    assert probe.probe_argmin(cd.data_ptr(), a.data_ptr(), ok.data_ptr(), n) == 0
    a, ok = a.cpu().numpy(), ok.cpu().numpy()
    val = lambda k, t: np.polyval(k[::-1], t)   # noqa: E731
    for k, t, f in zip(c, a, ok):
        d = np.trim_zeros(np.array([4 * k[4], 3 * k[3], 2 * k[2], k[1]]), "f")
        roots = np.roots(d)
        real = [z.real for z in roots if abs(z.imag) <= 1e-7 * max(1.0, abs(z)) and z.real > 0]
        assert bool(f) == bool(real)
        if real:
            best = min(val(k, z) for z in real)
            scale = sum(abs(k[i]) * t ** i for i in range(5))
            assert val(k, t) <= best + 1e-12 * scale
            assert abs(np.polyval(d, t)) <= 1e-9 * sum(abs(q) * t ** i for i, q in enumerate(d[::-1]))
