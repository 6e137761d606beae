"""The FP32 contractions against FP32 fused multiply-adds where a sum of truncations
or the three-way split could be worse: same-signed terms, sums of few products,
values near FP32's smallest, and non-finite values over long sums."""
import numpy as np
import pytest

import paper_2412_14973_gb300 as T
import tlr_synth as synth
from oracle import layout, operator

from _gpu import Gpu, rel

pytestmark = pytest.mark.gpu


def _fma(V, Dt):
    """V Dt^H by FP32 fused multiply-adds along the sources (products exact in 64 bits)."""
    re = np.zeros((V.shape[0], Dt.shape[0]), np.float32)
    im = re.copy()
    for s in range(V.shape[1]):
        a, b = V[:, s:s + 1].astype(np.complex128), np.conj(Dt[:, s].astype(np.complex128))[None]
        re = (re + a.real * b.real).astype(np.float32)
        re = (re - a.imag * b.imag).astype(np.float32)
        im = (im + a.real * b.imag).astype(np.float32)
        im = (im + a.imag * b.real).astype(np.float32)
    return re + 1j * im.astype(np.complex64)


def _adjoint(V, D):
    nr = V.shape[0]
    gp = Gpu(D, D, layout.make_layout(nr, 16, 2, "lowrank"), perm=list(range(nr)), alpha=1.0)
    Dt = gp.data()[2]
    got = gp.adjoint(V)
    want = V.astype(np.complex128) @ Dt.astype(np.complex128).conj().T
    gp.close()
    return got, _fma(V, Dt).astype(np.complex128), want


@pytest.mark.parametrize("ns", [1, 2, 7, 12, 13, 16, 33, 96, 512])
@pytest.mark.parametrize("kind", ["gram", "positive"])
def test_same_signed_sums(kind, ns):
    nr = 144
    g = synth.rng(ns)
    if kind == "gram":
        D = synth.cn(g, (ns, nr)).astype(np.complex64)
        V = np.ascontiguousarray(D.T)
    else:
        D = (0.1 + g.random((ns, nr))).astype(np.complex64)
        V = (0.1 + g.random((nr, ns))).astype(np.complex64)
    got, fma, want = _adjoint(V, D)
    e, ef = rel(got, want), rel(fma, want)
    bias = float(np.mean(((got - want) / np.abs(want)).real[np.eye(nr, dtype=bool)]))
    print(f"{kind} ns {ns}: {e:.2e}, FMA {ef:.2e}; signed mean on the diagonal {bias:+.2e}")
    # no larger than that of fused multiply-adds (5 %: two samples of rounding errors)
    assert e <= 1.05 * ef
    # a drained chunk's last two products are cut toward zero, each by less than an ulp
    assert abs(bias) <= 2.0 ** -23


@pytest.mark.parametrize("scale", [-100, -109, -112, -118, -124, -140])
@pytest.mark.parametrize("ns", [48, 131])
def test_small_values_keep_their_bits(scale, ns):
    nr = 144
    g = synth.rng(7)
    V = (synth.cn(g, (nr, ns)) * 2.0 ** scale).astype(np.complex64)
    D = (synth.cn(g, (ns, nr)) * 2.0 ** 60).astype(np.complex64)
    got, fma, want = _adjoint(V, D)
    e, ef = rel(got, want), rel(fma, want)
    print(f"2^{scale}, ns {ns}: {e:.2e}, FMA {ef:.2e}")
    assert e <= 1.05 * ef


def test_small_results_and_small_values_among_others():
    nr, ns = 144, 64
    g = synth.rng(8)
    V = synth.cn(g, (nr, ns)).astype(np.complex64)
    D = synth.cn(g, (ns, nr)).astype(np.complex64)
    V[5] *= np.float32(2.0 ** -70)       # results of 2^-140
    D[:, 9] *= np.float32(2.0 ** -70)
    V[100, :] = 0
    V[100, 3] = 1.2345678e-36            # one value, one product each
    got, fma, want = _adjoint(V, D)
    assert abs(got[5, 9] - fma[5, 9]) <= 64 * 2.0 ** -149
    for rows in ([100], [5], list(range(6, 100))):
        assert rel(got[rows], want[rows]) <= 1.05 * rel(fma[rows], want[rows])


def test_unbalanced_factors():
    # X = L R^T with L at 2^-115 and R at 2^105: the products keep their 24 bits
    nr, ns, b, k = 96, 70, 24, 5
    lay = layout.make_layout(nr, b, k, "lowrank")
    g = synth.rng(9)
    D, U = synth.cn(g, (ns, nr)).astype(np.complex64), synth.cn(g, (ns, nr)).astype(np.complex64)
    th = synth.cn(g, lay.size).astype(np.complex64)
    N = nr // b
    q = N * b * k                        # the diagonal's factors: zero here
    p = (lay.size - q) // 2
    th[:q] = 0
    un = th.copy()
    un[q:q + p] *= np.float32(2.0 ** -115)
    un[q + p:] *= np.float32(2.0 ** 105)
    gp = Gpu(D, U, lay, nx=12, ny=8)
    Dh, _, _ = operator.normalise(D, U, np.asarray(gp.data()[0]))
    want = operator.apply_y(un.astype(np.complex128), lay, Dh)
    assert rel(gp.apply(un), want) <= 1e-6


def test_nan_over_a_long_sum():
    nr, ns = 256, 20000
    g = synth.rng(10)
    V = synth.cn(g, (nr, ns)).astype(np.complex64)
    D = synth.cn(g, (ns, nr)).astype(np.complex64)
    D[17, 40] = np.nan
    D[18, 41] = np.inf
    gp = Gpu(D, D, layout.make_layout(nr, 16, 2, "lowrank"), perm=list(range(nr)), alpha=1.0)
    got = gp.adjoint(V)
    bad = np.zeros(nr, bool)
    bad[40:42] = True
    assert not np.isfinite(got[:, bad]).any()
    Dt = gp.data()[2][~bad].astype(np.complex128)
    assert rel(got[:, ~bad], V.astype(np.complex128) @ Dt.conj().T) <= 2e-7
