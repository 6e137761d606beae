"""The FP32 contractions on the tensor cores (exact three-way BF16 split): errors
against 64 bits over ragged shapes, against those of plain FP32 accumulation,
and Inf / NaN / near-overflow operands."""
import numpy as np
import pytest
import torch

import paper_2412_14973_gb300 as T
import tlr_synth as synth
from oracle import layout, operator

from _gpu import Gpu, dev, host, rel

pytestmark = pytest.mark.gpu


def _fma_adjoint(V, Dt):
    """V Dt^H with one FP32 multiply-add after the other along the sources."""
    G = np.zeros((V.shape[0], Dt.shape[0]), np.complex64)
    for s in range(V.shape[1]):
        a, b = V[:, s:s + 1], np.conj(Dt[:, s])[None]
        G.real += a.real * b.real
        G.real -= a.imag * b.imag
        G.imag += a.real * b.imag
        G.imag += a.imag * b.real
    return G


@pytest.mark.parametrize("nr,ns", [(16, 16), (16, 1), (112, 129), (128, 512), (144, 1031), (256, 2048)])
def test_adjoint_error_is_that_of_fp32_or_less(nr, ns):
    # tile edges (128 rows, 16-deep chunks), odd source counts (rows not 16-byte
    # aligned), one to 32 splits of the contraction
    g = synth.rng(nr + ns)
    D = synth.cn(g, (ns, nr)).astype(np.complex64)
    V = synth.cn(g, (nr, ns)).astype(np.complex64)
    lay = layout.make_layout(nr, 16, 2, "lowrank")
    gp = Gpu(D, D, lay, nx=nr // 4, ny=4, alpha=1.0)
    Dt = gp.data()[2]
    want = V.astype(np.complex128) @ Dt.astype(np.complex128).conj().T
    got = gp.adjoint(V)
    e, ef = rel(got, want), rel(_fma_adjoint(V, Dt).astype(np.complex128), want)
    print(f"nr {nr} ns {ns}: tensor cores {e:.2e}, plain FP32 {ef:.2e}")
    # FP32 rounds each of 2 ns terms; a one-term sum has only its products' rounding (2^-24 each, two per part)
    assert e <= max(1.25 * ef, 2.0 ** -23)


@pytest.mark.parametrize("ns", [96, 131])
def test_apply_and_gradient_shapes(ns):
    # panels of 5 .. 150 columns (one ragged and two N tiles), a dense tile, a rank-0 pair
    nr, b = 160, 40
    ks = [3, 0, 7, 20] + [1, 0, 38, 5, 16, 40]
    lay = layout.make_layout(nr, b, ks, [False, False, True, False])
    g = synth.rng(ns)
    D, U = synth.cn(g, (ns, nr)).astype(np.complex64), synth.cn(g, (ns, nr)).astype(np.complex64)
    th = synth.cn(g, lay.size).astype(np.complex64)
    gp = Gpu(D, U, lay, nx=16, ny=10)
    perm = np.asarray(gp.data()[0])
    Dh, Uh, _ = operator.normalise(D, U, perm)
    f, gr = gp.grad(th)
    th64 = th.astype(np.complex128)
    assert rel(gp.apply(th), (Dh @ operator.assemble_xh(th64, lay)).T) <= 1e-6
    assert abs(f - operator.misfit(th64, lay, Dh, Uh)) <= 1e-6 * f
    assert rel(gr, operator.gradient(th64, lay, Dh, Uh)) <= 1.5e-6


def test_inf_nan_and_near_overflow_as_fp32():
    # an element of each kind in V; column s of Dt has zeros, a one and a negative
    # value, so a product is Inf, -Inf, NaN (Inf times zero) or finite by FP32 rules
    nr, ns = 48, 40
    D = np.zeros((ns, nr), np.complex64)
    g = synth.rng(3)
    D[:, 1:] = synth.cn(g, (ns, nr - 1)).astype(np.complex64)
    D[0, :3] = [1.0, 0.0, -1.0]
    V = synth.cn(g, (nr, ns)).astype(np.complex64)
    V[3, 0], V[5, 7], V[9, 0], V[11, 2] = np.inf, np.nan, 3.4e38, -np.inf
    V.imag[3, 0] = V.imag[9, 0] = V.imag[11, 2] = 0.0
    lay = layout.make_layout(nr, 16, 2, "lowrank")
    gp = Gpu(D, D, lay, perm=list(range(nr)), alpha=1.0)
    Dt = gp.data()[2]
    got = gp.adjoint(V).astype(np.complex64)
    with np.errstate(all="ignore"):
        want = _fma_adjoint(V, Dt)
    for part in ("real", "imag"):
        x, y = getattr(got, part), getattr(want, part)
        assert np.array_equal(np.isnan(x), np.isnan(y))
        assert np.array_equal(x[np.isinf(y)], y[np.isinf(y)])
        fin = np.isfinite(y)
        assert np.array_equal(fin, np.isfinite(x))
        # row 9: one product of the order of 3.4e38 (the finite rest is the other tests' matter)
        big = fin[9] & (np.abs(y[9]) > 1e30)
        assert np.all(np.abs(x[9][big] - y[9][big]) <= 1e-5 * np.abs(y[9][big]))
