"""Packing at the ends of rows and chunks, at tolerances that see a plane: BF16x3 keeps
16 bits of each operand (a term is off by about 2^-16, rms over many terms less: 5e-5
of the norm, 2e-4 of the rms per element), TF32 11 bits (1e-3 and 5e-3); the dense
adjoint runs in BF16x3 on either kind of handle.  A missing low plane costs 2.4e-3
in norm, operands of 6 bits 4.7e-3."""
import numpy as np
import pytest

import tlr_synth as synth
from oracle import operator
from tests._cases import problem

pytestmark = pytest.mark.gpu
T = pytest.importorskip("paper_2412_14973_gb300")
from tests._gpu import Gpu, elem, rel  # noqa: E402

TOL = {"bf16x3": (5e-5, 2e-4), "tf32": (1e-3, 5e-3)}


@pytest.mark.parametrize("nx,ny,b,k,ns", [(8, 8, 16, 3, 33), (13, 10, 65, 5, 127), (16, 16, 32, 4, 129),
                                          (15, 17, 51, 7, 95), (9, 57, 171, 17, 257)])
@pytest.mark.parametrize("prec", ["bf16x3", "tf32"])
def test_every_plane_of_packed_operands(nx, ny, b, k, ns, prec):
    D, U, perm, lay, _ = problem(nx, ny, b, k, "lowrank", ns=ns, snr_db=10, planted=False)
    th = (synth.cn(synth.rng(nx * ny + ns), lay.size) * 0.2).astype(np.complex64).astype(np.complex128)
    Dh, Uh, alpha = operator.normalise(D, U, perm)
    g = Gpu(D, U, lay, nx=nx, ny=ny, alpha=alpha,
            precision=T.TLR_PREC_BF16X3 if prec == "bf16x3" else T.TLR_PREC_TF32)
    V = synth.cn(synth.rng(17), (lay.nr, Dh.shape[0])).astype(np.complex64).astype(np.complex128)
    for what, got, want, tol in [("apply", g.apply(th), operator.apply_y(th, lay, Dh), TOL[prec]),
                                 ("gradient", g.grad(th)[1], operator.gradient(th, lay, Dh, Uh), TOL[prec]),
                                 ("adjoint", g.adjoint(V), operator.adjoint_g(V, Dh), TOL["bf16x3"])]:
        print(f"{what}: norm {rel(got, want):.2e}, element {elem(got, want):.2e}")
        assert rel(got, want) <= tol[0], what
        assert elem(got, want) <= tol[1], what
    g.close()
