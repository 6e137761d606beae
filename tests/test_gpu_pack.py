"""Packing of operands for the tensor cores where its rows and chunks run out: odd
leading dimensions (no 16-byte loads), odd and short K, rows on either side of a
128-row tile, for the operator, its adjoint and the gradient.

Tolerances: BF16x3 keeps 16 significant bits of each operand, so a term of a
contraction is off by at most 2^-15 of its size; 1e-3 of the result's norm, and of
its rms per element, is 32 of these.  TF32 keeps 11 bits: 2^-10 a term, 32 of these."""
import numpy as np
import pytest

import tlr_synth as synth
from oracle import operator
from tests._cases import problem

pytestmark = pytest.mark.gpu
T = pytest.importorskip("paper_2412_14973_gb300")
from tests._gpu import Gpu, elem, rel  # noqa: E402

TOL = {"bf16x3": 32 * 2.0**-15, "tf32": 32 * 2.0**-10}


# nx, ny, b, rank, ns
@pytest.mark.parametrize("nx,ny,b,k,ns", [(2, 2, 2, 1, 1), (8, 8, 16, 3, 33), (13, 10, 65, 5, 127), (16, 16, 32, 4, 129),
                                          (15, 17, 51, 7, 95), (9, 57, 171, 17, 257)])
@pytest.mark.parametrize("prec", ["bf16x3", "tf32"])
def test_packed_operands_at_the_ends_of_tiles(nx, ny, b, k, ns, prec):
    nt = nx * ny // b
    D, U, perm, lay, _ = problem(nx, ny, b, k, "lowrank", ns=ns, snr_db=10, planted=False)
    th = (synth.cn(synth.rng(nx * ny + ns), lay.size) * 0.2).astype(np.complex64).astype(np.complex128)
    Dh, Uh, alpha = operator.normalise(D, U, perm)
    g = Gpu(D, U, lay, nx=nx, ny=ny, alpha=alpha,
            precision=T.TLR_PREC_BF16X3 if prec == "bf16x3" else T.TLR_PREC_TF32)
    V = synth.cn(synth.rng(17), (lay.nr, Dh.shape[0])).astype(np.complex64).astype(np.complex128)
    pairs = [(g.apply(th), operator.apply_y(th, lay, Dh)), (g.grad(th)[1], operator.gradient(th, lay, Dh, Uh)),
             (g.adjoint(V), operator.adjoint_g(V, Dh))]
    g.close()
    assert nt * b == nx * ny
    for got, want in pairs:
        assert rel(got, want) <= TOL[prec]
        assert elem(got, want) <= TOL[prec]
