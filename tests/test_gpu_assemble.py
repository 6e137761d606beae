"""X from its factors at the edges of the assembly's 64 x 64 blocks and 32-deep
stages, and alpha over values at the edges of its FP32 filter."""
import numpy as np
import pytest
import torch

import paper_2412_14973_gb300 as T
import tlr_synth as synth
from oracle import layout, operator

from _gpu import Gpu, dev, host, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tiles,k", [([1, 63, 64], 1), ([65, 128, 7], 5), ([130, 33], 33), ([64, 64], 64), ([16] * 9, 0)])
def test_blocks_and_depths(tiles, k):
    # a sum of at most 64 products of unit values in FP32: 64 2^-24 of their size at worst, 1e-5 of the norm
    nr, n = sum(tiles), len(tiles)
    kd = [min(k, t) for t in tiles]
    kp = [min(k, tiles[i], tiles[j]) for j in range(n) for i in range(j + 1, n)]
    lay = layout.make_layout(nr, None, kd + kp, [i == 1 for i in range(n)], tiles=tiles)
    th = synth.cn(synth.rng(nr + k), lay.size).astype(np.complex64)
    D = synth.cn(synth.rng(1), (16, nr)).astype(np.complex64)
    perm = list(synth.rng(2).permutation(nr))
    gp = Gpu(D, D, lay, perm=perm)
    X = gp.unpermute(th)
    Xo = operator.unpermute(operator.assemble_xh(th.astype(np.complex128), lay), np.asarray(perm))
    assert np.array_equal(X, X.T)
    assert np.linalg.norm(X - Xo) <= 1e-5 * max(np.linalg.norm(Xo), 1e-30)


@pytest.mark.parametrize("n", [1, 2, 4097, 700001])
def test_alpha_is_the_fp64_maximum(n):
    # many entries within a few ulp of the maximum, tiny, huge and zero entries
    for scale in (1.0, 1e-22, 3e18, 1e25):
        g = synth.rng(n)
        z = np.exp(2j * np.pi * g.random(n)) * (1 + 1e-7 * g.standard_normal(n)) * scale
        z[g.random(n) < 0.2] = 0
        z[n // 2] = 0.99 * scale
        z = z.astype(np.complex64)
        want = np.sqrt(np.max(z.real.astype(np.float64) ** 2 + z.imag.astype(np.float64) ** 2))
        buf = torch.from_numpy(np.concatenate([[0], z]).astype(np.complex64)).cuda()
        assert T.tlr_mdd_stack_alpha(torch.from_numpy(z).cuda(), n) == pytest.approx(want, rel=1e-15)
        assert T.tlr_mdd_stack_alpha(buf[1:], n) == pytest.approx(want, rel=1e-15)   # 8-byte aligned
