"""What the workspace pool keeps of the calls' scratch: at most 256 MB above what the
handles have taken, after any number of calls (on the fake runtime and on a GPU)."""
import numpy as np
import pytest

import paper_2412_14973_gb300 as T

from _fakecuda import fake, handle

KEEP = 256 << 20
NR, NS = 4096, 16   # 5 nr^2 complex values of scratch in FP32: 671 MB


def _calls(h, X):
    reserved = lambda: T.tlr_mdd_trim_pool(1 << 62)   # noqa: E731
    before = reserved()
    for _ in range(4):
        T.tlr_mdd_benchmark_solve(h, 0.1, 1, 0.0, X)
        assert reserved() <= before + KEEP
    T.tlr_mdd_tile_ranks(X, NR, 256)
    assert reserved() <= before + KEEP
    return before, reserved


def test_repeated_calls_keep_a_bounded_reserve():
    with fake():
        h, _ = handle(T.TLR_PREC_FP32, nr=NR, ns=NS, b=256)
        X = np.zeros((NR, NR), np.complex64)
        before, reserved = _calls(h, X)
        h2, _ = handle(T.TLR_PREC_FP32, nr=NR, ns=NS, b=256)
        T.tlr_mdd_destroy(h2)
        for _ in range(3):
            T.tlr_mdd_benchmark_solve(h, 0.1, 1, 0.0, X)
            assert before < reserved() <= 2 * before + KEEP
        assert T.tlr_mdd_trim_pool(0) < before + KEEP
        T.tlr_mdd_benchmark_solve(h, 0.1, 1, 0.0, X)
        assert reserved() <= before + KEEP      # handing the reserve back resets the bound
        T.tlr_mdd_destroy(h)
        assert T.tlr_mdd_trim_pool(0) == 0


@pytest.mark.gpu
def test_repeated_calls_keep_a_bounded_reserve_on_the_gpu():
    import torch
    T.tlr_mdd_trim_pool(0)
    D = torch.randn(NS, NR, dtype=torch.complex64, device="cuda")
    d = T.desc(NR, NS, 256, rank=3, nx=64, ny=64, diag_mode=T.TLR_DIAG_LOWRANK)
    h = T.tlr_mdd_create(d, D, D)
    _calls(h, torch.empty(NR, NR, dtype=torch.complex64, device="cuda"))
    T.tlr_mdd_destroy(h)
    T.tlr_mdd_trim_pool(0)
