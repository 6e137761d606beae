"""Uploads from pageable memory: the runtime may read the source at any time until
the stream is waited for, so the host tables of a call have to outlive its copies."""
import numpy as np
import pytest

import paper_2412_14973_gb300 as T

from _fakecuda import fake, handle


@pytest.mark.parametrize("precision", [T.TLR_PREC_FP32, T.TLR_PREC_BF16X3, T.TLR_PREC_TF32])
@pytest.mark.parametrize("alpha", [0.0, 2.0])
def test_sources_live_until_the_stream_is_waited_for(precision, alpha):
    with fake() as F:
        F.fake_fill_freed(1)
        try:
            n0, s0 = F.fake_uploads(), F.fake_stale_uploads()
            h, D = handle(precision, alpha=alpha)
            assert F.fake_stale_uploads() == s0, "creation"
            T.tlr_mdd_set_data(h, D, D)
            nr, ns = D.shape[1], D.shape[0]
            T.tlr_mdd_adjoint(h, np.zeros((nr, ns), np.complex64), np.zeros((nr, nr), np.complex64))
            X = np.zeros((nr, nr), np.complex64)
            T.tlr_mdd_benchmark_solve(h, 0.1, 2, 0.0, X)
            d = T.desc(nr, ns, 16, rank=3, diag_mode=T.TLR_DIAG_LOWRANK)
            th = np.zeros(T.tlr_mdd_theta_size(d), np.complex64)
            T.tlr_mdd_warm_start(h, X, th)
            T.tlr_mdd_unpermute_dense(h, th, X)
            T.tlr_mdd_destroy(h)
            assert F.fake_uploads() > n0
            assert F.fake_stale_uploads() == s0
        finally:
            F.fake_fill_freed(0)


def test_batch_tables_live_until_the_stream_is_waited_for():
    with fake() as F:
        F.fake_fill_freed(1)
        try:
            s0 = F.fake_stale_uploads()
            hs = [handle(T.TLR_PREC_BF16X3, nr=nr)[0] for nr in (64, 128)]
            b = T.tlr_mdd_batch_create(hs)
            assert F.fake_stale_uploads() == s0
            T.tlr_mdd_batch_destroy(b)
            for h in hs:
                T.tlr_mdd_destroy(h)
        finally:
            F.fake_fill_freed(0)
