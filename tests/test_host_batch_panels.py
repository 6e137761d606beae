"""The adjoint of a batch's member keeps its tables, packed operands and partials out of
the work panels while the batched solve runs on them (it only read the data there
before they lay in the panels)."""
import numpy as np

import paper_2412_14973_gb300 as T

from _fakecuda import fake, handle


def test_adjoint_beside_a_batched_solve():
    with fake() as F:
        hs, D = [], None
        for _ in range(2):
            h, D = handle(T.TLR_PREC_BF16X3)
            hs.append(h)
        nr, ns = D.shape[1], D.shape[0]
        V, G = np.zeros((nr, ns), np.complex64), np.zeros((nr, nr), np.complex64)
        th = np.zeros(T.tlr_mdd_theta_size(T.desc(nr, ns, 16, rank=3, diag_mode=T.TLR_DIAG_LOWRANK)), np.complex64)

        def block(h):
            T.tlr_mdd_adjoint(h, V, G)
            return F.fake_last_upload_block()

        arenas = [block(h) for h in hs]          # the handles' own memory
        b = T.tlr_mdd_batch_create(hs)
        opts = T.solve_opts(stages=1, admm_iters=1, lbfgs_iters=1)
        T.tlr_mdd_batch_solve_async(b, [th.copy(), th.copy()], opts)
        assert not {block(h) for h in hs} & set(arenas)
        T.tlr_mdd_batch_wait(b)
        assert [block(h) for h in hs] == arenas
        # a batch that is destroyed without a wait
        T.tlr_mdd_batch_solve_async(b, [th.copy(), th.copy()], opts)
        T.tlr_mdd_batch_destroy(b)
        assert [block(h) for h in hs] == arenas
        for h in hs:
            T.tlr_mdd_destroy(h)
