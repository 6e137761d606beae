"""A contraction that gives up on a bounded wait records it in an error word on the
device: the next synchronising call reports TLR_ERR_TIMEOUT, and the handle works
again.  On the fake runtime, whose contractions write the word when told to."""
import numpy as np
import pytest

import paper_2412_14973_gb300 as T

from _fakecuda import fake, handle

# the kernel's name and its argument that points to the word
WORD = {T.TLR_PREC_FP32: (b"k_cgemm_f32", 1), T.TLR_PREC_BF16X3: (b"k_cgemm_tcp", 6), T.TLR_PREC_TF32: (b"k_cgemm_tcp", 6)}


def _buffers(D):
    nr, ns = D.shape[1], D.shape[0]
    th = np.zeros(T.tlr_mdd_theta_size(T.desc(nr, ns, 16, rank=3, diag_mode=T.TLR_DIAG_LOWRANK)), np.complex64)
    return th, np.zeros((nr, ns), np.complex64), np.zeros((nr, nr), np.complex64)


def _times_out(f):
    with pytest.raises(T.TLRError) as e:
        f()
    return e.value.code == T.TLR_ERR_TIMEOUT


@pytest.mark.parametrize("precision", list(WORD))
def test_every_synchronising_call_reads_the_word(precision):
    name, arg = WORD[precision]
    with fake() as F:
        h, D = handle(precision)
        th, V, G = _buffers(D)
        calls = {"adjoint": lambda: T.tlr_mdd_adjoint(h, V, G), "grad": lambda: T.tlr_mdd_grad(h, th, th.copy()),
                 "solve": lambda: T.tlr_mdd_solve(h, th, T.solve_opts(stages=1, admm_iters=1, lbfgs_iters=1)),
                 "benchmark": lambda: T.tlr_mdd_benchmark_solve(h, 0.1, 1, 0.0, G)}
        for what, f in calls.items():
            F.fake_fail(name, arg, 7)
            assert _times_out(f), what
            F.fake_fail(b"", 0, 0)
            f()
            # left by an asynchronous call
            F.fake_fail(name, arg, 7)
            T.tlr_mdd_apply(h, th, V)
            T.tlr_mdd_grad(h, th, th.copy(), want_f=False)
            F.fake_fail(b"", 0, 0)
            assert _times_out(f), what
            f()
        T.tlr_mdd_destroy(h)


def test_a_batch_reads_and_clears_its_members_words():
    with fake() as F:
        made = [handle(T.TLR_PREC_BF16X3) for _ in range(2)]
        hs = [m[0] for m in made]
        th, V, G = _buffers(made[0][1])
        b = T.tlr_mdd_batch_create(hs)
        opts = T.solve_opts(stages=1, admm_iters=1, lbfgs_iters=1)
        F.fake_fail(b"k_cgemm_tcp", 6, 7)
        T.tlr_mdd_batch_solve_async(b, [th.copy(), th.copy()], opts)
        F.fake_fail(b"", 0, 0)
        assert _times_out(lambda: T.tlr_mdd_batch_wait(b))
        for h in hs:
            T.tlr_mdd_grad(h, th, th.copy())
        # a member's own word alone
        F.fake_fail(b"k_cgemm_tcp", 6, 7)
        T.tlr_mdd_apply(hs[1], th, V)
        F.fake_fail(b"", 0, 0)
        T.tlr_mdd_batch_solve_async(b, [th.copy(), th.copy()], opts)
        assert _times_out(lambda: T.tlr_mdd_batch_wait(b))
        T.tlr_mdd_batch_solve_async(b, [th.copy(), th.copy()], opts)
        T.tlr_mdd_batch_wait(b)
        T.tlr_mdd_batch_destroy(b)
        for h in hs:
            T.tlr_mdd_destroy(h)
