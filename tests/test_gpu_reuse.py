"""What handles share or reuse: recycled pinned blocks and pool memory on several threads
and streams, launches that start early beside another stream's, split-K partials that
fill the panels they lie over exactly."""
import threading

import numpy as np
import pytest
import torch

import paper_2412_14973_gb300 as T
import tlr_synth as synth
from oracle import operator, solver

from _cases import problem
from _gpu import Gpu, dev, host, rel

pytestmark = pytest.mark.gpu

OPTS = dict(stages=1, admm_iters=2, lbfgs_iters=4)


def test_handles_come_and_go_on_two_threads():
    shapes = [(8, 8, 16, 3, 70, T.TLR_PREC_FP32), (16, 16, 64, 5, 130, T.TLR_PREC_BF16X3),
              (16, 8, 32, 4, 99, T.TLR_PREC_TF32)]
    cases = []
    for nx, ny, b, k, ns, prec in shapes:
        D, U, perm, lay, _ = problem(nx, ny, b, k, "lowrank", ns=ns, snr_db=10, planted=False)
        th = (0.2 * synth.cn(synth.rng(ns), lay.size)).astype(np.complex64)
        cases.append((D, U, lay, nx, ny, prec, th))

    def once(c, stream=None):
        D, U, lay, nx, ny, prec, th = c
        g = Gpu(D, U, lay, nx=nx, ny=ny, precision=prec, stream=stream)
        td = dev(th)
        torch.cuda.current_stream().synchronize()
        gr = torch.empty_like(td)
        f = T.tlr_mdd_grad(g.h, td, gr)
        st = T.tlr_mdd_solve(g.h, td, T.solve_opts(**OPTS))
        out = (f, gr.cpu().numpy(), td.cpu().numpy(), list(st.f_hist)[:st.n_hist], st.iters)
        g.close()
        return out

    want = [once(c) for c in cases]
    wrong = []

    def work(seed):
        s = torch.cuda.Stream()
        order = np.random.default_rng(seed).integers(0, len(cases), 24)
        with torch.cuda.stream(s):
            for i in order:
                got = once(cases[i], s)
                if not (got[0] == want[i][0] and np.array_equal(got[1], want[i][1]) and
                        np.array_equal(got[2], want[i][2]) and got[3:] == want[i][3:]):
                    wrong.append(int(i))

    ts = [threading.Thread(target=work, args=(n,)) for n in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not wrong


def test_early_launches_beside_another_stream():
    # gradients small enough to start early, on streams side by side, with no waits between
    D, U, perm, lay, _ = problem(16, 16, 64, 5, "lowrank", ns=200, snr_db=10, planted=False)
    n = 3
    streams = [torch.cuda.Stream() for _ in range(n)]
    hs = [Gpu(D, U, lay, nx=16, ny=16, precision=p, stream=s)
          for p, s in zip((T.TLR_PREC_BF16X3, T.TLR_PREC_FP32, T.TLR_PREC_TF32), streams)]
    ths = [dev(0.2 * synth.cn(synth.rng(i), lay.size)) for i in range(8)]
    out = [[torch.empty_like(t) for t in ths] for _ in range(n)]
    torch.cuda.synchronize()
    for m in range(n):
        for i, t in enumerate(ths):
            T.tlr_mdd_grad(hs[m].h, t, out[m][i], want_f=False)
            torch.cuda.synchronize()
    want = [[g.clone() for g in o] for o in out]
    for o in out:
        for g in o:
            g.zero_()
    torch.cuda.synchronize()
    for _ in range(5):
        for i, t in enumerate(ths):
            for m in range(n):
                T.tlr_mdd_grad(hs[m].h, t, out[m][i], want_f=False)
        torch.cuda.synchronize()
        for m in range(n):
            for a, b in zip(out[m], want[m]):
                assert torch.equal(torch.view_as_real(a), torch.view_as_real(b))
    for h in hs:
        h.close()


# one dense tile of 256 x 256: the partials of a split over s chunks of the sources take
# s 65536 values of the 2 nr ns = 512 ns that they lie over
@pytest.mark.parametrize("ns", [128, 255, 256, 383, 384, 512])
@pytest.mark.parametrize("prec", [T.TLR_PREC_FP32, T.TLR_PREC_BF16X3])
def test_partials_fill_their_panels(ns, prec):
    D, U, perm, lay, _ = problem(16, 16, 256, 8, "dense", ns=ns, snr_db=10, planted=False)
    assert lay.size == 65536
    th = (0.1 * synth.cn(synth.rng(ns), lay.size)).astype(np.complex64).astype(np.complex128)
    Dh, Uh, alpha = operator.normalise(D, U, perm)
    g = Gpu(D, U, lay, nx=16, ny=16, alpha=alpha, precision=prec)
    f, gr = g.grad(th)
    tol = 1e-6 if prec == T.TLR_PREC_FP32 else 5e-5
    assert abs(f - operator.misfit(th, lay, Dh, Uh)) <= tol * f
    assert rel(gr, operator.gradient(th, lay, Dh, Uh)) <= tol
    got, st = g.solve(th, **OPTS)
    prob = solver.Problem(lay, Dh.T, Uh.T)
    want, _, _, sto = solver.admm(prob, th, solver.SolveOpts(**OPTS))
    g.close()
    # 8 steps, each of a few contractions at tol, through the line searches
    assert st.iters == 8
    assert rel(got, want) <= 200 * tol
