"""The transforms in shared memory: every kind of length (each factor, chirp, the
largest of both, one beyond), trace counts that end within a pair and within a
CTA, bands at both ends, and pairs of very different or non-finite traces."""
import numpy as np
import pytest
import torch

import paper_2412_14973_gb300 as T
import tlr_synth as synth
from oracle import fourier

pytestmark = pytest.mark.gpu


def _forward(x, f0, nf):
    S = torch.empty((nf, x.shape[0]), dtype=torch.complex64, device="cuda")
    T.tlr_mdd_time_to_freq(torch.from_numpy(x).cuda(), *x.shape, f0, nf, S)
    return S


def _inverse(S, nt, f0):
    y = torch.empty((S.shape[1], nt), dtype=torch.float32, device="cuda")
    T.tlr_mdd_freq_to_time(S, S.shape[1], nt, f0, S.shape[0], y)
    return y


@pytest.mark.parametrize("nt", [1, 2, 3, 4, 5, 7, 11, 13, 16, 17, 30, 121, 169, 1001, 1125, 1021, 2047, 2048, 4096, 4097])
@pytest.mark.parametrize("ntr", [1, 35])
def test_lengths(nt, ntr):
    # FFT errors are a few 2^-24 per factor (at most 12; 25 passes for a chirp) of
    # a trace's 2-norm: 1e-5 of its own norm is far above, a wrong term far beyond
    x = synth.rng(nt + ntr).standard_normal((ntr, nt)).astype(np.float32)
    nh = nt // 2 + 1
    for f0, nf in {(0, nh), (nh // 3, max(1, nh // 2)), (nh - 1, 1)}:
        S = _forward(x, f0, nf)
        So = fourier.time_to_freq(x, f0, nf)
        err = np.abs(S.cpu().numpy() - So).max(axis=0) / (np.linalg.norm(x, axis=1) + 1e-30)
        assert err.max() <= 1e-5, (f0, nf, err.max())
        yo = fourier.freq_to_time(S.cpu().numpy(), nt, f0)
        y = _inverse(S, nt, f0).cpu().numpy()
        assert np.abs(y - yo).max() <= 1e-5 * max(1e-30, np.abs(yo).max())


def test_traces_of_a_pair_do_not_meet():
    # neighbours 1e12 apart, a zero trace, Inf, NaN, and magnitudes beyond the
    # scaling's range: each trace as accurate as alone, zeros stay zeros
    nt, nh = 240, 121
    x = synth.rng(9).standard_normal((12, nt)).astype(np.float32)
    x[1] *= 1e12
    x[3] = 0.0
    x[5, 7], x[8, 0] = np.inf, np.nan
    x[10] *= 1e20
    S = _forward(x, 0, nh).cpu().numpy()
    bad = [5, 8]
    good = [i for i in range(12) if i not in bad]
    So = np.fft.rfft(x[good].astype(np.float64), axis=1).T
    err = np.abs(S[:, good] - So).max(axis=0) / np.maximum(np.linalg.norm(x[good].astype(np.float64), axis=1), 1e-30)
    assert err.max() <= 1e-6, err
    assert not S[:, 3].any()
    assert not np.isfinite(S[:, bad]).all(axis=0).any()
    Sx = np.ascontiguousarray(S)
    y = _inverse(torch.from_numpy(Sx).cuda(), nt, 0).cpu().numpy()
    err = np.abs(y[good] - x[good]).max(axis=1) / np.maximum(np.abs(x[good]).max(axis=1), 1e-30)
    assert err.max() <= 1e-5, err
    assert not y[3].any()
    assert not np.isfinite(y[bad]).all(axis=1).any()
