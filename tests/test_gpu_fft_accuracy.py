"""Errors of the time <-> frequency transforms against 64 bits are no larger than those
of cuFFT's FP32 transforms, over lengths of every kind on both sides of the lines
between the two; and magnitudes at the ends of FP32's range."""
import numpy as np
import pytest
import torch

import paper_2412_14973_gb300 as T

pytestmark = pytest.mark.gpu

LENGTHS = ([3, 4, 5, 7, 21, 32, 63, 64, 78, 90, 99, 100, 128, 256, 512, 1024, 2048, 4096]      # small; powers of two
           + [17, 19, 34, 62, 68, 85, 124, 246, 247, 456, 1007, 1462, 1998, 2006, 2046, 2047]              # a largest prime factor of 17 .. 127
           + [131, 262, 1021, 1383, 1964, 2042]                                               # above
           + [88, 105, 198, 360, 405, 625, 720, 990, 1000, 1001, 1080, 1125, 1155, 1296, 1300, 1536, 1920, 2187, 2401,
              3000, 3125, 4000])


def _rel(a, b):
    return (torch.linalg.norm(a - b) / torch.linalg.norm(b)).item()


@pytest.mark.parametrize("nt", LENGTHS)
def test_no_less_accurate_than_the_library(nt):
    torch.manual_seed(nt)
    ntr, nf = max(64, min(4096, 600000 // nt)) + 1, nt // 2 + 1
    x = torch.randn(ntr, nt, device="cuda")
    X = torch.empty(nf, ntr, dtype=torch.complex64, device="cuda")
    T.tlr_mdd_time_to_freq(x, ntr, nt, 0, nf, X)
    want = torch.fft.rfft(x.double(), dim=1)
    e, el = _rel(X.T.to(torch.complex128), want), _rel(torch.fft.rfft(x, dim=1).to(torch.complex128), want)
    S = want.to(torch.complex64)
    S[:, 0] = S[:, 0].real.to(torch.complex64)
    if nt % 2 == 0:
        S[:, -1] = S[:, -1].real.to(torch.complex64)
    y = torch.empty(ntr, nt, device="cuda")
    T.tlr_mdd_freq_to_time(S.T.contiguous(), ntr, nt, 0, nf, y)
    back = torch.fft.irfft(S.to(torch.complex128), n=nt, dim=1)
    lib = torch.fft.irfft(S, n=nt, dim=1, norm="forward") * torch.tensor(1.0 / nt, dtype=torch.float32, device="cuda")
    f, fl = _rel(y.double(), back), _rel(lib.double(), back)
    print(f"{nt}: forward {e:.3e} (library {el:.3e}), inverse {f:.3e} ({fl:.3e})")
    # 1 %: two samples of rounding errors of 6e5 values
    assert e <= 1.01 * el and f <= 1.01 * fl


@pytest.mark.parametrize("nt", [128, 1021, 1125, 1964])
def test_magnitudes_at_the_ends_of_the_range(nt):
    # a spike of 1e37 (every bin 1e37, while a chirp's sums go beyond FP32 unscaled), a
    # trace of 1e36 noise, one near the smallest normal values, and neighbours of order one
    nf = nt // 2 + 1
    x = np.random.default_rng(nt).standard_normal((6, nt)).astype(np.float32)
    x[1] = 0
    x[1, 5] = 1e37
    x[2] *= np.float32(1e36 / nt)
    x[4] *= np.float32(1e-36)
    X = torch.empty(nf, 6, dtype=torch.complex64, device="cuda")
    T.tlr_mdd_time_to_freq(torch.from_numpy(x).cuda(), 6, nt, 0, nf, X)
    want = np.fft.rfft(x.astype(np.float64), axis=1)
    got = X.cpu().numpy().T
    for i in range(6):
        assert np.linalg.norm(got[i] - want[i]) <= 1e-6 * np.linalg.norm(want[i]), i
    y = torch.empty(6, nt, device="cuda")
    T.tlr_mdd_freq_to_time(X, 6, nt, 0, nf, y)
    y = y.cpu().numpy().astype(np.float64)
    for i in range(6):
        assert np.linalg.norm(y[i] - x[i]) <= 1e-6 * np.linalg.norm(x[i].astype(np.float64)), i


@pytest.mark.parametrize("nt,ntr", [(51, 800001), (85, 800001), (247, 300001), (4097, 16385)])
def test_many_traces_of_odd_lengths(nt, ntr):
    # several chunks of the library's transforms (51, 4097) start on 8 bytes each
    torch.manual_seed(1)
    nf = 9
    x = torch.randn(ntr, nt, device="cuda")
    X = torch.empty(nf, ntr, dtype=torch.complex64, device="cuda")
    T.tlr_mdd_time_to_freq(x, ntr, nt, 3, nf, X)
    for part in (slice(0, 100), slice(ntr - 100, ntr)):
        want = torch.fft.rfft(x[part].double(), dim=1)[:, 3:3 + nf]
        assert _rel(X[:, part].T.to(torch.complex128), want) <= 1e-6
    y = torch.empty_like(x)
    T.tlr_mdd_freq_to_time(X, ntr, nt, 3, nf, y)
    S = torch.zeros(100, nt // 2 + 1, dtype=torch.complex128, device="cuda")
    S[:, 3:3 + nf] = X[:, ntr - 100:].T
    assert _rel(y[ntr - 100:].double(), torch.fft.irfft(S, n=nt, dim=1)) <= 1e-6


@pytest.mark.parametrize("nt", [51, 68])
def test_traces_that_start_on_four_bytes(nt):
    ntr, nf = 7, nt // 2 + 1
    x = torch.randn(ntr * nt + 1, device="cuda")[1:]
    X = torch.empty(nf, ntr, dtype=torch.complex64, device="cuda")
    T.tlr_mdd_time_to_freq(x, ntr, nt, 0, nf, X)
    want = torch.fft.rfft(x.view(ntr, nt).double(), dim=1)
    assert _rel(X.T.to(torch.complex128), want) <= 1e-6
