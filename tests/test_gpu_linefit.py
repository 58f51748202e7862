"""GPU peak fit (isr_peak_fit through the C ABI) against the FP64 peak-fit oracle."""
import numpy as np
import pytest
import torch

import synth
from gpu_helpers import gpu_integrate
from oracle import linefit
from paper_2311_18737_gb300 import isr

pytestmark = pytest.mark.gpu


def _gpu_fit(P, lo, hi):
    dev = torch.device("cuda:0")
    Pd = torch.from_numpy(np.ascontiguousarray(P, dtype=np.float32)).to(dev)
    R, N = P.shape
    f = torch.empty(R, dtype=torch.float64, device=dev)
    s = torch.empty(R, dtype=torch.float32, device=dev)
    isr.isr_peak_fit(Pd, R, N, lo, hi, f, s, torch.cuda.current_stream())
    torch.cuda.synchronize()
    return f.cpu().numpy(), s.cpu().numpy().astype(np.float64)


def test_random_spectra_with_peaks_and_ties():
    rng = np.random.default_rng(3)
    R, N = 300, 4096
    P = rng.gamma(50.0, 1.0, size=(R, N)).astype(np.float32)
    c = rng.uniform(400, 3600, R)
    f = np.arange(N)
    P += (300.0 * np.exp(-((f[None, :] - c[:, None]) ** 2) / 4.0)).astype(np.float32)
    P[7, 1000] = P[7, 1500] = 1e6          # tie
    P[8, :] = 3.0                          # flat
    got_f, got_s = _gpu_fit(P, 300, 3800)
    ref_f, ref_s = linefit.peak_fit(P, 300, 3800)
    assert np.abs(got_f - ref_f).max() <= 1e-9
    assert np.abs(got_s - ref_s).max() <= 1e-6 * np.abs(ref_s).max()


def test_fit_of_integrated_tones():
    w = synth.small(n_ipp=30, snap_to_bins=True)
    echo, code = w.echo_host(), w.code()
    P, _ = gpu_integrate(echo, code, nfft=w.nfft, n_ranges=w.n_ranges, range_step=w.range_step)
    got_f, _ = _gpu_fit(P, 0, w.nfft)
    ref_f, _ = linefit.peak_fit(P, 0, w.nfft)
    assert np.abs(got_f - ref_f).max() <= 1e-9
    true_bin = np.mod(np.round(w.base_freqs() * w.nfft), w.nfft)
    assert np.abs(got_f - true_bin).max() <= 0.5


@pytest.mark.parametrize("lo,hi,N", [(0, 8, 8), (3, 4, 64), (1, 256, 256), (5, 2054, 4096), (7, 4096, 4096), (11, 16384, 16384)])
def test_band_edges_and_odd_lengths(lo, hi, N):
    """Bands around one thread's, one warp's and one unrolled pass' share.  The ratio is one FP32
    rounding (2^-24) of a quotient whose band sum carries about 2^-44; 1.5e-7 covers both."""
    rng = np.random.default_rng(N + lo)
    P = rng.gamma(4.0, 1e9, size=(9, N)).astype(np.float32)
    got_f, got_s = _gpu_fit(P, lo, hi)
    ref_f, ref_s = linefit.peak_fit(P, lo, hi)
    assert np.abs(got_f - ref_f).max() <= 1e-9
    assert (np.abs(got_s - ref_s) <= 1.5e-7 * np.abs(ref_s)).all()


def test_non_finite_and_overflowing_bands():
    """Bands whose sum leaves FP32 (as values or as NaN and infinities) are summed in FP64."""
    N, lo, hi = 1024, 10, 1000
    P = np.full((4, N), 2.0, dtype=np.float32)
    P[0, :] = 3e38
    P[0, 500] = 3.2e38
    P[1, 400] = np.nan
    P[1, 300] = 5.0
    P[2, 200] = np.inf
    P[3, lo:hi] = np.nan
    got_f, got_s = _gpu_fit(P, lo, hi)
    ref_f, ref_s = linefit.peak_fit(P[:1], lo, hi)
    assert abs(got_f[0] - ref_f[0]) <= 1e-9 and abs(got_s[0] - ref_s[0]) <= 1.5e-7 * ref_s[0]
    assert list(got_f[1:]) == [300.0, 200.0, float(lo)]     # symmetric neighbours; NaN never wins
    assert got_s[1] == 0.0 and np.isnan(got_s[2]) and got_s[3] == 0.0
