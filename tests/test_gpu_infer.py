"""The fused inference kernel (BF16 storage, tcgen05): bands around its 488-position tiles, more tiles
than the chip has room for at once, and activations that overflow to infinity, whose products with the
zero taps of the widened convolution must not enter other positions' sums.  Inputs and convolution
weights are dyadic, so every convolution sum is exact and the predictions differ from the reference
with BF16 storage rounding by the head's FP32 arithmetic only (1e-3 bins, 1e-5 in presence)."""
import numpy as np
import pytest
import torch

from oracle import estimator as ref
from paper_2311_18737_gb300 import estimator as est_mod
from paper_2311_18737_gb300 import isr

pytestmark = pytest.mark.gpu


def _theta(seed):
    rng = np.random.default_rng(seed)
    d = ref.unpack(ref.init_params(seed))
    for l in range(1, 5):
        d[f"W{l}"] = rng.integers(-2, 3, d[f"W{l}"].shape) / 8.0
        d[f"b{l}"] = rng.integers(-2, 3, d[f"b{l}"].shape) / 8.0
    return d


def _predict(theta, x, precision=isr.ISR_EST_BF16):
    e = est_mod.Estimator(max_batch=x.shape[0], precision=precision, nfft=max(8, x.shape[1]), band_lo=0,
                          band_len=x.shape[1])
    e.set_params(theta)
    pos, pres = e.predict(torch.from_numpy(x).cuda())
    out = pos.cpu().numpy(), pres.cpu().numpy()
    e.close()
    return out


@pytest.mark.parametrize("B,L", [(1, 16), (3, 487), (2, 488), (2, 489), (3, 976), (2, 977), (1, 4608), (320, 1000)])
def test_tile_edges(B, L):
    theta = ref.pack(_theta(L)).astype(np.float32)
    x = (np.random.default_rng(B + L).integers(-8, 9, (B, L)) / 4.0).astype(np.float32)
    pos, pres = _predict(theta, x)
    rows = np.unique(np.linspace(0, B - 1, 24).astype(int))
    rpos, rpres = ref.predict(theta.astype(np.float64), x[rows], store=ref.round_bf16)
    assert np.abs(pos[rows] - rpos).max() <= 1e-3
    assert np.abs(pres[rows] - rpres).max() <= 1e-5


def test_infinite_activation_stays_within_its_taps():
    """One sample overflows channel 5 of the first layer at one position; the second layer's taps on that
    channel are negative or zero, so four positions on either side become 0 and the rest is finite.  The
    mma.sync engine multiplies the nine taps alone and is the reference."""
    rng = np.random.default_rng(4)
    d = _theta(4)
    d["W1"] = np.zeros_like(d["W1"])
    d["W1"][5, 0, 4] = 4.0
    d["b1"] = np.full_like(d["b1"], 0.5)
    d["W2"][:, 5, :] = -rng.integers(0, 3, d["W2"][:, 5, :].shape) / 8.0
    theta = ref.pack(d).astype(np.float32)
    x = (rng.integers(-8, 9, (4, 1000)) / 4.0).astype(np.float32)
    plain = _predict(theta, x)
    for row, at in ((0, 0), (1, 333), (2, 490), (3, 999)):
        x[row, at] = 2.0 ** 127
    got, want = _predict(theta, x), _predict(theta, x, isr.ISR_EST_BF16_MMASYNC)
    assert np.isfinite(want[0]).all() and np.isfinite(want[1]).all()
    assert np.abs(got[0] - want[0]).max() <= 1e-3 and np.abs(got[1] - want[1]).max() <= 1e-5
    assert np.abs(plain[1] - want[1]).max() > 1e-5      # the infinities do reach the head


@pytest.mark.parametrize("precision", [isr.ISR_EST_BF16, isr.ISR_EST_BF16_MMASYNC, isr.ISR_EST_FP32])
@pytest.mark.parametrize("L,max_batch,n", [(16, 2, 37), (488, 3, 100), (1101, 8, 37), (4608, 5, 77), (1000, 4, 4)])
def test_many_rows_as_their_batches(precision, L, max_batch, n):
    """A prediction of more rows than a batch, in one launch or several (77 and 100 rows pass what the
    buffers of 5 and 3 hold), against the rows batch by batch: bit for bit, since no row reads another's."""
    dev = torch.device("cuda:0")
    x = torch.randn((n, L), generator=torch.Generator(device="cuda").manual_seed(L), device=dev)
    e = est_mod.Estimator(max_batch=max_batch, precision=precision, nfft=8192, band_lo=7, band_len=L)
    e.set_params(ref.init_params(4).astype(np.float32))
    want = [torch.empty(n, device=dev) for _ in range(2)]
    for b in range(0, n, max_batch):
        m = min(max_batch, n - b)
        isr.isr_est_predict(e.h, x[b:b + m], m, want[0][b:b + m], want[1][b:b + m])
    got = [torch.full((n,), -1.0, device=dev) for _ in range(2)]
    isr.isr_est_predict_all(e.h, x, n, *got)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    assert all(torch.equal(a, b) for a, b in zip(e.predict(x), want))
    e.close()
