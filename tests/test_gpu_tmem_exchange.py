"""The fused kernel whose last exchange goes through tensor memory (nfft 1024 .. 16384) where it can go
wrong: several units per CTA (the next unit's window is staged while the last one ends), windows that
start at every offset within 16 bytes, codes a few chips shorter than nfft (what a rounded copy leaves
behind the last chip must not enter the transform), and packed chip signs over several launches.
Every bin is compared with the FP64 oracle at the per-bin bound RTOL."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import RTOL, assert_parity, gpu_integrate
from paper_2311_18737_gb300 import isr

pytestmark = pytest.mark.gpu


def _case(seed, nfft, R, P, start, step, L, kind, per):
    rng = np.random.default_rng(seed)
    stride = (start + (R - 1) * step + L + 3) // 4 * 4
    echo = np.clip(np.rint(rng.standard_normal((P, stride, 2)) * 1000), -32768, 32767).astype(np.int16)
    shape = (P, L) if per else (L,)
    if kind == "pm1":
        tx = np.where(rng.random(shape) < 0.5, -1, 1).astype(np.int8)
    elif kind == "ci16":
        tx = np.rint(rng.standard_normal(shape + (2,)) * 500).astype(np.int16)
    else:
        tx = rng.standard_normal(shape + (2,)).astype(np.float32)
    return echo, tx


@pytest.mark.parametrize("kind", ["pm1", "ci16", "c32"])
@pytest.mark.parametrize("log2n,short", [(10, 1), (11, 3), (12, 5), (13, 2), (14, 0), (14, 7)])
def test_several_units_per_cta_and_short_codes(log2n, short, kind):
    nfft = 1 << log2n
    G = 16384 // nfft
    R, P, step, L = 320 * G - 3, 4, 3, nfft - short      # at least two units for every CTA, the last ragged
    echo, tx = _case(log2n + short, nfft, R, P, 1, step, L, kind, False)
    got, info = gpu_integrate(echo, tx, nfft=nfft, n_ranges=R, range_start=1, range_step=step, code_len=L)
    assert info["kernel_launches"] == 1
    gates = np.unique(np.r_[0:5, np.linspace(0, R - 1, 24).astype(int), R - 5:R])
    ref = np.stack([oracle.integrate(echo, tx, nfft=nfft, n_ranges=1, range_start=1 + int(r) * step, range_step=1,
                                     code_len=L)[0] for r in gates])
    assert_parity(got[gates], ref, what=f"nfft={nfft} L={L} {kind}")


@pytest.mark.parametrize("log2n,L", [(10, 1024), (11, 2041), (14, 16384)])
def test_packed_signs_over_launches_and_calls(log2n, L):
    """Codes of their own per IPP at an odd row pitch; 7 IPPs in launches of 4 and calls of 5 + 2."""
    nfft = 1 << log2n
    R, P = 5, 7
    echo, tx = _case(3 * log2n, nfft, R, P, 2, 5, L + 3, "pm1", True)
    got, info = gpu_integrate(echo, tx, nfft=nfft, n_ranges=R, range_start=2, range_step=5, code_len=L,
                              per_ipp_tx=True, ipp_chunk=2, max_chunks=2, calls=[5, 2])
    ref = oracle.integrate(echo, tx, nfft=nfft, n_ranges=R, range_start=2, range_step=5, code_len=L, per_ipp_tx=True)
    assert_parity(got, ref, what=f"nfft={nfft} L={L}")


@pytest.mark.parametrize("order", [0, 6])
def test_orders_0_and_6_at_full_scale_samples(order):
    """Full-scale int16 samples and a line that fills one bin: the largest sums the decode meets."""
    nfft, R, P = 16384, 3, 2
    echo = np.full((P, 2 * 4 + nfft, 2), 32767, dtype=np.int16)
    echo[1] = -32768
    echo[:, 100:200] = np.random.default_rng(1).integers(-32768, 32768, (P, 100, 2)).astype(np.int16)
    tx = np.where(np.random.default_rng(2).random(nfft) < 0.5, -1, 1).astype(np.int8)
    dev = torch.device("cuda:0")
    with isr.Plan(nfft=nfft, n_ranges=R, echo_stride=echo.shape[1], range_step=3, device=0,
                  stream=torch.cuda.current_stream()) as plan:
        isr.isr_plan_set_order(plan.handle, order)
        plan.integrate(torch.from_numpy(echo).to(dev), torch.from_numpy(tx).to(dev), P)
        out, _ = plan.spectra()
    ref = oracle.integrate(echo, tx, nfft=nfft, n_ranges=R, range_start=0, range_step=3)
    # a bin may be small beside the rms bin, whose rounding it shares
    tol = RTOL * np.maximum(ref, ref.mean(axis=1, keepdims=True))
    assert (np.abs(out.numpy().astype(np.float64) - ref) <= tol).all()


@pytest.mark.parametrize("kind", ["ci16", "c32"])
@pytest.mark.parametrize("log2n", [11, 14])
def test_orders_of_full_length_complex_codes(log2n, kind):
    """The radix orders tell kernels of binary-phase codes apart; with any other code a plan takes orders
    1 to 3 as well, through the one kernel there is, and the autotuner times them on the caller's data."""
    nfft, R, P = 1 << log2n, 5, 3
    echo, tx = _case(5 * log2n, nfft, R, P, 1, 3, nfft, kind, False)
    ref = oracle.integrate(echo, tx, nfft=nfft, n_ranges=R, range_start=1, range_step=3)
    e, t = torch.from_numpy(echo).cuda(), torch.from_numpy(tx).cuda()
    with isr.Plan(nfft=nfft, n_ranges=R, echo_stride=echo.shape[1], range_start=1, range_step=3,
                  tx_type=isr.ISR_TX_CI16 if kind == "ci16" else isr.ISR_TX_C32, device=0,
                  stream=torch.cuda.current_stream()) as plan:
        for order in (1, 2, 3):
            isr.isr_plan_set_order(plan.handle, order)
            plan.integrate(e, t, P)
            out, _ = plan.spectra(flags=isr.ISR_RESET_AFTER)
            assert_parity(out.numpy().astype(np.float64), ref, what=f"nfft={nfft} {kind} order {order}")
        tuned = plan.autotune(e, t, P)
        assert tuned["order"] in range(4) and len(tuned["ms"]) == 4
        plan.integrate(e, t, P)
        assert_parity(plan.spectra()[0].numpy().astype(np.float64), ref, what=f"nfft={nfft} {kind} tuned")


def test_autotuner_times_each_kernel_once():
    """Orders 0 and 6 are one kernel: it is timed once, and reported as order 0."""
    nfft, R, P = 16384, 4, 2
    echo, tx = _case(7, nfft, R, P, 0, 1, nfft, "pm1", False)
    e, t = torch.from_numpy(echo).cuda(), torch.from_numpy(tx).cuda()
    with isr.Plan(nfft=nfft, n_ranges=R, echo_stride=echo.shape[1], range_step=1, device=0,
                  stream=torch.cuda.current_stream()) as plan:
        tuned = plan.autotune(e, t, P)
    assert len(tuned["ms"]) == isr.N_ORDERS and tuned["ms"][6] == tuned["ms"][0] and tuned["order"] != 6
