"""The read-back that sums chunk partials straight into the spectra, in every state the partials can be
in: none, some pending, scratch full and reduced, a read between calls, resets, a stream capture among
the calls, and an output that is not 16-byte aligned.  Bins against the FP64 oracle at RTOL."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import assert_parity
from gpu_helpers import RTOL
from paper_2311_18737_gb300 import isr

pytestmark = pytest.mark.gpu

NFFT, R, STEP = 1024, 5, 3


def _echo(seed, P):
    rng = np.random.default_rng(seed)
    stride = ((R - 1) * STEP + NFFT + 3) // 4 * 4
    return (np.clip(np.rint(rng.standard_normal((P, stride, 2)) * 1000), -32768, 32767).astype(np.int16),
            np.where(rng.random(NFFT) < 0.5, -1, 1).astype(np.int8))


def _ref(echo, tx):
    return oracle.integrate(echo, tx, nfft=NFFT, n_ranges=R, range_start=0, range_step=STEP)


def _plan(echo, stream, **kw):
    return isr.Plan(nfft=NFFT, n_ranges=R, echo_stride=echo.shape[1], range_step=STEP, device=0, stream=stream, **kw)


@pytest.mark.parametrize("max_chunks,ipp_chunk", [(0, 0), (1, 4), (2, 3), (3, 2)])
def test_reads_between_calls_and_resets(max_chunks, ipp_chunk):
    echo, tx = _echo(1, 23)
    e, t = torch.from_numpy(echo).cuda(), torch.from_numpy(tx).cuda()
    with _plan(echo, torch.cuda.current_stream(), max_chunks=max_chunks, ipp_chunk=ipp_chunk) as plan:
        out, n = plan.spectra()
        assert n == 0 and not out.any()
        done = 0
        for k in (4, 1, 7):
            plan.integrate(e[done:], t, k)
            done += k
            for _ in range(2):          # reading leaves the integration as it was
                out, n = plan.spectra(flags=isr.ISR_MEAN)
                assert n == done
                assert_parity(out.numpy().astype(np.float64), _ref(echo[:done], tx) / done, what=f"after {done}")
        plan.spectra(out, isr.ISR_RESET_AFTER)
        assert not plan.spectra()[0].any()
        plan.integrate(e[done:], t, 11)
        isr.isr_spectra(plan.handle, None, isr.ISR_RESET_AFTER)
        plan.integrate(e[:6], t, 6)
        buf = torch.zeros(R * NFFT + 1, device="cuda")          # an output that is only 4-byte aligned
        plan.spectra(buf[1:])
        assert buf[0] == 0
        assert_parity(buf[1:].reshape(R, NFFT).cpu().numpy().astype(np.float64), _ref(echo[:6], tx), what="unaligned")


def test_captured_integration_replayed_between_calls():
    """A captured isr_integrate adds to the integration at every replay, whatever was pending before it."""
    echo, tx = _echo(2, 12)
    e, t = torch.from_numpy(echo).cuda(), torch.from_numpy(tx).cuda()
    side = torch.cuda.Stream()
    with _plan(echo, side) as plan:
        side.wait_stream(torch.cuda.current_stream())
        plan.integrate(e, t, 4)                                   # pending when the capture starts
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            plan.integrate(e[4:], t, 5)
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            graph.replay()
            graph.replay()
        plan.integrate(e[9:], t, 3)
        out, _ = plan.spectra(flags=isr.ISR_RESET_AFTER)
        ref = _ref(echo[:4], tx) + 2 * _ref(echo[4:9], tx) + _ref(echo[9:], tx)
        assert_parity(out.numpy().astype(np.float64), ref, what="two replays")
        with torch.cuda.stream(side):
            graph.replay()
        out, _ = plan.spectra()
        assert_parity(out.numpy().astype(np.float64), _ref(echo[4:9], tx), what="a replay after the reset")


@pytest.mark.parametrize("gates,row", [(5001, 7168), (5001, 1 << 20), (2431, 1 << 20)])
def test_host_rows_in_blocks_and_gate_slices(gates, row):
    """Host rows to host spectra: blocks of rows (36 MB of them, or one block of the short rows) and,
    from 32 MB of spectra, a last launch in gate slices read back one by one (5001 gates: two, the last
    one ragged; 2431: none).  Against the device-resident call: every bin is a sum of nine powers, in
    FP32 in any order within 9 x 2^-24 of each other, twice over for two calls."""
    n, nfft = 9, 2048
    g = torch.Generator(device="cuda").manual_seed(3)
    echo = torch.randint(-300, 300, (n, row, 2), generator=g, device="cuda", dtype=torch.int16)
    code = torch.randint(0, 2, (nfft,), generator=g, device="cuda", dtype=torch.int8) * 2 - 1
    hosts = [t.cpu().pin_memory() for t in (echo, code)]
    with isr.Plan(nfft=nfft, n_ranges=gates, echo_stride=row, code_len=nfft, range_start=0, range_step=1,
                  tx_type=isr.ISR_TX_PM1, stream=torch.cuda.current_stream()) as plan:
        want = torch.empty((gates, nfft), device="cuda")
        plan.integrate(echo, code, n)
        plan.spectra(want, isr.ISR_RESET_AFTER)
        want = want.cpu()
        got = torch.empty((gates, nfft)).pin_memory()
        plan.integrate(*hosts, n)
        plan.spectra(got)
        assert torch.allclose(got, want, rtol=2e-6, atol=0)
        plan.integrate(echo, code, n)      # device rows on top: the slices are no longer the whole
        plan.spectra(got)
        assert torch.allclose(got, 2 * want, rtol=4e-6, atol=0)
        plan.integrate(*hosts, n)          # host rows on top of sums already there
        plan.spectra(got, isr.ISR_RESET_AFTER)
        assert torch.allclose(got, 3 * want, rtol=6e-6, atol=0)


@pytest.mark.parametrize("gates", [5001, 700])
def test_read_back_to_the_host_keeps_the_stream_order(gates):
    """Work that the caller queues on the plan's stream between isr_integrate (host rows) and isr_spectra
    comes before the copy into the host buffer, here an upload from that very buffer behind a long delay."""
    n, nfft = 9, 2048
    g = torch.Generator(device="cuda").manual_seed(4)
    echo = torch.randint(-300, 300, (n, 7168, 2), generator=g, device="cuda", dtype=torch.int16)
    code = torch.randint(0, 2, (nfft,), generator=g, device="cuda", dtype=torch.int8) * 2 - 1
    hosts = [t.cpu().pin_memory() for t in (echo, code)]
    buf = torch.full((gates, nfft), -5.0).pin_memory()
    before = torch.zeros((gates, nfft), device="cuda")
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with isr.Plan(nfft=nfft, n_ranges=gates, echo_stride=7168, code_len=nfft, range_start=0, range_step=1,
                  tx_type=isr.ISR_TX_PM1, stream=side) as plan:
        plan.integrate(*hosts, n)
        with torch.cuda.stream(side):
            torch.cuda._sleep(40_000_000)      # about 20 ms
            before.copy_(buf, non_blocking=True)
        plan.spectra(buf)
        assert (before == -5.0).all()
        assert (buf > 0.0).all()


@pytest.mark.parametrize("nfft", [512, 1024])
@pytest.mark.parametrize("max_chunks", [0, 2, 4])
def test_sums_over_calls_beyond_the_range_of_fp32(nfft, max_chunks):
    """Six calls whose sums leave FP32 together but not each (a float code of amplitude 1e14), pending all
    at once, two at a time, or two beside four reduced ones: the mean is finite and within RTOL of the oracle's, the sum infinite where
    it is beyond FP32."""
    rng = np.random.default_rng(8)
    R, calls = 4, 6
    echo = np.clip(np.rint(rng.standard_normal((1, nfft + 8, 2)) * 1000), -32768, 32767).astype(np.int16)
    tx = (1e14 * np.exp(2j * np.pi * rng.random(nfft))).astype(np.complex64).view(np.float32).reshape(nfft, 2)
    ref = oracle.integrate(echo, tx, nfft=nfft, n_ranges=R, range_start=0, range_step=2)
    assert ref.max() < 3.4e38 < calls * ref.max() and calls * ref.min() < 3.4e38
    e, t = torch.from_numpy(echo).cuda(), torch.from_numpy(tx).cuda()
    with isr.Plan(nfft=nfft, n_ranges=R, echo_stride=nfft + 8, range_step=2, tx_type=isr.ISR_TX_C32, device=0,
                  max_chunks=max_chunks, stream=torch.cuda.current_stream()) as plan:
        for _ in range(calls):
            plan.integrate(e, t, 1)
        out, _ = plan.spectra(flags=isr.ISR_MEAN)
        # a bin far below the mean shares the mean's rounding
        tol = RTOL * np.maximum(ref, 0.01 * ref.mean(axis=1, keepdims=True))
        assert (np.abs(out.numpy().astype(np.float64) - ref) <= tol).all()
        total = plan.spectra()[0].numpy()
        assert np.isposinf(total[calls * ref > 3.41e38]).all() and np.isfinite(total[calls * ref < 3.39e38]).all()
