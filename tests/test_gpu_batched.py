"""Batched uneven windows (one persistent launch) against one plan per window and against
the FP64 oracle on sampled gates; every radix order, graph replay, autotuning."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import RTOL, assert_parity
from paper_2311_18737_gb300 import batched, isr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bufs():
    ws = batched.config_windows(seed=5, n_windows=8, ipp_scale=0.006, max_gates=300)
    return batched.Buffers(ws)


@pytest.fixture(scope="module")
def reference(bufs):
    outs = batched.per_window(bufs)
    torch.cuda.synchronize()
    return [o.cpu().numpy().astype(np.float64) for o in outs]


@pytest.mark.parametrize("order", [0, 1, 2, 3])
def test_every_radix_order_matches_per_window_plans(bufs, reference, order):
    b = batched.Batch(bufs, flags=0, order=order)
    b.run()
    for i, (o, ref) in enumerate(zip(bufs.out, reference)):
        assert_parity(o.cpu().numpy().astype(np.float64), ref, what=f"order {order} window {i}")
    b.close()


def test_graph_replay_and_autotune(bufs, reference):
    b = batched.Batch(bufs, flags=isr.ISR_BATCH_GRAPH | isr.ISR_BATCH_AUTOTUNE)
    info = b.info()
    assert info["graph"] and info["n_windows"] == 8
    used = {w.nfft for w in bufs.w}
    for k, n in enumerate(batched.NFFTS):
        if n in used:
            assert info["order"][k] in (0, 1, 2, 3) and min(info["tune_ms"][k]) > 0
    b.run()
    first = [o.clone() for o in bufs.out]
    b.run()
    for a, c, ref in zip(first, bufs.out, reference):
        assert torch.equal(a, c)   # replays are deterministic
        assert_parity(c.cpu().numpy().astype(np.float64), ref, what="graph replay")
    b.close()


def test_sampled_gates_against_oracle(bufs):
    b = batched.Batch(bufs, flags=0)
    b.run()
    for i in (0, 1):   # one up-shifted, one down-shifted window
        w = bufs.w[i]
        echo = bufs.echo[i].cpu().numpy()
        code = bufs.code[i].cpu().numpy()
        sel = [0, w.n_ranges // 2, w.n_ranges - 1]
        ref = oracle.integrate(echo, code, nfft=w.nfft, n_ranges=w.n_ranges, range_start=w.range_start,
                               range_step=w.range_step, sel=sel)
        assert_parity(bufs.out[i].cpu().numpy().astype(np.float64)[sel], ref, rtol=RTOL, what=f"window {i}")
    b.close()


def test_bad_window_rejected(bufs):
    ws = bufs.windows()
    ws[3].nfft = 1024
    with pytest.raises(isr.IsrError) as ei:
        isr.isr_batch_create(ws, 0, 0, torch.cuda.current_stream())
    assert ei.value.status == isr.ISR_ERR_UNSUPPORTED


def test_reused_per_window_plans_match_fresh_plans(bufs, reference):
    # the batched comparison's baseline: plans created once and reused over two runs
    pw = batched.PerWindowPlans(bufs, orders={2048: 1, 4096: 0, 8192: 2, 16384: 1})
    try:
        for _ in range(2):
            outs = [torch.empty_like(o) for o in bufs.out]
            pw.run(outs)
            for i, (o, r) in enumerate(zip(outs, reference)):
                assert_parity(o.cpu().numpy().astype(np.float64), r, rtol=RTOL, what=f"reused plan, window {i}")
    finally:
        pw.close()


def test_mixed_code_lengths_and_gate_counts_in_one_launch():
    """Windows of one transform length with short and full codes in turn (a CTA takes units of several,
    and what a longer window left in its stage must not enter a shorter one), more CTAs than units for
    some lengths, several chunks (a reduction) for others, and per-IPP codes."""
    rng = np.random.default_rng(17)
    dev = torch.device("cuda:0")
    shapes = [(2048, 2048, 200, 3, 0), (2048, 1025, 700, 2, 0), (2048, 2041, 900, 2, 1), (2048, 2048, 1500, 2, 0),
              (4096, 4095, 3, 5, 0), (4096, 2049, 650, 2, 0), (4096, 4096, 700, 2, 1), (8192, 8190, 2, 600, 0),
              (16384, 9000, 160, 2, 0), (16384, 16384, 170, 2, 0), (16384, 16383, 180, 2, 0), (16384, 8193, 200, 2, 1)]
    keep, ws = [], []
    for nfft, L, R, P, per in shapes:
        stride = (2 + (R - 1) * 3 + L + 3) // 4 * 4
        echo = np.clip(np.rint(rng.standard_normal((P, stride, 2)) * 1000), -32768, 32767).astype(np.int16)
        code = np.where(rng.random((P, L) if per else (L,)) < 0.5, -1, 1).astype(np.int8)
        e, c = torch.from_numpy(echo).to(dev), torch.from_numpy(code).to(dev)
        o = torch.empty((R, nfft), device=dev)
        keep.append((echo, code, e, c, o))
        x = isr.IsrWindow()
        x.echo, x.tx_code, x.out = e.data_ptr(), c.data_ptr(), o.data_ptr()
        x.echo_stride, x.tx_stride, x.nfft, x.code_len = stride, L if per else 0, nfft, L
        x.n_ranges, x.range_start, x.range_step, x.n_ipp, x.order, x.reserved = R, 2, 3, P, -1, 0
        ws.append(x)
    torch.cuda.synchronize()
    h = isr.isr_batch_create(ws, 0, 0, torch.cuda.current_stream())
    for _ in range(2):
        isr.isr_batch_run(h)
        isr.isr_batch_wait(h)
    for (nfft, L, R, P, per), (echo, code, _, _, o) in zip(shapes, keep):
        sel = sorted({0, 1, R // 2, R - 1})
        ref = oracle.integrate(echo, code, nfft=nfft, n_ranges=R, range_start=2, range_step=3, code_len=L,
                               per_ipp_tx=bool(per), sel=sel)
        got = o.cpu().numpy().astype(np.float64)[sel]
        # few IPPs: a bin far below the mean shares the mean's rounding
        tol = RTOL * np.maximum(ref, 0.01 * ref.mean(axis=1, keepdims=True))
        assert (np.abs(got - ref) <= tol).all(), (nfft, L, R, P, per)
    isr.isr_batch_destroy(h)


def test_creation_leaves_the_outputs_alone():
    """Autotuning probes the windows at creation; only isr_batch_run writes `out`, of windows of one chunk
    (10 IPPs) and of several (600)."""
    rng = np.random.default_rng(23)
    dev = torch.device("cuda:0")
    keep, ws = [], []
    for nfft, R, P in [(2048, 40, 10), (16384, 30, 10), (4096, 9, 600)]:
        stride = (R + nfft + 3) // 4 * 4
        e = torch.from_numpy(rng.integers(-500, 500, (P, stride, 2)).astype(np.int16)).to(dev)
        c = torch.ones(nfft, dtype=torch.int8, device=dev)
        o = torch.full((R, nfft), -7.0, device=dev)
        keep.append((e, c, o))
        x = isr.IsrWindow()
        x.echo, x.tx_code, x.out = e.data_ptr(), c.data_ptr(), o.data_ptr()
        x.echo_stride, x.tx_stride, x.nfft, x.code_len = stride, 0, nfft, nfft
        x.n_ranges, x.range_start, x.range_step, x.n_ipp, x.order, x.reserved = R, 0, 1, P, -1, 0
        ws.append(x)
    torch.cuda.synchronize()
    for flags in (0, isr.ISR_BATCH_GRAPH | isr.ISR_BATCH_AUTOTUNE):
        h = isr.isr_batch_create(ws, flags, 0, torch.cuda.current_stream())
        torch.cuda.synchronize()
        assert all((o == -7.0).all() for _, _, o in keep), flags
        isr.isr_batch_run(h)
        isr.isr_batch_wait(h)
        assert all((o >= 0.0).all() for _, _, o in keep), flags
        isr.isr_batch_destroy(h)
        for _, _, o in keep:
            o.fill_(-7.0)
        torch.cuda.synchronize()


def test_outputs_that_share_memory_with_an_input():
    """A run reads every echo and code before it writes an output: a window integrated in place (its output
    over its own echo), one whose output lies over another's echo, one over its own code, and one that ends
    where an echo begins, all of one chunk, give the same sums as with outputs of their own."""
    dev = torch.device("cuda:0")
    stride, P, base = 70000, 6, 1 << 20
    shapes = [(2048, 100), (4096, 60), (2048, 77), (8192, 20)]

    def run(shared):
        rng = np.random.default_rng(31)
        pool = torch.from_numpy(rng.integers(-2**31, 2**31, base + 4 * stride * P).astype(np.int32)).to(dev)
        echoes = [pool[base + i * stride * P:][:stride * P] for i in range(4)]
        ws, outs = [], []
        for i, (nfft, R) in enumerate(shapes):
            n = R * nfft
            code = torch.from_numpy(np.where(rng.random(4 * n) < 0.5, -1, 1).astype(np.int8)).to(dev)
            o = torch.empty(n, device=dev)
            if shared:
                o = (echoes[0][:n], echoes[2][5:5 + n], code.view(torch.int32), pool[base - n:base])[i].view(torch.float32)
            x = isr.IsrWindow()
            x.echo, x.tx_code, x.out = echoes[i].data_ptr(), code.data_ptr(), o.data_ptr()
            x.echo_stride, x.tx_stride, x.nfft, x.code_len = stride, 0, nfft, nfft
            x.n_ranges, x.range_start, x.range_step, x.n_ipp, x.order, x.reserved = R, 1, 3, P, -1, 0
            ws.append(x)
            outs.append((o, code))
        torch.cuda.synchronize()
        h = isr.isr_batch_create(ws, 0, 0, torch.cuda.current_stream())
        isr.isr_batch_run(h)
        isr.isr_batch_wait(h)
        got = [o.cpu().numpy() for o, _ in outs]
        isr.isr_batch_destroy(h)
        return got

    for i, (a, b) in enumerate(zip(run(True), run(False))):
        assert np.isfinite(a).all() and np.array_equal(a, b), f"window {i}"
