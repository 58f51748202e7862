"""Plans made after the device was reset: what the library keeps in a CUDA context beside its handles (the
twiddle tables, the pinned page of status words) goes with the context and is made anew.  In a process of
its own, without torch; every plan is destroyed before the reset."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import ctypes
import numpy as np
from paper_2311_18737_gb300 import isr

cuda = ctypes.CDLL("libcuda.so.1")

def on_device(a):
    p = ctypes.c_uint64()
    assert cuda.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(a.nbytes)) == 0
    assert cuda.cuMemcpyHtoD_v2(p, a.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(a.nbytes)) == 0
    return p

def spectra(nfft, allocation_free):
    R, P, stride = 5, 3, nfft + 8
    pad = np.empty(P * stride * 2 + 8, dtype=np.int16)
    at = (-pad.ctypes.data % 16) // 2
    e = pad[at:at + P * stride * 2].reshape(P, stride, 2)
    e[:] = np.random.default_rng(nfft).integers(-900, 900, e.shape)
    code = np.where(np.random.default_rng(nfft + 1).random(nfft) < 0.5, -1, 1).astype(np.int8)
    out = np.zeros((R, nfft), dtype=np.float32)
    if allocation_free:
        ctx = ctypes.c_void_p()
        assert cuda.cuDevicePrimaryCtxRetain(ctypes.byref(ctx), 0) == 0 and cuda.cuCtxSetCurrent(ctx) == 0
        d = isr.IsrPlanDesc()
        d.nfft, d.code_len, d.n_ranges, d.range_start, d.range_step = nfft, nfft, R, 0, 2
        d.tx_type, d.echo_stride, d.device = isr.ISR_TX_PM1, stride, 0
        bufs = [on_device(a) for a in (e, code, out)]
        isr.isr_integrate_static(d, bufs[0].value, bufs[1].value, P, bufs[2].value)
        assert cuda.cuMemcpyDtoH_v2(out.ctypes.data_as(ctypes.c_void_p), bufs[2], ctypes.c_size_t(out.nbytes)) == 0
        for b in bufs:
            assert cuda.cuMemFree_v2(b) == 0
        assert cuda.cuDevicePrimaryCtxRelease_v2(0) == 0
    else:
        plan = isr.Plan(nfft=nfft, n_ranges=R, echo_stride=stride, range_step=2, device=0)
        plan.integrate(e, code, P)
        plan.spectra(out)
        plan.close()
    x = np.stack([e[:, 2 * r:2 * r + nfft].astype(np.float64) for r in range(R)])
    z = np.fft.fft((x[..., 0] + 1j * x[..., 1]) * code, axis=2)
    ref = (np.abs(z) ** 2).sum(1)
    assert (np.abs(out - ref) <= 1e-5 * np.maximum(ref, 0.01 * ref.mean(axis=1, keepdims=True))).all(), nfft
    return out

calls = [(1024, False), (512, False), (1024, True), (16384, True), (16384, False)]
first = [spectra(*c) for c in calls]
for order in (1, -1):
    assert cuda.cuDevicePrimaryCtxReset_v2(0) == 0
    for c, want in list(zip(calls, first))[::order]:
        assert np.array_equal(spectra(*c), want), (order, c)
    spectra(4096, order == 1)
print("same spectra")
"""


def test_plans_after_a_device_reset():
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same spectra" in r.stdout, r.stdout + r.stderr
