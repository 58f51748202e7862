"""The learned estimator's kernels (through the C ABI) against the FP64 reference:
features, loss and every parameter's gradient (FP32 storage), the BF16 variant (tensor-core
convolutions) against the reference with BF16 storage rounding, the prediction, and a short
end-to-end training on spectra the integrator produces."""
import numpy as np
import pytest
import torch

from oracle import estimator as ref
from paper_2311_18737_gb300 import estimator as est_mod
from paper_2311_18737_gb300 import isr

pytestmark = pytest.mark.gpu

# Both BF16 engines: tcgen05 (convolutions in 256-position CTAs of two M = 128 tiles, the weight
# gradient in 256-position chunks) and mma.sync.
ENGINES = [isr.ISR_EST_BF16, isr.ISR_EST_BF16_MMASYNC]


def _setup(precision, B=4, L=256, seed=0):
    rng = np.random.default_rng(seed)
    theta = (ref.init_params(seed) + 0.05 * rng.standard_normal(ref.N_PARAMS)).astype(np.float32)
    x = rng.standard_normal((B, L)).astype(np.float32)
    f = rng.uniform(3, L - 3, B).astype(np.float32)
    y = np.array([1, 0, 1, 1][:B], dtype=np.float32)
    f[1] = -320.0                      # a gate without a line: its position is meaningless
    e = est_mod.Estimator(max_batch=8, precision=precision, nfft=512, band_lo=0, band_len=L)
    e.set_params(theta)
    dev = torch.device("cuda:0")
    return e, theta, x, f, y, [torch.from_numpy(a).to(dev) for a in (x, f, y)]


def test_gradients_match_fp64_reference_fp32_storage():
    e, theta, x, f, y, (xd, fd, yd) = _setup(isr.ISR_EST_FP32)
    loss, g = e.grad(xd, fd, yd)
    rl, rg = ref.loss_and_grad(theta.astype(np.float64), x, f, y)
    assert abs(loss - rl) <= 1e-5 * abs(rl)
    gd, rd = ref.unpack(g.astype(np.float64)), ref.unpack(rg)
    gmax = np.abs(rg).max()
    for name, _ in ref.SHAPES:
        # b5 shifts every location logit equally, so its exact gradient is 0: measure such
        # blocks against the overall gradient scale
        scale = max(np.abs(rd[name]).max(), 1e-3 * gmax)
        err = np.abs(gd[name] - rd[name]).max() / scale
        assert err <= 2e-4, f"{name}: max error {err:.2e} of the block's largest gradient"
    e.close()


def test_bf16_storage_close_to_reference():
    e, theta, x, f, y, (xd, fd, yd) = _setup(isr.ISR_EST_BF16, seed=1)
    loss, g = e.grad(xd, fd, yd)
    rl, rg = ref.loss_and_grad(theta.astype(np.float64), x, f, y)
    assert abs(loss - rl) <= 3e-2 * abs(rl)
    cos = float(g @ rg / (np.linalg.norm(g) * np.linalg.norm(rg)))
    assert cos > 0.98, cos
    e.close()


@pytest.mark.parametrize("precision", ENGINES)
def test_bf16_gradients_per_block_against_rounding_reference(precision):
    """Random inputs (not dyadic): the BF16 variant against the FP64 reference that rounds to
    BF16 exactly where the variant stores (input, conv weights, activations).  What is left is
    FP32 accumulation order and the hi + lo split of the gradient entering the backward passes
    (~16 significant bits), which can move an activation across a BF16 rounding boundary now and
    then; so every parameter block's gradient must agree in norm to 2 % and in direction to
    cosine 0.999, and the loss to 1e-3."""
    e, theta, x, f, y, (xd, fd, yd) = _setup(precision, seed=3)
    loss, g = e.grad(xd, fd, yd)
    rl, rg = ref.loss_and_grad(theta.astype(np.float64), x, f, y, store=ref.round_bf16)
    assert abs(loss - rl) <= 1e-3 * abs(rl), (loss, rl)
    gd, rd = ref.unpack(g.astype(np.float64)), ref.unpack(rg)
    gmax = np.abs(rg).max()
    for name, _ in ref.SHAPES:
        a, b = gd[name].ravel(), rd[name].ravel()
        nb = np.linalg.norm(b)
        if nb <= 1e-3 * gmax:
            # b5: exactly zero in exact arithmetic; bound it by the overall gradient scale
            assert np.abs(a).max() <= 1e-3 * gmax, name
            continue
        rel = np.linalg.norm(a - b) / nb
        cos = float(a @ b / (np.linalg.norm(a) * nb))
        assert rel <= 2e-2 and cos >= 0.999, f"{name}: relative error {rel:.2e}, cosine {cos:.6f}"
    e.close()


def _dyadic_case(B=4, L=600, seed=7, precision=isr.ISR_EST_BF16):
    """Conv weights and biases in multiples of 1/8 within [-1/4, 1/4] and inputs in multiples
    of 1/4: every product and FP32 partial sum of the convolutions is exact, so the BF16
    variant's activations are the BF16 roundings of exact values on both sides.  L = 600 spans
    two full 256-position tiles of the tensor-core convolution and a ragged third."""
    rng = np.random.default_rng(seed)
    d = ref.unpack(ref.init_params(seed))
    for l in range(1, 5):
        d[f"W{l}"] = rng.integers(-2, 3, d[f"W{l}"].shape) / 8.0
        d[f"b{l}"] = rng.integers(-2, 3, d[f"b{l}"].shape) / 8.0
    theta = ref.pack(d).astype(np.float32)
    x = (rng.integers(-8, 9, (B, L)) / 4.0).astype(np.float32)
    f = rng.uniform(3, L - 3, B).astype(np.float32)
    y = np.resize(np.array([1, 0, 1, 1], dtype=np.float32), B)
    e = est_mod.Estimator(max_batch=max(8, B), precision=precision, nfft=2048, band_lo=0, band_len=L)
    e.set_params(theta)
    dev = torch.device("cuda:0")
    return e, theta, x, f, y, [torch.from_numpy(a).to(dev) for a in (x, f, y)]


# Lengths: 600 spans full tiles and a ragged rest; 37 is odd (unpaired stores), one partial
# tile; 1100 gives three tcgen05 CTAs with a length that is not a multiple of 8 (the
# word-by-word staging path).
@pytest.mark.parametrize("precision", ENGINES)
@pytest.mark.parametrize("L", [600, 37, 1100])
def test_bf16_tensor_core_forward_matches_bf16_storage_reference(L, precision):
    e, theta, x, f, y, (xd, fd, yd) = _dyadic_case(L=L, precision=precision)
    pos, pres = e.predict(xd)
    rpos, rpres = ref.predict(theta.astype(np.float64), x, store=ref.round_bf16)
    assert np.abs(pos.cpu().numpy() - rpos).max() <= 1e-3
    assert np.abs(pres.cpu().numpy() - rpres).max() <= 1e-5
    e.close()


@pytest.mark.parametrize("precision", ENGINES)
@pytest.mark.parametrize("L", [600, 37, 1100])
def test_bf16_tensor_core_gradients_match_bf16_storage_reference(L, precision):
    """The backward-data convolution splits the FP32 gradient into two BF16 parts (~16
    significant bits): every parameter block within 1e-3 of its largest gradient."""
    e, theta, x, f, y, (xd, fd, yd) = _dyadic_case(L=L, seed=8, precision=precision)
    loss, g = e.grad(xd, fd, yd)
    rl, rg = ref.loss_and_grad(theta.astype(np.float64), x, f, y, store=ref.round_bf16)
    assert abs(loss - rl) <= 1e-4 * abs(rl)
    gd, rd = ref.unpack(g.astype(np.float64)), ref.unpack(rg)
    gmax = np.abs(rg).max()
    for name, _ in ref.SHAPES:
        scale = max(np.abs(rd[name]).max(), 1e-3 * gmax)
        err = np.abs(gd[name] - rd[name]).max() / scale
        assert err <= 1e-3, f"{name}: max error {err:.2e} of the block's largest gradient"
    e.close()


def test_prediction_matches_reference():
    e, theta, x, f, y, (xd, fd, yd) = _setup(isr.ISR_EST_FP32, seed=2)
    pos, pres = e.predict(xd)
    rpos, rpres = ref.predict(theta.astype(np.float64), x)
    assert np.abs(pos.cpu().numpy() - rpos).max() <= 1e-3
    assert np.abs(pres.cpu().numpy() - rpres).max() <= 1e-5
    e.close()


def test_features_match_reference():
    rng = np.random.default_rng(5)
    P = rng.gamma(30.0, 2.0, size=(6, 512)).astype(np.float32)
    e = est_mod.Estimator(max_batch=8, precision=isr.ISR_EST_FP32, nfft=512, band_lo=40, band_len=300)
    x = e.features(torch.from_numpy(P).cuda()).cpu().numpy()
    assert np.abs(x - ref.features(P, 40, 300)).max() <= 1e-5
    e.close()


@pytest.mark.parametrize("L", [16, 37, 511, 513, 5120, 5121, 12000])
def test_features_band_lengths_and_floors(L):
    """Bands within and beyond the bins a thread keeps in registers, with bins at, below and far above
    the 1e-30 floor.  The logarithms carry about 2^-42, so a feature is one FP32 rounding (2^-24
    relative) of the exact one plus 2^-42 / std; 1.2e-7 |x| + 1e-9 covers both at std >= 0.01."""
    rng = np.random.default_rng(L)
    P = rng.gamma(30.0, 2.0, size=(4, L + 3)).astype(np.float32)
    P[1] *= np.exp(rng.uniform(-60, 60, L + 3)).astype(np.float32)
    P[2, 1:6] = [0.0, -4.0, 1e-30, 1e-31, 3e38]
    P[3, 4] = np.nan
    e = est_mod.Estimator(max_batch=4, precision=isr.ISR_EST_FP32, nfft=L + 3, band_lo=1, band_len=L)
    x = e.features(torch.from_numpy(P).cuda()).cpu().numpy()
    e.close()
    P[3, 4] = 0.0                       # NaN counts as the floor
    want = ref.features(P, 1, L)
    assert (np.abs(x - want) <= 1.2e-7 * np.abs(want) + 1e-9).all()


@pytest.mark.parametrize("B,L", [(1, 16), (2, 129), (5, 1153)])
def test_fp32_gradients_over_spans_and_rows(B, L):
    """FP32 storage where the weight gradient splits its rows differently: one short tile, and one position
    into a second tile or span; the bound of the other FP32 gradient test (2e-4 of each block's largest
    gradient)."""
    rng = np.random.default_rng(B + L)
    theta = (ref.init_params(3) + 0.05 * rng.standard_normal(ref.N_PARAMS)).astype(np.float32)
    x = rng.standard_normal((B, L)).astype(np.float32)
    f = rng.uniform(3, L - 3, B).astype(np.float32)
    y = np.resize(np.array([1, 0, 1, 1], dtype=np.float32), B)
    e = est_mod.Estimator(max_batch=B, precision=isr.ISR_EST_FP32, nfft=L, band_lo=0, band_len=L)
    e.set_params(theta)
    loss, g = e.grad(*[torch.from_numpy(a).cuda() for a in (x, f, y)])
    e.close()
    rl, rg = ref.loss_and_grad(theta.astype(np.float64), x, f, y)
    assert abs(loss - rl) <= 1e-5 * abs(rl)
    gd, rd = ref.unpack(g.astype(np.float64)), ref.unpack(rg)
    gmax = np.abs(rg).max()
    for name, _ in ref.SHAPES:
        scale = max(np.abs(rd[name]).max(), 1e-3 * gmax)
        err = np.abs(gd[name] - rd[name]).max() / scale
        assert err <= 2e-4, f"{name}: max error {err:.2e} of the block's largest gradient"


def test_fp32_batch_gradient_is_the_mean_over_its_rows():
    """300 rows at once (spans of 128 positions, several waves) against the same rows one at a time (one
    span per tile): the forward pass and its masks are the same per row, so the batch gradient is the
    mean of the rows' up to FP32 summation, 300 x 130 terms in any order: 1e-4 of each block's largest."""
    B, L = 300, 130
    rng = np.random.default_rng(B + L)
    theta = (ref.init_params(3) + 0.05 * rng.standard_normal(ref.N_PARAMS)).astype(np.float32)
    arrays = [torch.from_numpy(a).cuda() for a in (rng.standard_normal((B, L)).astype(np.float32),
                                                   rng.uniform(3, L - 3, B).astype(np.float32),
                                                   np.resize(np.array([1, 0, 1, 1], dtype=np.float32), B))]
    e = est_mod.Estimator(max_batch=B, precision=isr.ISR_EST_FP32, nfft=L, band_lo=0, band_len=L)
    e.set_params(theta)
    _, g = e.grad(*arrays)
    rows = np.zeros(ref.N_PARAMS)
    for r in range(B):
        rows += e.grad(*[a[r:r + 1].contiguous() for a in arrays])[1].astype(np.float64)
    e.close()
    gd, rd = ref.unpack(g.astype(np.float64)), ref.unpack(rows / B)
    gmax = np.abs(rows / B).max()
    for name, _ in ref.SHAPES:
        scale = max(np.abs(rd[name]).max(), 1e-3 * gmax)
        assert np.abs(gd[name] - rd[name]).max() <= 1e-4 * scale, name


@pytest.mark.slow
def test_training_gains_over_peak_fit():
    """Short training on integrator-made spectra (reduced from the full 200k-spectrum run):
    the network must beat the peak fit's presence decision and agree with the peak fit
    within one bin on strong lines."""
    e = est_mod.Estimator(max_batch=128, precision=isr.ISR_EST_BF16)
    e.set_params(est_mod.init_params(0))
    tr = est_mod.make_dataset(16, seed=11, est=e)
    te = est_mod.make_dataset(4, seed=12, est=e)
    hist = est_mod.train(e, tr, steps=600, batch=128, lr=2e-3, log_every=100)
    assert hist[-1][1] < 0.7 * hist[0][1], hist
    res = est_mod.evaluate(e, te, est_mod.presence_threshold(tr))
    print(res)
    assert res["presence_accuracy"]["network"] >= res["presence_accuracy"]["peak_fit"]
    assert res["agreement_with_peak_fit_above_-10dB"] >= 0.9
    e.close()


@pytest.mark.parametrize("precision", ENGINES)
def test_bf16_gradients_many_rows_several_chunks_per_cta(precision):
    """64 rows x 1100 positions: the tcgen05 weight gradient then spreads 320 chunks of 256
    positions over one CTA per SM (two or three per CTA through its double-buffered staging, most
    ranges crossing from one row into the next), and the persistent tcgen05 convolutions take
    several 256-position tiles per CTA; exact (dyadic) inputs, the same bound as the other BF16
    gradient tests."""
    e, theta, x, f, y, (xd, fd, yd) = _dyadic_case(B=64, L=1100, seed=9, precision=precision)
    loss, g = e.grad(xd, fd, yd)
    rl, rg = ref.loss_and_grad(theta.astype(np.float64), x, f, y, store=ref.round_bf16)
    assert abs(loss - rl) <= 1e-4 * abs(rl)
    gd, rd = ref.unpack(g.astype(np.float64)), ref.unpack(rg)
    gmax = np.abs(rg).max()
    for name, _ in ref.SHAPES:
        scale = max(np.abs(rd[name]).max(), 1e-3 * gmax)
        err = np.abs(gd[name] - rd[name]).max() / scale
        assert err <= 1e-3, f"{name}: max error {err:.2e} of the block's largest gradient"
    e.close()


@pytest.mark.parametrize("B,L", [(1, 16), (3, 487), (2, 488), (2, 489), (3, 976), (2, 977), (320, 1000)])
def test_bf16_fused_gradients_at_tile_edges(B, L):
    """Forward and backward passes of the tcgen05 engine work in tiles of 488 positions, two to
    a CTA: one short, one full and one position more, rows that are not whole groups of four
    positions, and more tiles than CTAs take at a time.  The bound of the other exact-input
    gradient tests."""
    e, theta, x, f, y, (xd, fd, yd) = _dyadic_case(B=B, L=L, seed=11)
    loss, g = e.grad(xd, fd, yd)
    rl, rg = ref.loss_and_grad(theta.astype(np.float64), x, f, y, store=ref.round_bf16)
    assert abs(loss - rl) <= 1e-4 * abs(rl)
    gd, rd = ref.unpack(g.astype(np.float64)), ref.unpack(rg)
    gmax = np.abs(rg).max()
    for name, _ in ref.SHAPES:
        scale = max(np.abs(rd[name]).max(), 1e-3 * gmax)
        err = np.abs(gd[name] - rd[name]).max() / scale
        assert err <= 1e-3, f"{name}: max error {err:.2e} of the block's largest gradient"
    e.close()


@pytest.mark.parametrize("B,L", [(37, 1101), (152, 128), (19, 1000)])
def test_fp32_batches_as_their_rows(B, L):
    """FP32 convolutions take 8, 12 or 16 positions per warp, by the batch (here 12, 16 and 16 on 152 SMs, 8
    for a single row), with ragged last tiles: predictions bit for bit as row by row (the sums' order
    is the same), the batch gradient the mean of the rows' up to FP32 summation (1e-4 of each block's
    largest)."""
    rng = np.random.default_rng(B + L)
    theta = (ref.init_params(3) + 0.05 * rng.standard_normal(ref.N_PARAMS)).astype(np.float32)
    arrays = [torch.from_numpy(a).cuda() for a in (rng.standard_normal((B, L)).astype(np.float32),
                                                   rng.uniform(3, L - 3, B).astype(np.float32),
                                                   np.resize(np.array([1, 0, 1, 1], dtype=np.float32), B))]
    e = est_mod.Estimator(max_batch=B, precision=isr.ISR_EST_FP32, nfft=L, band_lo=0, band_len=L)
    e.set_params(theta)
    whole = e.predict(arrays[0])
    _, g = e.grad(*arrays)
    rows = np.zeros(ref.N_PARAMS)
    for r in range(B):
        row = [a[r:r + 1].contiguous() for a in arrays]
        assert all(torch.equal(a[r:r + 1], b) for a, b in zip(whole, e.predict(row[0])))
        rows += e.grad(*row)[1].astype(np.float64)
    e.close()
    gd, rd = ref.unpack(g.astype(np.float64)), ref.unpack(rows / B)
    gmax = np.abs(rows / B).max()
    for name, _ in ref.SHAPES:
        scale = max(np.abs(rd[name]).max(), 1e-3 * gmax)
        assert np.abs(gd[name] - rd[name]).max() <= 1e-4 * scale, name


@pytest.mark.parametrize("B,L", [(32, 1101), (256, 300)])
def test_fp32_weight_gradients_round_no_worse_than_their_rows(B, L):
    """The weight gradients of layers 2 to 4 of a batch against the FP64 mean of its rows' (B a power of
    two, so a row's terms are the same bit for bit up to that factor; rows of up to 12 spans round little).
    n partial sums added one after the other in FP32 leave a relative RMS error of about
    sqrt(n / 3) 2^-24 / sqrt(3): 3.4e-7 and 4.4e-7 for the 288 and 512 or more spans here.  In 16 copies
    that are added in more bits it is a quarter of that, the spans' own sums and the rows' add about
    5e-8: 1.5e-7 lies between."""
    rng = np.random.default_rng(7)
    spec = 1 + rng.standard_normal((B, L)) / 16
    at = rng.uniform(4, L - 5, B)
    snr = np.where(rng.random(B) < 0.85, 10 ** rng.uniform(-3, 0, B), 0)
    spec += (snr * L / np.pi)[:, None] / (1 + (np.arange(L)[None] - at[:, None]) ** 2)
    x = ref.features(spec.astype(np.float32), 0, L).astype(np.float32)
    arrays = [torch.from_numpy(a.astype(np.float32)).cuda() for a in (x, at, snr > 0)]
    e = est_mod.Estimator(max_batch=B, precision=isr.ISR_EST_FP32, nfft=L, band_lo=0, band_len=L)
    e.set_params(ref.init_params(3).astype(np.float32))
    _, g = e.grad(*arrays)
    rows = np.zeros(ref.N_PARAMS)
    for r in range(B):
        rows += e.grad(*[a[r:r + 1].contiguous() for a in arrays])[1].astype(np.float64)
    e.close()
    gd, rd = ref.unpack(g.astype(np.float64)), ref.unpack(rows / B)
    for name in ("W2", "W3", "W4"):
        err = np.linalg.norm(gd[name] - rd[name]) / np.linalg.norm(rd[name])
        assert err <= 1.5e-7, f"{name}: relative error {err:.2e}"


@pytest.mark.parametrize("L", [4608, 4601])
def test_bf16_gradients_where_memory_holds_two_gradient_buffers(L):
    """With device memory for the activations and two full gradient buffers, but not four, a tcgen05
    estimator is still created, and its gradient, taken in two halves of the rows (the second ragged), is
    that of one with memory for all, at the bound of the gradient tests against the reference (1e-3 of
    each block's largest)."""
    B, n = 256, 251
    rng = np.random.default_rng(13)
    arrays = [torch.from_numpy(a).cuda() for a in (rng.standard_normal((n, L)).astype(np.float32),
                                                   rng.uniform(3, L - 3, n).astype(np.float32),
                                                   (rng.random(n) < 0.8).astype(np.float32))]
    theta = ref.init_params(3).astype(np.float32)

    def grad():
        e = est_mod.Estimator(max_batch=B, precision=isr.ISR_EST_BF16, nfft=L, band_lo=0, band_len=L)
        e.set_params(theta)
        out = e.grad(*arrays)
        e.close()
        return out

    loss, g = grad()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    row = 2 * L * (1 + 4 * 32) + 4 * L * 4 + 12 * 32 * (L // 488 + 1)      # activations, masks, logits, statistics
    one = 4 * 32 * L * B                                                    # a full gradient buffer
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (row * B + 2 * one + one), dtype=torch.uint8, device="cuda")
    try:
        loss2, g2 = grad()
    finally:
        del hog
        torch.cuda.empty_cache()
    assert abs(loss2 - loss) <= 1e-6 * abs(loss)
    gd, rd = ref.unpack(g2.astype(np.float64)), ref.unpack(g.astype(np.float64))
    gmax = np.abs(g).max()
    for name, _ in ref.SHAPES:
        scale = max(np.abs(rd[name]).max(), 1e-3 * gmax)
        assert np.abs(gd[name] - rd[name]).max() <= 1e-3 * scale, name


@pytest.mark.parametrize("which", [0, 1, 2])
def test_bounded_waits_for_products_are_reported(which):
    """Products left out in the forward pass, the backward pass or the weight gradient: the wait
    for them runs out and the call, or the next one, reports it instead of returning incomplete numbers; a
    train step leaves the parameters alone; afterwards everything works as before."""
    e, theta, x, f, y, (xd, fd, yd) = _dyadic_case(L=600, seed=12)
    want_pos, want_pres = (t.clone() for t in e.predict(xd))
    want_loss, want = e.grad(xd, fd, yd)

    def times_out(call):
        with pytest.raises(isr.IsrError) as ei:
            call()
        assert ei.value.status == isr.ISR_ERR_TIMEOUT

    isr.isr_est_test_drop_products(e.h, which, 20000)
    times_out(lambda: e.grad(xd, fd, yd))
    times_out(lambda: e.train_step(xd, fd, yd, 1e-2, want_loss=True))
    e.train_step(xd, fd, yd, 1e-2)
    times_out(e.get_params)
    if which == 0:
        e.predict(xd)
        torch.cuda.synchronize()
        times_out(lambda: e.predict(xd))
    isr.isr_est_test_drop_products(e.h, -1, 0)
    assert np.array_equal(e.get_params(), theta)
    pos, pres = e.predict(xd)
    assert torch.equal(pos, want_pos) and torch.equal(pres, want_pres)
    loss, g = e.grad(xd, fd, yd)
    assert abs(loss - want_loss) <= 1e-6 * abs(want_loss)
    assert np.linalg.norm(g - want) <= 1e-5 * np.linalg.norm(want)
    with pytest.raises(isr.IsrError) as ei:
        isr.isr_est_test_drop_products(e.h, 3, 1)
    assert ei.value.status == isr.ISR_ERR_INVALID_ARG
    e.close()


@pytest.mark.parametrize("L,at", [(16, 0), (700, 699), (5121, 5120), (6000, 17)])
def test_features_of_a_band_with_an_infinite_bin(L, at):
    """The mean is infinite and the variance, infinity less infinity, counts as 0: every finite bin gives
    minus infinity and the infinite one NaN, and other gates of the launch are not touched by it."""
    rng = np.random.default_rng(L)
    P = rng.gamma(30.0, 2.0, size=(3, L)).astype(np.float32)
    P[1, at] = np.inf
    e = est_mod.Estimator(max_batch=4, precision=isr.ISR_EST_FP32, nfft=L, band_lo=0, band_len=L)
    x = e.features(torch.from_numpy(P).cuda()).cpu().numpy()
    e.close()
    assert np.isnan(x[1, at]) and np.isneginf(np.delete(x[1], at)).all()
    assert np.abs(x[[0, 2]] - ref.features(P[[0, 2]], 0, L)).max() <= 1e-5
