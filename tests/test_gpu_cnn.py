"""rad_cnn_step against the convolutional oracle: the 32x32x3 / 16-32-64 / 1024-128-10 net of the
CNN configuration (bf16, batch 128) and smaller nets in both types and both sampling variants."""
import numpy as np
import pytest
import torch

from oracle import cnn as orc
from workloads import cnn_inputs

from gpu_util import TOL, rel_err, to_dev

pytestmark = pytest.mark.gpu

CASES = [
    # B, hw, cin, channels, fc, dtype
    (5, 8, 3, (8, 16), (24, 5), "f32"),
    (70, 16, 3, (8, 8), (32, 10), "bf16"),          # two row slabs in the stores
    (128, 32, 3, (16, 32, 64), (128, 10), "bf16"),  # the CNN configuration
    (37, 16, 16, (32, 24, 8), (16, 4), "bf16"),     # ragged pixel tiles; tensor-core kernels from the first convolution on
]


@pytest.fixture
def conv_kernel(request):
    """Forces the CUDA-core or the tensor-core convolution kernels for the test, then restores the automatic choice."""
    import paper_2007_10412_b200 as rad
    prev = rad.rad_set_conv_kernel(request.param)
    yield request.param
    rad.rad_set_conv_kernel(prev)


@pytest.mark.parametrize("conv_kernel", ["simt", "tensor"], indirect=True)
@pytest.mark.parametrize("B,hw,cin,channels,fc,dtype", CASES)
@pytest.mark.parametrize("variant", ["different", "same"])
@pytest.mark.parametrize("p", [0.1, 1.0])
def test_cnn_step_matches_oracle(B, hw, cin, channels, fc, dtype, variant, p, conv_kernel):
    import paper_2007_10412_b200 as rad
    X, y, cW, cb, fW, fb = cnn_inputs(B, hw, cin, channels, fc, dtype, seed=B + hw, bias_zero=False)
    ref = orc.cnn_step(X, y, cW, cb, fW, fb, dtype=dtype, variant=variant, p=p, seed=3, step=2)
    ctx = rad.CNNStep(B, hw, cin, channels, fc, dtype, variant, p)
    ctx(to_dev(X, dtype), torch.from_numpy(y).cuda(), [to_dev(w, dtype) for w in cW], [to_dev(b, "f32") for b in cb],
        [to_dev(w, dtype) for w in fW], [to_dev(b, "f32") for b in fb], seed=3, step=2)
    torch.cuda.synchronize()
    assert ctx.dev_status.item() == 0
    tol = TOL[dtype]
    assert abs(ctx.loss.item() - ref.loss) <= (1e-5 if dtype == "f32" else 2e-3) * abs(ref.loss)
    nnz = ctx.nnz.cpu().numpy().reshape(-1, 2)
    for l, want in enumerate(ref.nnz):
        assert nnz[l, 0] == (want if variant == "different" else want // B)
    got_all = ctx.dconv_W + ctx.dconv_b + ctx.dfc_W + ctx.dfc_b
    want_all = ref.dW_conv + ref.db_conv + ref.dW_fc + ref.db_fc
    # Frobenius error within the stated tolerance.  The largest single deviation gets twice that in bf16: one ReLU
    # decision of the 16384 outputs of the first linear layer that falls the other way (its pre-activation is a
    # last-bit rounding away from zero, and a different but equally valid summation order in a convolution
    # before it is enough) moves single entries of a 128-term sum by a percent or two while the tensor as a
    # whole moves by a fraction of a percent; it happens with either set of convolution kernels.
    for i, (got, want) in enumerate(zip(got_all, want_all)):
        fro, mx = rel_err(got.double().cpu().numpy(), want)
        assert fro <= tol and mx <= (tol if dtype == "f32" else 2 * tol), (i, fro, mx)


def test_cnn_stored_bytes():
    import paper_2007_10412_b200 as rad
    ctx = rad.CNNStep(128, 32, 3, (16, 32, 64), (128, 10), "bf16", "different", 0.1)
    s = ctx.stats
    per_sample_inputs = 3072 + 4096 + 2048 + 1024 + 128
    assert s.full_backprop_bytes == 128 * per_sample_inputs * 2 + 128 * 10 * 4
    assert s.relu_bytes == 128 * (32 * 32 * 16 + 16 * 16 * 32 + 8 * 8 * 64) // 8 + 128 * 4 * 4
    assert s.value_bytes < 0.16 * 128 * per_sample_inputs * 2


@pytest.mark.parametrize("B,hw,cin,channels,fc,dtype", [(1, 4, 1, (8,), (3,), "f32"), (800, 4, 2, (16,), (5,), "f32"),
                                                        (66, 16, 4, (64,), (6,), "bf16"), (65, 12, 3, (24,), (4,), "f32"),
                                                        (9, 16, 5, (8,), (3,), "f32")])
@pytest.mark.parametrize("variant", ["different", "same"])
def test_first_convolution_backward_over_channels_and_rows(B, hw, cin, channels, fc, dtype, variant):
    """The one-launch backward of the first convolution at one to four input channels, at channel counts that leave one
    to eight parts of the list of kept entries, with more rows than CTAs, and beside it the route of five channels."""
    import paper_2007_10412_b200 as rad
    X, y, cW, cb, fW, fb = cnn_inputs(B, hw, cin, channels, fc, dtype, seed=B + hw, bias_zero=False)
    ref = orc.cnn_step(X, y, cW, cb, fW, fb, dtype=dtype, variant=variant, p=0.3, seed=4, step=1)
    ctx = rad.CNNStep(B, hw, cin, channels, fc, dtype, variant, 0.3)
    ctx(to_dev(X, dtype), torch.from_numpy(y).cuda(), [to_dev(w, dtype) for w in cW], [to_dev(b, "f32") for b in cb],
        [to_dev(w, dtype) for w in fW], [to_dev(b, "f32") for b in fb], seed=4, step=1)
    torch.cuda.synchronize()
    assert ctx.dev_status.item() == 0
    for got, want in zip(ctx.dconv_W + ctx.dconv_b, ref.dW_conv + ref.db_conv):
        fro, mx = rel_err(got.double().cpu().numpy(), want)
        assert fro <= TOL[dtype] and mx <= TOL[dtype] * (1 if dtype == "f32" else 2)


@pytest.mark.parametrize("cin", [3, 5])
def test_padding_is_not_multiplied_with_an_infinite_filter(cin):
    """A tap outside the image contributes nothing, whatever the filter holds there: with -inf in a corner tap of one output
    channel and a positive image, the outputs whose tap lies inside are -inf before the ReLU (0 after it) and those on
    the upper and left border stay what the other taps make of them: the net of a filter with -1e30 in that place."""
    import paper_2007_10412_b200 as rad
    B, hw, channels, fc = 3, 4, (8,), (3,)
    X, y, cW, cb, fW, fb = cnn_inputs(B, hw, cin, channels, fc, "f32", seed=21, bias_zero=False)
    X = np.abs(X) + np.float32(0.1)
    cW = [np.abs(cW[0])]                       # so that the border outputs are positive
    cW[0][0, 0, 0, 2] = -1e30
    ref = orc.cnn_step(X, y, cW, cb, fW, fb, dtype="f32", variant="different", p=1.0, seed=3, step=2)
    cW[0][0, 0, 0, 2] = -np.inf
    ctx = rad.CNNStep(B, hw, cin, channels, fc, "f32", "different", 1.0)
    ctx(to_dev(X, "f32"), torch.from_numpy(y).cuda(), [to_dev(w, "f32") for w in cW], [to_dev(b, "f32") for b in cb],
        [to_dev(w, "f32") for w in fW], [to_dev(b, "f32") for b in fb], seed=3, step=2)
    torch.cuda.synchronize()
    assert abs(ctx.loss.item() - ref.loss) <= 1e-5 * abs(ref.loss)
    for got, want in zip(ctx.dconv_W + ctx.dconv_b + ctx.dfc_W + ctx.dfc_b, ref.dW_conv + ref.db_conv + ref.dW_fc + ref.db_fc):
        fro, mx = rel_err(got.double().cpu().numpy(), want)
        assert fro <= TOL["f32"] and mx <= TOL["f32"]


@pytest.mark.parametrize("cin", [1, 3])
@pytest.mark.parametrize("where", ["gradient", "gradient of a unit that was not active", "input"])
def test_first_convolution_backward_keeps_infinities_where_they_belong(cin, where):
    """Backward of the first convolution with one infinity: in the gradient of a pooled output (it reaches the filter entries
    whose kept inputs its four pixels see, and the bias gradient of its channel), in the gradient of an output none of
    whose pixels passed the ReLU (it reaches nothing), in a kept input at the corner of the image (it reaches its own
    channel's taps that lie inside).  Reference: the kept entries one by one, taps outside the image left out."""
    import paper_2007_10412_b200 as rad
    from oracle import rad as orad
    hw, co, p, seed, step, C = 4, 8, (1.0 if where == "input" else 0.3), 6, 2, 2
    X, _, cW, cb, fW, fb = cnn_inputs(1, hw, cin, (co,), (C,), "f32", seed=5, bias_zero=False)
    y = np.array([1], np.int32)
    W = cW[0].copy()
    if where == "input":
        X[0, 0, 0, 0] = np.inf
        W[:, :, 0, :] = -np.abs(W[:, :, 0, :])              # its outputs are -inf before the ReLU, 0 after it
    X64, W64 = X.astype(np.float64), W.astype(np.float64)
    Z = np.zeros((hw, hw, co)) + cb[0]
    taps = [(yy, xx, ky, kx) for yy in range(hw) for xx in range(hw) for ky in range(3) for kx in range(3)
            if 0 <= yy + ky - 1 < hw and 0 <= xx + kx - 1 < hw]       # output pixel and tap; the input lies inside
    for yy, xx, ky, kx in taps:
        Z[yy, xx] += X64[0, yy + ky - 1, xx + kx - 1] @ W64[ky, kx]
    on = Z > 0
    active = on.reshape(hw // 2, 2, hw // 2, 2, co).sum(axis=(1, 3)).reshape(-1)              # pixels of a window that passed
    P = np.where(on, Z, 0.0).reshape(hw // 2, 2, hw // 2, 2, co).mean(axis=(1, 3)).reshape(-1)
    # logits one of which is far above the other: softmax - onehot is exactly (1, -1), so dP = F[:, 0] - F[:, 1]
    F = fW[0] * np.float32(1e-3)
    F[int(np.argmax(P))] = (1e6, -1e6)
    hot = int(np.argmin(np.where(active > 0, P, np.inf))) if where == "gradient" else int(np.argmin(active))
    assert (active[hot] > 0) == (where == "gradient") and P[hot] < 0.9
    if where != "input":
        F[hot] = (1.8e38, -1.8e38)
    with np.errstate(all="ignore"):
        dP = (F[:, 0].astype(np.float32) - F[:, 1].astype(np.float32)).astype(np.float32)
        assert np.isinf(dP[hot]) == (where != "input")
        dZ = np.where(on, np.repeat(np.repeat(0.25 * dP.astype(np.float64).reshape(hw // 2, hw // 2, co), 2, 0), 2, 1), 0.0)
        keep = orad.keep_mask("different", 1, hw * hw * cin, p, seed, 0, step).reshape(hw, hw, cin)
        A = X64[0] * float(orad.scale_factor(p))
        want = np.zeros((3, 3, cin, co))
        for yy, xx, ky, kx in taps:
            for ci in range(cin):
                if keep[yy + ky - 1, xx + kx - 1, ci]:
                    want[ky, kx, ci] += A[yy + ky - 1, xx + kx - 1, ci] * dZ[yy, xx]
        want_b = dZ.sum(axis=(0, 1))
    ctx = rad.CNNStep(1, hw, cin, (co,), (C,), "f32", "different", p)
    ctx(to_dev(X, "f32"), torch.from_numpy(y).cuda(), [to_dev(W, "f32")], [to_dev(cb[0], "f32")], [to_dev(F, "f32")],
        [torch.zeros(C, device="cuda")], seed=seed, step=step)
    torch.cuda.synchronize()
    for got, ref in ((ctx.dconv_W[0], want), (ctx.dconv_b[0], want_b)):
        got = got.double().cpu().numpy()
        assert (np.isfinite(got) == np.isfinite(ref)).all()
        ok = np.isfinite(ref)
        assert ok.any() and (np.abs(got[ok] - ref[ok]) <= 1e-5 * np.abs(ref[ok]).max()).all()
