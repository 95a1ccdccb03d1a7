"""Per-layer backward calls against the oracle: dW from the store, exact dX / db, forward, loss."""
import numpy as np
import pytest
import torch

from oracle import rad as orc
from workloads import layer_inputs, mlp_inputs

from gpu_util import TOL, rel_err, to_dev, to_host_f32, u32

pytestmark = pytest.mark.gpu

LAYERS = [
    (150, 784, 300, "f32"),
    (150, 300, 10, "f32"),
    (150, 300, 10, "bf16"),     # unaligned bf16: CUDA-core kernels
    (33, 17, 5, "f32"),
    (328, 640, 520, "bf16"),    # aligned bf16: tensor-core kernels
    (328, 392, 200, "bf16"),
    (1024, 256, 512, "bf16"),
    (900, 520, 600, "f32"),     # float32 with enough tiles for the CUDA-core GEMM's larger tile
]


@pytest.mark.parametrize("B,D,H,dtype", LAYERS)
@pytest.mark.parametrize("variant", ["different", "same"])
@pytest.mark.parametrize("p", [0.1, 1.0, 0.5])
def test_weight_grad_matches_oracle(B, D, H, dtype, variant, p):
    import paper_2007_10412_b200 as rad
    A, dZ = layer_inputs(B, D, H, dtype=dtype, seed=B + D + H)
    ref_st = orc.forward_store(A, dtype, variant, p, 11, 2, 0)
    ref = orc.weight_grad(ref_st, dZ)
    st = rad.Store(variant, dtype, B, D, p, seed=11, layer=2, step=0, relu_bits=False)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    rad.rad_linear_forward_store(to_dev(A, dtype), st, status)
    dW = torch.full((D, H), float("nan"), dtype=torch.float32, device="cuda")
    rad.rad_linear_weight_grad(st, to_dev(dZ, dtype), dW, dev_status=status)
    torch.cuda.synchronize()
    assert status.item() == 0
    got = to_host_f32(dW)
    fro, mx = rel_err(got, ref)
    assert fro <= TOL[dtype] and mx <= TOL[dtype], (fro, mx)
    if variant == "same":
        kept = np.zeros(D, bool)
        kept[ref_st.idx] = True
        assert (got[~kept] == 0).all()          # Sec. 4.3: rows of unsampled columns are untouched
    # run to run reproducibility (fixed accumulation order)
    dW2 = torch.empty_like(dW)
    rad.rad_linear_weight_grad(st, to_dev(dZ, dtype), dW2, dev_status=status)
    torch.cuda.synchronize()
    assert torch.equal(dW, dW2)


@pytest.mark.parametrize("B,D,H,dtype", LAYERS)
@pytest.mark.parametrize("act", ["relu", "gelu"])
def test_input_grad_matches_oracle(B, D, H, dtype, act):
    import paper_2007_10412_b200 as rad
    rng = np.random.default_rng(B * 7 + D)
    _, dZ = layer_inputs(B, D, H, dtype=dtype, seed=5)
    W = rng.standard_normal((D, H), dtype=np.float32) * np.float32(np.sqrt(2.0 / D))
    Zp = rng.standard_normal((B, D), dtype=np.float32)
    if dtype == "bf16":
        from workloads import to_bf16_grid
        W, Zp = to_bf16_grid(W), to_bf16_grid(Zp)
    bits = orc.pack_bits(Zp > 0)
    if act == "relu":
        ref_dA, ref_db = orc.input_grad(dZ, W, relubits_prev=bits, dtype=dtype)
    else:
        ref_dA, ref_db = orc.input_grad(dZ, W, Z_prev=Zp, act="gelu", dtype=dtype)
    tdt = torch.float32 if dtype == "f32" else torch.bfloat16
    out = torch.full((B, D), float("nan"), dtype=tdt, device="cuda")
    db = torch.full((H,), float("nan"), dtype=torch.float32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    rad.rad_linear_input_grad(to_dev(dZ, dtype), to_dev(W, dtype),
                              relubits_prev=torch.from_numpy(bits.view(np.int32)).cuda() if act == "relu" else None,
                              z_prev=to_dev(Zp, dtype) if act == "gelu" else None,
                              dZ_prev=out, db=db, dev_status=status)
    torch.cuda.synchronize()
    assert status.item() == 0
    fro, mx = rel_err(to_host_f32(out), ref_dA)
    assert fro <= TOL[dtype] and mx <= TOL[dtype], (fro, mx)
    fro, mx = rel_err(to_host_f32(db), ref_db)
    assert fro <= 1e-5 and mx <= 1e-5, (fro, mx)
    if act == "relu":
        assert (to_host_f32(out)[~(Zp > 0)] == 0).all()


@pytest.mark.parametrize("B,D,H,dtype", LAYERS)
@pytest.mark.parametrize("act", ["relu", "gelu", "none"])
def test_forward_matches_oracle(B, D, H, dtype, act):
    import paper_2007_10412_b200 as rad
    X, _, Ws, bs = mlp_inputs((D, H), B, dtype=dtype, x_dist="normal", seed=3, bias_zero=False)
    z = X.astype(np.float64) @ Ws[0].astype(np.float64) + bs[0]
    a = orc.act_forward(z, act)
    tdt = torch.float32 if dtype == "f32" else torch.bfloat16
    out_act = torch.empty(B, H, dtype=tdt, device="cuda")
    out_z = torch.empty(B, H, dtype=torch.float32, device="cuda")
    out_zl = torch.empty(B, H, dtype=tdt, device="cuda")
    w32 = (H + 31) // 32
    rb = torch.zeros(B * w32, dtype=torch.int32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    rad.rad_linear_forward(to_dev(X, dtype), to_dev(Ws[0], dtype), to_dev(bs[0], "f32"), act, out_act=out_act,
                           out_z=out_z, out_zlow=out_zl, relubits=rb, dev_status=status)
    torch.cuda.synchronize()
    assert status.item() == 0
    tol = TOL[dtype]
    assert max(rel_err(to_host_f32(out_z), z)) <= 1e-5
    assert max(rel_err(to_host_f32(out_act), a)) <= (1e-5 if dtype == "f32" else 8e-3)
    assert max(rel_err(to_host_f32(out_zl), z)) <= (1e-5 if dtype == "f32" else 8e-3)
    assert tol >= 1e-5
    # the ReLU bits are those of the activation the call wrote
    assert np.array_equal(u32(rb).reshape(B, w32), orc.pack_bits(to_host_f32(out_act) > 0))


@pytest.mark.parametrize("B,C,dtype", [(150, 10, "f32"), (150, 10, "bf16"), (513, 1000, "bf16"), (3, 2, "f32")])
def test_softmax_xent_matches_oracle(B, C, dtype):
    import paper_2007_10412_b200 as rad
    rng = np.random.default_rng(C)
    logits = (rng.standard_normal((B, C)) * 3).astype(np.float32)
    labels = rng.integers(0, C, B).astype(np.int32)
    loss_ref, dz_ref = orc.softmax_xent(logits, labels)
    tdt = torch.float32 if dtype == "f32" else torch.bfloat16
    dz = torch.empty(B, C, dtype=tdt, device="cuda")
    loss = torch.zeros(1, device="cuda")
    rad.rad_softmax_xent(torch.from_numpy(logits).cuda(), torch.from_numpy(labels).cuda(), loss, dz)
    torch.cuda.synchronize()
    assert abs(loss.item() - loss_ref) <= 1e-5 * abs(loss_ref)
    assert max(rel_err(to_host_f32(dz), dz_ref)) <= (1e-5 if dtype == "f32" else 8e-3)


@pytest.mark.parametrize("B,H,dtype", [(700, 10, "f32"), (700, 40, "bf16"), (5000, 64, "bf16"), (40000, 16, "bf16"),
                                       (700, 300, "f32"), (700, 301, "bf16"), (2100, 1000, "bf16"), (130, 1000, "bf16")])
def test_bias_gradient_alone_on_every_column_sum_route(B, H, dtype):
    """db = sum over the minibatch of dZ (Sec. 4.2: exact, never sampled), asked for without the input gradient:
    few rows (one launch), narrow matrices (row lanes x columns), wide bf16 matrices (16-byte loads) and the
    plain two-stage route, against float64 sums of the same numbers."""
    import paper_2007_10412_b200 as rad
    rng = np.random.default_rng(B + H)
    dZ = rng.standard_normal((B, H), dtype=np.float32)
    if dtype == "bf16":
        from workloads import to_bf16_grid
        dZ = to_bf16_grid(dZ)
    W = torch.zeros(8, H, dtype=torch.float32 if dtype == "f32" else torch.bfloat16, device="cuda")
    db = torch.full((H,), float("nan"), dtype=torch.float32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    rad.rad_linear_input_grad(to_dev(dZ, dtype), W, db=db, dev_status=status)
    torch.cuda.synchronize()
    assert status.item() == 0
    want = dZ.astype(np.float64).sum(axis=0)
    bound = 2e-6 * np.abs(dZ.astype(np.float64)).sum(axis=0)
    assert (np.abs(to_host_f32(db).astype(np.float64) - want) <= bound).all()


@pytest.mark.parametrize("B,H,ld,dtype", [(1, 1, 1, "f32"), (33, 8, 8, "bf16"), (1025, 24, 32, "bf16"), (257, 65, 65, "f32"),
                                          (4097, 72, 72, "f32"), (300001, 8, 8, "bf16"), (300001, 7, 7, "f32"),
                                          (140000, 20, 24, "bf16"), (70000, 132, 132, "f32"), (8192, 601, 601, "f32"),
                                          (8193, 601, 601, "bf16"), (40001, 603, 605, "f32"), (33000, 1201, 1201, "bf16")])
def test_bias_gradient_over_clusters_and_slabs(B, H, ld, dtype):
    """Column sums by one CTA, by a cluster of CTAs along the rows and by slabs of rows added in a second launch, with
    vector and single-element loads (padded rows, odd widths, tall ones of many column blocks), against float64 sums of the same numbers.  Every chain
    of float32 additions is shorter than 4096 terms of a 2^-24 relative rounding each; the bound allows 33 in a row."""
    import paper_2007_10412_b200 as rad
    tdt = torch.float32 if dtype == "f32" else torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(B + H)
    wide = torch.randn(B, ld, generator=g, device="cuda").to(tdt)
    dZ = wide[:, :H]
    W = torch.zeros(8, ld, dtype=tdt, device="cuda")[:, :H]
    db = torch.full((H,), float("nan"), dtype=torch.float32, device="cuda")
    rad.rad_linear_input_grad(dZ, W, db=db)
    torch.cuda.synchronize()
    d64 = dZ.double()
    assert ((db.double() - d64.sum(0)).abs() <= 2e-6 * d64.abs().sum(0)).all()


@pytest.mark.parametrize("B,C,dtype", [(1, 1, "f32"), (33, 32, "bf16"), (257, 33, "f32"), (256, 257, "bf16"), (2048, 1024, "bf16"),
                                       (2049, 1025, "f32"), (300, 2500, "f32")])
def test_softmax_xent_over_clusters_and_row_lengths(B, C, dtype):
    """The loss of one CTA, of a cluster of CTAs and of many rows, with rows that fit the registers of a warp (32, 256,
    1024 logits) and longer ones, logits of -inf among them, against float64."""
    import paper_2007_10412_b200 as rad
    g = torch.Generator(device="cuda").manual_seed(B + C)
    logits = torch.randn(B, C, generator=g, device="cuda") * 3
    labels = torch.randint(0, C, (B,), generator=g, device="cuda", dtype=torch.int32)
    if C > 2:
        drop = torch.rand(B, C, generator=g, device="cuda") < 0.1
        drop[torch.arange(B), labels.long()] = False
        logits[drop] = float("-inf")
    dz = torch.full((B, C), float("nan"), dtype=torch.float32 if dtype == "f32" else torch.bfloat16, device="cuda")
    loss = torch.zeros(1, device="cuda")
    rad.rad_softmax_xent(logits, labels, loss, dz)
    torch.cuda.synchronize()
    lp = torch.log_softmax(logits.double(), 1)
    rows = torch.arange(B, device="cuda")
    want = -lp[rows, labels.long()].mean().item()
    ref = lp.exp()
    ref[rows, labels.long()] -= 1
    ref /= B
    assert abs(loss.item() - want) <= 1e-5 * max(abs(want), 1e-3)
    assert max(rel_err(to_host_f32(dz), ref.cpu().numpy())) <= (1e-5 if dtype == "f32" else 8e-3) or C == 1
    if C == 1:
        assert (dz == 0).all()


# The forms the CUDA-core GEMM takes, by forward and input gradient: one CTA that walks all of k ("walk", tiles of 32 or 64),
# or k split over thread groups and up to eight CTAs of a cluster ("split"); from 297 tiles on the walk has several waves.
CUDA_CORE_FORMS = [
    # B, D, H, type, forward, input gradient
    (1, 1, 1, "f32", "walk32", "walk32"),
    (33, 130, 31, "f32", "split32x8", "walk32"),
    (65, 1001, 33, "f32", "split32x8", "walk32"),
    (150, 784, 300, "f32", "split32x2", "split32x1"),
    (700, 257, 203, "f32", "split32x1", "split32x1"),
    (2000, 68, 1500, "f32", "walk64", "split64x4"),
    (129, 3000, 70, "f32", "split32x8", "walk64"),
    (90, 100, 30, "bf16", "split32x4", "walk32"),
    (700, 515, 333, "bf16", "split32x1", "walk64"),
    (4100, 10, 300, "f32", "walk64", "split32x1"),
    (3000, 20, 10, "f32", "walk32", "walk32"),
    (130, 33, 9, "bf16", "walk32", "walk32"),
    (1000, 41, 1001, "bf16", "walk64", "split32x4"),
    (2100, 203, 601, "bf16", "walk64", "walk64"),
]


@pytest.mark.parametrize("B,D,H,dtype", [c[:4] for c in CUDA_CORE_FORMS])
def test_cuda_core_contractions_over_tiles_and_splits(B, D, H, dtype):
    """Forward, input gradient and weight gradients (either mask) on CUDA cores, in the form that walks the contraction index
    and in the one that splits it, from one CTA to clusters that share it, 32 and 64 wide tiles with remainders, one wave
    of tiles and several, aligned and odd leading dimensions, against float64.
    Bound per output: sqrt(K) + 16 roundings of 2^-24 of the sum of magnitudes, plus one bf16 rounding of the result."""
    import paper_2007_10412_b200 as rad
    tdt = torch.float32 if dtype == "f32" else torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(B + D + H)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda").to(tdt)
    A, W, dZ = rnd(B, D), rnd(D, H), rnd(B, H)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = torch.full((B, H), float("nan"), dtype=torch.float32, device="cuda")
    rad.rad_linear_forward(A, W, None, "none", out_z=out, dev_status=status)
    dX = torch.full((B, D), float("nan"), dtype=tdt, device="cuda")
    rad.rad_linear_input_grad(dZ, W, dZ_prev=dX, dev_status=status)
    st = rad.Store("same", dtype, B, D, 1.0, relu_bits=False)
    rad.rad_linear_forward_store(A, st, status)
    dW = torch.full((D, H), float("nan"), dtype=torch.float32, device="cuda")
    rad.rad_linear_weight_grad(st, dZ, dW, dev_status=status)
    sd = rad.Store("different", dtype, B, D, 0.3, seed=3, relu_bits=False)
    rad.rad_linear_forward_store(A, sd, status)
    dWd = torch.full((D, H), float("nan"), dtype=torch.float32, device="cuda")
    rad.rad_linear_weight_grad(sd, dZ, dWd, dev_status=status)
    torch.cuda.synchronize()
    assert status.item() == 0
    keep = torch.from_numpy(orc.keep_mask("different", B, D, 0.3, 3, 0, 0)).cuda()
    Ah = torch.where(keep, (A.float() * float(orc.scale_factor(0.3))).to(tdt), torch.zeros((), dtype=tdt, device="cuda")).double()
    A, W, dZ = A.double(), W.double(), dZ.double()
    for got, x, y, low in ((out, A, W, False), (dX, dZ, W.T, dtype == "bf16"), (dW, A.T, dZ, False), (dWd, Ah.T, dZ, False)):
        ref, mag, K = x @ y, x.abs() @ y.abs(), x.shape[1]
        bound = (K ** 0.5 + 16) * 2.0 ** -24 * mag + (2.0 ** -8 * ref.abs() if low else 0)
        assert ((got.double() - ref).abs() <= bound + 1e-30).all()


DENSE_WIDTHS = [
    # B, D, H, columns of a tile of the forward (H wide) and of the input gradient (D wide), on 66 to 74 SM pairs
    (64, 64, 64, 64, 64),
    (300, 72, 200, 64, 64),
    (257, 2048, 136, 64, 64),
    (200, 2056, 72, 64, 64),            # above 2048 inputs: eight epilogue warps
    (1024, 640, 1000, 64, 64),
    (1280, 520, 1032, 128, 64),
    (1280, 1032, 520, 64, 128),
    (1280, 2056, 1032, 128, 256),       # eight epilogue warps
    (2500, 2056, 1032, 256, 256),
    (5000, 128, 1096, 256, 64),
]


def dense_tile_width(M, N, pairs):
    """The narrowest of 64, 128 and 256 columns with which the tiles of 256 rows are one wave of SM pairs, else 256."""
    return next((w for w in (64, 128) if -(-M // 256) * -(-N // w) <= pairs), 256)


@pytest.mark.parametrize("B,D,H,fwd_width,dx_width", DENSE_WIDTHS)
@pytest.mark.parametrize("act", ["relu", "gelu"])
def test_dense_tile_widths(B, D, H, fwd_width, dx_width, act):
    """Forward with the next layer's store and input gradient on the tensor cores at tiles of 64, 128 and 256 columns with
    remainders, and with either number of epilogue warps: the forward's store is the store of its own output bit for
    bit, the forward without a store (whose epilogue warps are counted by another rule) gives the same output, values against
    float64 within one bf16 rounding and the float32 sums' error."""
    import paper_2007_10412_b200 as rad
    pairs = rad.rad_sm_pairs()
    assert dense_tile_width(B, H, pairs) == fwd_width and dense_tile_width(B, D, pairs) == dx_width
    _check_dense(B, D, H, act)


@pytest.mark.parametrize("B,D,H", [(20000, 200, 64), (19500, 128, 72), (20001, 72, 128), (38000, 64, 64)])
@pytest.mark.parametrize("act", ["relu", "gelu"])
def test_narrow_outputs_of_many_rows(B, D, H, act):
    """More tiles than SM pairs in one column of tiles, of 64 or 128 columns as the matrix needs and of 128 where a store is
    filled: the same checks as for the other tile widths."""
    import paper_2007_10412_b200 as rad
    assert -(-B // 256) > rad.rad_sm_pairs()
    _check_dense(B, D, H, act)


def _check_dense(B, D, H, act):
    import paper_2007_10412_b200 as rad
    bf = torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(B + D + H)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda").to(bf)
    A, W, dZ, zp, b = rnd(B, D), rnd(D, H), rnd(B, H), rnd(B, D), rnd(H).float()
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    fill = rad.Store("different", "bf16", B, H, 0.2, seed=9, layer=2, step=3, relu_bits=True)
    own = rad.Store("different", "bf16", B, H, 0.2, seed=9, layer=2, step=3, relu_bits=True)
    for st in (fill, own):
        st.values.zero_()
    out, zl = torch.empty(B, H, dtype=bf, device="cuda"), torch.empty(B, H, dtype=bf, device="cuda")
    rad.rad_linear_forward_fill(A, W, b, act, out, fill, out_zlow=zl, relubits=fill.relubits, dev_status=status)
    rad.rad_linear_forward_store(out, own, status)
    plain = torch.empty_like(out)
    rad.rad_linear_forward(A, W, b, act, out_act=plain, dev_status=status)
    dX = torch.empty(B, D, dtype=bf, device="cuda")
    rad.rad_linear_input_grad(dZ, W, z_prev=zp if act == "gelu" else None, dZ_prev=dX, dev_status=status)
    torch.cuda.synchronize()
    assert status.item() == 0
    for x, y in ((fill.values, own.values), (fill.keepbits, own.keepbits), (fill.offsets, own.offsets), (fill.nnz, own.nnz),
                 (fill.relubits, own.relubits), (plain, out)):
        assert torch.equal(x, y)
    z = A.double() @ W.double() + b.double()
    tol = (max(D, H) ** 0.5 + 16) * 2.0 ** -24
    mag = A.double().abs() @ W.double().abs() + b.abs()
    assert ((zl.double() - z).abs() <= tol * mag + 2.0 ** -8 * z.abs()).all()
    dx, mx = dZ.double() @ W.double().T, dZ.double().abs() @ W.double().abs().T
    if act == "gelu":
        x = zp.double()
        d = 0.5 * (1 + torch.erf(x / 2 ** 0.5)) + x * torch.exp(-0.5 * x * x) / (2 * np.pi) ** 0.5
        dx, mx = dx * d, mx * (d.abs() + 1e-3)
    assert ((dX.double() - dx).abs() <= 8 * tol * mx + 2.0 ** -8 * dx.abs()).all()


@pytest.mark.parametrize("B", [40, 130, 640])
def test_different_sample_dw_of_several_units_per_sm_pair(B):
    """dW of 4000 x 4104 from a different-sample store: 144 tiles of 256 x 512 or 272 half as wide on at most 74 SM pairs, with one K block per tile
    (the expanders run several tiles ahead of the epilogue), a few, and more than the ring of stages holds; tiles that
    reach past either edge.  Against float64; the bound is that of a float32 sum of B products in any order."""
    import paper_2007_10412_b200 as rad
    D, H, p = 4000, 4104, 0.3
    assert -(-D // 256) * -(-H // 512) > rad.rad_sm_pairs()
    bf = torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(B)
    A, dZ = (torch.randn(B, n, generator=g, device="cuda").to(bf) for n in (D, H))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    st = rad.Store("different", "bf16", B, D, p, seed=3, layer=1, step=2, relu_bits=False)
    rad.rad_linear_forward_store(A, st, status)
    dW = torch.full((D, H), float("nan"), device="cuda")
    rad.rad_linear_weight_grad(st, dZ, dW, dev_status=status)
    torch.cuda.synchronize()
    assert status.item() == 0
    keep = torch.from_numpy(orc.keep_mask("different", B, D, p, 3, 1, 2)).cuda()
    Ah = torch.where(keep, (A.float() * float(orc.scale_factor(p))).to(bf), torch.zeros((), dtype=bf, device="cuda")).double()
    ref, mag = Ah.T @ dZ.double(), Ah.abs().T @ dZ.double().abs()
    assert ((dW.double() - ref).abs() <= B * 2.0 ** -24 * mag).all()


@pytest.mark.parametrize("B,D,H", [(64, 64, 64), (300, 72, 136), (2500, 64, 1032)])
@pytest.mark.parametrize("p,shift", [(0.05, 0), (0.05, 1), (0.9, 0)])
def test_outputs_in_chunks_and_the_store_beside_them(B, D, H, p, shift):
    """Outputs with rows longer than the layer's width keep what lies past it; every combination of outputs gives the same
    bits; the next store is the same whether a warp stages its entries (16-byte aligned values, few of them) or not."""
    import paper_2007_10412_b200 as rad
    bf = torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(B + H)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    A, W, b = rnd(B, D).to(bf), rnd(D, H).to(bf), rnd(H)
    new = lambda dt, ld: torch.full((B, ld), -7.0, dtype=dt, device="cuda")
    act, zl, z = new(bf, H + 24), new(bf, H + 8), new(torch.float32, H + 4)
    rad.rad_linear_forward(A, W, b, "gelu", out_act=act[:, :H], out_zlow=zl[:, :H], out_z=z[:, :H])
    a2, z2 = new(bf, H), new(torch.float32, H)
    rad.rad_linear_forward(A, W, b, "gelu", out_act=a2)
    rad.rad_linear_forward(A, W, b, "none", out_z=z2)
    st = rad.Store("different", "bf16", B, H, p, seed=3, layer=1, step=2, relu_bits=False)
    own = rad.Store("different", "bf16", B, H, p, seed=3, layer=1, step=2, relu_bits=False)
    room = torch.zeros(st.values.numel() + 8, dtype=bf, device="cuda")
    st.c.values = room[shift:].data_ptr()
    own.values.zero_()
    a3 = new(bf, H)
    rad.rad_linear_forward_fill(A, W, b, "gelu", a3, st)
    rad.rad_linear_forward_store(a3, own)
    torch.cuda.synchronize()
    for full, width in ((act, H), (zl, H), (z, H)):
        assert (full[:, width:] == -7.0).all()
    assert torch.equal(act[:, :H], a2) and torch.equal(z[:, :H], z2) and torch.equal(zl[:, :H], z2.to(bf)) and torch.equal(a3, a2)
    assert torch.equal(room[shift:shift + own.values.numel()], own.values)
    want = A.double() @ W.double() + b.double()
    mag = A.double().abs() @ W.double().abs() + b.double().abs()
    assert ((z2.double() - want).abs() <= (D ** 0.5 + 16) * 2.0 ** -24 * mag).all()      # float32 sums in any order


@pytest.mark.parametrize("act", ["none", "relu", "gelu"])
@pytest.mark.parametrize("B,D,H", [(64, 64, 64), (300, 72, 136), (2500, 64, 1032)])
def test_pre_activations_as_the_only_output(B, D, H, act):
    """The forward pass on the tensor cores with its bf16 pre-activations as the only output: the same bits as beside others."""
    import paper_2007_10412_b200 as rad
    bf = torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(B + H)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    A, W, b = rnd(B, D).to(bf), rnd(D, H).to(bf), rnd(H)
    alone, beside, out = (torch.full((B, H), -7.0, dtype=bf, device="cuda") for _ in range(3))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    rad.rad_linear_forward(A, W, b, act, out_zlow=alone, dev_status=status)
    rad.rad_linear_forward(A, W, b, act, out_act=out, out_zlow=beside, dev_status=status)
    torch.cuda.synchronize()
    assert status.item() == 0 and torch.equal(alone, beside)


BIAS_ROUTES = [
    # B, D, H, row stride of dZ, are the column sums made by the input gradient's launch?
    (64, 64, 64, 64, True),
    (130, 72, 200, 208, False),
    (300, 1032, 200, 208, True),
    (2049, 128, 1184, 1184, False),
    (2100, 64, 1192, 1192, False),
    (20000, 1096, 264, 264, False),
    (1024, 64, 4744, 4744, False),
    (256, 64, 4096, 4096, False),
    (200, 4096, 8192, 8192, True),          # four groups of columns per CTA
    (1100, 2048, 4104, 4104, True),         # ... of two steps down the rows each
    (9000, 2048, 1032, 1032, True),         # five steps, four tiles per SM pair
]


@pytest.mark.parametrize("B,D,H,ld", [r[:4] for r in BIAS_ROUTES])
@pytest.mark.parametrize("act", ["relu", "gelu"])
def test_bias_gradient_beside_the_input_gradient(B, D, H, ld, act):
    """Column sums asked for with the input gradient, made by its launch (one group of 8 or 16 columns per CTA and several, rows
    that end inside a step, several tiles per SM pair) or by one of their own; the input gradient is the same with and without them.  Bound: eight rows as a tree, then
    at most B / 1024 + 1 steps, lanes and warps, each a float32 rounding of the sum of magnitudes."""
    import paper_2007_10412_b200 as rad
    bf = torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(B + H)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda").to(bf)
    dZ, W = rnd(B, ld)[:, :H], rnd(D, H)
    z = rnd(B, D) if act == "gelu" else None
    bits = torch.randint(-2 ** 31, 2 ** 31, (B * ((D + 31) // 32),), generator=g, device="cuda", dtype=torch.int64).to(torch.int32)
    kw = dict(z_prev=z, relubits_prev=None if act == "gelu" else bits)
    db, dX, dX2 = torch.full((H,), float("nan"), device="cuda"), torch.empty(B, D, dtype=bf, device="cuda"), torch.empty(B, D, dtype=bf, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    rad.rad_linear_input_grad(dZ, W, dZ_prev=dX, db=db, dev_status=status, **kw)
    rad.rad_linear_input_grad(dZ, W, dZ_prev=dX2, **kw)
    torch.cuda.synchronize()
    assert status.item() == 0 and torch.equal(dX, dX2)
    x = dZ.double()
    assert ((db.double() - x.sum(0)).abs() <= (3 + 2 * (B / 1024 + 1) + 5 + 8) * 2.0 ** -24 * x.abs().sum(0)).all()


@pytest.mark.parametrize("D,ldp", [(64, 72), (256, 264)])
def test_gelu_derivative_is_the_same_function_on_both_routes(D, ldp):
    """The input gradient of a GELU net at every bf16 pre-activation there is, infinities and NaN among them.  dZ has one 1 in a
    row, so the float32 sum is an entry of W on the tensor cores and on the CUDA cores (taken where the output's row stride
    is odd), and what is left is the product with GELU': the two routes give the same bits."""
    import paper_2007_10412_b200 as rad
    bf = torch.bfloat16
    B, H = 65536 // D, 64
    g = torch.Generator(device="cuda").manual_seed(D)
    z = torch.arange(-32768, 32768, device="cuda").to(torch.int16)[torch.randperm(65536, generator=g, device="cuda")].view(bf).view(B, D)
    W = torch.randn(D, H, generator=g, device="cuda").to(bf)
    dZ = torch.zeros(B, H, dtype=bf, device="cuda")
    dZ[torch.arange(B, device="cuda"), torch.arange(B, device="cuda") % H] = 1
    outs = [torch.zeros(B, ld, dtype=bf, device="cuda")[:, :D] for ld in (ldp, ldp + 1)]
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for out in outs:
        rad.rad_linear_input_grad(dZ, W, z_prev=z, dZ_prev=out, dev_status=status)
    torch.cuda.synchronize()
    assert status.item() == 0
    tensor, cuda = (out.contiguous() for out in outs)
    nan = torch.isnan(cuda)
    assert torch.equal(torch.isnan(tensor), nan)
    assert torch.equal(tensor[~nan].view(torch.int16), cuda[~nan].view(torch.int16))


@pytest.mark.parametrize("B,D,H", [(64, 64, 64), (328, 264, 136), (1000, 520, 264), (4160, 256, 264), (1024, 2048, 2040), (70, 1032, 520)])
@pytest.mark.parametrize("p", [0.1, 0.7])
def test_different_sample_dw_over_tile_widths(B, D, H, p):
    """dW from a different-sample store of few and of many tiles, sparse and dense, with rows and columns that end inside a tile."""
    _check_dw(B, D, H, p)


DW_TILES = [
    # B, D, H, p, columns of a tile, K splits
    (328, 264, 136, 0.1, 128, 6),
    (200, 520, 136, 0.1, 128, 1),
    (200, 2056, 1032, 0.1, 256, 1),
    (700, 264, 1544, 0.7, 256, 4),
    (200, 2056, 2056, 0.1, 512, 1),
    (4096, 2040, 2040, 0.1, 512, 2),
    (1500, 520, 2056, 0.7, 512, 4),
]


@pytest.mark.parametrize("B,D,H,p", [c[:4] for c in DW_TILES])
def test_different_sample_dw_at_every_tile_width_and_split(B, D, H, p):
    """Tiles of 128, 256 and 512 columns, each with and without a split of the rows, none a whole number of tiles."""
    _check_dw(B, D, H, p)


def _check_dw(B, D, H, p):
    """Against float64: the sum of B products in any order."""
    import paper_2007_10412_b200 as rad
    bf = torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(B + D + H)
    A, dZ = (torch.randn(B, n, generator=g, device="cuda").to(bf) for n in (D, H))
    st = rad.Store("different", "bf16", B, D, p, seed=5, layer=1, step=2, relu_bits=False)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    rad.rad_linear_forward_store(A, st, status)
    dW = torch.full((D, H), float("nan"), device="cuda")
    rad.rad_linear_weight_grad(st, dZ, dW, dev_status=status)
    torch.cuda.synchronize()
    assert status.item() == 0
    keep = torch.from_numpy(orc.keep_mask("different", B, D, p, 5, 1, 2)).cuda()
    kept = torch.where(keep, (A.float() * rad.rad_scale(p)).to(bf), torch.zeros((), dtype=bf, device="cuda")).double()
    mag = kept.abs().T @ dZ.double().abs()
    assert ((dW.double() - kept.T @ dZ.double()).abs() <= (B ** 0.5 + 16) * 2.0 ** -24 * mag).all()
