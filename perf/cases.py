"""Timed cases of the library: what a training program calls, over the sizes it calls it with.

Kinds of case
  mlp    one training step of a fully connected net (MLPStep): loss, dW and db of every layer
  irnn   one training step of the sequential-pixel recurrent net (IRNNStep)
  cnn    one training step of the 3x3-convolution net (CNNStep)
  store  the compact store of one layer input (Store + rad_linear_forward_store)
  layer  a hidden layer of a net, both directions: forward with the next layer's store filled, weight gradient
         from the layer's own store, input gradient and bias gradient
"""
import math

import torch

import paper_2007_10412_b200 as rad

DEV = "cuda"
TORCH_DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16}


def _mlp(name, dims, batch, dtype, act, variant, p, law="bernoulli"):
    return dict(name=name, kind="mlp", dims=dims, batch=batch, dtype=dtype, act=act, variant=variant, p=p, law=law)


def _layer(name, B, D, H, dtype, act, variant, p):
    return dict(name=name, kind="layer", B=B, D=D, H=H, dtype=dtype, act=act, variant=variant, p=p)


def _store(name, B, D, dtype, variant, p, law="bernoulli", relu=False):
    return dict(name=name, kind="store", B=B, D=D, dtype=dtype, variant=variant, p=p, law=law, relu=relu)


def _cnn(name, batch, dtype, variant, p):
    return dict(name=name, kind="cnn", batch=batch, hw=32, cin=3, channels="16,32,64", fc="128,10", dtype=dtype,
                variant=variant, p=p)


def listed():
    return [
        # the MNIST-shaped net of the paper's App. A at its batch of 150, both sampling variants: the smallest step
        # anybody takes, where latency and launches count
        _mlp("mlp_mnist_different", "784,300,300,10", 150, "f32", "relu", "different", 0.1),
        _mlp("mlp_mnist_same", "784,300,300,10", 150, "f32", "relu", "same", 0.1),
        # the wide net cut to sizes that are multiples of nothing but 8: ragged tiles in every dimension
        _mlp("mlp_ragged_bf16", "640,520,392,200", 328, "bf16", "relu", "different", 0.1),
        # the recurrent net of App. A: one scalar per step, 784 steps, 100 hidden units
        dict(name="irnn_mnist", kind="irnn", batch=150, steps=784, hidden=100, classes=10, variant="different", p=0.1),
        # the convolutional net on 32 x 32 x 3 images, at an ordinary and at a large batch
        _cnn("cnn_b128", 128, "bf16", "different", 0.1),
        _cnn("cnn_b4096", 4096, "bf16", "different", 0.1),
        # the store of one wide layer input: the network input of the wide net; the static mask shared by the batch
        _store("store_wide_different", 65536, 8192, "bf16", "different", 0.1),
        # hidden layers of an ordinary net in both directions: bf16 with either mask, float32 at an odd size
        _layer("layer_bf16_different", 4096, 2048, 2048, "bf16", "gelu", "different", 0.1),
        _layer("layer_bf16_same", 2048, 1024, 1024, "bf16", "relu", "same", 0.1),
        _layer("layer_f32_odd", 1500, 1001, 777, "f32", "relu", "different", 0.1),
        # a middle-sized net from end to end
        _mlp("mlp_middle_bf16", "1024,1024,1024,1024,1000", 4096, "bf16", "relu", "different", 0.1),
        # the default workload of the benchmark: 8192 x 4 -> 1000, batch 65536
        _mlp("mlp_wide", "8192,8192,8192,8192,8192,1000", 65536, "bf16", "gelu", "different", 0.1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mult(n, m):
    return max(m, n // m * m)


def draw(rng):
    kind = rng.choice(["mlp", "mlp", "mlp", "irnn", "cnn", "store", "layer", "layer", "layer"])
    p = rng.choice([0.01, 0.05, 0.1, 0.1, 0.1, 0.2, 0.5])
    variant = rng.choice(["different", "different", "same"])
    dtype = rng.choice(["f32", "bf16", "bf16"])
    if kind == "mlp":
        act = rng.choice(["relu", "relu", "gelu"])
        depth = rng.randint(2, 4)
        if dtype == "f32":
            dims = [_log(rng, 64, 1200)] + [_log(rng, 64, 700) for _ in range(depth - 1)] + [rng.randint(5, 100)]
            c = _mlp("", "", _log(rng, 16, 1024), "f32", act, variant, p)
        else:
            dims = [_mult(_log(rng, 256, 4096), 8) for _ in range(depth)] + [_mult(rng.randint(16, 1000), 8)]
            c = _mlp("", "", _log(rng, 128, 16384), "bf16", act, variant, p)
        c["dims"] = ",".join(str(d) for d in dims)
    elif kind == "irnn":
        c = dict(kind="irnn", batch=_log(rng, 16, 400), steps=_log(rng, 28, 784), hidden=rng.randint(32, 128),
                 classes=rng.randint(5, 20), variant=variant, p=p)
    elif kind == "cnn":
        c = _cnn("", _log(rng, 32, 4096), dtype, variant, p)
        if dtype == "f32":
            c["batch"] = min(c["batch"], 512)
        c["hw"] = rng.choice([16, 32, 32])
    elif kind == "store":
        B, D = _log(rng, 256, 65536), _log(rng, 200, 8192)
        c = _store("", B, _mult(D, 8) if dtype == "bf16" else D, dtype, variant, p,
                   rng.choice(["bernoulli", "bernoulli", "bernoulli", "replace", "fixed"]), rng.random() < 0.5)
    else:
        act = rng.choice(["relu", "gelu"])
        if dtype == "f32":
            c = _layer("", _log(rng, 64, 4096), _log(rng, 64, 2048), _log(rng, 64, 2048), "f32", act, variant, p)
        else:
            c = _layer("", _log(rng, 128, 16384), _mult(_log(rng, 128, 4096), 8), _mult(_log(rng, 128, 4096), 8), "bf16",
                       act, variant, p)
    c.pop("name", None)
    return c


def _ints(text):
    return [int(v) for v in text.split(",")]


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 2654435761 % (1 << 31) + 17)


def _normal(g, shape, dtype, std=1.0):
    """N(0, std^2), drawn row block by row block so that large bf16 inputs need no large float32 copy."""
    out = torch.empty(shape, dtype=dtype, device=DEV)
    rows = max(1, (1 << 26) // max(1, math.prod(shape[1:])))
    for r in range(0, shape[0], rows):
        n = min(rows, shape[0] - r)
        out[r:r + n] = torch.randn((n,) + tuple(shape[1:]), generator=g, device=DEV) * std
    return out


def _labels(g, batch, classes):
    return torch.randint(0, classes, (batch,), generator=g, device=DEV, dtype=torch.int32)


MASK_STEP = 7       # the step number in the masks' key


def _inputs(case, seed):
    """Inputs and weights alone, from the seed alone."""
    g, k = _gen(seed), case["kind"]
    dt = TORCH_DTYPE[case.get("dtype", "f32")]
    if k == "mlp":
        dims, B = _ints(case["dims"]), case["batch"]
        # pixels in [0, 1) for the float32 nets, normal inputs for the wide ones
        X = torch.rand((B, dims[0]), generator=g, device=DEV) if case["dtype"] == "f32" else _normal(g, (B, dims[0]), dt)
        Ws = [_normal(g, (dims[l], dims[l + 1]), dt, math.sqrt(2.0 / dims[l])) for l in range(len(dims) - 1)]
        bs = [_normal(g, (d,), torch.float32, 0.1) for d in dims[1:]]
        return dict(X=X, Ws=Ws, bs=bs, y=_labels(g, B, dims[-1]))
    if k == "irnn":
        B, T, H, C = case["batch"], case["steps"], case["hidden"], case["classes"]
        return dict(x=torch.rand((B, T), generator=g, device=DEV), y=_labels(g, B, C), W_ih=_normal(g, (H,), torch.float32, 1e-3),
                    b_ih=torch.zeros(H, device=DEV), W_hh=torch.eye(H, device=DEV), b_hh=torch.zeros(H, device=DEV),
                    W_out=_normal(g, (H, C), torch.float32, 1e-3), b_out=torch.zeros(C, device=DEV))
    if k == "cnn":
        ch, fc, hw, c = _ints(case["channels"]), _ints(case["fc"]), case["hw"], case["cin"]
        X = _normal(g, (case["batch"], hw, hw, c), dt)
        cW, cb, fW, fb = [], [], [], []
        for co in ch:
            cW.append(_normal(g, (3, 3, c, co), dt, math.sqrt(2.0 / (9 * c))))
            cb.append(_normal(g, (co,), torch.float32, 0.1))
            c = co
        d = (hw >> len(ch)) ** 2 * c
        for h in fc:
            fW.append(_normal(g, (d, h), dt, math.sqrt(2.0 / d)))
            fb.append(_normal(g, (h,), torch.float32, 0.1))
            d = h
        return dict(X=X, y=_labels(g, case["batch"], fc[-1]), cW=cW, cb=cb, fW=fW, fb=fb)
    if k == "store":
        A = _normal(g, (case["B"], case["D"]), dt)
        return dict(A=A.relu_() if case["relu"] else A)
    B, D, H = case["B"], case["D"], case["H"]
    z = _normal(g, (B, D), dt)
    return dict(A=z.relu() if case["act"] == "relu" else torch.nn.functional.gelu(z), z=z,
                W=_normal(g, (D, H), dt, math.sqrt(2.0 / D)), b=_normal(g, (H,), torch.float32, 0.1),
                dZ=_normal(g, (B, H), dt, 1.0 / B))


def _new_store(case, B, D, seed, layer, relu_bits):
    st = rad.Store(case["variant"], case["dtype"], B, D, case["p"], seed=seed, layer=layer, step=MASK_STEP, relu_bits=relu_bits,
                   law=case.get("law", "bernoulli"))
    for t in (st.values, st.keepbits, st.offsets, st.relubits):
        if t is not None:
            t.zero_()              # the reserve beyond what is kept is compared too
    return st


def prepare(case, seed):
    k = case["kind"]
    s = dict(case=case, seed=seed, **_inputs(case, seed))
    if k == "mlp":
        s["ctx"] = rad.MLPStep(_ints(case["dims"]), case["batch"], case["dtype"], case["act"], case["variant"], case["p"],
                               law=case["law"])
    elif k == "irnn":
        s["ctx"] = rad.IRNNStep(case["batch"], case["steps"], case["hidden"], case["classes"], case["variant"], case["p"])
    elif k == "cnn":
        s["ctx"] = rad.CNNStep(case["batch"], case["hw"], case["cin"], _ints(case["channels"]), _ints(case["fc"]), case["dtype"],
                               case["variant"], case["p"])
    elif k == "store":
        s["st"] = _new_store(case, case["B"], case["D"], seed, 0, case["relu"])
        s["status"] = torch.zeros(1, dtype=torch.int32, device=DEV)
    else:
        B, D, H, dt = case["B"], case["D"], case["H"], TORCH_DTYPE[case["dtype"]]
        relu = case["act"] == "relu"
        s["status"] = torch.zeros(1, dtype=torch.int32, device=DEV)
        s["st"] = _new_store(case, B, D, seed, 1, relu)
        rad.rad_linear_forward_store(s["A"], s["st"], s["status"])       # what the layer before left behind
        s["next"] = _new_store(case, B, H, seed, 2, False)
        s["out"] = torch.empty(B, H, dtype=dt, device=DEV)
        s["zlow"] = None if relu else torch.empty(B, H, dtype=dt, device=DEV)
        s["bits"] = torch.zeros(B * ((H + 31) // 32), dtype=torch.int32, device=DEV) if relu else None
        s["dW"] = torch.empty(D, H, dtype=torch.float32, device=DEV)
        s["dZp"] = torch.empty(B, D, dtype=dt, device=DEV)
        s["db"] = torch.empty(H, dtype=torch.float32, device=DEV)
        s["ws_w"] = torch.empty(max(256, rad.rad_weight_grad_workspace(s["st"], H)), dtype=torch.uint8, device=DEV)
        s["ws_x"] = torch.empty(rad.rad_input_grad_workspace(B, H), dtype=torch.uint8, device=DEV)
    return s


def run(s):
    k = s["case"]["kind"]
    if k == "mlp":
        c = s["ctx"](s["X"], s["y"], s["Ws"], s["bs"], seed=s["seed"], step=MASK_STEP)
        return dict(loss=c.loss, dW=c.dW, db=c.db, nnz=c.nnz, status=c.dev_status)
    if k == "irnn":
        c = s["ctx"](s["x"], s["y"], s["W_ih"], s["b_ih"], s["W_hh"], s["b_hh"], s["W_out"], s["b_out"], seed=s["seed"],
                     step0=MASK_STEP)
        return dict(loss=c.loss, dW_ih=c.dW_ih, db=c.db, dW_hh=c.dW_hh, dW_out=c.dW_out, db_out=c.db_out, nnz=c.nnz,
                    status=c.dev_status)
    if k == "cnn":
        c = s["ctx"](s["X"], s["y"], s["cW"], s["cb"], s["fW"], s["fb"], seed=s["seed"], step=MASK_STEP)
        return dict(loss=c.loss, conv_dW=c.dconv_W, conv_db=c.dconv_b, fc_dW=c.dfc_W, fc_db=c.dfc_b, nnz=c.nnz,
                    status=c.dev_status)
    if k == "store":
        st = s["st"]
        rad.rad_linear_forward_store(s["A"], st, s["status"])
        return dict(values=st.values, keepbits=st.keepbits, offsets=st.offsets, nnz=st.nnz, relubits=st.relubits,
                    status=s["status"])
    st, nx, act = s["st"], s["next"], s["case"]["act"]
    rad.rad_linear_forward_fill(s["A"], s["W"], s["b"], act, s["out"], nx, out_zlow=s["zlow"], relubits=s["bits"],
                                dev_status=s["status"])
    rad.rad_linear_weight_grad(st, s["dZ"], s["dW"], s["ws_w"], s["status"])
    rad.rad_linear_input_grad(s["dZ"], s["W"], relubits_prev=st.relubits, z_prev=s["z"] if act == "gelu" else None,
                              dZ_prev=s["dZp"], db=s["db"], workspace=s["ws_x"], dev_status=s["status"])
    return dict(out=s["out"], zlow=s["zlow"], bits=s["bits"], next_values=nx.values, next_keepbits=nx.keepbits,
                next_offsets=nx.offsets, next_nnz=nx.nnz, dW=s["dW"], dZ_prev=s["dZp"], db=s["db"], status=s["status"])


def work(case):
    """Contractions: the exact ones whole, the weight gradients on the kept entries; every input and result once."""
    k, p = case["kind"], case["p"]
    es = 2 if case.get("dtype") == "bf16" else 4
    if k == "mlp":
        dims, B = _ints(case["dims"]), case["batch"]
        flops = nbytes = 0.0
        for l in range(len(dims) - 1):
            DH = dims[l] * dims[l + 1]
            flops += 2.0 * B * DH * (1 + p + (1 if l > 0 else 0))
            nbytes += DH * (es + 4.0)
        return dict(bytes=nbytes + B * dims[0] * es, flops=flops)
    if k == "irnn":
        B, T, H, C = case["batch"], case["steps"], case["hidden"], case["classes"]
        return dict(bytes=4.0 * (B * T + 2 * H * H + 2 * H * C + B), flops=2.0 * B * T * H * H * (2 + p))
    if k == "cnn":
        ch, fc, hw, c, B = _ints(case["channels"]), _ints(case["fc"]), case["hw"], case["cin"], case["batch"]
        flops, nbytes = 0.0, float(B * hw * hw * c * es)
        for l, co in enumerate(ch):
            flops += 2.0 * B * hw * hw * 9 * c * co * (1 + p + (1 if l > 0 else 0))
            nbytes += 9 * c * co * (es + 4.0)
            c, hw = co, hw // 2
        d = hw * hw * c
        for h in fc:
            flops += 2.0 * B * d * h * (2 + p)
            nbytes += d * h * (es + 4.0)
            d = h
        return dict(bytes=nbytes, flops=flops)
    if k == "store":
        B, D = case["B"], case["D"]
        index = B * D / 8.0 if case["variant"] == "different" else D * 4.0
        return dict(bytes=B * D * es * (1 + p) + index + (B * D / 8.0 if case["relu"] else 0.0), flops=0.0)
    B, D, H = case["B"], case["D"], case["H"]
    bits = 1.0 / 8 if case["variant"] == "different" else 0.0
    held = 1.0 / 8 if case["act"] == "relu" else es              # derivative bits, or the pre-activation whole
    nbytes = B * D * (es * (1 + p) + bits + held + es)           # A, its store, the derivative of its activation, dZ_prev
    nbytes += B * H * (es * (1 + p) + bits + held + es)          # the activation, its store, its derivative, dZ
    return dict(bytes=nbytes + D * H * (es + 4.0), flops=2.0 * B * D * H * (2 + p))


def tolerance(case):
    if case["kind"] == "store":
        return "exact"
    bf16 = case.get("dtype") == "bf16"
    if case["kind"] == "layer":
        # float32 sums in another order; bf16 results round the same sums, and a rounding or a sign at zero falls
        # the other way now and then
        return dict(rel=2e-3, max=0.05, differ=2e-3) if bf16 else dict(rel=1e-5, max=4e-4, differ=1e-3)
    if case["kind"] == "irnn":
        return dict(rel=1e-5, max=4e-4)
    # Whole nets: one ReLU whose pre-activation is a last-bit rounding away from zero may fall the other way and
    # move a row's share of the gradients before it: a small part of a tensor's norm, but single entries of a
    # gradient that sums a few sampled rows move by as much as they are (against exact(), both sides' bf16 nets
    # are off by up to 5e-2 and such entries by more than 1).
    return dict(rel=2e-2, max=0.99) if bf16 else dict(rel=4e-3, max=0.99)


# ---- the same results in 64 bits ------------------------------------------------------------------------------------
def _philox(c0, c1, c2, c3, seed):
    """Philox-4x32-10 (Salmon et al., SC'11) on int64 tensors that hold 32-bit words."""
    m = 0xFFFFFFFF
    k0, k1 = seed & m, (seed >> 32) & m
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & m) ^ c1 ^ k0, p1 & m, ((p0 >> 32) & m) ^ c3 ^ k1, p0 & m
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return [c0, c1, c2, c3]


def _keep(variant, B, D, p, seed, layer, step):
    """(keep mask B x D, 1 / p_eff): column c of group g of a row has a 12-bit number, bit 11 - i of it the complement
    of bit c of word i of the outputs for counters (3 g + j, row, layer | stream << 24, step); kept where it is
    below rint(4096 p)."""
    T = min(max(round(p * 4096), 1), 4096)
    G, rows = (D + 31) // 32, B if variant == "different" else 1
    g = torch.arange(G, device=DEV, dtype=torch.int64)[None, :].expand(rows, G)
    r = torch.arange(rows, device=DEV, dtype=torch.int64)[:, None].expand(rows, G)
    c2 = torch.full_like(g, layer | ((0 if variant == "different" else 1) << 24))
    words = []
    for j in range(3):
        words += _philox(3 * g + j, r, c2, torch.full_like(g, step), seed)
    x = torch.full_like(g, 0xFFFFFFFF if T == 4096 else 0)
    for i in range(11, -1, -1):                      # u < T, from the lowest digit up
        x = (words[i] | x) if T == 4096 or (T >> (11 - i)) & 1 else (words[i] & x)
    mask = torch.empty(rows, G, 32, dtype=torch.bool, device=DEV)
    for c in range(32):
        mask[:, :, c] = ((x >> c) & 1).bool()
    return mask.view(rows, G * 32)[:, :D].expand(B, D), 4096.0 / T


def _dact(act, z):
    """Derivative of the activation at pre-activation z."""
    if act == "relu":
        return (z > 0).double()
    return 0.5 * (1 + torch.erf(z / math.sqrt(2))) + z * torch.exp(-0.5 * z * z) / math.sqrt(2 * math.pi)


def _act(act, z):
    return z.relu() if act == "relu" else 0.5 * z * (1 + torch.erf(z / math.sqrt(2)))


def _xent(z, y):
    lp = torch.log_softmax(z, 1)
    n = torch.arange(z.shape[0], device=DEV)
    loss = -lp[n, y.long()].mean().reshape(1)
    dz = lp.exp()
    dz[n, y.long()] -= 1
    return loss, dz / z.shape[0]


def _sampled(case, A, seed, layer, step=MASK_STEP):
    keep, scale = _keep(case["variant"], A.shape[0], A[0].numel(), case["p"], seed, layer, step)
    return torch.where(keep.view(A.shape), A * scale, torch.zeros((), dtype=A.dtype, device=DEV))


def _exact_mlp(case, i, seed):
    A, As, zs = i["X"].double(), [], []
    L = len(i["Ws"])
    for l in range(L):
        As.append(A)
        z = A @ i["Ws"][l].double() + i["bs"][l].double()
        zs.append(z)
        A = _act(case["act"], z) if l < L - 1 else z
    loss, dz = _xent(zs[-1], i["y"])
    dW, db = [None] * L, [None] * L
    for l in range(L - 1, -1, -1):
        # a sign that falls the other way in 32 bits says nothing of the precision: float32 ReLU nets are
        # compared down to their last hidden layer, bf16 nets (whose rounding dominates) and GELU nets whole
        if l == L - 1 or case["dtype"] == "bf16" or case["act"] == "gelu":
            dW[l], db[l] = _sampled(case, As[l], seed, l).T @ dz, dz.sum(0)
        if l > 0:
            dz = (dz @ i["Ws"][l].double().T) * _dact(case["act"], zs[l - 1])
        As[l] = None
    return dict(loss=loss, dW=dW, db=db, nnz=None, status=None)


def _exact_irnn(case, i, seed):
    d = {n: v.double() for n, v in i.items() if n != "y"}
    T, hs = case["steps"], [torch.zeros(case["batch"], case["hidden"], device=DEV, dtype=torch.float64)]
    for t in range(T):
        hs.append((d["x"][:, t:t + 1] * d["W_ih"] + d["b_ih"] + hs[-1] @ d["W_hh"] + d["b_hh"]).relu())
    loss, dl = _xent(hs[T] @ d["W_out"] + d["b_out"], i["y"])
    dW_out, dh = _sampled(case, hs[T], seed, 1).T @ dl, dl @ d["W_out"].T
    dW_hh, dW_ih, db = torch.zeros_like(d["W_hh"]), torch.zeros_like(d["W_ih"]), torch.zeros_like(d["b_ih"])
    for t in range(T, 0, -1):
        dz = dh * (hs[t] > 0)
        dW_hh += _sampled(case, hs[t - 1], seed, 0, MASK_STEP + t).T @ dz
        dW_ih += d["x"][:, t - 1] @ dz
        db += dz.sum(0)
        dh = dz @ d["W_hh"].T
    return dict(loss=loss, dW_ih=dW_ih, db=db, dW_hh=dW_hh, dW_out=dW_out, db_out=dl.sum(0), nnz=None, status=None)


def _taps(X):
    """The nine shifted views of an NHWC tensor under zero padding 1, tap by tap."""
    B, H, W, C = X.shape
    P = torch.zeros(B, H + 2, W + 2, C, dtype=X.dtype, device=DEV)
    P[:, 1:-1, 1:-1] = X
    return [(ky, kx, P[:, ky:ky + H, kx:kx + W].reshape(-1, C)) for ky in range(3) for kx in range(3)]


def _exact_cnn(case, i, seed):
    A, ins, signs, whole = i["X"].double(), [], [], case["dtype"] == "bf16"
    nc, nf = len(i["cW"]), len(i["fW"])
    for l in range(nc):
        B, H, W, _ = A.shape
        ins.append(A)
        z = sum(x @ i["cW"][l][ky, kx].double() for ky, kx, x in _taps(A)) + i["cb"][l].double()
        z = z.view(B, H, W, -1)
        signs.append(z > 0)
        A = z.relu().view(B, H // 2, 2, W // 2, 2, -1).mean((2, 4))
    shape, F, zs = A.shape, [A.reshape(A.shape[0], -1)], []
    for l in range(nf):
        zs.append(F[l] @ i["fW"][l].double() + i["fb"][l].double())
        F.append(zs[l].relu())
    loss, dz = _xent(zs[-1], i["y"])
    fdW, fdb, cdW, cdb = [None] * nf, [None] * nf, [None] * nc, [None] * nc
    for l in range(nf - 1, -1, -1):
        if whole or l == nf - 1:
            fdW[l], fdb[l] = _sampled(case, F[l], seed, nc + l).T @ dz, dz.sum(0)
        dz = dz @ i["fW"][l].double().T
        if l > 0:
            dz = dz * (zs[l - 1] > 0)
    dP = dz.view(shape)
    for l in range(nc - 1, -1, -1) if whole else ():
        dZ = 0.25 * dP.repeat_interleave(2, 1).repeat_interleave(2, 2) * signs[l]
        flat, Wt = dZ.reshape(-1, dZ.shape[3]), i["cW"][l].double()
        cdW[l] = torch.stack([x.T @ flat for _, _, x in _taps(_sampled(case, ins[l], seed, l))]).view(Wt.shape)
        cdb[l] = flat.sum(0)
        if l > 0:
            dP = sum(x @ Wt[2 - ky, 2 - kx].T for ky, kx, x in _taps(dZ)).view(ins[l].shape)
    return dict(loss=loss, conv_dW=cdW, conv_db=cdb, fc_dW=fdW, fc_db=fdb, nnz=None, status=None)


def _exact_layer(case, i, seed):
    act = case["act"]
    z = i["A"].double() @ i["W"].double() + i["b"].double()
    dZ = i["dZ"].double()
    dZp = (dZ @ i["W"].double().T) * ((i["A"] > 0) if act == "relu" else _dact(act, i["z"].double()))
    return dict(out=_act(act, z), zlow=None if act == "relu" else z, bits=None, next_values=None, next_keepbits=None,
                next_offsets=None, next_nnz=None, dW=_sampled(case, i["A"].double(), seed, 1).T @ dZ, dZ_prev=dZp,
                db=dZ.sum(0), status=None)


def exact(case, seed):
    if case["kind"] == "store" or case.get("law", "bernoulli") != "bernoulli":
        return None
    fn = dict(mlp=_exact_mlp, irnn=_exact_irnn, cnn=_exact_cnn, layer=_exact_layer)[case["kind"]]
    return fn(case, _inputs(case, seed), seed)
