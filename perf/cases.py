"""What is measured: the work that a user of this library has it do, as cases of plain values.

A case is one of five kinds:

* ``dense``   a few steps of local / post-local SGD on a dense network and the read of the model they
              end with: the library's main path (lsgd_run on a resident dataset, lsgd_run_batch on
              mini-batches that the caller holds on the GPU);
* ``resnet``  the same on ResNet-20;
* ``gemm``    one dense layer's three products (forward, data gradient, weight gradient) for all
              workers through lsgd_grouped_gemm_bf16;
* ``conv``    one 3x3 convolution layer: forward with BatchNorm statistics, data gradient, weight
              gradient;
* ``update``  the local update and the K-way average over a caller's own K x d buffers.

A training case's outputs are the model after its last average and every worker's loss of every
step.  Its steps include at least one update that uses the momentum of an earlier one where there are two
or more, so the optimizer's state shows in the model.
"""
import math

import numpy as np
import torch

import paper_1808_07217_gb300 as lsgd

# ------------------------------------------------------------------------------------- the cases


def _dense(name, widths, K, B, steps, H, **kw):
    c = dict(name=name, kind="dense", widths=",".join(str(w) for w in widths), K=K, B=B, steps=steps,
             H=H, t_switch=-1, precision="bf16", fused=True, momentum=0.9, nesterov=True, lr=0.02,
             weight_decay=5e-4, sync="plain", source="dataset", N=4096)
    c.update(kw)
    return c


def _resnet(name, K, B, steps, H, **kw):
    c = dict(name=name, kind="resnet", K=K, B=B, steps=steps, H=H, t_switch=-1, precision="bf16",
             momentum=0.9, nesterov=True, lr=0.02, weight_decay=1e-4, source="batch")
    c.update(kw)
    return c


def listed():
    return [
        # the smallest training job: softmax regression in fp32 on few workers, one round of local
        # steps.  Latency and the number of launches count.
        _dense("softmax_fp32", (3072, 10), K=4, B=32, steps=4, H=4, precision="fp32", fused=False,
               momentum=0.0, nesterov=False, lr=0.05),
        # the K x H trade-off's network: small layers, many short steps, heavy ball
        _dense("mlp512_round", (3072, 512, 512, 10), K=8, B=32, steps=4, H=4, nesterov=False),
        # the ordinary job: local SGD on the 1024-wide network, one round of four steps
        _dense("mlp1024_round", (3072, 1024, 1024, 10), K=16, B=128, steps=4, H=4),
        # the largest: post-local SGD across its switch (two steps that each end with the average,
        # then a round of two local steps)
        _dense("mlp4096_postlocal", (3072, 4096, 4096, 4096, 100), K=16, B=128, steps=4, H=2, t_switch=2),
        # the paper's own precision: everything in fp32
        _dense("mlp1024_fp32", (3072, 1024, 1024, 10), K=4, B=64, steps=2, H=2, precision="fp32",
               fused=False, source="batch"),
        # ragged widths and batch, an odd number of workers, compressed averaging with error
        # feedback, the stand-alone update, mini-batches from the caller
        _dense("ragged_ef_sign", (776, 520, 264, 17), K=5, B=50, steps=4, H=2, fused=False,
               sync="ef_sign", source="batch"),
        # ResNet-20 on 32 x 32 images at the paper's K and B, one round of two steps
        _resnet("resnet20_round", K=16, B=128, steps=2, H=2),
        # the same network in fp32 on a few workers
        _resnet("resnet20_fp32", K=4, B=64, steps=2, H=2, precision="fp32"),
        # a dense layer's products on their own, ragged in every extent
        dict(name="gemm_ragged", kind="gemm", G=6, B=100, n_in=1032, n_out=776),
        # a first-stage ResNet-20 layer for 16 workers
        dict(name="conv_stage1", kind="conv", G=16, B=128, hw=32, cin=16, cout=16, stride=1),
        # a stage's first layer: stride 2, twice the channels, an odd batch
        dict(name="conv_stride2", kind="conv", G=5, B=51, hw=32, cin=16, cout=32, stride=2),
        # update and average of a caller's own buffers, an odd number of workers
        dict(name="update_average", kind="update", K=11, d=3_000_004, nesterov=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("dense", "dense", "dense32", "resnet", "resnet32", "gemm", "conv", "update"))
    if kind in ("dense", "dense32"):
        fp32 = kind == "dense32"
        K = _log_int(rng, 1, 6 if fp32 else 16)
        B = _log_int(rng, 4, 96) if fp32 else _log_int(rng, 8, 160)
        layers = rng.randint(1, 4)
        top = 1024 if fp32 else 2304
        widths = [_log_int(rng, 48, 3072)] + [_log_int(rng, 48, top) for _ in range(layers - 1)]
        if not fp32:  # bf16 layers take inputs that are a multiple of 8 wide
            widths = [max(8, w // 8 * 8) for w in widths]
        widths.append(_log_int(rng, 2, 200))
        steps = rng.randint(2, 4)
        sync = rng.choice(("plain", "plain", "ef_sign", "global_momentum"))
        momentum = rng.choice((0.0, 0.9, 0.9))
        c = _dense("", widths, K, B, steps, rng.randint(1, steps), precision="fp32" if fp32 else "bf16",
                   fused=not fp32 and rng.random() < 0.75, momentum=momentum,
                   nesterov=momentum > 0 and rng.random() < 0.5, sync=sync,
                   t_switch=rng.choice((-1, 1)), source=rng.choice(("dataset", "batch")),
                   N=rng.randint(1024, 4096))
        del c["name"]
        return c
    if kind in ("resnet", "resnet32"):
        fp32 = kind == "resnet32"
        c = _resnet("", _log_int(rng, 2, 4) if fp32 else _log_int(rng, 1, 12),
                    _log_int(rng, 24, 64) if fp32 else _log_int(rng, 8, 96), 2, rng.randint(1, 2),
                    precision="fp32" if fp32 else "bf16")
        del c["name"]
        return c
    if kind == "gemm":
        return dict(kind="gemm", G=_log_int(rng, 1, 16), B=_log_int(rng, 16, 300),
                    n_in=8 * _log_int(rng, 8, 384), n_out=8 * _log_int(rng, 8, 256))
    if kind == "conv":
        hw, cin, cout, stride = rng.choice(((32, 3, 16, 1), (32, 16, 16, 1), (32, 16, 32, 2), (16, 32, 32, 1),
                                            (16, 32, 64, 2), (8, 64, 64, 1)))
        return dict(kind="conv", G=_log_int(rng, 1, 16), B=2 * _log_int(rng, 4, 64), hw=hw, cin=cin,
                    cout=cout, stride=stride)
    return dict(kind="update", K=_log_int(rng, 2, 32), d=4 * _log_int(rng, 4096, 1_000_000),
                nesterov=rng.random() < 0.5)


# --------------------------------------------------------------------------- inputs from the seed


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _randint(g, hi, *shape):
    return torch.randint(0, hi, shape, generator=g, device="cuda", dtype=torch.int32)


def _mixture(g, n, dim, classes):
    """n points of a Gaussian mixture with one centre per class, and their labels."""
    y = _randint(g, classes, n)
    return _randn(g, n, dim) + 0.5 * _randn(g, classes, dim)[y.long()], y


def _widths(case):
    return [int(w) for w in case["widths"].split(",")]


# ResNet-20's 3x3 convolutions (cin, cout, stride), stem first
_CONVS = [(3, 16, 1)] + [(cin, cout, s) for st in range(3) for b in range(3)
                         for cin, cout, s in ((16 << (st - 1) if st and not b else 16 << st, 16 << st,
                                               2 if st and not b else 1), (16 << st, 16 << st, 1))]


def _start_model(case, g):
    """A start model in the library's packed order: He-normal weights, zero biases (a little away
    from zero so that every parameter matters)."""
    parts = []
    if case["kind"] == "dense":
        w = _widths(case)
        for i, o in zip(w[:-1], w[1:]):
            parts += [math.sqrt(2.0 / i) * _randn(g, o * i), 0.01 * _randn(g, o)]
    else:
        for cin, cout, _ in _CONVS:
            parts += [math.sqrt(2.0 / (9 * cin)) * _randn(g, cout * 9 * cin),
                      1 + 0.1 * _randn(g, cout), 0.1 * _randn(g, cout)]
        parts += [0.1 * _randn(g, 10 * 64), 0.01 * _randn(g, 10)]
    return torch.cat(parts)


def _train_inputs(case, seed):
    """(start model, data, labels): a dataset of N points, or the mini-batches of every step."""
    g = _gen(seed)
    w0 = _start_model(case, g)
    dim, classes = (_widths(case)[0], _widths(case)[-1]) if case["kind"] == "dense" else (3072, 10)
    if case["source"] == "dataset":
        x, y = _mixture(g, case["N"], dim, classes)
    else:
        n = case["steps"] * case["K"] * case["B"]
        x, y = _mixture(g, n, dim, classes)
        x = x.reshape(case["steps"], case["K"], case["B"], dim)
        y = y.reshape(case["steps"], case["K"], case["B"])
    return w0, x.contiguous(), y.contiguous()


_SYNC = {"plain": {}, "ef_sign": dict(compress=lsgd.COMPRESS_EF_SIGN), "global_momentum": dict(global_momentum=0.3)}


def _train_state(case, seed):
    w0, x, y = _train_inputs(case, seed)
    data = case["source"] == "dataset"
    kw = dict(K=case["K"], B_loc=case["B"], H=case["H"], t_switch=case["t_switch"],
              total_steps=case["steps"], N=case["N"] if data else max(case["K"], 64), base_lr=case["lr"],
              momentum=case["momentum"], nesterov=case["nesterov"], weight_decay=case["weight_decay"],
              seed=seed, precision=lsgd.BF16 if case["precision"] == "bf16" else lsgd.FP32)
    if case["kind"] == "dense":
        kw.update(kind=lsgd.MLP, widths=_widths(case), fused_update=case["fused"], **_SYNC[case["sync"]])
    else:
        kw.update(kind=lsgd.RESNET20)
    ctx = lsgd.lsgd_create(lsgd.make_config(init=lsgd.INIT_ZERO, **kw))
    lsgd.lsgd_set_params(ctx, -1, w0.cpu().numpy())
    if data:
        lsgd.lsgd_set_dataset(ctx, x.cpu().numpy(), y.cpu().numpy())
    return dict(case=case, ctx=ctx, x=x, y=y, model=torch.empty_like(w0),
                losses=torch.empty(case["steps"], case["K"], pin_memory=True))


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("dense", "resnet"):
        return _train_state(case, seed)
    g = _gen(seed)
    if kind == "gemm":
        G, B, i, o = case["G"], case["B"], case["n_in"], case["n_out"]
        return dict(case=case, act=torch.relu(_randn(g, G, B, i)).bfloat16(),
                    w=(_randn(g, G, o, i) * math.sqrt(2.0 / i)).bfloat16(),
                    dz=(_randn(g, G, B, o) / B).bfloat16(), z=torch.empty(G, B, o, device="cuda"),
                    da=torch.empty(G, B, i, device="cuda"), dw=torch.empty(G, o, i, device="cuda"))
    if kind == "conv":
        G, B, hw, ci, co, s = (case[k] for k in ("G", "B", "hw", "cin", "cout", "stride"))
        ho = hw // s
        x = _randn(g, G, B, hw, hw, ci) if ci < 16 else torch.relu(_randn(g, G, B, hw, hw, ci))
        e = dict(device="cuda")
        return dict(case=case, x=x.bfloat16(), w=(_randn(g, G, co, 3, 3, ci) * math.sqrt(2.0 / (9 * ci))).bfloat16(),
                    dy=(_randn(g, G, B, ho, ho, co) / B).bfloat16(), y=torch.empty(G, B, ho, ho, co, **e),
                    mean=torch.empty(G, co, **e), rstd=torch.empty(G, co, **e),
                    dx=torch.empty(G, B, hw, hw, ci, **e), dw=torch.empty(G, co, 3, 3, ci, **e))
    K, d = case["K"], case["d"]
    w0 = 0.03 * _randn(g, d)
    return dict(case=case, w=(w0 + 1e-3 * _randn(g, K, d)).contiguous(), u=1e-2 * _randn(g, K, d),
                g=1e-2 * _randn(g, K, d), wb=torch.empty(K, d, device="cuda", dtype=torch.bfloat16))


# ------------------------------------------------------------------------------------- one pass

_LR, _MOM, _WD = 0.1, 0.9, 5e-4  # the update case's step


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("dense", "resnet"):
        ctx, steps = state["ctx"], case["steps"]
        lsgd.lsgd_set_step(ctx, 0)
        if case["source"] == "dataset":
            lsgd.lsgd_run(ctx, steps)
        else:
            for s in range(steps):
                lsgd.lsgd_run_batch(ctx, state["x"][s], state["y"][s])
        lsgd.lsgd_losses_async(ctx, state["losses"], steps)
        lsgd.lsgd_params(ctx, 0, state["model"])
        return dict(model=state["model"], losses=state["losses"])
    if kind == "gemm":
        G, B, i, o = case["G"], case["B"], case["n_in"], case["n_out"]
        lsgd.lsgd_grouped_gemm_bf16(state["act"], False, state["w"], False, state["z"], B, o, i, G)
        lsgd.lsgd_grouped_gemm_bf16(state["dz"], False, state["w"], True, state["da"], B, i, o, G)
        lsgd.lsgd_grouped_gemm_bf16(state["dz"], True, state["act"], True, state["dw"], o, i, B, G)
        return dict(z=state["z"], da=state["da"], dw=state["dw"])
    if kind == "conv":
        G, B, hw, ci, co, s = (case[k] for k in ("G", "B", "hw", "cin", "cout", "stride"))
        lsgd.lsgd_conv3x3_bn_bf16(state["x"], state["w"], state["y"], state["mean"], state["rstd"], G, B,
                                  hw, hw, ci, co, s)
        out = dict(y=state["y"], mean=state["mean"], rstd=state["rstd"])
        if ci >= 16:  # the stem has no data gradient, and its weight gradient is the network's own
            lsgd.lsgd_conv3x3_bf16(lsgd.CONV_DGRAD, state["dy"], state["w"], state["dx"], G, B, hw, hw, ci,
                                   co, s)
            lsgd.lsgd_conv_wgrad_bf16(state["x"], state["dy"], state["dw"], G, B, hw // s, hw // s, ci, co, s)
            out.update(dx=state["dx"], dw=state["dw"])
        return out
    K, d = case["K"], case["d"]
    lsgd.lsgd_sgd_update(state["w"], state["u"], state["g"], state["wb"], K * d, _LR, _MOM, case["nesterov"],
                         _WD)
    lsgd.lsgd_kway_average(state["w"], state["wb"], K, d)
    return dict(w=state["w"], u=state["u"], wb=state["wb"])


# ------------------------------------------------------------------- bytes and operations of one


def _round_ends(case):
    """For every step, whether the average follows it."""
    T, t, H = case["steps"], case["t_switch"], case["H"]
    return [s == T - 1 or s < t or (s + 1 - max(t, 0)) % H == 0 for s in range(T)]


def work(case):
    kind = case["kind"]
    if kind in ("dense", "resnet"):
        K, B = case["K"], case["B"]
        if kind == "dense":
            w = _widths(case)
            d = sum(i * o + o for i, o in zip(w[:-1], w[1:]))
            dim = w[0]
            macs = 3 * sum(i * o for i, o in zip(w[:-1], w[1:])) - w[0] * w[1]
        else:
            d = sum(9 * i * o + 2 * o for i, o, _ in _CONVS) + 650
            dim, macs, hw = 3072, 3 * 640, 32
            for n, (i, o, s) in enumerate(_CONVS):
                hw //= s
                macs += 9 * i * o * hw * hw * (2 if n == 0 else 3)
        # per step: the mini-batch and the momentum, once in and (momentum) out; a worker's own
        # model in and out, or one model where all workers hold the same
        nbytes, same = 0, True
        for end in _round_ends(case):
            nbytes += 4 * K * B * dim + (8 * K * d if case["momentum"] else 0)
            nbytes += 4 * d * ((1 if same else K) + (1 if end else K))
            same = end
        return {"bytes": nbytes, "flops": 2 * macs * K * B * case["steps"]}
    if kind == "gemm":
        G, B, i, o = case["G"], case["B"], case["n_in"], case["n_out"]
        return {"bytes": G * (2 * (B * i + o * i + B * o) + 4 * (B * o + B * i + o * i)), "flops": 6 * G * B * i * o}
    if kind == "conv":
        G, B, hw, ci, co, s = (case[k] for k in ("G", "B", "hw", "cin", "cout", "stride"))
        pi, po, wn = B * hw * hw * ci, B * (hw // s) ** 2 * co, 9 * ci * co
        fl = 2 * G * B * (hw // s) ** 2 * wn
        if ci < 16:
            return {"bytes": G * (2 * (pi + wn) + 4 * po), "flops": fl}
        return {"bytes": G * (2 * (pi + po + wn) + 4 * (pi + po + wn)), "flops": 3 * fl}
    # w, u, g in; u out; the mean and its bf16 copy out for every worker
    return {"bytes": case["K"] * case["d"] * (12 + 4 + 4 + 2), "flops": 8 * case["K"] * case["d"]}


def tolerance(case):
    """Four times what two correct implementations (the tensor-core and the SIMT products, both with
    bf16 operands), or where there is one only this one and 64 bits, were seen to differ by."""
    kind = case["kind"]
    if kind == "gemm":  # 7e-7 from 64 bits
        return {"rel": 6e-6, "max": 1e-4}
    if kind == "conv":  # 6e-6 (a weight gradient over 131,072 pixels)
        return {"rel": 2.4e-5, "max": 2e-4}
    if kind == "update":  # a few bf16 copies off by their last bit
        return {"rel": 1e-4, "max": 8e-3}
    if case.get("sync") == "ef_sign":  # differences near zero change sign
        return {"rel": 4e-3, "max": 0.3} if case["precision"] == "bf16" else {"rel": 2e-5, "max": 0.3}
    if case["precision"] == "fp32":  # ResNet-20: pre-activations near zero pass the ReLU or do not
        return {"rel": 4e-7, "max": 4e-6} if kind == "dense" else {"rel": 1e-4, "max": 5e-3}
    return {"rel": 1.2e-3, "max": 4e-2} if kind == "dense" else {"rel": 2.2e-3, "max": 8e-2}


# -------------------------------------------------------------- the same in 64 bits, in plain torch

_F64 = dict(dtype=torch.float64, device="cuda")


def _philox(ctr, key):
    """Philox4x32-10 (Salmon et al. 2011) on arrays of 32-bit counter words."""
    x, y, z, w = (np.asarray(v, dtype=np.uint64) for v in ctr)
    k0, k1 = key & 0xFFFFFFFF, key >> 32
    mask = np.uint64(0xFFFFFFFF)
    for _ in range(10):
        a, b = np.uint64(0xD2511F53) * x, np.uint64(0xCD9E8D57) * z
        x, y, z, w = (b >> np.uint64(32)) ^ y ^ np.uint64(k0), b & mask, (a >> np.uint64(32)) ^ w ^ np.uint64(k1), a & mask
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return [x, y, z, w]


def _indices(case, seed, step):
    """Every worker's mini-batch of a step: B uniform draws from its own shard of the dataset."""
    K, B, S = case["K"], case["B"], case["N"] // case["K"]
    j, k = np.meshgrid(np.arange((B + 3) // 4), np.arange(K))
    zero = np.zeros_like(j)
    words = np.stack(_philox((j, zero + step, k, zero), seed), -1).reshape(K, -1)[:, :B]
    return torch.from_numpy((np.arange(K)[:, None] * S + ((words * np.uint64(S)) >> np.uint64(32)).astype(np.int64))).cuda()


def _softmax_grad(z, y):
    """Mean loss per worker and its gradient with respect to the logits z [K][B][C]."""
    lse = torch.logsumexp(z, -1, keepdim=True)
    one = torch.nn.functional.one_hot(y.long(), z.shape[-1])
    loss = (lse.squeeze(-1) - (z * one).sum(-1)).mean(-1)
    return loss, (torch.exp(z - lse) - one) / z.shape[1]


def _dense_grad(case, w, x, y):
    """Losses [K] and gradients [K][d] of the dense ReLU network with parameters w [K][d]."""
    wd, acts, layers, at = _widths(case), [x], [], 0
    for i, o in zip(wd[:-1], wd[1:]):
        layers.append((at, i, o))
        at += i * o + o
    W = lambda l: w[:, l[0]:l[0] + l[1] * l[2]].reshape(-1, l[2], l[1])  # noqa: E731
    for n, l in enumerate(layers):
        z = torch.bmm(acts[-1], W(l).transpose(1, 2)) + w[:, l[0] + l[1] * l[2]:l[0] + l[1] * l[2] + l[2]].unsqueeze(1)
        acts.append(z if n == len(layers) - 1 else torch.relu(z))
    loss, dz = _softmax_grad(acts[-1], y)
    g = torch.empty_like(w)
    for n in range(len(layers) - 1, -1, -1):
        a, i, o = layers[n]
        g[:, a:a + i * o] = torch.bmm(dz.transpose(1, 2), acts[n]).reshape(len(g), -1)
        g[:, a + i * o:a + i * o + o] = dz.sum(1)
        if n:
            dz = torch.bmm(dz, W(layers[n])) * (acts[n] > 0)
    return loss, g


def _conv(x, w, stride):
    """3x3 convolution, padding 1: x [B][H][W][ci], w [co][3][3][ci]."""
    ho, wo = (x.shape[1] - 1) // stride + 1, (x.shape[2] - 1) // stride + 1
    p = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1))
    cols = [p[:, kh:kh + (ho - 1) * stride + 1:stride, kw:kw + (wo - 1) * stride + 1:stride]
            for kh in range(3) for kw in range(3)]
    return torch.cat(cols, -1) @ w.reshape(w.shape[0], -1).t()


def _resnet_grad(w, x, y):
    """Loss and gradient of one worker's ResNet-20 (w [d], x [B][3072])."""
    w = w.clone().requires_grad_(True)
    at, par = 0, []

    def take(*shape):
        nonlocal at
        n = math.prod(shape)
        at += n
        return w[at - n:at].reshape(shape)

    for ci, co, _ in _CONVS:
        par.append((take(co, 3, 3, ci), take(co), take(co)))
    fw, fb = take(10, 64), take(10)

    def unit(h, n, extra=None):
        z = _conv(h, par[n][0], _CONVS[n][2])
        mu, var = z.mean((0, 1, 2)), z.var((0, 1, 2), unbiased=False)
        z = (z - mu) / torch.sqrt(var + 1e-5) * par[n][1] + par[n][2]
        return torch.relu(z if extra is None else z + extra)

    h = unit(x.reshape(-1, 32, 32, 3), 0)
    for n in range(1, 19, 2):
        s, grow = _CONVS[n][2], _CONVS[n][1] - _CONVS[n][0]
        short = torch.nn.functional.pad(h[:, ::s, ::s], (0, grow))
        h = unit(unit(h, n), n + 1, short)
    z = h.mean((1, 2)) @ fw.t() + fb
    loss = torch.nn.functional.cross_entropy(z, y.long())
    loss.backward()
    return loss.detach(), w.grad


def _train_exact(case, seed):
    w0, x, y = _train_inputs(case, seed)
    K, lr, m = case["K"], case["lr"], case["momentum"]
    w = w0.double().repeat(K, 1)
    wref, e, ug = w[0].clone(), torch.zeros_like(w), torch.zeros_like(w[0])
    u = torch.zeros_like(w)
    decay = torch.full_like(w[0], case["weight_decay"])
    if case["kind"] == "resnet":  # none on BatchNorm's scale and shift
        at = 0
        for ci, co, _ in _CONVS:
            decay[at + 9 * ci * co:at + 9 * ci * co + 2 * co] = 0
            at += 9 * ci * co + 2 * co
    losses = []
    for s, end in enumerate(_round_ends(case)):
        if case["source"] == "dataset":
            idx = _indices(case, seed, s)
            xs, ys = x[idx].double(), y[idx]
        else:
            xs, ys = x[s].double(), y[s]
        if case["kind"] == "dense":
            loss, g = _dense_grad(case, w, xs, ys)
        else:
            one = [_resnet_grad(w[k], xs[k], ys[k]) for k in range(K)]
            loss, g = torch.stack([a for a, _ in one]), torch.stack([b for _, b in one])
        losses.append(loss)
        g += decay * w
        u = m * u + g
        w -= lr * (g + m * u if case["nesterov"] else u)
        if not end:
            continue
        sync = case.get("sync", "plain")
        if sync == "plain":
            w[:] = w.mean(0)
        elif sync == "global_momentum":
            ug = 0.3 * ug + (wref - w.mean(0)) / lr
            wref = wref - lr * ug
            w[:] = wref
        else:
            delta = wref - w + e
            p = delta.abs().mean(1, keepdim=True)
            e = delta - torch.sign(delta) * p
            wref = wref - (torch.sign(delta) * p).mean(0)
            w[:] = wref
    return dict(model=w[0].clone(), losses=torch.stack(losses).cpu())


def exact(case, seed):
    kind = case["kind"]
    if kind in ("dense", "resnet"):
        return _train_exact(case, seed)
    s = prepare(case, seed)
    if kind == "gemm":
        a, w, dz = s["act"].double(), s["w"].double(), s["dz"].double()
        return dict(z=a @ w.transpose(1, 2), da=dz @ w, dw=dz.transpose(1, 2) @ a)
    if kind == "conv":
        y, mean, rstd, dx, dw = [], [], [], [], []
        for g in range(case["G"]):
            x, w = s["x"][g].double().requires_grad_(True), s["w"][g].double().requires_grad_(True)
            v = _conv(x, w, case["stride"])
            v.backward(s["dy"][g].double())
            v = v.detach()
            y.append(v)
            mean.append(v.mean((0, 1, 2)))
            rstd.append(1 / torch.sqrt(v.var((0, 1, 2), unbiased=False) + 1e-5))
            dx.append(x.grad)
            dw.append(w.grad)
        out = dict(y=torch.stack(y), mean=torch.stack(mean), rstd=torch.stack(rstd))
        if case["cin"] >= 16:
            out.update(dx=torch.stack(dx), dw=torch.stack(dw))
        return out
    w, u, g = s["w"].double(), s["u"].double(), s["g"].double()
    g = g + _WD * w
    u = _MOM * u + g
    w = w - _LR * (g + _MOM * u if case["nesterov"] else u)
    w = w.mean(0, keepdim=True).expand_as(w).contiguous()
    return dict(w=w, u=u, wb=w)
