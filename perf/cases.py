"""Work that a user has this library do: local SGD steps of sub-ResNets (grouped or one worker's), whole rounds, the
synchronisation alone, evaluation of the reassembled network, and single layers.

Architectures, batch sizes and S are those of `synth.config` (tiny fp32 net, CIFAR ResNet-110, wide CIFAR bottleneck net,
ImageNet-shaped ResNet-101, reassembly set) or other sizes of the same families.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2107_00961_b200 as resist
import synth

# A warm-up learning rate: at 0.1 from a random start, the second of two steps already amplifies single bf16 roundings (a flipped
# ReLU mask is a changed gradient) beyond what two correct implementations can be compared on.
LR = 0.001


def listed():
    return [
        # the smallest training call: the 8x8 fp32 net of the protocol tests, S = 2, batch 8; launches and latency count
        dict(name="step_tiny_f32", kind="step", net="basic", n=2, width=8, hw=8, classes=10, policy="stage", S=2, B=8, dtype="f32"),
        # the inner loop of CIFAR training with ResNet-110 (narrow layers, long chain), all four sub-ResNets at once
        dict(name="step_resnet110", kind="step", net="basic", n=18, width=16, hw=32, classes=10, policy="stage", S=4, B=128, dtype="bf16"),
        # one worker stepping alone on the last, smaller batch of its shard (50000 images / 4 = 97 batches of 128 and one of 84)
        dict(name="worker_resnet110_b84", kind="worker", net="basic", n=18, width=16, hw=32, classes=10, policy="stage", S=4, B=84, dtype="bf16"),
        # the flagship workload: wide bottleneck net, S = 8, batch 128
        dict(name="step_wide", kind="step", net="wide", d2=4, d3=23, width=64, hw=32, classes=100, policy="section3", S=8, B=128, dtype="bf16"),
        # the local-SGD mode on the same net (no block dealt out), ragged batch
        dict(name="step_wide_localsgd", kind="step", net="wide", d2=4, d3=23, width=64, hw=32, classes=100, policy="none", S=3, B=100, dtype="bf16"),
        # ImageNet-shaped training: large maps, 7x7 stem, max-pool
        dict(name="step_imagenet", kind="step", net="imagenet", d2=4, d3=23, width=64, hw=224, classes=1000, policy="section3", S=4, B=64, dtype="bf16"),
        # a whole round with a single local step at batch 32: partition, first step on the new partition, reassembly
        dict(name="round_resnet101", kind="round", net="imagenet", d2=4, d3=23, width=64, hw=224, classes=1000, policy="section3", S=4, B=32, dtype="bf16"),
        # the synchronisation alone on the ResNet-101 parameters: reassembly, then the next partition
        dict(name="sync_resnet101", kind="sync", net="imagenet", d2=4, d3=23, width=64, hw=224, classes=1000, policy="section3", S=8, B=2, dtype="bf16"),
        # validation between rounds: the full ResNet-110 on 1000 test images
        dict(name="eval_resnet110", kind="eval", net="basic", n=18, width=16, hw=32, classes=10, policy="stage", S=4, B=1000, dtype="bf16"),
        # validation on ImageNet shapes with the shorter third section of ResNet-50, in batches of 50 (1000 of them cover 50000 images)
        dict(name="eval_imagenet_b50", kind="eval", net="imagenet", d2=4, d3=6, width=64, hw=224, classes=1000, policy="section3", S=4, B=50, dtype="bf16"),
        # one 3x3 layer of the wide net's second section on its own: forward, data gradient and weight gradient
        dict(name="layer_conv3x3", kind="conv", N=128, H=16, W=16, C=128, K=128, ksz=3, stride=1, dtype="bf16"),
        # one BN+ReLU on its own (the wide net's first section at batch 64), forward and backward, odd number of rows
        dict(name="layer_bn", kind="bn", m=65535, C=64, dtype="bf16"),
    ]


def draw(rng):
    """The same kinds of work at other sizes: batch, S, depth, width, input size, dtype and layer shapes."""
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step"] * 5 + ["worker", "round", "sync", "eval", "conv", "bn"])
    if kind == "conv":
        hw, s = log(4, 56), rng.choice([1, 1, 1, 2])
        C = 8 * log(2, 64)
        K = rng.choice([C, C, 4 * C, max(16, C // 4 // 8 * 8)])
        return dict(kind="conv", N=log(1, 256 if hw < 33 else 48), H=hw, W=max(4, hw + rng.choice([0, 0, -1, 3])), C=C, K=min(K, 1024),
                    ksz=3 if K == C else rng.choice([1, 1, 3]), stride=s, dtype="bf16")
    if kind == "bn":
        C = rng.choice([16, 32, 64, 128, 256, 512, 1024, 24, 72, 100])
        return dict(kind="bn", m=log(64, 2 ** 26 // C), C=C, dtype=rng.choice(["bf16", "bf16", "f32"]))
    net = rng.choice(["basic", "wide", "imagenet"] if kind != "sync" else ["wide", "imagenet"])
    S = rng.randint(1, 8)
    c = dict(kind=kind, net=net, classes=rng.choice([10, 100, 1000]), S=S, policy=rng.choice(["stage", "section3", "section3"]), dtype="bf16")
    if net == "basic":
        c.update(n=rng.randint(4, 18), width=rng.choice([8, 16, 16, 16]), hw=rng.choice([24, 28, 32, 32, 36]), B=log(8, 256), policy="stage")
        if rng.random() < 0.25:
            c.update(dtype="f32", n=rng.randint(2, 4), width=8, hw=rng.choice([8, 16]), S=min(S, 3), B=log(4, 64))
    elif net == "wide":
        c.update(d2=rng.randint(2, 4), d3=rng.randint(9, 12), width=rng.choice([32, 64]), hw=rng.choice([24, 32, 32]), B=log(16, 128))
    else:
        c.update(d2=rng.randint(2, 4), d3=rng.randint(9, 12), width=rng.choice([32, 64]), hw=rng.choice([96, 112, 160, 192, 224]), B=log(16, 64))
    if kind == "eval":
        c["B"] = min(4 * c["B"], 512)
    if kind == "sync":
        c["B"] = 2
    if kind == "step" and net != "basic" and rng.random() < 0.2:
        c.update(policy="none", S=min(S, 3))
    most = work(listed()[3])
    while c["B"] > 8 and (work(c)["flops"] > 0.9 * most["flops"] or work(c)["bytes"] > 0.9 * most["bytes"]):
        c["B"] = max(8, c["B"] * 2 // 3)
    return c


# ---- what a case is made of -----------------------------------------------------------------
POLICY = {"stage": "stage_first_shared", "section3": "paper_section3", "none": "none"}


def arch_of(c):
    w, policy = c["width"], POLICY[c["policy"]]
    if c["net"] == "basic":
        ws = (w, 2 * w, 4 * w)
        blocks = synth._stack(synth.BASIC, w, (c["n"],) * 3, ws, ws, policy)
        return synth.Arch(c["hw"], c["hw"], 3, c["classes"], 3, 1, w, 0, 0, blocks)
    mids = (w, 2 * w, 4 * w, 8 * w)
    blocks = synth._stack(synth.BOTTLENECK, w, (3, c["d2"], c["d3"], 3), tuple(4 * x for x in mids), mids, policy)
    if c["net"] == "wide":
        return synth.Arch(c["hw"], c["hw"], 3, c["classes"], 3, 1, w, 0, 0, blocks)
    return synth.Arch(c["hw"], c["hw"], 3, c["classes"], 7, 2, w, 1, 1, blocks)


def _batches(c, arch, dtype, gen, count):
    """`count` minibatches: Gaussian pixels (NHWC), uniform labels."""
    B = c["B"]
    xs = [torch.randn(B, arch.in_h, arch.in_w, arch.in_c, device="cuda", generator=gen).to(dtype) for _ in range(count)]
    ys = [torch.randint(0, arch.classes, (B,), device="cuda", generator=gen, dtype=torch.int32) for _ in range(count)]
    return xs, ys


def _align(n, a):
    return (n + a - 1) // a * a


def _state_views(ctx, S):
    """The library's flat arrays, in place: the context takes its device memory from torch, so the updated parameters can be
    looked at where they are.  Global vector [n] and running statistics; working copies [S][n'] of parameters, momentum and
    gradients and [S][nb'] of running statistics (n', nb': rounded up to 64 elements; one more copy serves evaluation)."""
    n, nb = ctx.n_params, ctx.n_buffers
    np_, nbp = _align(n, 64), _align(nb, 64)
    gsize = _align(4 * n, 256) + _align(4 * nb, 256)
    one, oneb = _align((S + 1) * np_ * 4, 256), _align((S + 1) * nbp * 4, 256)
    shadow = _align((S + 1) * np_ * 2, 256) if ctx.dtype == resist.BF16 else 0
    held = {t.numel(): t for t in ctx._held.values()}
    g, c = held[gsize], held[3 * one + shadow + oneb]
    f = lambda t, at, count: t[at:at + 4 * count].view(torch.float32)  # noqa: E731
    return dict(global_params=f(g, 0, n), global_stats=f(g, _align(4 * n, 256), nb),
                params=f(c, 0, S * np_).view(S, np_), momentum=f(c, one, S * np_).view(S, np_), grads=f(c, 2 * one, S * np_).view(S, np_),
                stats=f(c, 3 * one + shadow, S * nbp).view(S, nbp))


def _eval_stats(arch, S):
    """Running statistics as a trained context has them, to first order: mean 0 and, per BN, the variance that He-normal layers
    give its input (a residual branch adds 1, or 1/S^2 where the block is dealt out)."""
    out, v = [], 2.0
    put = lambda ch, var: out.extend([np.zeros(ch, np.float32), np.full(ch, var, np.float32)])  # noqa: E731
    if arch.stem_bn_relu:
        put(arch.stem_cout, v)
        v = 1.0
    for b in arch.blocks:
        put(b.cin, v)
        for _ in range(1 if b.kind == synth.BASIC else 2):
            put(b.cmid, 1.0)
        v = (1.0 if b.has_projection else v) + (1.0 / S ** 2 if b.partitionable else 1.0)
    put(arch.blocks[-1].cout, v)
    return np.concatenate(out)


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda").manual_seed(seed)
    bf = c["dtype"] == "bf16"
    dt = torch.bfloat16 if bf else torch.float32
    if c["kind"] == "conv":
        N, H, W, C, K, k, s = (c[x] for x in ("N", "H", "W", "C", "K", "ksz", "stride"))
        P, Q = (H - 1) // s + 1, (W - 1) // s + 1
        r = lambda *shape: torch.randn(*shape, device="cuda", generator=gen)  # noqa: E731
        return dict(case=c, geom=(N, H, W, C, K, k, s), a=torch.relu(r(N, H, W, C)).to(dt), w=(r(K, k, k, C) * math.sqrt(2 / (k * k * C))).to(dt),
                    dy=r(N, P, Q, K).to(dt))
    if c["kind"] == "bn":
        m, C = c["m"], c["C"]
        r = lambda *shape: torch.randn(*shape, device="cuda", generator=gen)  # noqa: E731
        return dict(case=c, x=(1.7 * r(m, C) + r(C)).to(dt), da=r(m, C).to(dt), gamma=1 + 0.2 * r(C), beta=0.3 * r(C),
                    rm=torch.zeros(C, device="cuda"), rv=torch.ones(C, device="cuda"))
    arch, S, kind = arch_of(c), c["S"], c["kind"]
    ctx = resist.Context(arch.to_int32(), dtype=resist.BF16 if bf else resist.F32, seed=seed)
    round0 = 1000 * seed + 17
    ctx.partition(round0, S)
    st = dict(case=c, ctx=ctx, round=round0, S=S, loss=torch.zeros(S, device="cuda"), view=_state_views(ctx, S))
    if kind == "eval":
        ctx.set_params(None, _eval_stats(arch, S))
        st["x"], st["y"] = (v[0] for v in _batches(c, arch, dt, gen, 1))
    elif kind == "sync":
        # working copies as after local steps: each sub-ResNet's own deviation from the global parameters, N(0, 1e-3)
        w, b = st["view"]["params"], st["view"]["stats"]
        w.add_(torch.randn(w.shape, device="cuda", generator=gen), alpha=1e-3)
        b.add_(torch.randn(b.shape, device="cuda", generator=gen), alpha=1e-3)
    else:
        st["x"], st["y"] = _batches(c, arch, dt, gen, 1 if kind == "worker" else S)
        st["sub"] = seed % S
    return st


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "conv":
        g = state["geom"]
        y, _ = resist.resist_conv2d(0, state["a"], state["w"], g)
        da, _ = resist.resist_conv2d(1, state["dy"], state["w"], g)
        dw, _ = resist.resist_conv2d(2, state["a"], state["dy"], g)
        return dict(y=y, da=da, dw=dw)
    if kind == "bn":
        a, stat = resist.resist_bn_relu_forward(state["x"], state["gamma"], state["beta"], state["rm"], state["rv"])
        C = c["C"]
        mean_invstd = stat[:2 * C].clone()
        dx, dg, db = resist.resist_bn_relu_backward(state["x"], state["da"], state["gamma"], state["beta"], stat)
        return dict(a=a, stat=mean_invstd, run_mean=state["rm"], run_var=state["rv"], dx=dx, dgamma=dg, dbeta=db)
    ctx, v, S = state["ctx"], state["view"], state["S"]
    if kind == "step":
        ctx.local_step_grouped(state["x"], state["y"], LR, state["loss"])
        out = dict(loss=state["loss"], params=v["params"], stats=v["stats"])
        # in bf16 a gradient of a whole net is not comparable element by element between two correct implementations (an activation
        # rounded the other way flips a ReLU mask); in fp32 it is
        return out if c["dtype"] == "bf16" else dict(out, grads=v["grads"], momentum=v["momentum"])
    if kind == "worker":
        s = state["sub"]
        ctx.local_step(s, state["x"][0], state["y"][0], LR, state["loss"][s:s + 1])
        out = dict(loss=state["loss"], params=v["params"][s], stats=v["stats"][s])
        return out if c["dtype"] == "bf16" else dict(out, grads=v["grads"][s], momentum=v["momentum"][s])
    if kind == "round":
        state["round"] += 1
        mask = ctx.partition(state["round"], S)
        ctx.local_step_grouped(state["x"], state["y"], LR, state["loss"])
        ctx.aggregate()
        return dict(mask=mask.astype(np.int64), loss=state["loss"], params=v["global_params"], stats=v["global_stats"])
    if kind == "sync":
        state["round"] += 1
        ctx.aggregate()
        mask = ctx.partition(state["round"], S)
        return dict(mask=mask.astype(np.int64), params=v["global_params"], stats=v["global_stats"], copies=v["params"])
    # eval: the number of hits is left out, it follows from the logits and turns on near ties
    logits, loss, _ = ctx.eval(state["x"], state["y"])
    return dict(logits=logits, loss=loss)


# ---- what a pass cannot do without ----------------------------------------------------------
def _net_cost(c, arch):
    """Per kind of block membership (held by every sub-ResNet / dealt to one): parameters, and per image: multiply-adds of the
    forward convolutions and head, and elements of the tensors that the backward pass needs (the input of every BN)."""
    h, w = (arch.in_h - 1) // arch.stem_stride + 1, (arch.in_w - 1) // arch.stem_stride + 1
    rows = h * w
    n = [arch.stem_cout * arch.stem_k ** 2 * arch.in_c, 0]
    mac = [rows * n[0], 0]
    act = [rows * arch.stem_cout * (arch.stem_bn_relu + 1), 0]
    if arch.stem_maxpool:
        h, w = (h - 1) // 2 + 1, (w - 1) // 2 + 1
    ch = arch.stem_cout
    for b in arch.blocks:
        p = b.partitionable
        rin = h * w
        h, w = (h - 1) // b.stride + 1, (w - 1) // b.stride + 1
        rout = h * w
        if b.kind == synth.BASIC:
            convs = [(9 * b.cin * b.cout, rout), (9 * b.cout * b.cout, rout)]
            acts = rin * b.cin + rout * b.cout
        else:
            convs = [(b.cin * b.cmid, rin), (9 * b.cmid * b.cmid, rout), (b.cmid * b.cout, rout)]
            acts = rin * (b.cin + b.cmid) + rout * b.cmid
        if b.has_projection:
            convs.append((b.cin * b.cout, rout))
        n[p] += sum(k for k, _ in convs)
        mac[p] += sum(k * r for k, r in convs)
        act[p] += acts
        ch = b.cout
    n[0] += ch * arch.classes
    mac[0] += ch * arch.classes
    act[0] += h * w * ch
    return n, mac, act


def work(case):
    """Bytes: inputs, parameters, momentum and results once each, and in training the saved activations (they exceed what stays
    on the chip) written once and read once.  Flops: convolutions and head, forward once and backward twice."""
    c = case
    es = 2 if c["dtype"] == "bf16" else 4
    if c["kind"] == "conv":
        N, H, W, C, K, k, s = (c[x] for x in ("N", "H", "W", "C", "K", "ksz", "stride"))
        rin, rout = N * H * W, N * ((H - 1) // s + 1) * ((W - 1) // s + 1)
        return dict(bytes=es * (2 * rin * C + 2 * rout * K + k * k * C * K) + 4 * k * k * C * K, flops=3 * 2 * rout * k * k * C * K)
    if c["kind"] == "bn":
        return dict(bytes=4 * es * c["m"] * c["C"], flops=20 * c["m"] * c["C"])
    arch, S, B = arch_of(c), c["S"], c["B"]
    n, mac, act = _net_cost(c, arch)
    total = n[0] + n[1]
    copies = S * n[0] + n[1]                                   # parameters held by the S sub-ResNets
    sync_bytes = 4 * copies + 4 * total + 4 * total + (4 + 4 + (2 if es == 2 else 0)) * copies   # means, then copies, momentum, bf16 copies
    image = es * arch.in_h * arch.in_w * arch.in_c
    if c["kind"] == "sync":
        return dict(bytes=sync_bytes, flops=2 * copies)
    if c["kind"] == "eval":
        return dict(bytes=B * image + es * total + 4 * B * arch.classes, flops=2 * B * (mac[0] + mac[1]))
    subs, held = (S, copies) if c["kind"] != "worker" else (1, n[0] + n[1] / S)
    dealt = 1 if c["kind"] != "worker" else 1 / S
    step_bytes = subs * B * (image + 4) + held * (4 * 4 + (2 if es == 2 else 0)) + 2 * es * B * (subs * act[0] + dealt * act[1])
    step_flops = 3 * 2 * B * (subs * mac[0] + dealt * mac[1])
    return dict(bytes=step_bytes + (sync_bytes if c["kind"] == "round" else 0), flops=step_flops)


def tolerance(case):
    c = case
    if c["kind"] == "sync":
        return "exact"                                         # the order of the mean's additions is part of the interface
    if c["dtype"] == "f32":
        return dict(rel=1e-4)
    if c["kind"] in ("conv", "bn"):
        return dict(rel=5e-3)                                  # outputs are bf16 (half an ulp: 2^-9), sums are fp32
    return dict(rel=1e-2)                                      # whole nets in bf16: roundings of a hundred layers, two steps deep
