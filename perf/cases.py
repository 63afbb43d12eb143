"""What is measured: the calls that a program which trains or runs a sigmoid
multi-layer perceptron with this library makes, through its Python binding.

A case is a dict of plain values:
  call       "train"    a net kept on the GPU: `epochs` passes of bp_train_epoch (or of
                        bp_train_batch, where the group is the whole set) over resident patterns,
                        then the weights are read back, as a program does that saves or scores them;
             "host"     the same through bp_train_epoch_host: patterns in pinned host memory;
             "noalloc"  bp_train_epoch_noalloc: the caller's own weight and velocity buffers;
             "split"    bp_forward + bp_backward over three groups (a pooled change larger than one
                        call), bp_update, and the weights read back;
             "forward"  bp_forward: outputs for a set of patterns;
  sizes      layer sizes n_0-...-n_L;  dtype "f32" or "bf16";
  n          patterns per pass (per group for "split");  mb: patterns per update (0: no update)
  epochs     passes over the patterns in one run;  lr: learning rate, per pattern (summed change)
             for f32 and per mean change for bf16, as in this repository's tests of many updates.

Patterns have the structure of the repository's workloads: nets of 203 inputs and 26 outputs take
one-hot letter windows and three-hot targets, all others N(0, 1) inputs and binary targets.
"""
import math

import numpy as np
import torch

from paper_1801_01554_gb300 import bp

MOMENTUM = 0.9
DEV = "cuda"


def _case(call, sizes, dtype, n, mb, epochs=1, lr=0.05):
    return dict(call=call, sizes=sizes, dtype=dtype, n=n, mb=mb, epochs=epochs, lr=lr)


def listed():
    return [
        # one pattern through a trained letter-to-phoneme net, as an interactive program asks for it
        dict(_case("forward", "203-120-26", "f32", 1, 0), name="f32_forward_1"),
        # a caller that owns all device memory updates a small net by a few small groups
        dict(_case("noalloc", "203-60-26", "f32", 250, 32, lr=0.1), name="f32_noalloc_mb32"),
        # the per-pattern update (online learning)
        dict(_case("train", "203-120-26", "f32", 1000, 1), name="f32_online_mb1"),
        # gradient accumulation through the separate calls, deeper net, odd sizes and groups
        dict(_case("split", "64-33-17-9", "f32", 300, 0), name="f32_split_300"),
        # the small net's full-batch training: ten updates of 1,024 patterns
        dict(_case("train", "203-60-26", "f32", 1024, 1024, epochs=10, lr=0.01), name="f32_full_1024"),
        # the headline workload: an epoch of 65,536 patterns in minibatches of 512
        dict(_case("train", "203-120-26", "f32", 65536, 512), name="f32_epoch_mb512"),
        # the same epoch from pinned host memory, copies included, in odd-sized groups
        dict(_case("host", "203-120-26", "f32", 60001, 500), name="f32_host_mb500"),
        # the largest group: whole-set updates over 65,536 patterns
        dict(_case("train", "203-120-26", "f32", 65536, 65536, epochs=8, lr=0.0005), name="f32_full_65536"),
        # a bf16 net of moderate width in minibatches of 512, the last one ragged
        dict(_case("train", "208-1024-32", "bf16", 16200, 512, epochs=2, lr=0.05), name="bf16_epoch_mb512"),
        # outputs of a trained wide net for an odd number of patterns
        dict(_case("forward", "1024-2048-2048-512", "bf16", 1001, 0), name="bf16_forward_1001"),
        # wide-net training, full batch of 8,192
        dict(_case("train", "1024-2048-2048-512", "bf16", 8192, 8192, epochs=25, lr=0.05), name="bf16_wide3"),
        # the widest net, full batch of 16,384, fifty updates
        dict(_case("train", "4096-4096-4096-4096-4096", "bf16", 16384, 16384, epochs=50, lr=0.05),
             name="bf16_wide4096"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    if rng.random() < 0.5:
        # letter-window nets and generic small ones, one or two hidden layers
        if rng.random() < 0.6:
            sizes = [203, _log(rng, 20, 300), 26]
        else:
            sizes = [_log(rng, 16, 256)] + [_log(rng, 8, 200) for _ in range(rng.randint(1, 2))]
            sizes += [rng.randint(3, 40)]
        call = rng.choice(["train", "train", "train", "host", "split", "forward", "noalloc"])
        if call == "forward":
            n, mb, epochs = _log(rng, 1, 65536), 0, 1
        elif call == "split":
            n, mb, epochs = _log(rng, 1, 20000), 0, 1
        else:
            mb = _log(rng, 1, 1000 if call == "noalloc" else 65536)
            groups = rng.randint(2, 40 if call == "noalloc" else 120)
            n = min(65536, mb * groups - rng.randrange(mb))
            mb, epochs = min(mb, n), max(1, min(8, 65536 // n)) if mb > 4 else 1
        lr = min(0.05, 8.0 / max(mb, 3 * n if call == "split" else 1))
        return _case(call, "-".join(map(str, sizes)), "f32", n, mb, epochs, lr)
    depth = rng.randint(2, 4)
    wide = rng.random() < 0.4
    sizes = [8 * _log(rng, 96 if wide else 16, 512 if wide else 128) for _ in range(depth)]
    sizes += [8 * _log(rng, 4, 256 if wide else 32)]
    call = rng.choice(["train", "train", "train", "forward", "split", "host"])
    if call == "forward":
        return _case(call, "-".join(map(str, sizes)), "bf16", _log(rng, 1, 16384), 0)
    if call == "split":
        return _case(call, "-".join(map(str, sizes)), "bf16", _log(rng, 16, 8192), 0)
    mb = _log(rng, 64, 16384)
    n = min(16384, mb * rng.randint(1, 16) - rng.randrange(mb // 4 + 1))
    mb = min(mb, n)
    return _case(call, "-".join(map(str, sizes)), "bf16", n, mb, 1 if call == "host" else rng.randint(2, 8))


def _sizes(case):
    return tuple(int(s) for s in case["sizes"].split("-"))


def _inputs(case, seed):
    """Patterns, targets (float32 on the GPU; bf16 values for bf16 nets) and start weights."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    sizes = _sizes(case)
    n = case["n"] * (3 if case["call"] == "split" else 1)
    if sizes[0] == 203 and sizes[-1] == 26 and case["dtype"] == "f32":
        letters = torch.randint(0, 29, (n, 7), generator=g, device=DEV) + 29 * torch.arange(7, device=DEV)
        X = torch.zeros(n, 203, device=DEV).scatter_(1, letters, 1.0)
        ones = torch.rand(n, 26, generator=g, device=DEV).topk(3, dim=1).indices
        T = torch.zeros(n, 26, device=DEV).scatter_(1, ones, 1.0)
    else:
        X = torch.randn(n, sizes[0], generator=g, device=DEV)
        T = (torch.rand(n, sizes[-1], generator=g, device=DEV) < 0.3).float()
    parts = []
    for i, o in zip(sizes[:-1], sizes[1:]):
        if case["dtype"] == "f32":
            parts.append(torch.rand((i + 1) * o, generator=g, device=DEV) * 0.6 - 0.3)
        else:
            parts.append(torch.randn(i * o, generator=g, device=DEV) / math.sqrt(i))
            parts.append(torch.rand(o, generator=g, device=DEV) * 0.2 - 0.1)
    if case["dtype"] == "bf16":
        X, T = X.bfloat16(), T.bfloat16()
    return X, T, torch.cat(parts)


def _scale(case):
    """Factor on the pooled change: a sum for f32, a mean for bf16."""
    if case["dtype"] == "f32":
        return 1.0
    return 1.0 / (3 * case["n"] if case["call"] == "split" else max(1, case["mb"]))


def prepare(case, seed):
    sizes, call, n, mb = _sizes(case), case["call"], case["n"], case["mb"]
    X, T, theta = _inputs(case, seed)
    s = dict(case=case, X=X, T=T)
    if call == "noalloc":
        s.update(theta=theta, V=torch.zeros_like(theta), sse=torch.zeros(-(-n // mb), device=DEV),
                 status=torch.zeros(1, dtype=torch.int32, device=DEV))
        return s
    net = bp.Net(sizes, case["lr"], MOMENTUM, dtype=bp.BP_BF16 if case["dtype"] == "bf16" else bp.BP_F32,
                 max_batch=mb or n, grad_scale=_scale(case))
    net.set_weights(theta.cpu().numpy())
    s["net"] = net
    if call == "forward":
        s["Y"] = torch.empty(n, sizes[-1], dtype=X.dtype, device=DEV)
    elif call == "host":
        s.update(X=X.cpu().pin_memory(), T=T.cpu().pin_memory())
    elif call == "split":
        s["sse"] = torch.zeros(3, device=DEV)
    else:
        s["sse"] = torch.zeros(case["epochs"], -(-n // mb), device=DEV)
    return s


def run(s):
    c = s["case"]
    call, n, mb = c["call"], c["n"], c["mb"]
    X, T = s["X"], s["T"]
    if call == "noalloc":
        for _ in range(c["epochs"]):
            bp.bp_train_epoch_noalloc(_sizes(c), c["lr"], MOMENTUM, 1.0, s["theta"], s["V"], X, T, n, mb,
                                      s["sse"], s["status"])
        return dict(theta=s["theta"], V=s["V"], sse=s["sse"])
    net = s["net"]
    if call == "forward":
        net.forward(X, n, s["Y"])
        return s["Y"]
    if call == "split":
        for k in range(3):
            net.forward(X[k * n:(k + 1) * n], n)
            net.backward(T[k * n:(k + 1) * n], n, s["sse"][k:k + 1])
        net.update()
        return dict(theta=net.get_weights(), sse=s["sse"])
    if call == "host":
        sse = np.empty(-(-n // mb) * c["epochs"], dtype=np.float32).reshape(c["epochs"], -1)
        for k in range(c["epochs"]):
            net.train_epoch_host(X, T, n, mb, sse[k])
        return dict(theta=net.get_weights(), sse=sse)
    for k in range(c["epochs"]):
        if mb == n:
            net.train_batch(X, T, n, s["sse"][k])
        else:
            net.train_epoch(X, T, n, mb, s["sse"][k])
    return dict(theta=net.get_weights(), sse=s["sse"])


def _weights(sizes):
    return sum((i + 1) * o for i, o in zip(sizes[:-1], sizes[1:]))


def work(case):
    """Patterns, targets and start state in, weights (velocity) and outputs out; flops as the
    repository's benchmark counts them, and five per weight and update."""
    sizes, n, call = _sizes(case), case["n"], case["call"]
    W, Wi, e = _weights(sizes), (sizes[0] + 1) * sizes[1], 2 if case["dtype"] == "bf16" else 4
    if call == "forward":
        return dict(bytes=n * (sizes[0] + sizes[-1]) * e + 4 * W, flops=2 * W * n)
    patterns = 3 * n if call == "split" else n
    updates = 1 if call == "split" else case["epochs"] * -(-n // case["mb"])
    return dict(bytes=patterns * (sizes[0] + sizes[-1]) * e + 16 * W + 4 * updates,
                flops=(6 * W - 2 * Wi) * patterns * case["epochs"] + 5 * W * updates)


def tolerance(case):
    # float32: sums of up to 65,536 terms in another order, through every update of the run;
    # bf16: activations, deltas and weight copies are rounded to 8 bits in every layer
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-3}
    return {"rel": 1e-2, "max": 0.3}


def exact(case, seed):
    """The run in float64: plain sums, the logistic, and the momentum update."""
    sizes, call, n = _sizes(case), case["call"], case["n"]
    if work(case)["flops"] > 1.5e13:
        return None
    X, T, theta = _inputs(case, seed)
    X, T, theta = X.double(), T.double(), theta.double()
    V = torch.zeros_like(theta)

    def layers(vec):
        at, out = 0, []
        for i, o in zip(sizes[:-1], sizes[1:]):
            out.append((vec[at:at + i * o].view(o, i), vec[at + i * o:at + (i + 1) * o]))
            at += (i + 1) * o
        return out

    def activations(x):
        a = [x]
        for W, b in layers(theta):
            a.append(torch.sigmoid(torch.addmm(b, a[-1], W.t())))
        return a

    def change(x, t, G):
        a = activations(x)
        err = t - a[-1]
        d = err * a[-1] * (1 - a[-1])
        for l in range(len(sizes) - 2, -1, -1):
            layers(G)[l][0].addmm_(d.t(), a[l])
            layers(G)[l][1].add_(d.sum(0))
            if l:
                d = (d @ layers(theta)[l][0]) * a[l] * (1 - a[l])
        return err.square().sum()

    def update(G):
        V.mul_(MOMENTUM).add_(G, alpha=case["lr"] * _scale(case))
        theta.add_(V)

    if call == "forward":
        return activations(X)[-1]
    sse = []
    if call == "split":
        G = torch.zeros_like(theta)
        for k in range(3):
            sse.append(change(X[k * n:(k + 1) * n], T[k * n:(k + 1) * n], G))
        update(G)
        return dict(theta=theta, sse=torch.stack(sse))
    for _ in range(case["epochs"]):
        for p in range(0, n, case["mb"]):
            G = torch.zeros_like(theta)
            sse.append(change(X[p:p + case["mb"]], T[p:p + case["mb"]], G))
            update(G)
    sse = torch.stack(sse)
    if call == "noalloc":   # the buffer holds the last pass's error sums
        return dict(theta=theta, V=V, sse=sse[-(-(-n // case["mb"])):])
    return dict(theta=theta, sse=sse.view(case["epochs"], -1))
