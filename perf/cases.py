"""The work whose speed is measured: steps of Algorithm 2 through the package's public calls.

A pass of every case but one is what a training program does once it has the
M workers' gradients: the batched worker step (`workers_compress_all`, or one
`worker_compress` per worker), the server step (`server_aggregate_update`) and,
where the handle keeps the lookahead offsets, `worker_lookahead` for every
worker, which gives the points of the next gradients.  The remaining case is
the worker step without a handle (`topk_compress_noalloc`).

Every result is fixed bit for bit by the entry points' own rules (one rounding
per operation, sums in one order), so every case is compared exactly.
"""
from __future__ import annotations

import math
import random

import torch

import paper_2010_13359_gb300 as P
from paper_2010_13359_gb300 import dqgan

COMPRESSORS = {"sign": P.SIGN, "topk": P.TOPK, "squant": P.SQUANT, "identity": P.IDENTITY, "qsgd": P.QSGD}
BUCKETED = ("sign", "squant", "qsgd")
LR = 1e-3
# Optimistic Adam as GAN training sets it: a small step, b1 = 0.5, b2 = 0.9.
OADAM = dict(alpha=1e-4, beta1=0.5, beta2=0.9, eps=1e-8)


def _case(name, q, d, M, **kw):
    """bucket, bits, k: of the compressor.  layers: layer segments, each with its own gradient scale;
    layer_buckets: the buckets restart at each of them.  lookahead: the handle keeps the lookahead
    offsets.  server: omd or oadam.  grads: gaussian or student (t, 3 degrees).  host: gradients in
    pinned host memory.  each: one worker_compress per worker.  noalloc: the call without a handle."""
    case = dict(name=name, q=q, d=d, M=M, bucket=512, bits=8, k=1, layers=16, layer_buckets=False, lookahead=False,
                server="omd", grads="gaussian", host=False, each=False, noalloc=False)
    case.update(kw)
    return case


def listed():
    return [
        # The smallest step, as the closed loop around a min-max game takes it: latency and launches.
        _case("tiny_sign_loop", "sign", 65_536, 4, bucket=512, layers=4, lookahead=True),
        # DCGAN-sized generator + discriminator, scaled sign.
        _case("dcgan_sign", "sign", 3_600_000, 8, bucket=1024),
        # The same vector, 1 % of the entries kept.
        _case("dcgan_topk", "topk", 3_600_000, 8, k=36_000),
        # The same vector uncompressed with Optimistic Adam on the server: the full-precision system
        # that the compressed ones are compared with.
        _case("dcgan_identity_oadam", "identity", 3_600_000, 8, server="oadam"),
        # Gradients that a data loader or another process left in pinned host memory.
        _case("dcgan_squant_b4_host", "squant", 3_600_000, 8, bucket=512, bits=4, host=True),
        # ResNet-GAN-sized vector: the 4-bit quantiser, the 8-bit one with a scale per layer bucket,
        # and 1 % top-k.
        _case("resnet_squant_b4", "squant", 25_000_000, 16, bucket=512, bits=4, layers=64),
        _case("resnet_squant_b8_layers", "squant", 25_000_000, 16, bucket=512, bits=8, layers=64, layer_buckets=True),
        _case("resnet_topk", "topk", 25_000_000, 16, k=250_000, layers=64),
        # The largest: heavy-tailed gradients, 32 workers.
        _case("stress_sign", "sign", 100_000_000, 32, bucket=4096, layers=1, grads="student"),
        # Ragged sizes and worker counts that are no power of two, small buckets, many workers.
        _case("ragged_sign_many", "sign", 1_234_567, 64, bucket=128, lookahead=True),
        _case("ragged_qsgd_layers", "qsgd", 5_000_011, 12, bucket=256, bits=8, layers=64, layer_buckets=True,
              lookahead=True),
        # The worker step of a program that may not allocate device memory.
        _case("noalloc_topk", "topk", 1_000_003, 1, k=10_000, noalloc=True),
    ]


def draw(rng):
    """Sizes over four decades (d from 2^12, at most 2e8 elements over all workers, 3e7 in host
    memory), 1 to 64 workers, every compressor, bucket and option.  Combinations whose residual grows
    without bound under error feedback (2 bits over large buckets, few bits over QSGD's l2 scale, 4
    bits over large buckets of heavy-tailed values) are drawn with buckets that keep it bounded."""
    q = rng.choice(("sign", "sign", "topk", "topk", "squant", "squant", "qsgd", "identity"))
    M = rng.choice((1, 2, 3, 4, 5, 8, 8, 12, 16, 16, 24, 32, 48, 64))
    host = rng.random() < 0.1
    noalloc = q == "topk" and not host and rng.random() < 0.25
    if noalloc:
        M = 1
    top = (1 << 20) if noalloc else min(50_000_000, int(3e7 if host else 2e8) // M)
    d = int(math.exp(rng.uniform(math.log(4096), math.log(top))))
    bits = rng.choice((2, 4, 8))
    bucket = 1 << rng.randint(5, 12)
    if q == "squant" and bits == 2 or q == "qsgd" and bits < 8:
        bits, bucket = max(bits, 4 if q == "qsgd" else 2), 32
    grads = rng.choice(("gaussian", "gaussian", "student"))
    if q == "squant" and bits == 4 and grads == "student":
        bucket = min(bucket, 512)
    layers = min(rng.choice((1, 4, 16, 64)), max(1, d // 2048))
    return _case("drawn", q, d, M, bucket=bucket, bits=bits, k=max(1, int(d * math.exp(rng.uniform(math.log(1e-3), math.log(5e-2))))),
                 layers=layers, layer_buckets=q in BUCKETED and rng.random() < 0.4,
                 lookahead=not noalloc and rng.random() < 0.4, server="oadam" if not noalloc and rng.random() < 0.2 else "omd",
                 grads=grads, host=host, each=not noalloc and rng.random() < 0.2,
                 noalloc=noalloc) | {"name": "%s_%d_%d" % (q, d, M)}


def _ld(case):
    return (case["d"] + 3) // 4 * 4


def _layer_offsets(case):
    """0 = o_0 < ... < o_n = d: weights 2^U(-3, 3), the inner offsets multiples of 32; the same for every seed."""
    d, n = case["d"], case["layers"]
    rng = random.Random("%d layers of %d" % (n, d))
    weights = [2.0 ** rng.uniform(-3, 3) for _ in range(n)]
    offsets = [0]
    for x in weights[:-1]:
        offsets.append(offsets[-1] + max(32, int(x / sum(weights) * d) // 32 * 32))
    if offsets[-1] >= d:
        offsets = [0]
    return offsets + [d]


def _generator(seed, *which):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(random.Random("%d %s" % (seed, which)).getrandbits(60))
    return gen


def _gradient(case, seed, worker, std, out):
    """Layer l's entries: N(0, std_l^2) or heavy-tailed with that scale."""
    gen = _generator(seed, "gradient", worker)
    torch.randn(out.shape, generator=gen, device=out.device, out=out)
    if case["grads"] == "student":
        chi, z = torch.zeros_like(out), torch.empty_like(out)
        for _ in range(3):
            torch.randn(out.shape, generator=gen, device=out.device, out=z)
            chi.addcmul_(z, z)
        out.div_(chi.div_(3.0).sqrt_())
    return out.mul_(std)


def _inputs(case, seed):
    """Yields worker by worker (gradient, residual from the steps before), then the parameters."""
    offsets = _layer_offsets(case)
    rng = random.Random("scales %d" % seed)
    stds = [1e-3] if len(offsets) == 2 else [math.exp(rng.uniform(math.log(1e-4), math.log(1e-1))) for _ in offsets[1:]]
    std = torch.repeat_interleave(torch.tensor(stds, device="cuda"),
                                  torch.tensor([b - a for a, b in zip(offsets, offsets[1:])], device="cuda"))
    for i in range(case["M"]):
        g = _gradient(case, seed, i, std, torch.empty(case["d"], device="cuda"))
        e = torch.randn(case["d"], generator=_generator(seed, "residual", i), device="cuda").mul_(std).mul_(LR)
        yield g, e
    yield torch.randn(case["d"], generator=_generator(seed, "parameters"), device="cuda").mul_(0.02), None


def prepare(case, seed):
    """The gradients, the message and parameter buffers and the handle (residuals of a run under way)."""
    d, M, ld = case["d"], case["M"], _ld(case)
    stream = torch.cuda.current_stream().cuda_stream
    g = torch.zeros((M, ld), pin_memory=True) if case["host"] else torch.zeros((M, ld), device="cuda")
    state = dict(case=case, g=g, ld=ld, stream=stream)
    inputs = _inputs(case, seed)
    if case["noalloc"]:
        g_row, e = next(inputs)
        g[0, :d] = g_row
        state.update(e=e, msgs=torch.zeros(8 * case["k"], dtype=torch.uint8, device="cuda"))
        return state
    h = P.create(P.make_config(d=d, M=M, compressor=COMPRESSORS[case["q"]], lr=LR, bucket=case["bucket"], k=case["k"],
                               bits=case["bits"], seed=seed, flags=P.KEEP_LOOKAHEAD if case["lookahead"] else 0,
                               cuda_stream=stream))
    if case["layer_buckets"]:
        h.set_segments(_layer_offsets(case))
    if case["server"] == "oadam":
        h.set_server_optimizer(dqgan.oadam(**OADAM))
    for i in range(M):
        g_row, e = next(inputs)
        g[i, :d] = g_row
        h.set_residual(i, e)
    w = next(inputs)[0]
    state.update(handle=h, msgs=torch.zeros((M, h.message_bytes()), dtype=torch.uint8, device="cuda"), w=w)
    if case["lookahead"]:
        state["w_half"] = torch.zeros((M, ld), device="cuda")
    return state


def run(state):
    case, g, msgs = state["case"], state["g"], state["msgs"]
    if case["noalloc"]:
        dqgan.topk_compress_noalloc(g, state["e"], msgs, case["d"], case["k"], LR, state["stream"])
        return {"msgs": msgs, "e": state["e"]}
    h, w = state["handle"], state["w"]
    if case["each"]:
        for i in range(case["M"]):
            h.worker_compress(i, g[i], msgs[i])
    else:
        h.workers_compress_all(g, state["ld"], msgs)
    h.server_aggregate_update(msgs, w)
    if not case["lookahead"]:
        return {"msgs": msgs, "w": w}
    for i in range(case["M"]):
        h.worker_lookahead(i, w, state["w_half"][i])
    return {"msgs": msgs, "w": w, "w_half": state["w_half"]}


def _buckets(case):
    """The buckets' starts and the end of the last."""
    offsets = _layer_offsets(case) if case["layer_buckets"] else [0, case["d"]]
    return [j for a, b in zip(offsets, offsets[1:]) for j in range(a, b, case["bucket"])] + [case["d"]]


def work(case):
    """Worker step: gradient and residual read, residual (and lookahead offset) and message written;
    server: messages read, parameters (and the optimiser's three vectors) read and written; lookahead:
    offset read, point written, parameters read."""
    d, M = case["d"], case["M"]
    if case["q"] == "topk":
        message = 8 * case["k"]
    elif case["q"] == "identity":
        message = 4 * d
    else:
        message = d * (1 if case["q"] == "sign" else case["bits"]) // 8 + 4 * (len(_buckets(case)) - 1)
    if case["noalloc"]:
        return {"bytes": 12 * d + message, "flops": 2 * d}
    total = M * (12 * d + message) + M * message + (8 * case["k"] * M if case["q"] == "topk" and case["server"] == "omd" else 8 * d)
    if case["server"] == "oadam":
        total += 24 * d
    if case["lookahead"]:
        total += M * 12 * d + 4 * d
    summed = M * (case["k"] if case["q"] == "topk" else d)
    return {"bytes": total, "flops": 4 * M * d + summed + 2 * d + (12 * d if case["server"] == "oadam" else 0)}


def tolerance(case):
    """Messages, residuals, offsets and parameters are reproducible bit for bit: each operation is
    rounded once and each sum has one order, which the calls' documentation states."""
    return "exact"


def _philox(counter, worker, step, key):
    """Four 32-bit words per counter of Philox4x32-10 (Salmon et al., SC'11), in 64-bit integers."""
    def mul(a, x):
        low, high = (a & 0xFFFF) * x, (a >> 16) * x
        return (high + (low >> 16)) >> 16, (((high & 0xFFFF) << 16) + low) & 0xFFFFFFFF

    k0, k1 = key & 0xFFFFFFFF, key >> 32
    x = [counter, torch.full_like(counter, worker), torch.full_like(counter, step), torch.full_like(counter, 0x51)]
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
        h0, l0 = mul(0xD2511F53, x[0])
        h1, l1 = mul(0xCD9E8D57, x[2])
        x = [h1 ^ x[1] ^ k0, l1, h0 ^ x[3] ^ k1, l0]
    return x


def _quantised(case, seed, worker, p, p32, bucket_of, counts):
    """Q(p) in 64 bits; which entries are sent and which signs they have is decided on the 32-bit p."""
    d = case["d"]
    if case["q"] == "identity":
        return p
    if case["q"] == "topk":
        key = p32.abs()
        T = torch.topk(key, case["k"]).values[-1]
        keep = key > T
        ties = torch.nonzero(key == T).flatten()[:case["k"] - int(keep.sum())]
        keep[ties] = True
        return torch.where(keep, p, torch.zeros_like(p))
    starts = torch.cumsum(counts, 0) - counts
    at = starts[:, None] + torch.arange(case["bucket"], device="cuda")
    rows = torch.where(at < (starts + counts)[:, None], p[at.clamp_(max=d - 1)], torch.zeros((), dtype=p.dtype, device="cuda")).abs_()
    del at
    if case["q"] == "sign":
        s = (rows.sum(1) / counts)[bucket_of]
        return torch.where(p32 < 0, -s, s)
    s = (rows.amax(1) if case["q"] == "squant" else rows.square().sum(1).sqrt())[bucket_of]
    del rows
    K = (1 << (case["bits"] - 1)) - 1
    t = torch.where(s > 0, p.abs() * K / s, torch.zeros_like(p)).clamp_(max=K)
    words = _philox(torch.arange((d + 3) // 4, device="cuda"), worker, 1, seed)
    u = torch.stack([x >> 8 for x in words], 1).flatten()[:d].double() / 2.0 ** 24
    level = t.floor() + (u < t - t.floor())
    return torch.where(p32 < 0, -1.0, 1.0) * s * level / K


def exact(case, seed):
    """The same step in 64 bits.  The messages are packed bytes, so nothing stands in their place."""
    d, M = case["d"], case["M"]
    lr = float(torch.tensor(LR))
    bucket_of = counts = None
    if case["q"] in BUCKETED:
        starts = torch.tensor(_buckets(case), device="cuda")
        counts = starts[1:] - starts[:-1]
        bucket_of = torch.repeat_interleave(torch.arange(len(counts), device="cuda"), counts)
    q_sum = torch.zeros(d, dtype=torch.float64, device="cuda")
    offsets = torch.zeros((M, _ld(case)), dtype=torch.float64, device="cuda") if case["lookahead"] else None
    inputs = _inputs(case, seed)
    for i in range(M):
        g, e = next(inputs)
        p = g.double() * lr + e.double()
        quantised = _quantised(case, seed, i, p, g * lr + e, bucket_of, counts)
        q_sum += quantised
        if case["noalloc"]:
            return {"msgs": None, "e": p - quantised}
        if case["lookahead"]:
            offsets[i, :d] = g.double() * lr + (p - quantised)
    w = next(inputs)[0].double()
    q = q_sum / M
    if case["server"] == "omd":
        w = w - q
    else:  # the first step: the moments' bias corrections cancel their weights
        w = w - OADAM["alpha"] * 2 * torch.where(q == 0, q, q / (q.abs() + OADAM["eps"]))
    if not case["lookahead"]:
        return {"msgs": None, "w": w}
    offsets[:, :d] = w - offsets[:, :d]
    return {"msgs": None, "w": w, "w_half": offsets}
