"""The top-k worker step where its sampled threshold, its candidate lists and
its counting rounds change course, against the selection's definition.

The k records are fixed by the definition alone (the k largest |p_j|, equal
ones lowest index first, in index order), so they, e and h are compared bit
for bit with numpy on the same fp32 p:

* few parameters (one CTA keeps them on chip), more (clusters of 8 and of 16
  CTAs do), parts that end in the last CTA, and d on both sides of the sizes
  from which the sampled kernels run; few candidates (selected in one launch,
  also where they turn out too many for its shared memory) and many;
* a gradient that is large exactly at the sampled runs, so that too few
  elements reach the threshold and the candidates are taken again;
* a few dense tiles among thousands with one candidate each;
* a k-th key far above the threshold, so many equal keys that their list
  overflows, k = 1 and k = d;
* sparse gradients: fewer than k non-zero entries (the k-th key is 0 and
  almost every element equals it) and a few more than k (every element is a
  candidate and T far above the threshold 0), also with more workers than
  there are clusters for them.  These are ordinary inputs, so their time is
  held against a dense gradient's too.
"""
from __future__ import annotations

import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def P():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2010_13359_gb300 as P
    return P


def sampled(d):
    """The elements the threshold's sample reads: one run of 8 in each of 8192 strata."""
    runs, s = d >> 3, np.arange(8192, dtype=np.uint64)
    lo, hi = runs * s // 8192, runs * (s + 1) // 8192
    at = lo + (((s * 0x9E3779B1) & 0xFFFFFFFF) * (hi - lo) >> np.uint64(32))
    return (at[:, None] * 8 + np.arange(8, dtype=np.uint64)).ravel().astype(np.int64)


def gradient(kind, d, k, rng):
    g = rng.standard_normal(d).astype(np.float32)
    if kind == "trap":
        g *= np.float32(1e-3)
        g[sampled(d)] = 10
    elif kind == "sparse tiles":  # one large value in each of the first tiles, the rest in the last ones
        nt = -(-d // 4096)
        g *= np.float32(1e-6)
        g[np.arange(nt - 90) * 4096 + 17] = 3
        tail = np.arange((nt - 90) * 4096, d)
        g[rng.choice(tail, 20_000, replace=False)] = 5
    elif kind == "outliers":
        g[rng.choice(d, 3, replace=False)] *= np.float32(1e25)
    elif kind == "ties":
        g = np.sign(g) * (rng.integers(1, 4, d) * 0.5).astype(np.float32)
    elif kind == "zeros":
        g[:] = 0
    elif kind in ("sparse", "just enough"):  # -0 and +0 elsewhere
        g[rng.random(d) >= (0.5 if kind == "sparse" else 1.1) * k / d] *= 0
    return g


CASES = [(1, 1, 2, "gauss"), (3, 2, 2, "gauss"), (2_049, 2_049, 2, "ties"), (20_001, 333, 40, "ties"),
         (49_152, 10, 20, "gauss"), (9_999, 1, 2, "gauss"), (32_767, 400, 2, "outliers"), (40_000, 30_000, 9, "ties"),
         (393_215, 4_000, 9, "gauss"), (65_535, 65_535, 20, "gauss"), (65_536, 300, 20, "gauss"),
         (200_003, 200_003, 9, "gauss"), (786_431, 9_000, 4, "ties"), (300_005, 2, 20, "outliers"),
         (300_005, 150_000, 20, "ties"), (1_000_003, 1, 2, "gauss"), (1_000_003, 990_000, 2, "gauss"),
         (1_000_003, 200_000, 2, "trap"), (9_000_001, 400_000, 2, "ties"), (9_000_001, 21_000, 2, "sparse tiles"),
         (200_003, 9_000, 2, "sparse"), (1_000_003, 20_000, 3, "sparse"), (1_000_003, 20_000, 3, "just enough"),
         (1_000_003, 300_000, 2, "just enough"), (90_001, 1_000, 64, "sparse"), (1_000_003, 60_000, 2, "zeros"), (35_000_001, 50_000, 1, "sparse"),
         (35_000_001, 50_000, 1, "trap"), (90_001, 30_000, 64, "ties"),
         # selected in one launch, up to its last size, and the next
         (1_000_003, 20_000, 2, "trap"), (9_000_001, 20_000, 2, "ties"), (1_000_003, 500, 15, "gauss"),
         (1_000_003, 500, 16, "gauss"), (1_000_003, 60_000, 2, "ties"), (1_000_003, 95_000, 3, "gauss"),
         (4096 * 4096, 2_000, 1, "gauss"), (4096 * 4096 + 1, 2_000, 1, "gauss"), (600_001, 1, 3, "outliers")]


@pytest.mark.parametrize("keep", [False, True])
@pytest.mark.parametrize("d,k,M,kind", CASES)
def test_records_residual_and_offsets(P, d, k, M, kind, keep):
    stream = torch.cuda.current_stream()
    rng = np.random.default_rng(d + k)
    lr = np.float32(0.25)
    h = P.create(P.make_config(d=d, M=M, compressor=P.TOPK, lr=float(lr), k=k,
                               flags=P.KEEP_LOOKAHEAD if keep else 0, cuda_stream=stream.cuda_stream))
    ld = (d + 3) // 4 * 4
    i = M - 1  # the worker looked at; the others get zeros
    e = np.zeros(d, np.float32)
    if kind in ("sparse", "just enough"):
        e = -e  # -0: with -0 in the gradient, p is -0 there
        h.set_residual(i, e)
    g_dev = torch.zeros((M, ld), device="cuda")
    msgs = torch.zeros((M, h.message_bytes()), dtype=torch.uint8, device="cuda")
    for step in range(2):
        g = gradient(kind, d, k, rng)
        g_dev[i, :d] = torch.from_numpy(g)
        h.workers_compress_all(g_dev, ld, msgs)
        h.synchronize()
        s = lr * g
        p = s + e
        key = p.view(np.uint32) & np.uint32(0x7FFFFFFF)
        T = np.partition(key, d - k)[d - k]
        kept = key > T
        ties = np.flatnonzero(key == T)[:k - int(kept.sum())]
        kept[ties] = True
        idx = np.flatnonzero(kept)
        rec = msgs[i, :8 * k].cpu().numpy().view(np.uint32).reshape(k, 2)
        assert np.array_equal(rec[:, 0], idx.astype(np.uint32)), step
        assert np.array_equal(rec[:, 1], p[idx].view(np.uint32)), step
        if M > 1:  # all zero: the first k indices
            rec = msgs[0, :8 * k].cpu().numpy().view(np.uint32).reshape(k, 2)
            assert np.array_equal(rec[:, 0], np.arange(k, dtype=np.uint32)) and not rec[:, 1].any(), step
        e = np.where(kept, p - p, p)
        got = np.empty(d, np.float32)
        h.get_residual(i, got)
        assert np.array_equal(got.view(np.uint32), e.view(np.uint32)), step
        if keep:
            h.get_lookahead(i, got)
            assert np.array_equal(got.view(np.uint32), (s + e).view(np.uint32)), step
    h.destroy()


@pytest.mark.parametrize("d,M", [(400_000, 4), (3_600_000, 8)])  # on chip; the sampled kernels
def test_sparse_gradients_take_a_few_times_a_dense_one(P, d, M):
    """Fewer than k non-zero entries, so that almost every element equals the k-th key: no
    slower than a dense gradient but for a few passes.  Selected by one CTA per worker it
    took 120 times a dense gradient's time."""
    stream = torch.cuda.current_stream()
    k, ld = d // 100, (d + 3) // 4 * 4
    took = {}
    for kind in ("gauss", "sparse"):
        h = P.create(P.make_config(d=d, M=M, compressor=P.TOPK, lr=0.25, k=k, cuda_stream=stream.cuda_stream))
        gen = torch.Generator(device="cuda").manual_seed(5)
        g = torch.randn((M, ld), generator=gen, device="cuda")
        if kind == "sparse":
            g *= torch.rand((M, ld), generator=gen, device="cuda") < 0.005
        msgs = torch.zeros((M, h.message_bytes()), dtype=torch.uint8, device="cuda")
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        times = []
        for _ in range(5):
            a.record()
            for _ in range(4):
                h.workers_compress_all(g, ld, msgs)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) / 4)
        took[kind] = min(times)
        h.destroy()
    assert took["sparse"] < 5 * took["gauss"], took


@pytest.mark.parametrize("d", [300_005, 1_000_003])  # on chip; the sampled kernels
def test_gradients_from_another_stream(P, d):
    """The gradients are still being written on another stream when the call is made; an event
    orders the two."""
    M, k, lr = 2, 5_000, np.float32(0.25)
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    h = P.create(P.make_config(d=d, M=M, compressor=P.TOPK, lr=float(lr), k=k, cuda_stream=mine.cuda_stream))
    ld = (d + 3) // 4 * 4
    gen = torch.Generator(device="cuda").manual_seed(d)
    sources = [torch.randn((M, ld), generator=gen, device="cuda") * 10.0 ** -step for step in range(4)]
    g = torch.zeros((M, ld), device="cuda")
    msgs = torch.zeros((M, h.message_bytes()), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    got = []
    for src in sources:
        with torch.cuda.stream(other):
            other.wait_stream(mine)
            busy = torch.ones(1 << 24, device="cuda")
            for _ in range(8):
                busy = busy * 1.0001
            g.copy_(src)
            written = other.record_event()
        mine.wait_event(written)
        h.workers_compress_all(g, ld, msgs)
        with torch.cuda.stream(mine):
            got.append(msgs.clone())
    h.synchronize()
    torch.cuda.synchronize()
    e = np.zeros((M, d), np.float32)
    for step, src in enumerate(sources):
        p = lr * src[:, :d].cpu().numpy() + e
        for m in range(M):
            rec = got[step][m, :8 * k].cpu().numpy().view(np.uint32).reshape(k, 2)
            idx = np.sort(np.argpartition(np.abs(p[m]), d - k)[d - k:])  # no two keys are equal at the k-th
            assert np.array_equal(rec[:, 0], idx.astype(np.uint32)), (step, m)
            assert np.array_equal(rec[:, 1], p[m, idx].view(np.uint32)), (step, m)
            e[m] = p[m]
            e[m, idx] = 0
    h.destroy()


# run by a child process: the sizes that take clusters of CTAs, and those that would take them
NO_CLUSTERS = r"""
import numpy as np, torch
import paper_2010_13359_gb300 as P
import oracle
stream = torch.cuda.current_stream()
for d, M, k, launches in ((300_007, 1, 3_000, 5), (65_535, 2, 700, 5), (49_153, 1, 20, 5), (786_431, 3, 8_000, 5),
                          (65_536, 4, 60_000, 5), (40_000, 9, 400, 1), (33, 1, 3, 1)):
    h = P.create(P.make_config(d=d, M=M, compressor=P.TOPK, lr=0.5, k=k, cuda_stream=stream.cuda_stream))
    cfg = oracle.Config(d=d, M=M, compressor=oracle.TOPK, lr=0.5, k=k)
    st = oracle.State(cfg)
    ld = (d + 3) // 4 * 4
    g_dev = torch.zeros((M, ld), device="cuda")
    msgs = torch.zeros((M, h.message_bytes()), dtype=torch.uint8, device="cuda")
    for step in range(2):
        g = np.random.default_rng(step).standard_normal((M, d)).astype(np.float32)
        g_dev[:, :d] = torch.from_numpy(g)
        before = h.launch_count()
        h.workers_compress_all(g_dev, ld, msgs)
        assert h.launch_count() - before == launches, (d, M, h.launch_count() - before)
        want = st.compress_all(g)
        h.synchronize()
        got = msgs.cpu().numpy()
        for i in range(M):
            assert np.array_equal(got[i, :8 * k], want[i][:8 * k]), (d, M, step, i)
    h.destroy()
print("no clusters: ok")
"""


def test_a_device_part_without_room_for_clusters(P):
    """Where no cluster of 8 or 16 CTAs fits (a part of a device), their launch would fail;
    those sizes take the five kernels then, below the sample's size too."""
    env = dict(os.environ, DQGAN_TEST_NO_CLUSTERS="1")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    res = subprocess.run([sys.executable, "-c", NO_CLUSTERS], cwd=root, env=env, capture_output=True, text=True, timeout=600)
    assert res.returncode == 0 and "no clusters: ok" in res.stdout, res.stdout + res.stderr
