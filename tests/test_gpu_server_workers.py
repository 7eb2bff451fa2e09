"""The server kernels' worker sums at the edges of their groups: 1 worker to
more than two slabs of 32, every bucket size that has a form of its own, flat
and layer buckets, a vector that ends inside a word and a chunk; w against
the oracle bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from parity_helpers import assert_params_equal, oracle_config

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

D = 8 * 256 + 5 * 32 + 7
SEGMENTS = (0, 32, 96, 1056, 1088, 2112, D)


@pytest.fixture(scope="module")
def P():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2010_13359_gb300 as P
    return P


def run(P, comp, M, segments=None, d=D, hot=0, **kw):
    ocfg = oracle_config(d, M, comp, lr=0.03, seed=M, segments=segments, **kw)
    h = P.create(P.make_config(d=d, M=M, compressor=comp, lr=0.03, seed=M,
                               cuda_stream=torch.cuda.current_stream().cuda_stream, **kw))
    if segments:
        h.set_segments(segments)
    rng = np.random.default_rng(M)
    g = (rng.standard_normal((M, d)) * np.exp(rng.uniform(-3, 1, (M, d)))).astype(np.float32)
    g[:, :hot] *= 1e3
    ld = (d + 3) // 4 * 4
    g_dev = torch.zeros((M, ld), device="cuda")
    g_dev[:, :d] = torch.from_numpy(g)
    msgs = torch.zeros((M, h.message_bytes()), dtype=torch.uint8, device="cuda")
    w = (rng.standard_normal(d) * 0.02).astype(np.float32)
    w_gpu = torch.full((d + 64,), 12345.0, device="cuda")
    w_gpu[:d] = torch.from_numpy(w)
    h.workers_compress_all(g_dev, ld, msgs)
    h.server_aggregate_update(msgs, w_gpu[:d])
    st = oracle.State(ocfg)
    st.server(st.compress_all(g), w)
    h.synchronize()
    got = w_gpu.cpu().numpy()
    assert_params_equal(got[:d], w)
    assert np.all(got[d:] == 12345.0)
    h.destroy()


WORKERS = [1, 2, 3, 4, 5, 8, 9, 16, 17, 32, 33, 64, 65, 100]


@pytest.mark.parametrize("segments", [None, SEGMENTS], ids=["flat", "layers"])
@pytest.mark.parametrize("bucket", [32, 64, 128, 256, 2048])
@pytest.mark.parametrize("M", WORKERS)
def test_sign(P, M, bucket, segments):
    run(P, oracle.SIGN, M, segments, bucket=bucket)


@pytest.mark.parametrize("M", [*WORKERS, 129])
def test_identity(P, M):
    run(P, oracle.IDENTITY, M)


@pytest.mark.parametrize("M", [1, 3, 8, 17, 33, 65])
def test_identity_with_optimistic_adam(P, M):
    """Two steps of the pass that sums and updates, a vector that ends inside a chunk."""
    params = dict(alpha=1e-2, beta1=0.5, beta2=0.9, eps=1e-8)
    ocfg = oracle_config(D, M, oracle.IDENTITY, lr=0.03)
    h = P.create(P.make_config(d=D, M=M, compressor=P.IDENTITY, lr=0.03,
                               cuda_stream=torch.cuda.current_stream().cuda_stream))
    h.set_server_optimizer(P.dqgan.oadam(**params))
    rng = np.random.default_rng(M)
    w = (rng.standard_normal(D) * 0.02).astype(np.float32)
    w_gpu = torch.from_numpy(w.copy()).to("cuda")
    state = oracle.OAdamState(D, oracle.OAdam(**params))
    for step in range(1, 3):
        msgs = np.zeros((M, h.message_bytes()), np.uint8)
        msgs[:, :4 * D] = rng.standard_normal((M, D)).astype(np.float32).view(np.uint8)
        h.server_aggregate_update(torch.from_numpy(msgs).to("cuda"), w_gpu)
        state.server_step_range(ocfg, step, msgs, w, 0, D)
        h.synchronize()
        assert_params_equal(w_gpu.cpu().numpy(), w)
    h.destroy()


@pytest.mark.parametrize("segments", [None, SEGMENTS], ids=["flat", "layers"])
@pytest.mark.parametrize("bits", [2, 4, 8])
@pytest.mark.parametrize("M", [*WORKERS, 129])
def test_quantiser_small_buckets(P, M, bits, segments):
    run(P, oracle.SQUANT, M, segments, bucket=64, bits=bits)


@pytest.mark.parametrize("bits", [4, 8])
@pytest.mark.parametrize("M", WORKERS)
def test_quantiser_layer_buckets(P, M, bits):
    run(P, oracle.SQUANT, M, SEGMENTS, bucket=256, bits=bits)


@pytest.mark.parametrize("M", [1, 3, 8, 16, 17, 32])
def test_two_bits_beyond_the_small_sizes(P, M):
    run(P, oracle.SQUANT, M, d=262_144 + 519, bucket=512, bits=2)
    d = 524_288 + 519
    cuts = tuple(32 * c for c in np.sort(np.random.default_rng(M).choice(d // 32, 20, replace=False)) if c)
    run(P, oracle.SQUANT, M, (0, *cuts, d), d=d, bucket=512, bits=2)


@pytest.mark.parametrize("M", [1, 3, 8, 16, 17, 32])
def test_two_bits_past_the_line(P, M):
    """Flat vectors just above the size from which slices are staged by TMA."""
    run(P, oracle.SQUANT, M, d=max(262_144, 5_000_000 // max(M, 4)) + 519, bucket=512, bits=2)


@pytest.mark.parametrize("M", [1, 3, 6, 17])
def test_two_bits_with_layers_past_the_line(P, M):
    d = (8_000_000 if M > 4 else 1_500_000) + 519
    cuts = tuple(32 * c for c in np.sort(np.random.default_rng(M).choice(d // 32, 200, replace=False)) if c)
    run(P, oracle.SQUANT, M, (0, *cuts, d), d=d, bucket=512, bits=2)


def records(kind, M, d, k, rng):
    """M messages of k records."""
    common = rng.choice(d, 2 * k // 3, replace=False)
    msgs = np.zeros((M, (8 * k + 255) // 256 * 32, 2), np.uint32)
    for m in range(M):
        if kind == "spread":
            idx = rng.choice(d, k, replace=False)
        elif kind == "shared":
            own = rng.permutation(np.setdiff1d(rng.choice(d, 2 * k, replace=False), common))
            idx = np.concatenate([common, own[:k - len(common)]])
        elif kind == "edge":  # tiles of 4096 indices with 2048 records in all, 2049, and the rest at the end
            n = 2048 // M + (m < 2048 % M)
            idx = np.concatenate([rng.choice(4096, n, replace=False),
                                  4096 + rng.choice(4096, n + (m == 0), replace=False)])
            idx = np.concatenate([idx, d - 1 - rng.choice(d - 8192, k - len(idx), replace=False)])
        else:
            idx = d - 1 - rng.choice(k + k // 3, k, replace=False)
        msgs[m, :k, 0] = np.sort(idx)
        msgs[m, :k, 1] = rng.standard_normal(k).astype(np.float32).view(np.uint32)
    return msgs.view(np.uint8).reshape(M, -1)


@pytest.mark.parametrize("kind", ["spread", "shared", "dense"])
@pytest.mark.parametrize("M", [1, 2, 3, 8, 16, 17, 32, 33, 64])
def test_top_k_merged_by_tiles(P, M, kind):
    """Half a million records: spread over the vector; two in three of them at
    indices every worker sends; and all of them in a few tiles, more than a
    list holds."""
    top_k_server(P, 4_100_007, M, -(-510_000 // M), kind)


LISTS = [(M, kind, False) for M in (1, 3, 4, 8, 17, 32, 33, 64) for kind in ("spread", "shared", "dense", "edge")]
LISTS += [(M, kind, True) for M in (4, 17, 64) for kind in ("dense", "edge")]


@pytest.mark.parametrize("M,kind,oadam", LISTS)
def test_top_k_lists_and_dense_tiles(P, M, kind, oadam):
    """A million records, from where they are merged by tiles: also a tile with as many
    records as a list holds and one with one more, and with Optimistic Adam on the
    server, which wants +0 at the indices nobody sent."""
    top_k_server(P, 4_100_007, M, -(-1_010_000 // M), kind, oadam=oadam)


@pytest.mark.parametrize("kind", ["spread", "edge"])
@pytest.mark.parametrize("d,M,k", [(500_000, 21, 47_620), (499_999, 21, 47_620), (999_999, 64, 15_624)])
def test_top_k_at_the_smallest_merged(P, d, M, k, kind):
    """The smallest vector that is merged by tiles, and one parameter or record less."""
    top_k_server(P, d, M, k, kind)


@pytest.mark.parametrize("M", [16, 64])
def test_top_k_records_gathered_in_a_tenth_take_no_longer(P, M):
    """Layers differ in scale, so the records of a step often sit in a few tiles.  Those
    are shared out over the GPU; a CTA for each took four times as long as for the same
    number of records spread evenly."""
    d, k = 1_048_576, 104_857
    took = {}
    for kind in ("spread", "gathered"):
        h = P.create(P.make_config(d=d, M=M, compressor=P.TOPK, lr=0.03, k=k,
                                   cuda_stream=torch.cuda.current_stream().cuda_stream))
        gen = torch.Generator(device="cuda").manual_seed(M)
        msgs = torch.zeros((M, h.message_bytes()), dtype=torch.uint8, device="cuda")
        for m in range(M):
            p = torch.rand(d, generator=gen, device="cuda")
            if kind == "gathered":
                p[:k + 100] += 1
            msgs[m].view(torch.int32)[:2 * k:2] = torch.topk(p, k).indices.sort().values.int()
        w = torch.zeros(d, device="cuda")
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        times = []
        for _ in range(5):
            a.record()
            for _ in range(8):
                h.server_aggregate_update(msgs, w)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) / 8)
        took[kind] = min(times)
        h.destroy()
    assert took["gathered"] < 2.5 * took["spread"], took


def top_k_server(P, d, M, k, kind, oadam=False):
    rng = np.random.default_rng(M)
    ocfg = oracle_config(d, M, oracle.TOPK, lr=0.03, k=k)
    h = P.create(P.make_config(d=d, M=M, compressor=P.TOPK, lr=0.03, k=k,
                               cuda_stream=torch.cuda.current_stream().cuda_stream))
    params = dict(alpha=1e-2, beta1=0.5, beta2=0.9, eps=1e-8)
    if oadam:
        h.set_server_optimizer(P.dqgan.oadam(**params))
    w = (rng.standard_normal(d) * 0.02).astype(np.float32)
    w_gpu = torch.from_numpy(w.copy()).to("cuda")
    state = oracle.OAdamState(d, oracle.OAdam(**params)) if oadam else None
    for step in range(1, 3 if oadam else 2):
        msgs = records(kind, M, d, k, rng)
        h.server_aggregate_update(torch.from_numpy(msgs).to("cuda"), w_gpu)
        if oadam:
            state.server_step_range(ocfg, step, msgs, w, 0, d)
        else:
            oracle.server_step(ocfg, msgs, w)
        h.synchronize()
        assert_params_equal(w_gpu.cpu().numpy(), w)
    h.destroy()
