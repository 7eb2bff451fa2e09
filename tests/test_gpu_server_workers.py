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


@pytest.mark.parametrize("kind", ["spread", "shared", "dense"])
@pytest.mark.parametrize("M", [1, 2, 3, 8, 16, 17, 32, 33, 64])
def test_top_k_merged_by_tiles(P, M, kind):
    """Half a million records: spread over the vector; two in three of them at
    indices every worker sends; and all of them in a few tiles, more than a
    list holds."""
    d, k = 4_100_007, -(-510_000 // M)
    rng = np.random.default_rng(M)
    ocfg = oracle_config(d, M, oracle.TOPK, lr=0.03, k=k)
    h = P.create(P.make_config(d=d, M=M, compressor=P.TOPK, lr=0.03, k=k,
                               cuda_stream=torch.cuda.current_stream().cuda_stream))
    common = rng.choice(d, 2 * k // 3, replace=False)
    msgs = np.zeros((M, h.message_bytes() // 8, 2), np.uint32)
    for m in range(M):
        if kind == "spread":
            idx = rng.choice(d, k, replace=False)
        elif kind == "shared":
            own = rng.permutation(np.setdiff1d(rng.choice(d, 2 * k, replace=False), common))
            idx = np.concatenate([common, own[:k - len(common)]])
        else:
            idx = d - 1 - rng.choice(k + k // 3, k, replace=False)
        msgs[m, :k, 0] = np.sort(idx)
        msgs[m, :k, 1] = rng.standard_normal(k).astype(np.float32).view(np.uint32)
    msgs = msgs.view(np.uint8).reshape(M, -1)
    w = (rng.standard_normal(d) * 0.02).astype(np.float32)
    w_gpu = torch.from_numpy(w.copy()).to("cuda")
    h.server_aggregate_update(torch.from_numpy(msgs).to("cuda"), w_gpu)
    oracle.server_step(ocfg, msgs, w)
    h.synchronize()
    assert_params_equal(w_gpu.cpu().numpy(), w)
    h.destroy()
