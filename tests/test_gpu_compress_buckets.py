"""The bucketed compress kernels at the edges of their spans: every bucket
size, flat and layer buckets (partial buckets, layers shorter than a bucket),
vectors that end inside a chunk, a word, a row and a span; messages, residuals
and lookahead offsets over two steps against the oracle bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from parity_helpers import assert_bits_equal, assert_messages_equal, oracle_config

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def P():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2010_13359_gb300 as P
    return P


FORMS = [(oracle.SIGN, 8), (oracle.SQUANT, 2), (oracle.SQUANT, 4), (oracle.SQUANT, 8), (oracle.QSGD, 4)]


def run(P, comp, bits, bucket, keep, d, layers, M=2):
    rng = np.random.default_rng(bucket + bits + d)
    cuts = np.sort(rng.choice(np.arange(1, d // 32), layers, replace=False)) * 32 if layers else []
    segments = (0, *map(int, cuts), d) if layers else None
    ocfg = oracle_config(d, M, comp, lr=0.1, bucket=bucket, bits=bits, seed=d, keep=keep, segments=segments)
    h = P.create(P.make_config(d=d, M=M, compressor=comp, lr=0.1, bucket=bucket, bits=bits, seed=d,
                               flags=P.KEEP_LOOKAHEAD if keep else 0,
                               cuda_stream=torch.cuda.current_stream().cuda_stream))
    if segments:
        h.set_segments(segments)
    st = oracle.State(ocfg)
    ld = (d + 3) // 4 * 4
    g_dev = torch.zeros((M, ld), device="cuda")
    msgs = torch.zeros((M, h.message_bytes()), dtype=torch.uint8, device="cuda")
    row = np.empty(d, np.float32)
    for step in range(2):
        g = (rng.standard_normal((M, d)) * np.exp(rng.uniform(-4, 1, (M, d)))).astype(np.float32)
        g_dev[:, :d] = torch.from_numpy(g)
        h.workers_compress_all(g_dev, ld, msgs)
        want = st.compress_all(g)
        got = msgs.cpu().numpy()
        for i in range(M):
            ctx = f"d {d} worker {i} step {step}"
            assert_messages_equal(ocfg, got[i], want[i], ctx)
            h.get_residual(i, row)
            assert_bits_equal(row, st.e[i], ctx)
            if keep:
                h.get_lookahead(i, row)
                assert_bits_equal(row, st.h[i], ctx)
    h.synchronize()
    h.destroy()


@pytest.mark.parametrize("keep", [False, True])
@pytest.mark.parametrize("bucket", [32, 64, 128, 256, 512, 1024, 2048, 4096])
@pytest.mark.parametrize("comp,bits", FORMS)
def test_compress(P, comp, bits, bucket, keep):
    for d, layers in ((5, 0), (512, 0), (3 * 512 + 128 + 37, 0), (9 * 4096 + 1025, 0), (4096 + 512 + 21, 9)):
        run(P, comp, bits, bucket, keep, d, layers)


@pytest.mark.parametrize("layers", [0, 50])
@pytest.mark.parametrize("comp,bits", FORMS)
def test_compress_128_per_scale_with_a_span_per_warp(P, comp, bits, layers):
    run(P, comp, bits, 128, True, 2_097_152 + 677, layers)


@pytest.mark.parametrize("layers", [0, 50])
@pytest.mark.parametrize("comp,bits", FORMS[1:])
def test_quantisers_128_per_scale_about_the_line(P, comp, bits, layers):
    """A warp per bucket to 10,239 buckets of both workers, a span per warp from there."""
    for d in (128 * 5119 + 5, 128 * 5120 + 37):
        run(P, comp, bits, 128, True, d - 128 * layers, layers)
