"""worker_lookahead on a handle that keeps only some of the workers: the
worker's own row of the offsets, which start at the range's first worker."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_lookahead_of_a_local_range():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2010_13359_gb300 as P
    d, M, first, count = 4_100, 5, 3, 2
    h = P.create(P.make_config(d=d, M=M, compressor=P.SIGN, lr=0.5, bucket=512, flags=P.KEEP_LOOKAHEAD,
                               cuda_stream=torch.cuda.current_stream().cuda_stream))
    h.set_local_workers(first, count)
    g = torch.randn((count, d), device="cuda")
    msgs = torch.zeros((count, h.message_bytes()), dtype=torch.uint8, device="cuda")
    w, out = torch.randn(d, device="cuda"), torch.empty(d, device="cuda")
    h.workers_compress_range(first, count, g, d, msgs)
    offset = np.empty(d, np.float32)
    for i in range(first, first + count):
        h.worker_lookahead(i, w, out)
        h.get_lookahead(i, offset)
        assert np.array_equal(out.cpu().numpy(), w.cpu().numpy() - offset)
    h.destroy()
