"""Long codes of high rate: frames with thousands of codewords in their TEP space, whose first hit is light, take no
longer than in the TEP search, and have its outputs."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

AMPLE = 10 ** 10


@pytest.fixture(scope="module")
def g():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2405_01808_gb300 as grand

    grand.build()
    return grand


@pytest.mark.parametrize("N,R,M,S,cap,frames,snr", [
    (1024, 10, 16, 12, 300, 18000, 8.0),         # a cap between the TEPs of weight 1 and 2
    (1024, 10, 4096, 10, 300, 18000, 24.0),
    (1024, 36, 1024, 10, 1 << 20, 18000, 25.6),  # two syndrome words, most frames received without an error
    (1024, 33, 4096, 8, 1 << 20, 6000, 29.6),
])
def test_not_slower_than_the_search(g, N, R, M, S, cap, frames, snr):
    import torch

    code = g.Code.polar(N, N - R)
    _, frozen = g.polar_H(N, N - R)
    d = wl.qam_frames(N + R, 6, 1000, N, np.setdiff1d(np.arange(N), frozen), M, snr)
    x = torch.from_numpy(d["symbols"]).cuda()
    x = x.repeat(-(-frames // len(x)), 1)[:frames].contiguous()

    def run(ns):
        p = g.Params.make(M=M, S=S, query_cap=cap, deadline_ns=ns)
        ms = []
        for _ in range(12):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            r = g.decode_symbols(code, p, x)
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        return float(np.median(ms[2:])), r

    (one, got), (search, want) = run(0), run(AMPLE)
    for k in ("cw", "queries", "abandon"):
        assert torch.equal(want[k], got[k]), k
    assert one < search, (one, search)
    code.close()
