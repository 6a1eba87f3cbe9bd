"""Matrices not of polar form in batches that a warp per frame prepares (small ones, and demodulated arrays of any size):
the base syndromes by columns give the search's outputs for every number of syndrome words, and a call that a query cap
ends early is not slower than the search."""
from __future__ import annotations

import numpy as np
import pytest
from test_gpu_general_rows import random_code, symbols_of

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


def arrays(g, x, M, N):
    import torch

    F, L = x.shape
    o = {"y": torch.empty((F, N // 32), dtype=torch.int32, device="cuda"),
         "hard_idx": torch.empty((F, L), dtype=torch.int16, device="cuda"),
         "key": torch.empty((F, L), dtype=torch.int32, device="cuda"),
         "nmask": torch.empty((F, L), dtype=torch.uint8, device="cuda")}
    g.demod(x, M, N, outputs=o)
    return o["y"], o["hard_idx"], o["key"], o["nmask"]


# 1 to 16 syndrome words (whole and partial groups of four) of 1 to 32 words of a frame
@pytest.mark.parametrize("N,R,M", [(32, 20, 4), (32, 31, 64), (64, 33, 16), (64, 63, 4), (128, 100, 16), (256, 129, 64),
                                   (512, 224, 16), (512, 256, 64), (1024, 500, 256), (1024, 481, 16)])
def test_outputs(g, N, R, M):
    import torch

    code, H, at, free = random_code(g, N, R, N + R + 1)
    x = torch.from_numpy(symbols_of(g, H, at, free, N, M, 700, {4: 5.0, 16: 8.0, 64: 12.0, 256: 18.0}[M], R)).cuda()
    p, search = (g.Params.make(M=M, S=9, query_cap=1 << 16, deadline_ns=ns) for ns in (0, AMPLE))
    want = g.decode_symbols(code, search, x)
    for got in (g.decode_symbols(code, p, x), g.decode_batch(code, p, *arrays(g, x, M, N))):
        for k in ("cw", "queries", "abandon"):
            assert torch.equal(want[k], got[k]), k
    code.close()


@pytest.mark.parametrize("form,frames", [("symbols", 10000), ("arrays", 30000)])
def test_not_slower_than_the_search(g, form, frames):
    import torch

    N, M = 1024, 64
    code, H, at, free = random_code(g, N, 512, 2)
    x = torch.from_numpy(symbols_of(g, H, at, free, N, M, 500, 12.0, 2)).cuda().repeat(frames // 500, 1)
    args = arrays(g, x, M, N)

    def time(ns):
        p = g.Params.make(M=M, S=10, query_cap=30, deadline_ns=ns)
        ms = []
        for _ in range(12):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            g.decode_symbols(code, p, x) if form == "symbols" else g.decode_batch(code, p, *args)
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        return float(np.median(ms[2:]))

    one, search = time(0), time(AMPLE)
    assert one < search, (one, search)
    code.close()
