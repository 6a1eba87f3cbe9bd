"""Received symbols many times larger than the constellation (a receiver that does not know its gain; hard decisions and
the order of the reliabilities still mean something): keys beyond the packed range are selected exactly, also where one
lane of a warp holds more of the smallest than it keeps, and not much slower than the search's preparation selects."""
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


def frames_of(g, N, M, frames, snr, gain):
    import torch

    _, frozen = g.polar_H(N, N // 2)
    d = wl.qam_frames(N + M, 5, min(frames, 2000), N, np.setdiff1d(np.arange(N), frozen), M, snr)
    x = torch.from_numpy(d["symbols"] * np.float32(gain)).cuda()
    return x.repeat(-(-frames // len(x)), 1)[:frames].contiguous()


# frames of 3 to 512 symbols; 600 frames: a warp per frame, 17,000: a thread per frame
@pytest.mark.parametrize("frames", [600, 17000])
@pytest.mark.parametrize("N,M,S,gain", [(32, 4096, 12, 60.0), (64, 4, 10, 60.0), (512, 16, 12, 12.0), (1024, 4, 12, 60.0),
                                        (1024, 4, 8, 1e6), (1024, 64, 10, 3.0)])
def test_outputs(g, N, M, S, gain, frames):
    import torch

    code = g.Code.polar(N, N // 2)
    x = frames_of(g, N, M, frames, {4: 4.0, 16: 8.0, 64: 12.0, 4096: 24.0}[M], gain)
    if x.shape[1] >= 256:  # the small keys in one residue class of 32, fewer and more than a lane keeps
        f = torch.arange(frames, device="cuda")
        for k in range(8):
            at = (f % 3 == 0) & (f % 8 >= k)
            x[at, 5 + 32 * k] = x[at, 5 + 32 * k] / gain
    for order in (g.ORDER_QAM_NNE, g.ORDER_QAM_NEARER):
        kw = dict(order=order, M=M, S=S, query_cap=1 << 14)
        want = g.decode_symbols(code, g.Params.make(**kw, deadline_ns=AMPLE), x)
        got = g.decode_symbols(code, g.Params.make(**kw), x)
        for k in ("cw", "queries", "abandon"):
            assert torch.equal(want[k], got[k]), (order, k)
    code.close()


def test_not_slower_than_the_search(g):
    import torch

    code = g.Code.polar(1024, 512)
    x = frames_of(g, 1024, 4, 18000, 4.0, 60.0)

    def time(**kw):
        ms = []
        for _ in range(12):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            g.decode_symbols(code, g.Params.make(M=4, S=10, query_cap=1 << 20, **kw), x)
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        return float(np.median(ms[2:]))

    one, search = time(), time(deadline_ns=AMPLE)
    assert one < search, (one, search)
    code.close()
