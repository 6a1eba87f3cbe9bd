"""Few parity bits leave a frame up to millions of codewords in its TEP space: a query cap bounds what is looked at,
and the outputs stay those of the TEP search, with caps below, at and above the TEPs of the lightest weights."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

TABLE = (1, 0, 0, 0)


@pytest.fixture(scope="module")
def g():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2405_01808_gb300 as grand

    grand.build()
    return grand


def frames_of(g, N, K, M, frames, snr):
    import torch

    _, frozen = g.polar_H(N, K)
    d = wl.qam_frames(N + K, 0, frames, N, np.setdiff1d(np.arange(N), frozen), M, snr)
    return torch.from_numpy(d["symbols"]).cuda()


@pytest.mark.parametrize("N,K,M,S", [(128, 120, 16, 12), (128, 112, 16, 12), (64, 57, 4, 12), (32, 30, 4, 10),
                                     (1024, 1014, 16, 12), (128, 86, 16, 12)])
def test_outputs(g, N, K, M, S):
    """Caps inside every weight class up to the fourth (S = 12 ranks of three alternatives: 1, 37, 631, 6,571 TEPs)."""
    import torch

    code = g.Code.polar(N, K)
    x = frames_of(g, N, K, M, 600, {4: 2.0, 16: 5.0}[M])
    for cap in (1, 2, 37, 38, 300, 630, 631, 632, 6570, 6571, 6572, 40000):
        want = g.decode_symbols(code, g.Params.make(M=M, S=S, query_cap=cap, tiles=TABLE), x)
        for membership in (g.MEMBERSHIP_AUTO, g.MEMBERSHIP_SOLVE):
            got = g.decode_symbols(code, g.Params.make(M=M, S=S, query_cap=cap, membership=membership), x)
            for k in ("cw", "queries", "abandon"):
                assert torch.equal(want[k], got[k]), (cap, membership, k)
    code.close()


def time(g, code, x, **kw):
    import torch

    ms = []
    for _ in range(22):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        g.decode_symbols(code, g.Params.make(**kw), x)
        b.record()
        b.synchronize()
        ms.append(a.elapsed_time(b))
    return float(np.median(ms[2:]))


def test_a_small_cap_bounds_the_work(g):
    """10 parity bits: half of the frames have no codeword among the 300 TEPs of the cap, and their 2^14 solutions
    are not walked for one."""
    code = g.Code.polar(128, 118)
    x = frames_of(g, 128, 118, 16, 20000, 4.0)
    few, all_of_them = (time(g, code, x, M=16, S=12, query_cap=cap) for cap in (300, 1 << 24))
    assert few < 0.7 * all_of_them, (few, all_of_them)
    code.close()


def test_two_parity_bits_are_not_slower_than_the_search(g):
    """Two parity bits: nearly every frame has a codeword among the TEPs of one altered symbol. (A budget selects the
    preparation and the search.)"""
    code = g.Code.polar(32, 30)
    x = frames_of(g, 32, 30, 16, 20000, 10.0)
    one, search = (time(g, code, x, M=16, S=8, query_cap=1 << 16, deadline_ns=ns) for ns in (0, 10 ** 10))
    assert one < search, (one, search)
    code.close()
