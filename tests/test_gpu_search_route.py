"""The preparation and TEP search with automatic launch shapes, which calls with a deadline run: under a budget that no
call reaches its outputs are those of the one-kernel decode, for both register splits (S = 10: nibble tables; S = 12:
warp pairs, 7-rank B side), uniform and uneven batches, demodulated arrays, and twice in a row out of the fixed scratch
of the no-allocation entry point (records or counters left by the first call would show)."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

AMPLE = 10 ** 10
KEYS = ("cw", "queries", "abandon")


@pytest.fixture(scope="module")
def g():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2405_01808_gb300 as grand

    grand.build()
    return grand


def frames_of(g, N, M, frames, snr, seed):
    import torch

    _, frozen = g.polar_H(N, N // 2)
    d = wl.qam_frames(79, seed, frames, N, np.setdiff1d(np.arange(N), frozen), M, snr)
    return torch.from_numpy(d["symbols"]).cuda()


def same(a, b):
    import torch

    return all(torch.equal(a[k], b[k]) for k in KEYS)


CASES = [(128, 16, 10, 1 << 20, ((6000, 6.5), (2500, 9.0))), (512, 64, 12, 1 << 24, ((1500, 14.0), (700, 15.0)))]


@pytest.mark.parametrize("N,M,S,cap,batches", CASES)
def test_uniform(g, N, M, S, cap, batches):
    import torch

    code = g.Code.polar(N, N // 2)
    one, search = (g.Params.make(M=M, S=S, query_cap=cap, deadline_ns=ns) for ns in (0, AMPLE))
    for i, (frames, snr) in enumerate(batches):
        x = frames_of(g, N, M, frames, snr, i)
        want = g.decode_symbols(code, one, x)
        got = g.decode_symbols(code, search, x, stats=True)
        assert got["prep_ms"] > 0 and got["hard_frames"] > 0  # the two kernels, and frames searched by the second
        assert same(want, got)
        outs = {"cw": torch.full_like(want["cw"], -1), "queries": torch.full_like(want["queries"], -1),
                "abandon": torch.full_like(want["abandon"], 255)}
        g.decode_symbols_noalloc(code, search, x, *(outs[k] for k in KEYS))
        assert same(want, outs), f"no-allocation call {i}"
        dm = g.demod(x, M, N, outputs={"y": torch.empty((frames, N // 32), dtype=torch.int32, device="cuda"),
                                       "hard_idx": torch.empty(x.shape, dtype=torch.int16, device="cuda"),
                                       "key": torch.empty(x.shape, dtype=torch.int32, device="cuda"),
                                       "nmask": torch.empty(x.shape, dtype=torch.uint8, device="cuda")})
        assert same(want, g.decode_batch(code, search, dm["y"], dm["hard_idx"], dm["key"], dm["nmask"]))
        first = {10: 1 + 30 + 405, 12: 1 + 36 + 594}[S]  # TEPs of at most two altered symbols: the preparation's
        assert int(((want["abandon"] == 0) & (want["queries"] > first)).sum()) > 0
    assert g.stream_status(code) == 0
    code.close()


@pytest.mark.parametrize("S", [8, 10, 12])
def test_uneven(g, S):
    import torch

    Ns = wl.MIXED_N
    codes = [g.Code.polar(n, n // 2) for n in Ns]
    info = {n: np.setdiff1d(np.arange(n), g.polar_H(n, n // 2)[1]) for n in Ns}
    mx = wl.mixed_frames(79, S, 3000, info)
    desc = torch.from_numpy(g.frame_desc(np.searchsorted(np.array(Ns), mx["N"]), mx["M"], mx["sym_offset"],
                                         mx["cw_offset"]).view(np.uint8)).cuda()
    x = torch.from_numpy(mx["symbols"]).cuda()
    want, got = (g.decode_mixed(codes, g.Params.make(M=0, S=S, query_cap=1 << 20, deadline_ns=ns), desc, x,
                                mx["n_cw_words"], stats=ns > 0) for ns in (0, AMPLE))
    assert got["prep_ms"] > 0 and got["hard_frames"] > 0
    assert same(want, got)
    for code in codes:
        code.close()
