"""The linear solve under a deadline: frames with more than 2^8 codewords in their TEP space whose walk is reached
after the budget are returned with abandon 5, the hard word and the TEPs tested without a hit; every other frame is
that of a call without a deadline."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as wl
from test_gpu_deadline import prep_tested

pytestmark = pytest.mark.gpu

KEYS = ("cw", "queries", "abandon")


@pytest.fixture(scope="module")
def g():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2405_01808_gb300 as grand

    grand.build()
    return grand


def coded(N, K, M, frames, snr, oracle_lib):
    return wl.qam_frames(N + K, 3, frames, N, oracle_lib.info_set(N, K), M, snr)["symbols"]


# 2,000 frames: a warp per frame; 17,000: a thread per frame
@pytest.mark.parametrize("N,K,M,S,frames", [(128, 118, 16, 12, 2000), (128, 118, 16, 12, 17000), (64, 56, 4, 10, 2000),
                                            (32, 28, 4, 12, 17000)])
def test_late_walks_are_cut(g, oracle_lib, N, K, M, S, frames):
    import torch

    code = g.Code.polar(N, K)
    sym = coded(N, K, M, frames, {4: 0.0, 16: 4.0}[M], oracle_lib)
    x = torch.from_numpy(sym).cuda()

    def run(cap, ns):
        p = g.Params.make(M=M, S=S, query_cap=cap, membership=g.MEMBERSHIP_SOLVE, deadline_ns=ns)
        r = g.decode_symbols(code, p, x)
        status = g.stream_status(code)
        return {k: r[k].cpu().numpy() for k in KEYS}, status, p

    want, status, _ = run(1 << 24, 0)
    assert status == 0
    long, status, _ = run(1 << 24, 10 ** 10)
    assert status == 0 and all(np.array_equal(want[k], long[k]) for k in KEYS)
    got, status, p = run(1 << 24, 1)
    cut = got["abandon"] == 5
    assert cut.any() and not cut.all() and status == g.E_TIMEOUT
    for k in KEYS:
        assert np.array_equal(got[k][~cut], want[k][~cut]), k
    tested, y = prep_tested(oracle_lib, sym[cut], M, N, S, w0=1)
    assert np.array_equal(got["cw"][cut].view(np.uint32), y)
    assert np.array_equal(got["queries"][cut].astype(np.int64), tested)
    assert np.all((want["queries"][cut].astype(np.int64) > tested) | (want["abandon"][cut] == 1))
    # a cap of one query: nothing is left to walk
    one, status, _ = run(1, 1)
    assert status == 0 and not (one["abandon"] == 5).any()
    # a captured plan starts its clock at every replay
    outs = [torch.empty(frames, N // 32, dtype=torch.int32, device="cuda"),
            torch.empty(frames, dtype=torch.int32, device="cuda"), torch.empty(frames, dtype=torch.uint8, device="cuda")]
    plan = g.plan_symbols(code, p, x, *outs)
    for _ in range(2):
        for o in outs:
            o.zero_()
        g.stream_status(code)
        plan.launch()
        assert g.stream_status(code) == g.E_TIMEOUT
        for k, o in zip(KEYS, outs):
            assert np.array_equal(o.cpu().numpy().reshape(got[k].shape), got[k]), k
    plan.close()
    code.close()


# 3,000 frames in their own order; 50,000 put in order by length
@pytest.mark.parametrize("frames", [3000, 50000])
def test_uneven_batch_flags_the_code_it_cut(g, oracle_lib, frames):
    """Few parity bits beside a code of rate 1/2, whose frames have too few codewords to be cut."""
    import torch

    pairs = ((128, 118), (64, 32))
    codes = [g.Code.polar(n, k) for n, k in pairs]
    sym = [coded(n, k, 16, frames // 2, 4.0, oracle_lib) for n, k in pairs]
    f = np.arange(frames)
    c, i, h = f % 2, f // 2, frames // 2
    desc = g.frame_desc(c, np.full(frames, 16), np.where(c == 0, 32 * i, 32 * h + 16 * i),
                        np.where(c == 0, 4 * i, 4 * h + 2 * i))
    d = torch.from_numpy(desc.view(np.uint8)).cuda()
    x = torch.from_numpy(np.concatenate([s.reshape(-1) for s in sym])).cuda()
    out = []
    for ns in (0, 1):
        p = g.Params.make(M=16, S=12, query_cap=1 << 24, membership=g.MEMBERSHIP_SOLVE, deadline_ns=ns)
        r = g.decode_mixed(codes, p, d, x, 6 * h)
        out.append({k: r[k].cpu().numpy() for k in KEYS})
    assert [g.stream_status(c) for c in codes] == [g.E_TIMEOUT, 0]
    want, got = out
    cut = got["abandon"] == 5
    assert cut[c == 0].any() and not cut[c == 1].any()
    assert np.array_equal(got["queries"][~cut], want["queries"][~cut])
    assert np.array_equal(got["abandon"][~cut], want["abandon"][~cut])
    words = np.concatenate([np.repeat(cut[c == 0], 4), np.repeat(cut[c == 1], 2)])
    assert np.array_equal(got["cw"][~words], want["cw"][~words])
    for code in codes:
        code.close()
