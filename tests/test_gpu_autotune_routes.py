"""The autotuner times what its answer is used for: the TEP search for calls with a deadline, whose sample is never
cut, and shapes that leave the one-kernel decode alone for calls without; lines that an earlier version cached are
not used."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2405_01808_gb300 as grand

    grand.build()
    return grand


def frames_of(g, N, M, frames, snr):
    import torch

    _, frozen = g.polar_H(N, N // 2)
    d = wl.qam_frames(56, N, frames, N, np.setdiff1d(np.arange(N), frozen), M, snr)
    return torch.from_numpy(d["symbols"]).cuda()


@pytest.mark.parametrize("mixed", [False, True])
def test_deadline_tunes_the_search(g, tmp_path, mixed):
    """20,000 frames at 5 dB: the search takes more than four times the one kernel (300,000 at 6 / 8 / 10 dB: 33 times)."""
    import torch

    N, M = 128, 16
    code = g.Code.polar(N, N // 2)
    x = frames_of(g, N, M, 20000, 5.0)
    f = np.arange(len(x))
    desc = torch.from_numpy(g.frame_desc(np.zeros_like(f), np.full_like(f, M), 32 * f, 4 * f).view(np.uint8)).cuda()
    cache = str(tmp_path / "tiles.txt")

    def tune(ns):
        p = g.Params.make(M=M, S=10, query_cap=1 << 20, deadline_ns=ns)
        if mixed:
            return p, g.autotune_mixed([code], p, desc, x.reshape(-1), 4 * len(x), cache_path=cache)
        return p, g.autotune(code, p, x, cache_path=cache)

    _, plain = tune(0)
    p, search = tune(1)
    assert not search["from_cache"] and p.deadline_ns == 1
    assert g.stream_status(code) == 0  # nothing was cut
    assert search["best_ms"] > 4 * plain["best_ms"], (search, plain)
    for ns in (0, 10 ** 9):
        assert tune(ns)[1]["from_cache"]
    code.close()


@pytest.mark.parametrize("membership", ["AUTO", "FASTEST"])
def test_one_kernel_is_kept(g, tmp_path, membership):
    """S = 12 without a deadline: warps and split stay automatic; an earlier version's line with explicit warps, or
    with the hash join, is passed over."""
    import torch

    N, M = 256, 64
    code = g.Code.polar(N, N // 2)
    x = frames_of(g, N, M, 2000, 12.0)
    m = getattr(g, "MEMBERSHIP_" + membership)
    cache = tmp_path / "tiles.txt"
    name = torch.cuda.get_device_name().replace(" ", "_").replace("|", "_")
    cache.write_text(f"{name}|sym|N={N}|K={N // 2}|M={M}|S=12|cap={1 << 20}|lik=0|ord=1|mem={m} 4 0 2 4 0.1000 "
                     f"{g.MEMBERSHIP_HASH if membership == 'FASTEST' else g.MEMBERSHIP_AUTO}\n")
    p = g.Params.make(M=M, S=12, query_cap=1 << 20, membership=m)
    r = g.autotune(code, p, x, cache_path=str(cache))
    assert not r["from_cache"] and r["membership"] == g.MEMBERSHIP_AUTO
    assert tuple(p.tiles[:2]) == (0, 0) and p.tiles[2] in (2, 3) and p.tiles[3] in (4, 6)
    code.close()
