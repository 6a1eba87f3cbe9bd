"""Large batches of codes whose matrix is not of polar form (their syndromes are row parities, a thread per frame):
the same outputs as the same frames in batches small enough for the warp per frame (column sums) and as the TEP search,
with row counts around the eight rows taken at once and the 32 of a syndrome word, and hard words of 1 to 32 words."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

TABLE = (1, 0, 0, 0)
SMALL = 8000


@pytest.fixture(scope="module")
def g():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2405_01808_gb300 as grand

    grand.build()
    return grand


def random_code(g, N, R, seed):
    r = np.random.default_rng(seed)
    H = r.integers(0, 2, (R, N))
    at = r.permutation(N)[:R]
    H[:, at] = np.eye(R, dtype=np.int64)
    free = np.setdiff1d(np.arange(N), at)
    return g.Code(g.H_from_dense(H), N, N - R), H, at, free


def symbols_of(g, H, at, free, N, M, frames, snr, seed):
    """Codewords of H (information bits on the free positions) through the channel."""
    r = np.random.default_rng(seed)
    c = np.zeros((frames, N), dtype=np.int64)
    c[:, free] = r.integers(0, 2, (frames, free.size))
    c[:, at] = (c[:, free] @ H[:, free].T) & 1
    return wl.awgn(r, wl.qam_modulate(c, M), float(wl.ebn0_to_n0(snr))).astype(np.complex64)


@pytest.mark.parametrize("N,R,M,S,snr", [
    (32, 1, 4, 6, 4.0), (32, 31, 16, 8, 7.0), (64, 32, 4, 10, 5.0), (64, 33, 64, 10, 12.0), (128, 8, 16, 10, 8.0),
    (128, 65, 16, 12, 8.0), (256, 200, 64, 8, 12.0), (512, 7, 256, 8, 16.0), (1024, 505, 256, 10, 16.0),
    (1024, 505, 256, 10, 26.0), (1024, 512, 4, 10, 6.0),
])
def test_uniform(g, N, R, M, S, snr):
    import torch

    code, H, at, free = random_code(g, N, R, N + R)
    sym = symbols_of(g, H, at, free, N, M, 2048, snr, R)
    sym[3, 0] = np.complex64(complex(np.nan, 0.5))
    sym[4] *= np.float32(60.0)
    F = 16384 + 77
    x = torch.from_numpy(sym[np.random.default_rng(R).integers(0, 2048, F)]).cuda()
    p = g.Params.make(M=M, S=S, query_cap=1 << 16)
    got = g.decode_symbols(code, p, x)
    parts = [g.decode_symbols(code, p, x[i:i + SMALL]) for i in range(0, F, SMALL)]
    table = g.decode_symbols(code, g.Params.make(M=M, S=S, query_cap=1 << 16, tiles=TABLE), x[:2000])
    for k in ("cw", "queries", "abandon"):
        assert torch.equal(got[k], torch.cat([q[k] for q in parts])), k
        assert torch.equal(got[k][:2000], table[k]), k
    code.close()


def test_uneven(g):
    """General codes of different sizes and a polar one, neighbours in one warp."""
    import torch

    r = np.random.default_rng(2)
    made = [random_code(g, *nr, 5) for nr in ((64, 20), (64, 40), (128, 70), (1024, 300))]
    codes = [m[0] for m in made] + [g.Code.polar(64, 32)]
    F = 49152 + 333
    ci = r.choice(5, F, p=[0.3, 0.3, 0.25, 0.05, 0.1])
    N = np.asarray([c.N for c in codes])[ci]
    M = np.where(r.random(F) < 0.5, 16, 64)
    L = np.asarray([wl.symbols_per_frame(int(n), int(m)) for n, m in zip(N, M)])
    so, co = np.cumsum(L) - L, np.cumsum(N // 32) - N // 32
    sym = np.zeros(int(L.sum()), dtype=np.complex64)
    for c in range(5):
        for m in (16, 64):
            idx = np.nonzero((ci == c) & (M == m))[0]
            if c < 4:
                s = symbols_of(g, *made[c][1:], codes[c].N, m, idx.size, 9.0 if m == 16 else 13.0, c + m)
            else:
                s = wl.awgn(r, wl.qam_modulate(r.integers(0, 2, (idx.size, 64)), m), 0.1).astype(np.complex64)
            sym[so[idx][:, None] + np.arange(s.shape[1])] = s
    desc = g.frame_desc(ci, M, so, co)
    d = torch.from_numpy(desc.view(np.uint8).reshape(F, -1).copy()).cuda()
    x, words = torch.from_numpy(sym).cuda(), int((N // 32).sum())
    p = g.Params.make(S=9, query_cap=1 << 16)
    cw, cw_parts = (torch.zeros(words, dtype=torch.int32, device="cuda") for _ in range(2))
    got = g.decode_mixed(codes, p, d.view(-1), x, words, cw=cw)
    parts = [g.decode_mixed(codes, p, d[i:i + SMALL].reshape(-1), x, words, cw=cw_parts) for i in range(0, F, SMALL)]
    for k in ("queries", "abandon"):
        assert torch.equal(got[k], torch.cat([q[k] for q in parts])), k
    assert torch.equal(cw, cw_parts)
    for c in codes:
        c.close()


def test_not_slower_than_the_search(g):
    """20,000 frames of 1024 bits and 512 rows: the one kernel against the TEP search of the same frames."""
    import torch

    code, H, at, free = random_code(g, 1024, 512, 1)
    x = torch.from_numpy(symbols_of(g, H, at, free, 1024, 256, 500, 30.0, 1)).cuda().repeat(40, 1)

    def time(p):
        ms = []
        for _ in range(12):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            g.decode_symbols(code, p, x)
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        return float(np.median(ms[2:]))

    one = time(g.Params.make(M=256, S=10, query_cap=1 << 20))
    search = time(g.Params.make(M=256, S=10, query_cap=1 << 20, tiles=TABLE))
    assert one < search, (one, search)
    code.close()
