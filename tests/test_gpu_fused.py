"""The one-kernel decode (AUTO with automatic tiles, and SOLVE) against the two-kernel TEP search (an explicit
warps-per-CTA setting), which tests every TEP: same decoded words, query counts and abandon flags over the forms
both accept -- code rates and matrices that leave large solution sets, every constellation, orders, likelihood
readings, cut-offs, caps inside a weight class, odd batch sizes, demodulated arrays and uneven batches."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

TABLE = (1, 0, 0, 0)  # one warp per frame of the TEP-by-TEP search


@pytest.fixture(scope="module")
def g():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2405_01808_gb300 as grand

    grand.build()
    return grand


def host(r):
    return {k: r[k].cpu().numpy() for k in ("cw", "queries", "abandon")}


def assert_equal(a, b, label):
    a, b = host(a), host(b)
    for k in ("abandon", "queries", "cw"):
        bad = np.nonzero(a[k] != b[k])[0]
        assert bad.size == 0, f"{label}: {k} differs in {bad.size} places, first {bad[:6].tolist()}"


def symbols_of(N, M, frames, snr, seed):
    """Random bits through the mapper and the channel (the decoders need no codeword)."""
    r = np.random.default_rng(seed)
    rx = wl.awgn(r, wl.qam_modulate(r.integers(0, 2, (frames, N)), M), float(wl.ebn0_to_n0(snr)))
    return rx.astype(np.complex64)


def coded_symbols(g, N, K, M, frames, snr, seed):
    _, frozen = g.polar_H(N, K)
    r = np.random.default_rng(seed)
    c = wl.random_codewords(r, frames, N, np.setdiff1d(np.arange(N), frozen))
    return wl.awgn(r, wl.qam_modulate(c, M), float(wl.ebn0_to_n0(snr))).astype(np.complex64)


def matrix(kind, N, R, seed):
    """Parity-check matrices not of polar form, full row rank by an identity block."""
    r = np.random.default_rng(seed)
    H = r.integers(0, 2, (R, N)) if kind == "random" else np.zeros((R, N), dtype=np.int64)
    if kind == "units":  # every column a unit vector: few distinct columns, heavy first hits
        H[r.integers(0, R, N), np.arange(N)] = 1
    elif kind == "sparse":  # zero and repeated columns among random ones
        cols = r.integers(0, 2, (R, N // 4))
        H = cols[:, r.integers(0, N // 4, N)]
        H[:, r.random(N) < 0.2] = 0
    at = r.permutation(N)[:R]
    H[:, at] = np.eye(R, dtype=np.int64)
    return H


def both(g, code, sym, **kw):
    import torch

    x = torch.from_numpy(sym).cuda()
    out = []
    for extra in ({"tiles": TABLE}, {}, {"membership": g.MEMBERSHIP_SOLVE}):
        out.append(g.decode_symbols(code, g.Params.make(**kw, **extra), x))
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("N,K,M,S,cap,snr,frames,order,lik", [
    (32, 16, 4, 12, 1 << 24, 1.0, 333, 1, 0),
    (32, 16, 256, 12, 1 << 20, 12.0, 129, 2, 0),   # fewer symbols than S
    (32, 28, 4, 12, 1 << 20, 2.0, 257, 1, 0),      # 4 parity bits: kernels of 20 dimensions and more
    (32, 22, 16, 8, 300, 4.0, 128, 1, 0),          # 10 parity bits, cap inside a weight class
    (64, 32, 4, 10, 1 << 20, 3.0, 1000, 1, 0),
    (64, 20, 64, 11, 1 << 22, 8.0, 97, 2, 1),
    (64, 48, 4, 9, 5000, 3.0, 700, 1, 0),
    (128, 64, 16, 10, 1 << 20, 6.0, 4097, 1, 0),
    (128, 64, 16, 10, 1 << 20, 6.0, 1, 1, 0),
    (128, 100, 4, 10, 1 << 20, 4.0, 513, 1, 1),
    (128, 64, 1024, 12, 1 << 24, 19.0, 200, 2, 0),
    (256, 128, 64, 8, 4 ** 8, 12.0, 2050, 1, 0),   # padded last symbol
    (256, 128, 4096, 10, 1 << 20, 24.0, 300, 1, 0),
    (512, 256, 4, 6, 1 << 12, 5.0, 700, 2, 0),
    (1024, 512, 4, 10, 1 << 20, 6.0, 300, 1, 0),   # 512 symbols a frame
    (1024, 900, 256, 12, 1 << 20, 18.0, 130, 1, 0),
    (128, 64, 16, 0, 10, 9.0, 40, 1, 0),
    (128, 64, 16, 1, 10, 9.0, 40, 1, 0),
])
def test_polar_codes(g, N, K, M, S, cap, snr, frames, order, lik):
    code = g.Code.polar(N, K)
    sym = coded_symbols(g, N, K, M, frames, snr, N + K + M + S)
    want, auto, solve = both(g, code, sym, order=order, M=M, S=S, query_cap=cap, lik_variant=lik)
    assert_equal(auto, want, "auto")
    assert_equal(solve, want, "solve")
    code.close()


@pytest.mark.parametrize("kind,N,R,M,S,frames,cap", [
    ("random", 64, 20, 16, 10, 200, 1 << 20),
    ("random", 128, 64, 4, 10, 200, 1 << 20),
    ("random", 1024, 512, 256, 10, 60, 1 << 20),
    ("units", 64, 8, 4, 10, 100, 1 << 20),
    ("units", 128, 40, 16, 10, 100, 1 << 20),  # two syndrome words, dependent columns
    ("sparse", 128, 48, 64, 12, 100, 1 << 22),
    ("sparse", 256, 70, 4, 8, 100, 3000),
])
def test_general_matrices(g, kind, N, R, M, S, frames, cap):
    H = matrix(kind, N, R, 11 * N + R)
    code = g.Code(g.H_from_dense(H), N, N - R)
    want, auto, solve = both(g, code, symbols_of(N, M, frames, 6.0, R), M=M, S=S, query_cap=cap)
    assert_equal(auto, want, kind)
    assert_equal(solve, want, kind)
    code.close()


def test_selection_corner_cases(g):
    """The least reliable symbols all in one lane's share of a long frame; equal keys everywhere; keys beyond the
    packed range; non-finite symbols."""
    N, M = 1024, 4
    code = g.Code.polar(N, N // 2)
    sym = coded_symbols(g, N, N // 2, M, 70, 20.0, 5)
    sym[:20, 5::32] = np.complex64(0.01 + 0.02j) * np.arange(1, 17, dtype=np.float32)  # 16 symbols of lane 5
    sym[20:30, 64:200] = np.complex64(0.125 - 0.125j)                                  # ties
    sym[30:40] *= np.float32(40.0)                                                     # every key saturates
    sym[40, 3] = np.complex64(complex(np.inf, 1.0))
    sym[41, 511] = np.complex64(complex(0.0, np.nan))
    want, auto, solve = both(g, code, sym, M=M, S=10, query_cap=1 << 18)
    assert_equal(auto, want, "auto")
    assert_equal(solve, want, "solve")
    code.close()
    small = g.Code.polar(32, 16)
    sym = coded_symbols(g, 32, 16, 16, 64, 6.0, 6)
    sym[:30] *= np.logspace(0, 3, 30).astype(np.float32)[:, None]
    want, auto, _ = both(g, small, sym, M=16, S=8, query_cap=1 << 16)
    assert_equal(auto, want, "scaled")
    small.close()


@pytest.mark.parametrize("N,M,S", [(128, 16, 10), (256, 4096, 12), (512, 4, 8)])
def test_demodulated_arrays(g, N, M, S):
    import torch

    code = g.Code.polar(N, N // 2)
    sym = coded_symbols(g, N, N // 2, M, 301, wl.bits_per_symbol(M) + 3.0, N + M)
    sym[:20] *= np.float32(3.0)  # beyond the outermost levels
    x = torch.from_numpy(sym).cuda()
    for order in (g.ORDER_QAM_NNE, g.ORDER_QAM_NEARER):
        d = g.demod(x, M, N)
        args = (d["y"], d["hard_idx"], d["key"], d["nmask"])
        want = g.decode_batch(code, g.Params.make(order=order, M=M, S=S, query_cap=1 << 20, tiles=TABLE), *args)
        got = g.decode_batch(code, g.Params.make(order=order, M=M, S=S, query_cap=1 << 20), *args)
        fused = g.decode_symbols(code, g.Params.make(order=order, M=M, S=S, query_cap=1 << 20), x)
        assert_equal(got, want, "arrays")
        assert_equal(fused, want, "symbols")
    code.close()


def test_uneven_batch(g):
    """Polar and general codes, every constellation, a gap and invalid descriptors; an odd number of frames."""
    import torch

    codes = [g.Code.polar(n, n // 2) for n in (32, 128, 1024)]
    codes.append(g.Code(g.H_from_dense(matrix("random", 64, 30, 3)), 64, 34))
    r = np.random.default_rng(8)
    F = 1501
    ci = r.integers(0, len(codes), F)
    M = np.asarray([4, 16, 64, 256, 1024, 4096])[r.integers(0, 6, F)]
    N = np.asarray([c.N for c in codes])[ci]
    L = np.asarray([wl.symbols_per_frame(int(n), int(m)) for n, m in zip(N, M)])
    so = np.cumsum(L) - L + 3
    co = np.cumsum(N // 32) - N // 32
    sym = np.zeros(int(L.sum()) + 3, dtype=np.complex64)
    for f in range(F):
        sym[so[f]:so[f] + L[f]] = symbols_of(int(N[f]), int(M[f]), 1, 2.0 + 2 * wl.bits_per_symbol(int(M[f])), f)[0]
    desc = g.frame_desc(ci, M, so, co)
    desc["code"][7], desc["M"][8], desc["sym_offset"][9], desc["cw_offset"][1500] = 9, 8, -1, 10 ** 9
    desc["M"][64], desc["sym_offset"][65] = 0, sym.size - 1
    x, d = torch.from_numpy(sym).cuda(), torch.from_numpy(desc.view(np.uint8)).cuda()
    words = int((N // 32).sum())
    out = []
    for extra in ({"tiles": TABLE}, {}, {"membership": g.MEMBERSHIP_SOLVE}):
        cw = torch.zeros(words, dtype=torch.int32, device="cuda")
        out.append(g.decode_mixed(codes, g.Params.make(S=9, query_cap=1 << 18, **extra), d, x, words, cw=cw))
    assert_equal(out[1], out[0], "auto")
    assert_equal(out[2], out[0], "solve")
    ab = host(out[1])["abandon"]
    assert all(ab[f] == 3 for f in (7, 8, 9, 64, 65, 1500))
    for c in codes:
        c.close()
