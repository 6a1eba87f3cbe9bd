"""Coordinates whose product with the grid's scale rounds to a half: the hard level, the threshold and the existence
of an alternative follow the rounded product (round to even of it), not the exact one. Every route of the decode
against the preparation kernel's integer arithmetic (an explicit launch shape), and the demodulation against the
oracle."""
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


def half_coordinates(M):
    """Floats a with fl(a q) half an integer and a q not; those next to a level or a threshold apart."""
    side = 1 << (M.bit_length() - 1) // 2
    q = np.float32(256.0 / np.sqrt(1.5 * (M.bit_length() - 1) / (M - 1)))
    n = np.arange(-256 * side - 300, 256 * side + 300) + 0.5
    a = (n / np.float64(q)).astype(np.float32)
    out = []
    for step in range(-2, 3):
        v = a.copy()
        for _ in range(abs(step)):
            v = np.nextafter(v, np.float32(np.inf if step > 0 else -np.inf))
        keep = ((v * q) == n.astype(np.float32)) & (v.astype(np.float64) * np.float64(q) != n)
        out.append(np.stack([v[keep], n[keep].astype(np.float32)]))
    v, n = np.concatenate(out, axis=1)
    near = np.abs((n / 256.0) - np.rint(n / 256.0)) < 0.01
    return v, v[near]


def frames_of(M, N, frames, seed):
    r = np.random.default_rng(seed)
    L = wl.symbols_per_frame(N, M)
    every, near = half_coordinates(M)
    assert every.size > 20 and near.size > 0
    x = np.where(r.random((frames, L, 2)) < 0.5, r.choice(every, (frames, L, 2)), r.choice(near, (frames, L, 2)))
    # a quarter of the symbols in noise between them, so that the selections differ
    d = np.float32(1.0 / np.sqrt(1.5 * (M.bit_length() - 1) / (M - 1)))
    side = 1 << (M.bit_length() - 1) // 2
    noise = (r.random((frames, L, 1)) < 0.25)
    x = np.where(noise, (r.uniform(-side, side, (frames, L, 2)) / d).astype(np.float32), x)
    return np.ascontiguousarray(x.astype(np.float32)).view(np.complex64)[..., 0]


def assert_equal(a, b, label):
    for k in ("abandon", "queries", "cw"):
        x, y = a[k].cpu().numpy(), b[k].cpu().numpy()
        bad = np.nonzero(x != y)[0]
        assert bad.size == 0, f"{label}: {k} differs in {bad.size} places, first {bad[:6].tolist()}"


@pytest.mark.parametrize("M,N", [(16, 128), (16, 256), (64, 128), (64, 512), (256, 512), (1024, 128),
                                 (4096, 256)])
@pytest.mark.parametrize("frames", [1500, 17000])  # a warp per frame, a thread per frame
def test_decode(g, M, N, frames):
    import torch

    x = torch.from_numpy(frames_of(M, N, frames, M + N)).cuda()
    r = np.random.default_rng(N)
    R = N // 2
    # no codeword in reach (the query count is the number of valid TEPs), and one in most reaches
    codes = [g.Code(g.H_from_dense(np.concatenate([r.integers(0, 2, (R, N - R)), np.eye(R, dtype=int)], 1)), N, N - R),
             g.Code.polar(N, N - 9)]
    d = g.demod(x, M, N)
    args = (d["y"], d["hard_idx"], d["key"], d["nmask"])
    for code in codes:
        for lik in (0, 1):
            kw = dict(M=M, S=8, query_cap=4 ** 8, lik_variant=lik)
            want = g.decode_symbols(code, g.Params.make(**kw, tiles=TABLE), x)
            assert_equal(g.decode_symbols(code, g.Params.make(**kw), x), want, f"symbols K={code.K} lik={lik}")
            if lik == 0:
                assert_equal(g.decode_batch(code, g.Params.make(**kw), *args), want, f"arrays K={code.K}")
        code.close()


@pytest.mark.parametrize("frames", [1500, 49500])  # as it comes, in order of length
def test_uneven(g, frames):
    import torch

    r = np.random.default_rng(frames)
    codes = [g.Code.polar(64, 32), g.Code.polar(64, 55)]
    Ms = (16, 64, 256, 1024)
    M = np.repeat(Ms, -(-frames // 4))[:frames]
    L = np.asarray([wl.symbols_per_frame(64, int(m)) for m in M])
    so = np.cumsum(L) - L
    sym = np.concatenate([frames_of(m, 64, int((M == m).sum()), m).ravel() for m in Ms])
    order = r.permutation(frames)
    desc = g.frame_desc(r.integers(0, 2, frames), M[order], so[order], 2 * np.arange(frames))
    x, dd = torch.from_numpy(sym).cuda(), torch.from_numpy(desc.view(np.uint8)).cuda()
    kw = dict(M=0, S=8, query_cap=4 ** 8)
    want = g.decode_mixed(codes, g.Params.make(**kw, tiles=TABLE), dd, x, 2 * frames)
    assert_equal(g.decode_mixed(codes, g.Params.make(**kw), dd, x, 2 * frames), want, "uneven")
    for c in codes:
        c.close()


@pytest.mark.parametrize("M,N", [(16, 128), (64, 128), (256, 128), (1024, 128), (4096, 256)])
def test_demodulation(g, oracle_lib, M, N):
    import torch

    sym = frames_of(M, N, 3000, M)
    want = oracle_lib.demod(sym, M, N)
    got = g.demod(torch.from_numpy(sym).cuda(), M, N)
    for k in ("y", "hard_idx", "key", "nmask"):
        a = got[k].cpu().numpy()
        assert np.array_equal(a.view(want[k].dtype) if a.dtype.itemsize == want[k].dtype.itemsize else a, want[k]), k
