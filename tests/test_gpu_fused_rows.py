"""Large uniform batches are prepared by a thread per frame: the same outputs as the same frames in batches small
enough for the warp per frame, and the same as the TEP-by-TEP search on a prefix. Every constellation (frames of 3 to
512 symbols, whole and partial steps of 8), cut-offs of each kernel and beyond the frame, orders, likelihood readings,
a matrix not of polar form, and among the frames values that are not finite, keys beyond the packed range and ties."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

FRAMES = 16384 + 128 * 3 + 37  # a last tile and a last warp that are partly empty
SMALL = 8000  # below every size from which the thread per frame is used


@pytest.mark.parametrize("N,M,S,order,lik,matrix", [
    (32, 4, 10, "nne", 0, "polar"), (32, 256, 12, "nearer", 0, "polar"), (32, 4096, 8, "nne", 1, "polar"),
    (64, 64, 12, "nne", 0, "random"), (128, 16, 0, "nne", 0, "polar"), (128, 16, 10, "nne", 0, "polar"),
    (128, 1024, 9, "nearer", 1, "polar"), (256, 64, 8, "nne", 0, "polar"), (256, 16, 11, "nne", 1, "random"),
    (512, 64, 12, "nearer", 0, "polar"), (1024, 256, 12, "nne", 0, "polar"), (1024, 4, 10, "nne", 0, "polar"),
])
def test_thread_per_frame(N, M, S, order, lik, matrix):
    import torch

    import paper_2405_01808_gb300 as g

    r = np.random.default_rng(N + M + S)
    if matrix == "polar":
        code = g.Code.polar(N, N // 2)
    else:
        H = r.integers(0, 2, (24, N))
        H[:, r.permutation(N)[:24]] = np.eye(24, dtype=np.int64)
        code = g.Code(g.H_from_dense(H), N, N - 24)
    _, frozen = g.polar_H(N, N // 2)
    c = wl.random_codewords(r, 2048, N, np.setdiff1d(np.arange(N), frozen))
    snr = {4: 5.0, 16: 8.0, 64: 12.0, 256: 16.0, 1024: 20.0, 4096: 24.0}[M]
    sym = wl.awgn(r, wl.qam_modulate(c, M), float(wl.ebn0_to_n0(snr))).astype(np.complex64)
    L = sym.shape[1]
    sym[1] = np.complex64(0.125 - 0.125j)                # equal keys
    sym[2] *= np.float32(60.0)                           # every key saturates
    sym[3, L - 1] *= np.float32(1e30)
    sym[4, 0] = np.complex64(complex(np.inf, 0.5))
    sym[5, L - 1] = np.complex64(complex(0.5, np.nan))
    sym[6, L // 2] = np.complex64(complex(-np.inf, np.nan))
    x = torch.from_numpy(sym[r.integers(0, 2048, FRAMES)]).cuda()
    p = g.Params.make(order=g.ORDER_QAM_NNE if order == "nne" else g.ORDER_QAM_NEARER, M=M, S=S, query_cap=1 << 16,
                      lik_variant=lik)
    rows = g.decode_symbols(code, p, x)
    parts = [g.decode_symbols(code, p, x[i:i + SMALL]) for i in range(0, FRAMES, SMALL)]
    pt = g.Params.make(order=p.order, M=M, S=S, query_cap=1 << 16, lik_variant=lik, tiles=(1, 0, 0, 0))
    table = g.decode_symbols(code, pt, x[:3000])
    for k in ("cw", "queries", "abandon"):
        assert torch.equal(rows[k], torch.cat([q[k] for q in parts])), k
        assert torch.equal(rows[k][:3000], table[k]), k
    code.close()


@pytest.mark.parametrize("S,lik,membership", [(10, 0, "auto"), (8, 1, "auto"), (12, 0, "solve")])
def test_large_uneven_batch(S, lik, membership):
    """A large uneven batch is put in order by frame length and prepared by a thread per frame: the same outputs as its
    descriptors in slices small enough for the warp per frame. All constellations, polar codes and a random matrix,
    descriptors that name no frame, values that are not finite or saturate, words that no frame owns."""
    import torch

    import paper_2405_01808_gb300 as g

    r = np.random.default_rng(S)
    codes = [g.Code.polar(n, n // 2) for n in (32, 64, 128, 512, 1024)]
    H = r.integers(0, 2, (20, 64))
    H[:, r.permutation(64)[:20]] = np.eye(20, dtype=np.int64)
    codes.append(g.Code(g.H_from_dense(H), 64, 44))
    F = 49152 + 1111
    ci = r.integers(0, len(codes), F)
    M = np.asarray([4, 16, 64, 256, 1024, 4096])[r.integers(0, 6, F)]
    N = np.asarray([c.N for c in codes])[ci]
    L = np.asarray([wl.symbols_per_frame(int(n), int(m)) for n, m in zip(N, M)])
    so = np.cumsum(L + 1) - L
    co = np.cumsum(N // 32 + 1) - N // 32
    sym = np.zeros(int(so[-1] + L[-1]), dtype=np.complex64)
    for m in np.unique(M):
        for n in np.unique(N):
            idx = np.nonzero((M == m) & (N == n))[0]
            s = wl.qam_modulate(r.integers(0, 2, (idx.size, n)), int(m))
            snr = {4: 5.0, 16: 8.0, 64: 12.0, 256: 16.0, 1024: 20.0, 4096: 24.0}[int(m)]
            s = wl.awgn(r, s, float(wl.ebn0_to_n0(snr))).astype(np.complex64)
            s[0] *= np.float32(60.0)
            s[1, -1] = np.complex64(complex(np.nan, 0.5))
            s[2, 0] *= np.float32(1e30)
            sym[so[idx][:, None] + np.arange(s.shape[1])] = s
    desc = g.frame_desc(ci, M, so, co)
    words = int(co[-1] + N[-1] // 32)
    for f, (field, value) in {5: ("M", 8), 77: ("code", 6), 1234: ("sym_offset", len(sym)), 4321: ("cw_offset", words),
                              20000: ("sym_offset", -1), 32900: ("cw_offset", 2 ** 63 - 1)}.items():
        desc[f][field] = value
    d = torch.from_numpy(desc.view(np.uint8).reshape(F, -1).copy()).cuda()
    x = torch.from_numpy(sym).cuda()
    p = g.Params.make(S=S, query_cap=1 << 16, lik_variant=lik,
                      membership=g.MEMBERSHIP_AUTO if membership == "auto" else g.MEMBERSHIP_SOLVE)
    ps = g.Params.make(S=S, query_cap=1 << 16, lik_variant=lik)

    def buffers(n):
        return {"queries": torch.zeros(n, dtype=torch.int32, device="cuda"),
                "abandon": torch.zeros(n, dtype=torch.uint8, device="cuda")}

    cw, cw_parts = (torch.full((words,), 0x5A5A5A5A, dtype=torch.int32, device="cuda") for _ in range(2))
    got = g.decode_mixed(codes, p, d.view(-1), x, words, cw=cw, **buffers(F))
    parts = [g.decode_mixed(codes, ps, d[i:i + SMALL].reshape(-1), x, words, cw=cw_parts, **buffers(len(d[i:i + SMALL])))
             for i in range(0, F, SMALL)]
    for k in ("queries", "abandon"):
        assert torch.equal(got[k], torch.cat([q[k] for q in parts])), k
    assert torch.equal(cw, cw_parts)
    assert (got["abandon"] == 3).sum().item() == 6
    for c in codes:
        c.close()
