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
SMALL = 8000


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
