"""The five-point order with the library's choice of the test (the join of the two halves of the ranks) against the
TEP-by-TEP walk (membership DELTA): same words, query counts and abandon flags, from no searched rank to full sides,
with caps inside a weight class, codes with few parity bits (many codewords in the space) and general matrices."""
from __future__ import annotations

import numpy as np
import pytest

from test_gpu_fused import assert_equal, coded_symbols, g, matrix, symbols_of  # noqa: F401

pytestmark = pytest.mark.gpu


def pair(g, code, sym, **kw):
    import torch

    x = torch.from_numpy(sym).cuda()
    a = g.decode_symbols(code, g.Params.make(order=g.ORDER_QAM_NNE5, **kw), x, stats=True)
    b = g.decode_symbols(code, g.Params.make(order=g.ORDER_QAM_NNE5, membership=g.MEMBERSHIP_DELTA, **kw), x, stats=True)
    return a, b


@pytest.mark.parametrize("N,K,M,S,cap,snr,frames", [
    (32, 16, 4, 10, 1 << 20, 2.0, 130),
    (32, 26, 16, 8, 1 << 20, 3.0, 61),      # fewer parity bits than walked TEPs need
    (64, 52, 4, 9, 4000, 2.0, 61),          # cap inside a weight class
    (64, 32, 256, 8, 5 ** 8, 13.0, 200),
    (128, 64, 16, 10, 1 << 20, 6.0, 201),
    (128, 64, 16, 10, 1 << 20, 6.0, 1),
    (128, 64, 16, 3, 1 << 20, 6.0, 66),
    (128, 64, 16, 2, 1 << 20, 6.0, 66),     # nothing left for the join
    (128, 64, 16, 5, 300, 6.0, 67),         # cap reached by the walk
    (256, 128, 4096, 7, 5 ** 7, 23.0, 50),
    (1024, 512, 4, 6, 5 ** 6, 5.0, 50),
])
def test_join_equals_walk(g, N, K, M, S, cap, snr, frames):  # noqa: F811
    code = g.Code.polar(N, K)
    sym = coded_symbols(g, N, K, M, frames, snr, N + M + S)
    if frames > 60:
        sym[17, 1] = np.complex64(complex(np.nan, 0.0))
    a, b = pair(g, code, sym, M=M, S=S, query_cap=cap)
    assert_equal(a, b, "join")
    assert a["hard_frames"] == b["hard_frames"] and a["search_useful"] == b["search_useful"]
    assert a["evaluated_checks"] >= b["search_useful"]
    code.close()


@pytest.mark.parametrize("kind,N,R", [("units", 64, 20), ("sparse", 128, 40)])
def test_join_general_matrix(g, kind, N, R):  # noqa: F811
    code = g.Code(g.H_from_dense(matrix(kind, N, R, N)), N, N - R)
    a, b = pair(g, code, symbols_of(N, 16, 70, 6.0, 3), M=16, S=8, query_cap=5 ** 8)
    assert_equal(a, b, kind)
    code.close()
