"""The five-point order with the library's choice of the test is not slower than the walk of its TEPs (membership
DELTA) where the walk has little to do: small caps, and codes whose few parity bits fill the space with codewords."""
from __future__ import annotations

import numpy as np
import pytest

from test_gpu_fused import assert_equal, coded_symbols, g  # noqa: F401

pytestmark = pytest.mark.gpu


def both(g, N, K, S, cap, snr, frames, reps=12):
    """Median times of the library's choice and of the walk, their outputs compared."""
    import torch

    code = g.Code.polar(N, K)
    x = torch.from_numpy(coded_symbols(g, N, K, 16, frames, snr, N + K)).cuda()
    out, t = [], []
    for membership in (g.MEMBERSHIP_AUTO, g.MEMBERSHIP_DELTA):
        p = g.Params.make(order=g.ORDER_QAM_NNE5, M=16, S=S, query_cap=cap, membership=membership)
        ms = []
        for _ in range(reps):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            r = g.decode_symbols(code, p, x)
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        out.append(r)
        t.append(float(np.median(ms[2:])))
    assert_equal(out[0], out[1], f"K={K} cap={cap}")
    code.close()
    return t


@pytest.mark.parametrize("S,cap", [(10, 50), (10, 1500), (10, 3125), (9, 625), (2, 5)])
def test_small_caps(g, S, cap):  # noqa: F811
    chosen, walk = both(g, 128, 64, S, cap, 6.0, 3000, reps=32)
    assert chosen < 1.15 * walk, (chosen, walk)


@pytest.mark.parametrize("S,cap", [(10, 3126), (10, 3127), (9, 626), (8, 626), (1, 2)])
def test_first_caps_of_the_join(g, S, cap):  # noqa: F811
    both(g, 128, 64, S, cap, 6.0, 500, reps=3)


@pytest.mark.parametrize("N,K,S,cap,snr", [(128, 122, 10, 1 << 20, 8.0), (128, 120, 10, 1 << 20, 8.0),
                                           (128, 116, 10, 5000, 6.0), (32, 24, 8, 1 << 20, 3.0), (128, 118, 9, 1 << 20, 6.0)])
def test_few_parity_bits(g, N, K, S, cap, snr):  # noqa: F811
    chosen, walk = both(g, N, K, S, cap, snr, 300)
    assert chosen < 1.5 * walk, (chosen, walk)


@pytest.mark.parametrize("kind,N,R,S", [("units", 128, 40, 10), ("units", 64, 14, 10), ("sparse", 256, 36, 9),
                                        ("sparse", 128, 14, 10)])
def test_repeated_columns(g, kind, N, R, S):  # noqa: F811
    """Many lower codes of one syndrome, confirmed on one and two syndrome words."""
    import torch
    from test_gpu_fused import matrix, symbols_of

    code = g.Code(g.H_from_dense(matrix(kind, N, R, N + S)), N, N - R)
    x = torch.from_numpy(symbols_of(N, 4, 90, 4.0, R)).cuda()
    a, b = (g.decode_symbols(code, g.Params.make(order=g.ORDER_QAM_NNE5, M=4, S=S, query_cap=1 << 20, membership=m), x)
            for m in (g.MEMBERSHIP_AUTO, g.MEMBERSHIP_DELTA))
    assert_equal(a, b, kind)
    code.close()
