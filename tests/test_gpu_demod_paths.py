"""grand_demod's vector widths (four, two and one symbols per thread, by the outputs' alignment) and its path for
symbols far outside the constellation: the same arrays as the aligned call, and the oracle's."""
from __future__ import annotations

import numpy as np
import pytest

import workloads as wl
from test_gpu_fused import g, symbols_of  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lik", [0, 1])
@pytest.mark.parametrize("N,M", [(32, 4), (128, 16), (64, 64), (256, 256), (32, 1024), (64, 4096)])
def test_widths_and_far_symbols(g, oracle_lib, N, M, lik):  # noqa: F811
    import torch

    L = wl.symbols_per_frame(N, M)
    F = 67
    sym = symbols_of(N, M, F, wl.bits_per_symbol(M) + 3.0, N + M)
    sym[5:25] *= np.logspace(0, 6, 20).astype(np.float32)[:, None]  # through the int16 clamps
    sym[30, 0] = np.complex64(complex(np.inf, 0.1))
    sym[31, L - 1] = np.complex64(complex(0.1, np.nan))
    sym[32, :] = 0
    x = torch.from_numpy(sym).cuda()
    want = g.demod(x, M, N, lik_variant=lik)
    for f in list(range(5, 25)) + [32, 40, 66]:
        o = oracle_lib.demod(sym[f:f + 1], M, N, literal=bool(lik))
        for k in ("hard_idx", "key", "nmask", "y"):
            got = want[k][f].cpu().numpy().reshape(-1)
            assert np.array_equal(got.astype(np.int64) & 0xFFFFFFFF,
                                  np.asarray(o[k]).reshape(-1).astype(np.int64) & 0xFFFFFFFF), (f, k)
    for skip in (1, 2, 3):  # outputs at odd, even and odd element offsets: one or two symbols per thread
        n = F * L
        out = {"hard_idx": torch.zeros(n + 8, dtype=torch.int16, device="cuda")[skip:skip + n],
               "key": torch.zeros(n + 8, dtype=torch.int32, device="cuda")[skip:skip + n],
               "nmask": torch.zeros(n + 8, dtype=torch.uint8, device="cuda")[skip:skip + n],
               "rel": torch.zeros(n + 8, dtype=torch.float32, device="cuda")[skip:skip + n],
               "y": torch.full((F * (N // 32) + 8,), -1, dtype=torch.int32, device="cuda")[skip:skip + F * (N // 32)]}
        g.demod(x, M, N, lik_variant=lik, outputs=out)
        for k, t in out.items():
            assert torch.equal(t, want[k].reshape(-1)), (skip, k)
        part = g.demod(x, M, N, lik_variant=lik, outputs={"nmask": out["nmask"].clone(), "y": out["y"].clone()})
        assert torch.equal(part["y"], out["y"]) and torch.equal(part["nmask"], out["nmask"])
