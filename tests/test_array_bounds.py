"""What a caller's demodulated arrays can make the decoder address (the public call trusts their contents): the
flip positions of every hard index and mask byte stay inside the word, and a selection always finds a symbol. The
device functions are compiled for the host and run on the CPU; the GPU test compares whole calls."""
from __future__ import annotations

import os
import shutil
import subprocess

import numpy as np
import pytest

import workloads as wl

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

PROGRAM = r"""
#include <stdio.h>
#include "device_common.cuh"
using namespace grand;
// positions of grand_demod's own arrays by definition: neighbouring levels inside the constellation
static int gray(int l) { return l ^ (l >> 1); }
static uint32_t by_labels(int first, int m, int l, int dir, int N) {
  const int change = gray(l) ^ gray(l + dir);
  for (int b = 0; b < m; ++b)
    if (change == 1 << (m - 1 - b)) return first + b < N ? first + b : kNoPos;
  return 0;
}
int main() {
  for (int N = 32; N <= 1024; N <<= 1)
    for (int m = 1; m <= 6; ++m) {
      const int L = (N + 2 * m - 1) / (2 * m);
      for (int i = 0; i < L; ++i)
        for (int l = 0; l < 256; ++l)
          for (int dir = -1; dir <= 1; dir += 2) {
            const uint32_t I = flip_pos_I(i, m, l, dir, N), Q = flip_pos_Q(i, m, l, dir, N);
            // the one-kernel decode's form: threshold k = level + (direction up) - 1
            const uint32_t k = (uint32_t)l + (dir > 0) - 1u;
            if (flip_pos(2 * m * i + m, (int)(k + 1u), N) != I || flip_pos(2 * m * i + 2 * m, (int)(k + 1u), N) != Q)
              return printf("forms differ N=%d m=%d i=%d l=%d\n", N, m, i, l), 1;
            if ((I != kNoPos && I >= (uint32_t)N) || (Q != kNoPos && Q >= (uint32_t)N))
              return printf("outside the word N=%d m=%d i=%d l=%d dir=%d: %u %u\n", N, m, i, l, dir, I, Q), 1;
            if (l < 1 << m && l + dir >= 0 && l + dir < 1 << m &&
                (I != by_labels(2 * m * i, m, l, dir, N) || Q != by_labels(2 * m * i + m, m, l, dir, N)))
              return printf("not the label's bit N=%d m=%d i=%d l=%d dir=%d: %u %u\n", N, m, i, l, dir, I, Q), 1;
          }
    }
  const uint32_t keys[] = {0u, 5u, 0x7FFFFFFFu, 0xFFFFFFFDu, 0xFFFFFFFEu, 0xFFFFFFFFu};
  for (uint32_t k : keys)
    if (selection_key(k) >= 0xFFFFFFFFu || selection_key(k) > k || (k < 0xFFFFFFFFu && selection_key(k) != k))
      return printf("key %u\n", k), 1;
  puts("ok");
  return 0;
}
"""


@pytest.mark.skipif(not os.path.exists(NVCC), reason="no nvcc")
def test_flip_positions_of_any_array(tmp_path):
    src = tmp_path / "positions.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "positions")
    subprocess.run([NVCC, "-O1", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2405_01808_gb300", "csrc"),
                    "-o", exe, str(src)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("N,M", [(128, 16), (64, 4), (1024, 16), (512, 4)])  # at most 32 symbols a frame, and more
@pytest.mark.parametrize("tiles", [(0, 0, 0, 0), (1, 0, 0, 0)])              # one kernel; preparation and search
def test_largest_key(N, M, tiles):
    """Keys of 2^32 - 1 are the least reliable of all: a frame of nothing else takes its first symbols, as a frame
    of equal small keys does."""
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2405_01808_gb300 as g

    g.build()
    code = g.Code.polar(N, N // 2)
    _, frozen = g.polar_H(N, N // 2)
    d = wl.qam_frames(3, 0, 40, N, np.setdiff1d(np.arange(N), frozen), M, 6.0)
    a = g.demod(torch.from_numpy(d["symbols"]).cuda(), M, N)
    p = g.Params.make(M=M, S=10, query_cap=1 << 20, tiles=tiles)
    shape = a["key"].shape
    pairs = []
    for seed, kept in ((0, 0), (1, 3)):  # no smaller key, and three of them
        few = np.zeros(shape, dtype=bool)
        if kept:
            r = np.random.default_rng(seed)
            for f in range(shape[0]):
                few[f, r.permutation(shape[1])[:kept]] = True
        small = np.where(few, 1, 7).astype(np.uint32)
        huge = np.where(few, 1, 0xFFFFFFFF).astype(np.uint32)
        pairs.append([g.decode_batch(code, p, a["y"], a["hard_idx"], torch.from_numpy(k.view(np.int32)).cuda(),
                                     a["nmask"]) for k in (small, huge)])
    torch.cuda.synchronize()
    for want, got in pairs:
        for k in ("cw", "queries", "abandon"):
            assert torch.equal(want[k], got[k]), k
    code.close()
