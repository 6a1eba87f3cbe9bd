"""Performance cases: the calls a user of the decoder makes, at the sizes they are made with.

Every case goes through the public Python entry points. Inputs are what a receiver has in hand:
codewords of the library's polar codes, Gray-labelled M-QAM (or BPSK) points and white Gaussian noise
at the Eb/N0 range in which the constellation is used. Codes have rate 1/2. All decode outputs are
whole numbers; the demodulation's reported likelihood is the one floating-point output.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2405_01808_gb300 as g

MIX_N = (32, 64, 128, 256, 512, 1024)
MIX_M = (4, 16, 64, 256)
# Eb/N0 window of each constellation (nine 1 dB points of a block-error sweep)
SNR_RANGE = {4: (0.0, 8.0), 16: (4.0, 12.0), 64: (8.0, 16.0), 256: (12.0, 20.0), 1024: (16.0, 24.0),
             4096: (20.0, 28.0)}
ORDERS = {"nne": g.ORDER_QAM_NNE, "nearer": g.ORDER_QAM_NEARER, "nne5": g.ORDER_QAM_NNE5, "hamming": g.ORDER_HAMMING}
MEMBERSHIP = {"auto": g.MEMBERSHIP_AUTO, "solve": g.MEMBERSHIP_SOLVE}


def _symbols_call(name, frames, N, M, S, cap, snrs, order="nne", membership="auto", kind="symbols"):
    return {"name": name, "kind": kind, "frames": frames, "N": N, "M": M, "S": S, "cap": cap,
            "snrs": ",".join(str(float(s)) for s in snrs), "order": order, "membership": membership}


def _mixed_call(name, frames, S, cap, snr_lo, snr_hi, membership="auto"):
    return {"name": name, "kind": "mixed", "frames": frames, "S": S, "cap": cap, "snr_lo": snr_lo, "snr_hi": snr_hi,
            "membership": membership}


def listed():
    return [
        # one received frame decoded by its own call: the plain request-response receiver, all latency
        _symbols_call("one_frame_n128", 1, 128, 16, 10, 1 << 20, (8,)),
        # one batch of the serving loop's size under a few million requests/s: frames of every code and constellation
        _mixed_call("serving_batch_400", 400, 10, 1 << 20, 4.0, 14.0),
        # the hard-decision bit-level decoder on short BPSK frames
        {"name": "ab_n32_bpsk_10k", "kind": "ab", "frames": 10000, "N": 32, "snrs": "4.0", "weight": 3, "cap": 5489},
        # the benchmark's default batch: medium code, three Eb/N0 points
        _symbols_call("n128_16qam_300k", 300000, 128, 16, 10, 1 << 20, (6, 8, 10)),
        # long codes with the largest cut-off and query cap
        _symbols_call("n512_64qam_s12_80k", 80000, 512, 64, 12, 1 << 24, (10, 12, 14, 16)),
        _symbols_call("n1024_256qam_s12_20k", 20000, 1024, 256, 12, 1 << 24, (10, 12, 14, 16)),
        # an uneven batch of a million frames in one call
        _mixed_call("mixed_1m", 1000000, 10, 1 << 20, 4.0, 14.0),
        # the same kind of batch (an odd frame count) decided by the linear solve
        _mixed_call("mixed_solve_250k", 250001, 10, 1 << 20, 4.0, 14.0, membership="solve"),
        # one point of a block-error-rate sweep: padded last symbol (256 bits in 43 symbols of 6), paper's cut-off
        _symbols_call("bler_n256_64qam_250k", 250000, 256, 64, 8, 4 ** 8, (12,)),
        # the default batch arriving in and returning to host memory
        _symbols_call("host_n128_16qam_300k", 300000, 128, 16, 10, 1 << 20, (6, 8, 10), kind="host"),
        # soft demodulation alone (another decoder consumes the reliabilities)
        {"name": "demod_n128_16qam_300k", "kind": "demod", "frames": 300000, "N": 128, "M": 16, "snrs": "6.0,8.0,10.0"},
        # the five-point error model, as a study comparing TEP orders runs it
        _symbols_call("nne5_n128_6k", 6000, 128, 16, 10, 1 << 20, (6, 8, 10), order="nne5"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["symbols", "symbols", "symbols", "mixed", "mixed", "solve", "bler", "ab", "host", "demod", "nne5"])
    if kind == "mixed":
        c = _mixed_call("", _log_int(rng, 100, 500000), rng.randint(6, 10), 1 << rng.randint(16, 20), 4.0, 14.0,
                        membership=rng.choice(["auto", "solve"]))
    elif kind == "ab":
        c = {"kind": "ab", "frames": _log_int(rng, 100, 30000), "N": 32, "snrs": str(round(rng.uniform(2.0, 7.0), 2)),
             "weight": rng.randint(1, 3), "cap": 5489}
    else:
        M = rng.choice(sorted(SNR_RANGE))
        N = rng.choice(MIX_N)
        lo, hi = SNR_RANGE[M]
        snrs = [round(rng.uniform(lo, hi), 2) for _ in range(rng.randint(1, 3))]
        if kind == "demod":
            L = -(-N // (M.bit_length() - 1))
            c = {"kind": "demod", "frames": _log_int(rng, 1000, 9600000 // L), "N": N, "M": M,
                 "snrs": ",".join(str(s) for s in snrs)}
        elif kind == "nne5":
            c = _symbols_call("", _log_int(rng, 50, 1500), rng.choice((32, 64, 128, 256)), M, rng.randint(6, 10), 1 << 20,
                              snrs, order="nne5")
        elif kind == "bler":
            c = _symbols_call("", _log_int(rng, 5000, 250000 if N <= 512 else 120000), N, M, 8, 4 ** 8, snrs,
                              order=rng.choice(["nne", "nearer"]))
        else:
            S = rng.randint(6, 12)
            top = (300000 if N <= 128 else 100000) if S <= 10 else 25000
            c = _symbols_call("", _log_int(rng, 1 if kind == "symbols" else 2000, top), N, M, S,
                              1 << (20 if S <= 10 else 24), snrs,
                              membership="solve" if kind == "solve" else "auto",
                              kind="host" if kind == "host" else "symbols")
    c.pop("name", None)
    return c


# --------------------------------------------------------------------------
# transmitter and channel (on the GPU)
# --------------------------------------------------------------------------
def _info_positions(N):
    _, frozen = g.polar_H(N, N // 2)
    return np.setdiff1d(np.arange(N), frozen)


def _codewords(gen, frames, N, info, dev):
    """Uniform information bits through the polar transform: (frames, N) of 0/1."""
    c = torch.zeros((frames, N), dtype=torch.uint8, device=dev)
    c[:, torch.as_tensor(info, device=dev)] = torch.randint(0, 2, (frames, len(info)), generator=gen, device=dev,
                                                            dtype=torch.uint8)
    half = 1
    while half < N:
        v = c.view(frames, N // (2 * half), 2, half)
        v[:, :, 0, :] ^= v[:, :, 1, :]
        half *= 2
    return c


def _qam(gen, bits, M, sigma, dev):
    """Coded bits -> received complex64 symbols (frames, L); sigma per frame (frames, 1)."""
    frames, N = bits.shape
    b = int(M).bit_length() - 1
    m = b // 2
    L = -(-N // b)
    padded = torch.zeros((frames, L * b), dtype=torch.uint8, device=dev)
    padded[:, :N] = bits
    padded = padded.view(frames, L, 2, m).to(torch.int32)
    label = (padded << torch.arange(m - 1, -1, -1, device=dev, dtype=torch.int32)).sum(dim=3)
    side = 1 << m
    levels = torch.arange(side, device=dev)
    amp = torch.empty(side, dtype=torch.float64, device=dev)
    amp[levels ^ (levels >> 1)] = (2 * levels - (side - 1)).to(torch.float64) * math.sqrt(3.0 * m / (M - 1))
    x = amp[label]
    x += torch.randn(x.shape, generator=gen, device=dev, dtype=torch.float64) * sigma.view(-1, 1, 1)
    return torch.view_as_complex(x.to(torch.float32).contiguous())


def _sigma(snr_db):
    return np.sqrt(0.5 * np.power(10.0, -np.asarray(snr_db, dtype=np.float64) / 10.0))


def _frame_snrs(case):
    points = [float(s) for s in case["snrs"].split(",")]
    return np.array(points)[np.arange(case["frames"]) * len(points) // case["frames"]]


def _generator(seed, dev):
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    return gen


def _uniform_symbols(case, seed, dev):
    gen = _generator(seed, dev)
    bits = _codewords(gen, case["frames"], case["N"], _info_positions(case["N"]), dev)
    return _qam(gen, bits, case["M"], torch.as_tensor(_sigma(_frame_snrs(case)), device=dev), dev)


def _mixed_batch(case, seed, dev):
    F = case["frames"]
    r = np.random.default_rng(int(seed))
    # every (N, M) class in equal shares, in random order
    cls = r.permutation(F) % (len(MIX_N) * len(MIX_M))
    code = cls // len(MIX_M)
    M = np.asarray(MIX_M)[cls % len(MIX_M)]
    sigma = _sigma(r.uniform(case["snr_lo"], case["snr_hi"], F))
    N = np.asarray(MIX_N)[code]
    bps = np.rint(np.log2(M)).astype(np.int64)
    L = -(-N // bps)
    sym_off = np.concatenate(([0], np.cumsum(L)))
    cw_off = np.concatenate(([0], np.cumsum(N // 32)))
    gen = _generator(seed, dev)
    symbols = torch.empty(int(sym_off[-1]), dtype=torch.complex64, device=dev)
    for ci, n in enumerate(MIX_N):
        info = _info_positions(n)
        for m in MIX_M:
            idx = np.nonzero((code == ci) & (M == m))[0]
            if idx.size == 0:
                continue
            rx = _qam(gen, _codewords(gen, idx.size, n, info, dev), m, torch.as_tensor(sigma[idx], device=dev), dev)
            at = torch.as_tensor(sym_off[idx], device=dev).view(-1, 1) + torch.arange(rx.shape[1], device=dev)
            symbols[at.view(-1)] = rx.view(-1)
    desc = g.frame_desc(code, M, sym_off[:-1], cw_off[:-1])
    return symbols, torch.from_numpy(desc.view(np.uint8)).to(dev), int(cw_off[-1])


# --------------------------------------------------------------------------
# the measured calls
# --------------------------------------------------------------------------
def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    kind = case["kind"]
    st = {"kind": kind}
    if kind == "mixed":
        st["symbols"], st["desc"], st["cw_words"] = _mixed_batch(case, seed, dev)
        st["codes"] = [g.Code.polar(n, n // 2) for n in MIX_N]
        st["params"] = g.Params.make(S=case["S"], query_cap=case["cap"], membership=MEMBERSHIP[case["membership"]])
        return st
    N = case["N"]
    if kind == "ab":
        gen = _generator(seed, dev)
        tx = 1.0 - 2.0 * _codewords(gen, case["frames"], N, _info_positions(N), dev).to(torch.float64)
        sigma = torch.as_tensor(_sigma(_frame_snrs(case)), device=dev).view(-1, 1)
        st["symbols"] = (tx + torch.randn(tx.shape, generator=gen, device=dev, dtype=torch.float64) * sigma).float()
        st["params"] = g.Params.make(order=g.ORDER_HAMMING, M=2, max_weight=case["weight"], query_cap=case["cap"])
        st["code"] = g.Code.polar(N, N // 2)
        return st
    st["symbols"] = _uniform_symbols(case, seed, dev)
    if kind == "demod":
        st["M"], st["N"] = case["M"], N
        return st
    st["code"] = g.Code.polar(N, N // 2)
    st["params"] = g.Params.make(order=ORDERS[case["order"]], M=case["M"], S=case["S"], query_cap=case["cap"],
                                 membership=MEMBERSHIP[case["membership"]])
    if kind == "host":  # page-locked buffers, as the call's documentation asks for
        F = case["frames"]
        st["symbols"] = st["symbols"].cpu().pin_memory()
        st["cw"] = torch.empty((F, N // 32), dtype=torch.int32, pin_memory=True)
        st["queries"] = torch.empty(F, dtype=torch.int32, pin_memory=True)
        st["abandon"] = torch.empty(F, dtype=torch.uint8, pin_memory=True)
    return st


def run(state):
    kind = state["kind"]
    if kind == "mixed":
        return g.decode_mixed(state["codes"], state["params"], state["desc"], state["symbols"], state["cw_words"])
    if kind == "demod":
        return g.demod(state["symbols"], state["M"], state["N"])
    if kind == "host":
        return g.decode_symbols_host(state["code"], state["params"], state["symbols"], cw=state["cw"],
                                     queries=state["queries"], abandon=state["abandon"])
    return g.decode_symbols(state["code"], state["params"], state["symbols"])


def work(case):
    """Received symbols (and descriptors) read once, results written once. The decode's arithmetic is integer
    logic; the floating-point operations are the demodulation's: scaling both axes and the squared distance."""
    F = case["frames"]
    kind = case["kind"]
    if kind == "mixed":
        per = [(n, -(-n // (m.bit_length() - 1))) for n in MIX_N for m in MIX_M]
        L = sum(l for _, l in per) / len(per)
        N = sum(n for n, _ in per) / len(per)
        return {"bytes": F * (8 * L + 24 + N / 8 + 5), "flops": F * 5 * L}
    N = case["N"]
    if kind == "ab":
        return {"bytes": F * (4 * N + N / 8 + 5), "flops": F * N}
    L = -(-N // (case["M"].bit_length() - 1))
    if kind == "demod":
        return {"bytes": F * (8 * L + 11 * L + N / 8), "flops": F * 12 * L}
    return {"bytes": F * (8 * L + N / 8 + 5), "flops": F * 5 * L}


def exact(case, seed):
    """The reported likelihood of the demodulation in 64 bits. The other outputs are whole numbers."""
    if case["kind"] != "demod":
        return None
    dev = torch.device("cuda", torch.cuda.current_device())
    x = torch.view_as_real(_uniform_symbols(case, seed, dev))
    M = case["M"]
    m = (M.bit_length() - 1) // 2
    side = 1 << m
    d = math.sqrt(3.0 * m / (M - 1))
    # the hard level is decided on the fixed-point grid of 1/256 (a part of the call's definition)
    aq = torch.round(x * torch.tensor(256.0 / d, dtype=torch.float32, device=dev)).clamp(-32768, 32767).to(torch.float64)
    level = torch.floor((aq + 256 * side) / 512).clamp(0, side - 1)
    A = 2 * level - (side - 1)
    outside = ((level == 0) & (aq < 256 * A)) | ((level == side - 1) & (aq > 256 * A))
    mag = (A - x.to(torch.float64) / d).abs()
    dist = torch.where(outside, 1 + mag, 1 - mag)
    rel = dist.pow(2).sum(dim=2).sqrt()
    return {"y": None, "hard_idx": None, "key": None, "nmask": None, "rel": rel}
