// Public demodulation call (Def. III.1, III.2; Alg. 2 Step 1): per-symbol hard
// level, ordering key, neighbour mask, FP32 likelihood, and the packed hard
// word.
#include <type_traits>

#include "axis.cuh"
#include "device_common.cuh"

namespace grand {
namespace {

constexpr unsigned kAll = 0xFFFFFFFFu;
constexpr int kThreads = 256;

struct DemodArgs {
  const float2* symbols;
  int64_t n_sym;
  int L, NW;
  AxisConst ax;
  float2 inv_d;   // 1/d, twice
  uint16_t* hard_idx;
  uint32_t* key;
  uint8_t* nmask;
  float* rel;
  uint32_t* y;
  uint64_t Lmagic;  // ceil(2^64 / L): frame of symbol s = high word of s * Lmagic (exact for s < 2^64 / L)
};

// Square root by the SFU's approximate instruction (relative error about
// 2^-22, far inside the 1e-5 tolerance of the reported likelihood).
__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

struct Out {
  uint32_t hard, key, nmask, label;  // label: Gray labels, I then Q, MSB first
  float rel;
};

// Symbols outside the plain range (beyond the outermost level by more than
// about six units, or not finite): integer arithmetic with the int16 clamps.
template <int kM, int kLit>
__device__ __noinline__ Out demod_far(float q, float inv_d, float2 v) {
  const bool nf = !(isfinite(v.x) && isfinite(v.y));
  if (nf) v = make_float2(0.0f, 0.0f);
  const AxisDemod I = demod_axis_q(v.x, q, 1 << kM, kLit), Q = demod_axis_q(v.y, q, 1 << kM, kLit);
  Out o;
  o.hard = (uint32_t)((I.level << 8) | Q.level);
  o.key = (uint32_t)I.dq * (uint32_t)I.dq + (uint32_t)Q.dq * (uint32_t)Q.dq;
  o.nmask = make_nmask(I, Q, nf);
  const float dI = axis_dist_f32(v.x, inv_d, I.amp, I.outside, kLit);
  const float dQ = axis_dist_f32(v.y, inv_d, Q.amp, Q.outside, kLit);
  o.rel = sqrt_approx(dI * dI + dQ * dQ);
  o.label = ((uint32_t)gray_code(I.level) << kM) | (uint32_t)gray_code(Q.level);
  return o;
}

// One symbol. Everything but the label's Gray map and the key's mask runs on
// the FMA pipe: truth values are floats 0 / 1 (a saturated difference of
// integers), combined by multiply-adds -- the integer form (157 instructions
// a symbol, the ALU pipe 88 % busy) bounded the kernel at 0.46 of the copy
// bandwidth.
template <int kM, int kLit>
__device__ __forceinline__ Out demod_one(const AxisRegs& ax, F2 inv_d, float2 v) {
  const F2 raw = pack2(v);
  const F2 x = grid2(raw, ax);
  const float2 xs = unpack2(x);
  if (!(fabsf(xs.x) <= ax.lim && fabsf(xs.y) <= ax.lim)) 
    return demod_far<kM, kLit>(unpack2(ax.q).x, unpack2(inv_d).x, v);
  const Axes t = axes_fast(x, ax);
  Out o;
  const float exI = __saturatef(257.0f - fabsf(t.e.x)), exQ = __saturatef(257.0f - fabsf(t.e.y));  // neighbour exists
  const float upI = __saturatef(t.e.x + 1.0f), upQ = __saturatef(t.e.y + 1.0f);                    // level above the threshold
  const float lI = __fadd_rn(t.k.x, upI), lQ = __fadd_rn(t.k.y, upQ);
  float dI = fabsf(t.e.x), dQ = fabsf(t.e.y);
  if (kLit) {
    dI = fmaxf(0.0f, 256.0f - fabsf(dI - 256.0f));
    dQ = fmaxf(0.0f, 256.0f - fabsf(dQ - 256.0f));
  }
  o.key = __float_as_uint(__fadd_rn(__fmaf_rn(dI, dI, __fmul_rn(dQ, dQ)), 8388608.0f)) & 0x7FFFFFu;
  const float lQm = __fadd_rn(lQ, kMagic);
  o.hard = __float_as_uint(__fmaf_rn(lI, 256.0f, lQm)) & 0xFFFFu;
  const uint32_t lv = __float_as_uint(__fmaf_rn(lI, (float)(1 << kM), lQm)) & ((1u << (2 * kM)) - 1u);
  o.label = lv ^ ((lv >> 1) & ~(1u << (kM - 1)));
  // direction of the neighbour: across the threshold, outward beyond the
  // outermost level
  const float dirI = __fmaf_rn(exI, 1.0f - 2.0f * upI, upI), dirQ = __fmaf_rn(exQ, 1.0f - 2.0f * upQ, upQ);
  float mask = __fmaf_rn(exQ, 2.0f, exI);
  mask = __fmaf_rn(exI * exQ, 4.0f, mask);
  mask = __fmaf_rn(dirI, 8.0f, mask);
  mask = __fmaf_rn(dirQ, 16.0f, mask);
  mask = __fmaf_rn(__saturatef(dI - dQ), 32.0f, mask);
  o.nmask = __float_as_uint(__fadd_rn(mask, kMagic)) & 0xFFu;
  // likelihood distance from the unquantised value: 1 - |A - a|, beyond the
  // outermost level 1 + |A - a| (threshold reading)
  const float2 xr = unpack2(mul2(raw, inv_d));
  constexpr float kTop = (float)((1 << kM) - 1);
  const float mI = fabsf(__fmaf_rn(lI, 2.0f, -kTop) - xr.x), mQ = fabsf(__fmaf_rn(lQ, 2.0f, -kTop) - xr.y);
  const float rI = kLit ? 1.0f - mI : __fmaf_rn(__fmaf_rn(exI, -2.0f, 1.0f), mI, 1.0f);
  const float rQ = kLit ? 1.0f - mQ : __fmaf_rn(__fmaf_rn(exQ, -2.0f, 1.0f), mQ, 1.0f);
  o.rel = sqrt_approx(rI * rI + rQ * rQ);
  return o;
}

// kV consecutive symbols per thread (4, 2 or 1, as the pointers' alignment
// allows, checked by the host: vector loads and stores). For 4^m with m = 1,
// 2, 4 a frame fills whole words, so the hard words are the labels' bits one
// after the other and are stored in whole bytes; for the others the label
// bits are ORed into zeroed words (a frame's last symbol may be padded).
// 9.6 M 16-QAM symbols (187 MB): 31 us, 6.0 TB/s, against 60 us of the integer
// form with two symbols per thread, a zeroing pass and an OR per pair.
template <int kV, int kM, int kLit>
__global__ void __launch_bounds__(kThreads, kV == 4 ? 6 : 8) k_demod(const __grid_constant__ DemodArgs a) {
  constexpr int kBits = 2 * kM * kV;  // label bits of the thread's symbols
  constexpr bool kStream = kM == 1 || kM == 2 || kM == 4;
  const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  const int64_t s0 = t * kV;
  const int n = (int)min((int64_t)kV, max((int64_t)0, a.n_sym - s0));  // symbols of this thread
  const AxisRegs ax = axis_regs(a.ax, a.ax.nz);
  const F2 inv_d = pack2(a.inv_d);
  float2 v[kV];
#pragma unroll
  for (int j = 0; j < kV; ++j) v[j] = make_float2(0.0f, 0.0f);
  if (n == kV) {
    if constexpr (kV >= 2) {
      const float4* p = reinterpret_cast<const float4*>(a.symbols + s0);
#pragma unroll
      for (int j = 0; j < kV / 2; ++j) {
        const float4 q = p[j];
        v[2 * j] = make_float2(q.x, q.y);
        v[2 * j + 1] = make_float2(q.z, q.w);
      }
    } else {
      v[0] = a.symbols[s0];
    }
  } else {
#pragma unroll
    for (int j = 0; j < kV; ++j)
      if (j < n) v[j] = a.symbols[s0 + j];
  }
  Out o[kV];
#pragma unroll
  for (int j = 0; j < kV; ++j) o[j] = demod_one<kM, kLit>(ax, inv_d, v[j]);
  if (n == kV) {
    if constexpr (kV == 4) {
      if (a.hard_idx)
        reinterpret_cast<uint2*>(a.hard_idx)[t] = make_uint2(o[0].hard | (o[1].hard << 16), o[2].hard | (o[3].hard << 16));
      if (a.key) reinterpret_cast<uint4*>(a.key)[t] = make_uint4(o[0].key, o[1].key, o[2].key, o[3].key);
      if (a.nmask)
        reinterpret_cast<uint32_t*>(a.nmask)[t] =
            o[0].nmask | (o[1].nmask << 8) | (o[2].nmask << 16) | (o[3].nmask << 24);
      if (a.rel) reinterpret_cast<float4*>(a.rel)[t] = make_float4(o[0].rel, o[1].rel, o[2].rel, o[3].rel);
    } else if constexpr (kV == 2) {
      if (a.hard_idx) reinterpret_cast<uint32_t*>(a.hard_idx)[t] = o[0].hard | (o[1].hard << 16);
      if (a.key) reinterpret_cast<uint2*>(a.key)[t] = make_uint2(o[0].key, o[1].key);
      if (a.nmask) reinterpret_cast<uint16_t*>(a.nmask)[t] = (uint16_t)(o[0].nmask | (o[1].nmask << 8));
      if (a.rel) reinterpret_cast<float2*>(a.rel)[t] = make_float2(o[0].rel, o[1].rel);
    } else {
      if (a.hard_idx) a.hard_idx[s0] = (uint16_t)o[0].hard;
      if (a.key) a.key[s0] = o[0].key;
      if (a.nmask) a.nmask[s0] = (uint8_t)o[0].nmask;
      if (a.rel) a.rel[s0] = o[0].rel;
    }
  } else {
#pragma unroll
    for (int j = 0; j < kV; ++j) {
      if (j >= n) continue;
      if (a.hard_idx) a.hard_idx[s0 + j] = (uint16_t)o[j].hard;
      if (a.key) a.key[s0 + j] = o[j].key;
      if (a.nmask) a.nmask[s0 + j] = (uint8_t)o[j].nmask;
      if (a.rel) a.rel[s0 + j] = o[j].rel;
    }
  }
  if (!a.y) return;
  if constexpr (kStream) {
    // labels first symbol highest, reversed at the end: bit k of the stream is
    // the k-th transmitted bit. The symbol count is a multiple of 16 / m.
    uint32_t w = 0;
#pragma unroll
    for (int j = 0; j < kV; ++j) w |= (j < n ? o[j].label : 0u) << (kBits - 2 * kM * (j + 1));
    constexpr int kGroup = kBits < 8 ? 8 / kBits : 1;  // lanes that fill a byte
    const int g = (int)(threadIdx.x % kGroup);
    if constexpr (kGroup > 1) {
      w <<= kBits * (kGroup - 1 - g);
#pragma unroll
      for (int d = 1; d < kGroup; d <<= 1) w |= __shfl_xor_sync(kAll, w, d);
    }
    constexpr int kAllBits = kBits * kGroup;
    const uint32_t r = __brev(w) >> (32 - kAllBits);
    if (n > 0 && g == 0) {
      if constexpr (kAllBits == 32) a.y[t] = r;
      else if constexpr (kAllBits == 16) reinterpret_cast<uint16_t*>(a.y)[t] = (uint16_t)r;
      else reinterpret_cast<uint8_t*>(a.y)[t / kGroup] = (uint8_t)r;
    }
  } else {
    if (n == 0) return;
    int64_t f = (int64_t)__umul64hi((uint64_t)s0, a.Lmagic);
    int i = (int)(s0 - f * a.L);
    // bits of up to kV symbols of one frame, 24 at most a time
#pragma unroll
    for (int j = 0; j < kV; ++j) {
      if (j >= n) break;
      const uint32_t bits = __brev(o[j].label) >> (32 - 2 * kM);
      const int p0 = 2 * kM * i, wd = p0 >> 5, sh = p0 & 31;
      uint32_t* yf = a.y + f * a.NW;
      const uint32_t lo = bits << sh, hi = sh ? bits >> (32 - sh) : 0u;
      if (wd < a.NW && lo) atomicOr(yf + wd, lo);
      if (hi && wd + 1 < a.NW) atomicOr(yf + wd + 1, hi);
      if (++i == a.L) {
        i = 0;
        ++f;
      }
    }
  }
}

// BPSK hard decisions: one warp per 32 samples
__global__ void __launch_bounds__(256) k_demod_bpsk(const float* r, int64_t n_words, uint32_t* y, uint8_t* nmask) {
  const int lane = threadIdx.x & 31;
  for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < n_words;
       w += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    float v = r[32 * w + lane];
    const bool nf = !isfinite(v);
    if (nf) v = 0.0f;
    const unsigned b = __ballot_sync(kAll, v < 0.0f);
    if (lane == 0 && y) y[w] = b;
    if (nmask) nmask[32 * w + lane] = nf ? 128 : 0;
  }
}

template <int kV, int kM>
void launch_lit(const DemodArgs& a, int lik, cudaStream_t st) {
  const int64_t per_block = (int64_t)kThreads * kV;
  const unsigned grid = (unsigned)((a.n_sym + per_block - 1) / per_block);
  if (lik == GRAND_LIK_LITERAL)
    k_demod<kV, kM, 1><<<grid, kThreads, 0, st>>>(a);
  else
    k_demod<kV, kM, 0><<<grid, kThreads, 0, st>>>(a);
}
template <int kV>
void launch_m(const DemodArgs& a, int m, int lik, cudaStream_t st) {
  switch (m) {
    case 1: launch_lit<kV, 1>(a, lik, st); break;
    case 2: launch_lit<kV, 2>(a, lik, st); break;
    case 3: launch_lit<kV, 3>(a, lik, st); break;
    case 4: launch_lit<kV, 4>(a, lik, st); break;
    case 5: launch_lit<kV, 5>(a, lik, st); break;
    default: launch_lit<kV, 6>(a, lik, st); break;
  }
}

}  // namespace
}  // namespace grand

using namespace grand;

extern "C" int grand_demod(const void* symbols, int64_t n_frames, int L, int M, float N0, int lik_variant,
                           uint16_t* hard_idx, uint32_t* key, uint8_t* nmask, float* rel, uint32_t* y, int N,
                           void* stream) {
  if ((!symbols && n_frames > 0) || n_frames < 0 || !(N0 > 0.0f) || !isfinite(N0)) return GRAND_E_INVALID;
  if (N < GRAND_N_MIN || N > GRAND_N_MAX || (N & (N - 1))) return GRAND_E_INVALID;
  if (lik_variant != GRAND_LIK_THRESHOLD && lik_variant != GRAND_LIK_LITERAL) return GRAND_E_INVALID;
  cudaStream_t st = (cudaStream_t)stream;
  if (M == 2) {
    if (L != N) return GRAND_E_INVALID;
    if (n_frames == 0) return GRAND_OK;
    const int64_t n_words = n_frames * (N / 32);
    const int64_t blocks = (n_words * 32 + 255) / 256;
    k_demod_bpsk<<<(int)(blocks < 65535 * 8 ? blocks : 65535 * 8), 256, 0, st>>>((const float*)symbols, n_words, y,
                                                                                  nmask);
    return cudaGetLastError() == cudaSuccess ? GRAND_OK : GRAND_E_CUDA;
  }
  const int m = m_of(M);
  if (!m || L != (N + 2 * m - 1) / (2 * m)) return GRAND_E_INVALID;
  if (n_frames == 0) return GRAND_OK;
  const QamConst qc = make_qam_const();
  DemodArgs a{};
  a.symbols = (const float2*)symbols;
  a.L = L;
  a.NW = N / 32;
  a.ax = axis_const(m, qc);
  a.inv_d = make_float2(qc.inv_d[m], qc.inv_d[m]);
  a.Lmagic = UINT64_MAX / (uint64_t)L + 1;  // L >= 3 for the supported N and M
  if (y && m != 1 && m != 2 && m != 4 &&
      cudaMemsetAsync(y, 0, sizeof(uint32_t) * (size_t)n_frames * (N / 32), st) != cudaSuccess)
    return GRAND_E_CUDA;
  auto aligned = [](const void* p, uintptr_t b) { return ((uintptr_t)p % b) == 0; };
  const bool by2 = aligned(symbols, 16) && aligned(hard_idx, 4) && aligned(key, 8) && aligned(nmask, 2) &&
                   aligned(rel, 8);
  const bool by4 = by2 && aligned(hard_idx, 8) && aligned(key, 16) && aligned(nmask, 4) && aligned(rel, 16);
  // 2^36 symbols a launch (the grid's limit is 2^31 blocks); a part is a
  // multiple of four whole frames, which keeps every pointer's alignment
  const int64_t part = ((int64_t)1 << 36) / L / 4 * 4;
  for (int64_t f0 = 0; f0 < n_frames; f0 += part) {
    const int64_t nf = n_frames - f0 < part ? n_frames - f0 : part, s0 = f0 * L;
    a.symbols = (const float2*)symbols + s0;
    a.n_sym = nf * L;
    a.hard_idx = hard_idx ? hard_idx + s0 : nullptr;
    a.key = key ? key + s0 : nullptr;
    a.nmask = nmask ? nmask + s0 : nullptr;
    a.rel = rel ? rel + s0 : nullptr;
    a.y = y ? y + f0 * a.NW : nullptr;
    if (by4) launch_m<4>(a, m, lik_variant, st);
    else if (by2) launch_m<2>(a, m, lik_variant, st);
    else launch_m<1>(a, m, lik_variant, st);
  }
  return cudaGetLastError() == cudaSuccess ? GRAND_OK : GRAND_E_CUDA;
}
