// The symbol-level decode in one kernel (Alg. 2 Steps 1-5 for the paper's
// four-alternative model), for the calls whose membership test is the
// library's choice (GRAND_MEMBERSHIP_AUTO with automatic tiles) or the linear
// solve (GRAND_MEMBERSHIP_SOLVE).
//
// The valid TEPs of a frame are the flip vectors x over its existing I / Q
// slots (bit 2r: the first single-axis slot of rank r, bit 2r+1: the second,
// both: the diagonal alternative), and H (y xor e(x)) = 0 reads
// XOR_{b in x} c_b = s(y) with c_b the syndrome change of slot b. The
// codewords of the TEP space are the solutions of this GF(2) system, and the
// first hit is the solution of smallest canonical position (none: abandoned
// after min(valid TEPs, cap) queries).
//
// k_decode works on tiles of 4 T frames per CTA in two mappings:
//   front  one warp per frame, T frames one after the other: symbols are read
//          coalesced (the next 32 are in flight while 32 are worked on), the
//          hard word is packed by byte stores, the S' least reliable symbols
//          are picked by warp minima. What is left of a frame is its hard
//          word and S' symbol records in shared memory.
//   solve  one thread per frame: the base syndrome by the polar transform of
//          the hard word, the slot columns' 32-bit projections, Gaussian
//          elimination with the columns in registers, the check of the
//          solution on the full syndrome, its canonical position in closed
//          form and the outputs. A warp instruction serves 32 frames here,
//          where a warp per frame spent a ballot and a shuffle per slot on one.
#include <type_traits>

#include "device_common.cuh"
#include "fused.cuh"
#include "host_util.cuh"

namespace grand {
namespace {

constexpr unsigned kAll = 0xFFFFFFFFu;
constexpr int kWarps = 4;               // warps per CTA
constexpr uint32_t kNone = 0xFFFFFFFFu;
constexpr uint32_t kKeySat = 0x7FFFFFu; // packed selection keys hold 23 bits of the reliability
constexpr int kLanePick = 3;            // smallest keys kept per lane of a long frame

// e_v(n1, n3): valid TEPs altering exactly v of n1 ranks with one alternative
// and n3 ranks with three = the coefficient of x^v in (1 + x)^n1 (1 + 3x)^n3;
// cum: the number with fewer than v altered ranks.
struct EspTable {
  uint32_t e[kSMax + 1][kSMax + 1][kSMax + 2];
  uint32_t cum[kSMax + 1][kSMax + 1][kSMax + 2];
};
constexpr EspTable make_esp() {
  EspTable t{};
  for (int a = 0; a <= kSMax; ++a)
    for (int b = 0; a + b <= kSMax; ++b) {
      if (a == 0 && b == 0) {
        t.e[0][0][0] = 1;
      } else {
        const int pa = a > 0 ? a - 1 : a, pb = a > 0 ? b : b - 1;
        const uint32_t k = a > 0 ? 1u : 3u;
        for (int v = 0; v <= kSMax + 1; ++v)
          t.e[a][b][v] = t.e[pa][pb][v] + (v > 0 ? k * t.e[pa][pb][v - 1] : 0u);
      }
      for (int v = 1; v <= kSMax + 1; ++v) t.cum[a][b][v] = t.cum[a][b][v - 1] + t.e[a][b][v - 1];
    }
  return t;
}
__device__ const EspTable g_esp = make_esp();

// One axis on the Q8.8 grid (the reading of demod_axis_q): k = the inner
// decision threshold nearest to the received value (k separates the levels
// k - 1 and k), e = the signed distance to it. Ties between two thresholds go
// to the lower one, so that the neighbour of a value on a level is the lower
// level; |e| > 256 says the value lies beyond the outermost level, where the
// neighbouring level across the far threshold does not exist.
struct Axis {
  int k, e;
};
__device__ __forceinline__ Axis axis_at(float a, float q, int side) {
  int aq;
  const float x = fminf(fmaxf(__fmul_rn(a, q), -32768.0f), 32767.0f);
  aq = __float2int_rn(x);
  const int t = aq + 256 * side;
  Axis r;
  r.k = min(max((t + 255) >> 9, 1), side - 1);
  r.e = t - (r.k << 9);
  return r;
}
// Distance of the ordering key (threshold or literal reading).
__device__ __forceinline__ int axis_dist(int e, int literal) {
  const int m = e < 0 ? -e : e;
  const int lit = max(0, 512 - m);
  return literal && m > 256 ? lit : min(m, 32767);
}

// A selected symbol: index (bits 0..8), threshold of each axis (9..14,
// 15..20), existing alternatives (21 I, 22 Q), Q nearer than I (23).
__device__ __forceinline__ uint32_t pack_rec(int i, int kI, int kQ, bool exI, bool exQ, bool near) {
  return (uint32_t)i | ((uint32_t)kI << 9) | ((uint32_t)kQ << 15) | (exI ? 1u << 21 : 0u) | (exQ ? 1u << 22 : 0u) |
         (near ? 1u << 23 : 0u);
}

__device__ __forceinline__ uint32_t transform_word(uint32_t x) {  // superset sums inside a word
  x ^= (x >> 1) & 0x55555555u;
  x ^= (x >> 2) & 0x33333333u;
  x ^= (x >> 4) & 0x0F0F0F0Fu;
  x ^= (x >> 8) & 0x00FF00FFu;
  x ^= (x >> 16) & 0x0000FFFFu;
  return x;
}

// Bits i of a word with i a subset of t: the polar transform of bit t.
__device__ __forceinline__ uint32_t subset_pattern(uint32_t t) {
  uint32_t p = 1u;
#pragma unroll
  for (int b = 0; b < 5; ++b)
    if ((t >> b) & 1u) p |= p << (1 << b);
  return p;
}

// Where a symbol's demodulation comes from.
enum { kFromUniform = 0, kFromMixed = 1, kFromArrays = 2 };

struct Sym {
  uint32_t key;    // full ordering key
  uint32_t rec;    // record bits without the index
  uint32_t label;  // Gray label bits in transmission order (bit k = label bit 2m-1-k)
  bool nf;         // a coordinate is not finite (read as 0)
};

__device__ __forceinline__ Sym demod_symbol(float2 v, float q, int m, int lik) {
  Sym s;
  const int side = 1 << m;
  s.nf = !(isfinite(v.x) && isfinite(v.y));
  if (s.nf) v = make_float2(0.0f, 0.0f);
  const Axis I = axis_at(v.x, q, side), Q = axis_at(v.y, q, side);
  const int dI = axis_dist(I.e, lik), dQ = axis_dist(Q.e, lik);
  s.key = (uint32_t)(dI * dI) + (uint32_t)(dQ * dQ);
  s.rec = pack_rec(0, I.k, Q.k, I.e >= -256 && I.e <= 256, Q.e >= -256 && Q.e <= 256, dQ < dI);
  const uint32_t lv = ((uint32_t)(I.k + (I.e >> 31)) << m) | (uint32_t)(Q.k + (Q.e >> 31));
  const uint32_t gray = lv ^ ((lv >> 1) & ~(1u << (m - 1)));
  s.label = __brev(gray) >> (32 - 2 * m);
  return s;
}

// One symbol of a call on demodulated arrays (its hard word is an input).
__device__ __forceinline__ Sym array_symbol(const DecodeArgs& a, int64_t o) {
  Sym s;
  const uint32_t h = a.hard_idx[o], nm = a.nmask[o];
  s.key = a.key[o];
  s.nf = (nm & 128u) != 0;
  // the threshold toward the neighbour (0 or 2^m: none there, and no alternative)
  const int kI = ((int)(h >> 8) + (int)((nm >> 3) & 1u)) & 63, kQ = ((int)(h & 0xFFu) + (int)((nm >> 4) & 1u)) & 63;
  s.rec = pack_rec(0, kI, kQ, nm & 1u, nm & 2u, nm & 32u);
  s.label = 0;
  return s;
}

template <int kFrom>
__device__ __forceinline__ Sym symbol_at(const DecodeArgs& a, int64_t base, int i, float q, int m) {
  if constexpr (kFrom == kFromArrays) return array_symbol(a, base + i);
  else return demod_symbol(a.symbols[base + i], q, m, a.lik);
}

// Exact selection of the S' smallest (key, index) pairs, S' scans of the
// frame: for the rare frame whose packed keys do not settle it (a selected
// key saturates, or one lane of a long frame ran out of kept keys). Lane r
// returns the index of rank r.
template <int kFrom>
__device__ __noinline__ int select_exact(const DecodeArgs& a, int64_t base, int L, int Sp, float q, int m) {
  const int lane = threadIdx.x & 31;
  uint32_t last_k = 0;
  int last_i = -1, sel = 0;
  for (int r = 0; r < Sp; ++r) {
    uint32_t bk = kNone, bi = kNone;
    for (int i = lane; i < L; i += 32) {
      const uint32_t k = symbol_at<kFrom>(a, base, i, q, m).key;
      const bool after = k > last_k || (k == last_k && i > last_i);
      if (after && k < bk) { bk = k; bi = (uint32_t)i; }
    }
    const uint32_t kmin = __reduce_min_sync(kAll, bk);
    const uint32_t imin = __reduce_min_sync(kAll, bk == kmin ? bi : kNone);
    if (lane == r) sel = (int)imin;
    last_k = kmin;
    last_i = (int)imin;
  }
  return sel;
}

// ---------------------------------------------------------------------------
// Solve helpers (one thread per frame)
// ---------------------------------------------------------------------------

// What a thread needs to look at its frame: its column of the shared words
// (masked transform of y for polar-form H, else the compact syndrome), the
// slot positions and the code.
struct Frame {
  uint32_t* buf;        // word w at buf[w * stride]
  const uint32_t* pos;  // rank r: positions of its two slots (16 bits each) at pos[r * pstride]
  int stride, pstride;
  const uint32_t* fmask;  // frozen bits of each word (polar form)
  const uint32_t* hcol;   // packed columns, W words each
  int W;
  const uint32_t* pat;  // shared: subset_pattern of 0..31
  int nw;               // syndrome words in buf
  int polar;
};

__device__ __forceinline__ uint32_t slot_pos(const Frame& f, int b) {
  return (f.pos[(b >> 1) * f.pstride] >> (16 * (b & 1))) & 0xFFFFu;
}

// Word w of slot b's syndrome change.
__device__ __forceinline__ uint32_t column_word(const Frame& f, uint32_t p, int w) {
  if (p == kNoPos) return 0u;
  if (f.polar) return ((uint32_t)w & ~(p >> 5)) ? 0u : f.pat[p & 31u] & __ldg(f.fmask + w);
  return __ldg(f.hcol + (size_t)p * f.W + w);
}

// XOR of the slot columns over x (and the base syndrome) is zero everywhere.
__device__ __noinline__ bool sum_zero(const Frame f, uint32_t x, bool base) {
  for (int w = 0; w < f.nw; ++w) {
    uint32_t acc = base ? f.buf[w * f.stride] : 0u;
    for (uint32_t t = x; t; t &= t - 1u) acc ^= column_word(f, slot_pos(f, __ffs(t) - 1), w);
    if (acc) return false;
  }
  return true;
}

// The same test of s(y) xor the columns of x for polar-form H, in place: a
// flipped bit p changes only the words that are subsets of p >> 5. The base
// syndrome is destroyed.
__device__ __forceinline__ bool consume_zero_polar(const Frame& f, uint32_t x) {
  for (uint32_t t = x; t; t &= t - 1u) {
    const uint32_t p = slot_pos(f, __ffs(t) - 1);
    if (p == kNoPos) continue;
    const uint32_t pt = f.pat[p & 31u], sup = p >> 5;
    uint32_t w = sup;
    for (;;) {
      f.buf[w * f.stride] ^= pt & __ldg(f.fmask + w);
      if (w == 0) break;
      w = (w - 1u) & sup;
    }
  }
  uint32_t orr = 0;
  for (int w = 0; w < f.nw; ++w) orr |= f.buf[w * f.stride];
  return orr == 0;
}

__device__ __forceinline__ uint32_t altered(uint32_t x) { return (x | (x >> 1)) & 0x55555555u; }

// Canonical order as an integer comparison: weight first, then colex order of
// the altered ranks (their mask as a number), then the alternatives from the
// heaviest digit down (the code itself: h = 1 < v = 2 < diag = 3).
__device__ __forceinline__ uint32_t order_key(uint32_t x) {
  const uint32_t m = altered(x);
  return ((uint32_t)__popc(m) << 24) | m;  // the mask of 12 ranks takes 24 bits
}
__device__ __forceinline__ bool comes_before(uint32_t k, uint32_t x, uint32_t bk, uint32_t bx) {
  return k < bk || (k == bk && x < bx);
}

// 1-based position of TEP x among the valid TEPs. one / both: ranks with one
// alternative and with three (bit 2r).
__device__ __forceinline__ uint32_t tep_position(uint32_t x, uint32_t one, uint32_t both) {
  const uint32_t m = altered(x);
  uint32_t acc = 0, alt = 0, low = 1;
  int i = 0;
  for (uint32_t t = m; t; t &= t - 1u) {
    const int b = __ffs(t) - 1;
    const uint32_t below = (1u << b) - 1u;
    const uint32_t three = (both >> b) & 1u;
    const uint32_t k = three ? 3u : 1u;
    ++i;
    acc = acc * k + g_esp.e[__popc(one & below)][__popc(both & below)][i];
    alt += (three ? ((x >> b) & 3u) - 1u : 0u) * low;
    low *= k;
  }
  return g_esp.cum[__popc(one)][__popc(both)][i] + acc + alt + 1u;
}

// The projection of slot b's column.
struct Proj {
  const uint32_t* tab;
  __device__ __forceinline__ uint32_t operator()(uint32_t p) const { return p == kNoPos ? 0u : __ldg(tab + p); }
};

// First TEP of weight <= wmax in canonical order whose projection equals f0
// and which passes the full test, or kNone.
__device__ __noinline__ uint32_t light_hit(const Frame f, const Proj proj, uint32_t ex, int Sp, uint32_t f0,
                                           bool exact, int wmax) {
  auto delta = [&](int r, int c) {
    uint32_t d = 0;
    if (c & 1) d ^= proj(slot_pos(f, 2 * r));
    if (c & 2) d ^= proj(slot_pos(f, 2 * r + 1));
    return d;
  };
  auto valid = [&](int r, int c) { return ((ex >> (2 * r)) & (uint32_t)c) == (uint32_t)c; };
  auto full = [&](uint32_t x) { return exact || sum_zero(f, x, true); };
  if (f0 == 0 && full(0u)) return 0u;
  for (int p = 0; wmax >= 1 && p < Sp; ++p)
    for (int c = 1; c <= 3; ++c)
      if (valid(p, c) && delta(p, c) == f0 && full((uint32_t)c << (2 * p))) return (uint32_t)c << (2 * p);
  for (int p = 1; wmax >= 2 && p < Sp; ++p)
    for (int o = 0; o < p; ++o)
      for (int c = 1; c <= 3; ++c) {
        if (!valid(p, c)) continue;
        const uint32_t z = f0 ^ delta(p, c);
        for (int d = 1; d <= 3; ++d) {
          const uint32_t x = ((uint32_t)c << (2 * p)) | ((uint32_t)d << (2 * o));
          if (valid(o, d) && delta(o, d) == z && full(x)) return x;
        }
      }
  for (int p = 2; wmax >= 3 && p < Sp; ++p)
    for (int o = 1; o < p; ++o)
      for (int n = 0; n < o; ++n)
        for (int c = 1; c <= 3; ++c) {
          if (!valid(p, c)) continue;
          const uint32_t z = f0 ^ delta(p, c);
          for (int d = 1; d <= 3; ++d) {
            if (!valid(o, d)) continue;
            const uint32_t zz = z ^ delta(o, d);
            for (int e = 1; e <= 3; ++e) {
              const uint32_t x = ((uint32_t)c << (2 * p)) | ((uint32_t)d << (2 * o)) | ((uint32_t)e << (2 * n));
              if (valid(n, e) && delta(n, e) == zz && full(x)) return x;
            }
          }
        }
  return kNone;
}

// First solution in canonical order among x0 + span(kv[0..d)), d >= 1 (a
// Gray-code walk; every solution is a valid TEP). exact: the projection
// decides. Else: when every kernel vector passes the full test the projected
// kernel is the true one, and x0 decides for all; otherwise (the projection
// lost rank on the columns) every candidate is tested.
// The walk costs 2^d steps; codes with few parity bits have large kernels,
// and then their first hit is light: weights <= 2 (630 TEPs at most), and
// above 2^11 solutions weight 3 (5,940), are tested first.
__device__ __noinline__ uint32_t first_solution(const Frame f, const Proj proj, uint32_t ex, int Sp, uint32_t f0,
                                                bool exact, uint32_t x0, const uint32_t* kv, int d,
                                                unsigned long long* ranked) {
  bool each = false;
  if (!exact) {
    for (int t = 0; t < d && !each; ++t) each = !sum_zero(f, kv[t], false);
    if (!each && !sum_zero(f, x0, true)) return kNone;
  }
  if (d > 8) {
    const uint32_t x = light_hit(f, proj, ex, Sp, f0, exact || !each, d > 11 ? 3 : 2);
    if (x != kNone) {
      *ranked += 1;
      return x;
    }
  }
  *ranked += 1ull << d;
  uint32_t x = x0, bk = kNone, bx = kNone;
  for (uint32_t i = 0;;) {
    const uint32_t k = order_key(x);
    if (comes_before(k, x, bk, bx) && (!each || sum_zero(f, x, true))) {
      bk = k;
      bx = x;
    }
    if (++i >> d) break;
    x ^= kv[__ffs(i) - 1];
  }
  return bx;
}

// ---------------------------------------------------------------------------
// The kernel
// ---------------------------------------------------------------------------
// kOne: every frame has at most 32 symbols (one per lane). kSlots: 2 x the
// largest S' (16, 20 or 24: the elimination is unrolled over it).
template <int kFrom, bool kOne, int kSlots>
__global__ void __launch_bounds__(32 * kWarps, 8) k_decode(const __grid_constant__ DecodeArgs a) {
  extern __shared__ __align__(16) char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int FT = kWarps * a.T;
  const int stride = FT + 1;  // odd: a frame's words fall into different banks
  constexpr int kRanks = kSlots / 2;
  int64_t* s_off = reinterpret_cast<int64_t*>(smem_raw);             // [FT] mixed: first symbol
  int64_t* s_cw = s_off + (kFrom == kFromMixed ? FT : 0);            // [FT] mixed: first output word
  uint32_t* s_par = reinterpret_cast<uint32_t*>(s_cw + (kFrom == kFromMixed ? FT : 0));  // [FT] mixed: L | m | code
  uint32_t* pat = s_par + (kFrom == kFromMixed ? FT : 0);            // [32]
  uint32_t* s_f0 = pat + 32;                                         // [FT] projection of s(y) (H not of polar form)
  uint32_t* s_flag = s_f0 + FT;                                      // [FT] 0, or the abandon flag of an undecodable frame
  uint32_t* rec = s_flag + FT;                                       // [kRanks][FT]
  uint32_t* buf = rec + kRanks * FT;                                 // [NWmax][stride]
  const int64_t tile = (int64_t)blockIdx.x * FT;
  const int n_here = (int)min((int64_t)FT, a.n_frames - tile);

  if (threadIdx.x < 32) pat[threadIdx.x] = subset_pattern(threadIdx.x);
  for (int t = threadIdx.x; t < a.NWmax * stride; t += 32 * kWarps) buf[t] = 0u;
  for (int t = threadIdx.x; t < FT; t += 32 * kWarps) s_flag[t] = 0u;
  if constexpr (kFrom == kFromMixed) {
    for (int t = threadIdx.x; t < n_here; t += 32 * kWarps) {
      const grand_frame_desc d = a.desc[tile + t];
      const int m = (31 - __clz(d.M)) >> 1;
      bool ok = d.code >= 0 && d.code < a.n_codes && m >= 1 && m <= 6 && d.M == 1 << (2 * m) && d.sym_offset >= 0 &&
                d.cw_offset >= 0;
      int L = 0;
      if (ok) {
        const int N = a.codes[d.code].N;
        L = (N + 2 * m - 1) / (2 * m);
        ok = d.sym_offset + L <= a.n_symbols && d.cw_offset + (N >> 5) <= a.n_cw_words;
      }
      s_off[t] = d.sym_offset;
      s_cw[t] = d.cw_offset;
      s_par[t] = ok ? (uint32_t)L | ((uint32_t)m << 10) | ((uint32_t)d.code << 13) : 1u << 10;  // L = 0: not decoded
    }
  }
  __syncthreads();

  // --- front: one warp per frame ---------------------------------------------
  int um = 0, uL = 0;
  if constexpr (kFrom != kFromMixed) {
    um = (31 - __clz(a.M)) >> 1;
    uL = a.L;
  }
  const int fr_end = min(n_here, (warp + 1) * a.T);
  auto frame_base = [&](int fr) { return kFrom == kFromMixed ? s_off[fr] : (tile + fr) * (int64_t)uL; };
  auto frame_len = [&](int fr) { return kFrom == kFromMixed ? (int)(s_par[fr] & 1023u) : uL; };
  float2 nxt = make_float2(0.0f, 0.0f);
  if constexpr (kFrom != kFromArrays) {
    const int fr = warp * a.T;
    if (fr < fr_end && lane < frame_len(fr)) nxt = a.symbols[frame_base(fr) + lane];
  }
  for (int fr = warp * a.T; fr < fr_end; ++fr) {
    const int64_t base = frame_base(fr);
    const int L = frame_len(fr);
    const int m = kFrom == kFromMixed ? (int)((s_par[fr] >> 10) & 7u) : um;
    const CodeDev* code = kFrom == kFromMixed ? a.codes + (s_par[fr] >> 13) : a.codes;
    const float q = a.qc.q[m];
    const int Sp = a.S < L ? a.S : L;
    const int b2 = 2 * m;
    uint32_t* y = buf + fr;
    uint32_t best[kOne ? 1 : kLanePick];
#pragma unroll
    for (int j = 0; j < (kOne ? 1 : kLanePick); ++j) best[j] = kNone;
    uint32_t info = 0;
    bool nf = false;
    const int nch = kOne ? 1 : max(1, (L + 31) >> 5);
    const int nbytes = kFrom == kFromMixed ? code->N >> 3 : a.NWmax * 4;
    for (int c = 0; c < nch; ++c) {
      const int i = 32 * c + lane;
      const bool on = i < L;
      const float2 cur = nxt;
      if constexpr (kFrom != kFromArrays) {  // the next 32 symbols, of this frame or the next one
        if (!kOne && c + 1 < nch) {
          if (i + 32 < L) nxt = a.symbols[base + i + 32];
        } else if (fr + 1 < fr_end) {
          if (lane < frame_len(fr + 1)) nxt = a.symbols[frame_base(fr + 1) + lane];
        }
      }
      Sym s{kNone, 0u, 0u, false};
      if constexpr (kFrom == kFromArrays) {
        if (on) s = array_symbol(a, base + i);
      } else {
        s = demod_symbol(cur, q, m, a.lik);
        if (!on) { s.label = 0u; s.nf = false; }
        // the group of symbols that fills whole bytes ORs its labels together
        // and stores them (4, 2, 1 symbols a byte for m = 1, 2, 4; 4 symbols
        // in 3 bytes for m = 3); m = 5, 6 OR into the word
        uint8_t* yb = reinterpret_cast<uint8_t*>(y);
        auto put = [&](int byte, uint32_t v) {
          if (byte < nbytes) yb[(byte >> 2) * (4 * stride) + (byte & 3)] = (uint8_t)v;
        };
        if (m == 1) {
          uint32_t v = s.label << (2 * (lane & 3));
          v |= __shfl_xor_sync(kAll, v, 1);
          v |= __shfl_xor_sync(kAll, v, 2);
          if ((lane & 3) == 0) put(i >> 2, v);
        } else if (m == 2) {
          uint32_t v = s.label << (4 * (lane & 1));
          v |= __shfl_xor_sync(kAll, v, 1);
          if ((lane & 1) == 0) put(i >> 1, v);
        } else if (m == 4) {
          put(i, s.label);
        } else if (m == 3) {
          uint32_t v = s.label << (6 * (lane & 3));
          v |= __shfl_xor_sync(kAll, v, 1);
          v |= __shfl_xor_sync(kAll, v, 2);
          if ((lane & 3) != 3) put((i >> 2) * 3 + (lane & 3), v >> (8 * (lane & 3)));
        } else if (on) {
          const int p0 = b2 * i, wd = p0 >> 5, sh = p0 & 31;
          if (4 * wd < nbytes) atomicOr(y + wd * stride, s.label << sh);
          if (sh + b2 > 32 && 4 * (wd + 1) < nbytes) atomicOr(y + (wd + 1) * stride, s.label >> (32 - sh));
        }
      }
      nf |= s.nf;
      const uint32_t kp = on ? (min(s.key, kKeySat) << 9) | (uint32_t)i : kNone;
      if constexpr (kOne) {
        best[0] = kp;
        info = s.rec;
      } else {
        const uint32_t t0 = max(best[0], kp);
        best[0] = min(best[0], kp);
        const uint32_t t1 = max(best[1], t0);
        best[1] = min(best[1], t0);
        best[2] = min(best[2], t1);
      }
    }
    if (L == 0) {  // not a decodable descriptor
      if (lane == 0) s_flag[fr] = 3u;
      continue;
    }
    if constexpr (kFrom == kFromArrays) {
      const int NW = a.NWmax;
      if (lane < NW) y[lane * stride] = a.y_in[(tile + fr) * NW + lane];
    }
    if (__any_sync(kAll, nf)) {
      if (lane == 0) s_flag[fr] = 2u;
      continue;
    }
    // Steps 2-3: the S' least reliable symbols by warp minima of the packed
    // (reliability, index) keys
    uint32_t sel = 0, kmin = 0;
    int pops = 0;
    for (int r = 0; r < Sp; ++r) {
      kmin = __reduce_min_sync(kAll, best[0]);
      if (lane == r) sel = kmin;
      if (best[0] == kmin) {
        if constexpr (kOne) {
          best[0] = kNone;
        } else {
          best[0] = best[1];
          best[1] = best[2];
          best[2] = kNone;
          ++pops;
        }
      }
    }
    bool redo = Sp > 0 && (kmin >> 9) >= kKeySat;
    if constexpr (!kOne) redo |= __any_sync(kAll, pops >= kLanePick && L > 32 * kLanePick + lane);
    sel &= 511u;
    if (redo) sel = (uint32_t)select_exact<kFrom>(a, base, L, Sp, q, m);
    if constexpr (kOne) {
      const uint32_t v = __shfl_sync(kAll, info, (int)(sel & 31u));
      if (lane < Sp) rec[lane * FT + fr] = v | sel;
    } else {
      if (lane < Sp) rec[lane * FT + fr] = sel;  // its alternatives are worked out in the solve
    }
    // H not of polar form: the base syndrome by the columns of y's one-bits
    if (!code->polar) {
      __syncwarp();
      const int W = code->W, NW = code->N >> 5;
      uint32_t yw = lane < NW ? y[lane * stride] : 0u;
      const int64_t co = kFrom == kFromMixed ? s_cw[fr] : (tile + fr) * (int64_t)NW;
      if (lane < NW) a.cw[co + lane] = yw;
      uint32_t f0 = 0;
      for (int w = 0; w < NW; ++w)
        if ((__shfl_sync(kAll, yw, w) >> lane) & 1u) f0 ^= __ldg(code->hf + 32 * w + lane);
      f0 = __reduce_xor_sync(kAll, f0);
      for (int v = 0; v < W; ++v) {
        uint32_t acc = 0;
        for (int w = 0; w < NW; ++w)
          if ((__shfl_sync(kAll, yw, w) >> lane) & 1u) acc ^= __ldg(code->hcol + (size_t)(32 * w + lane) * W + v);
        acc = __reduce_xor_sync(kAll, acc);
        if (lane == 0) y[v * stride] = acc;  // the hard word is no longer needed here
        if (W == 1) f0 = acc;
      }
      if (lane == 0) s_f0[fr] = f0;
    }
  }
  __syncthreads();

  // --- hard words out (decoded bits are flipped in place later) ---------------
  if constexpr (kFrom == kFromMixed) {
    for (int fr = warp; fr < n_here; fr += kWarps) {
      if (s_flag[fr] == 3u) continue;
      const CodeDev* code = a.codes + (s_par[fr] >> 13);
      if ((code->polar || s_flag[fr]) && lane < (code->N >> 5)) a.cw[s_cw[fr] + lane] = buf[lane * stride + fr];
    }
  } else {
    const int NW = a.NWmax, lg = 31 - __clz(NW), polar = a.codes->polar;
    for (int t = threadIdx.x; t < n_here * NW; t += 32 * kWarps) {
      const int fr = t >> lg, w = t & (NW - 1);
      if (polar || s_flag[fr]) a.cw[tile * NW + t] = buf[w * stride + fr];
    }
  }
  __syncthreads();

  // --- solve: one thread per frame ---------------------------------------------
  unsigned long long evaluated = 0, useful = 0;
  unsigned hard = 0;
  const int fr = threadIdx.x;
  if (fr < n_here) {
    const int64_t f = tile + fr;
    const uint32_t flag = s_flag[fr];
    if (flag) {
      a.queries[f] = 0;
      a.abandon[f] = (uint8_t)flag;
    } else {
      const int L = frame_len(fr);
      const int m = kFrom == kFromMixed ? (int)((s_par[fr] >> 10) & 7u) : um;
      const CodeDev* code = kFrom == kFromMixed ? a.codes + (s_par[fr] >> 13) : a.codes;
      const int N = code->N, NW = N >> 5;
      const int64_t cw_off = kFrom == kFromMixed ? s_cw[fr] : f * (int64_t)NW;
      const int Sp = a.S < L ? a.S : L;
      Frame F;
      F.buf = buf + fr;
      F.pos = rec + fr;
      F.stride = stride;
      F.pstride = FT;
      F.fmask = code->fmask;
      F.hcol = code->hcol;
      F.W = code->W;
      F.pat = pat;
      F.polar = code->polar;
      F.nw = F.polar ? NW : code->W;
      const bool exact = F.polar ? NW == 1 : code->W == 1;

      // the alternatives of each rank: flip positions, existing slots
      uint32_t ex = 0;
      {
        const float q = a.qc.q[m];
        const int64_t base = frame_base(fr);
        for (int r = 0; r < Sp; ++r) {
          uint32_t v = rec[r * FT + fr];
          if constexpr (!kOne) v |= symbol_at<kFrom>(a, base, (int)v, q, m).rec;
          const int i = (int)(v & 511u);
          bool eI = (v >> 21) & 1u, eQ = (v >> 22) & 1u;
          // the neighbour differs from the hard level in the Gray label's bit ctz(threshold)
          int pI = 2 * m * i + m - __ffs((int)((v >> 9) & 63u));
          int pQ = 2 * m * i + 2 * m - __ffs((int)((v >> 15) & 63u));
          if (!eI || pI >= N) pI = kNoPos;
          if (!eQ || pQ >= N) pQ = kNoPos;
          if (a.nearer && ((v >> 23) & 1u)) {  // the nearer (vertical) alternative takes the first slot
            const int tp = pI; pI = pQ; pQ = tp;
            const bool te = eI; eI = eQ; eQ = te;
          }
          rec[r * FT + fr] = (uint32_t)pI | ((uint32_t)pQ << 16);
          ex |= ((eI ? 1u : 0u) | (eQ ? 2u : 0u)) << (2 * r);
        }
      }

      // base syndrome (polar form: the transform of y on the frozen bits) and its projection
      uint32_t f0;
      if (F.polar) {
        uint32_t* b = F.buf;
        if (NW >= 4) {
          for (int w = 0; w < NW; w += 4) {
            uint32_t x0 = transform_word(b[w * stride]), x1 = transform_word(b[(w + 1) * stride]);
            uint32_t x2 = transform_word(b[(w + 2) * stride]), x3 = transform_word(b[(w + 3) * stride]);
            x0 ^= x1; x2 ^= x3;
            x0 ^= x2; x1 ^= x3;
            b[w * stride] = x0; b[(w + 1) * stride] = x1; b[(w + 2) * stride] = x2; b[(w + 3) * stride] = x3;
          }
          for (int dw = 4; dw < NW; dw <<= 1)
            for (int t = 0; t < NW / 2; ++t) {
              const int w = ((t & ~(dw - 1)) << 1) | (t & (dw - 1));
              b[w * stride] ^= b[(w + dw) * stride];
            }
        } else {
          const uint32_t x0 = transform_word(b[0]);
          b[0] = x0;
          if (NW == 2) {
            const uint32_t x1 = transform_word(b[stride]);
            b[stride] = x1;
            b[0] = x0 ^ x1;
          }
        }
        f0 = 0;
        for (int w = 0; w < NW; ++w) {
          const uint32_t s = b[w * stride] & __ldg(F.fmask + w);
          b[w * stride] = s;
          f0 = syndrome_fold(f0, s);
        }
      } else {
        f0 = s_f0[fr];
      }

      // elimination: column b reduced by the earlier pivots, its combination
      // of slots beside it; the base syndrome last
      const Proj proj{F.polar ? code->hx : (exact ? code->hcol : code->hf)};
      uint32_t c[kSlots], comb[kSlots];
      uint32_t real = 0;  // existing slots whose flip lies inside the word
#pragma unroll
      for (int b = 0; b < kSlots; ++b) {
        uint32_t p = kNoPos;
        if ((ex >> b) & 1u) p = slot_pos(F, b);
        c[b] = proj(p);
        comb[b] = 1u << b;
        real |= p != kNoPos ? 1u << b : 0u;
      }
      uint32_t s = f0, x0 = 0;
      uint32_t kv[kSlots];
      int d = 0;
#pragma unroll
      for (int j = 0; j < kSlots; ++j) {
        const uint32_t v = c[j], piv = v & (0u - v);
#pragma unroll
        for (int k = j + 1; k < kSlots; ++k)
          if (c[k] & piv) {
            c[k] ^= v;
            comb[k] ^= comb[j];
          }
        if (s & piv) {
          s ^= v;
          x0 ^= comb[j];
        }
        // a slot that changes nothing (padding) is never part of the first
        // solution: leaving it out lowers the position
        if (v == 0u && ((real >> j) & 1u)) kv[d++] = comb[j];
      }
      uint32_t x = kNone;
      unsigned long long ranked = 0;
      if (s == 0u) {
        if (d == 0) {
          const bool ok = exact || (F.polar ? consume_zero_polar(F, x0) : sum_zero(F, x0, true));
          if (ok) x = x0;
          ranked = ok ? 1 : 0;
        } else {
          x = first_solution(F, proj, ex, Sp, f0, exact, x0, kv, d, &ranked);
        }
      }

      // outputs
      const uint32_t exh = ex & 0x55555555u, exv = (ex >> 1) & 0x55555555u;
      const uint32_t one = exh ^ exv, both = exh & exv;
      const uint32_t total = 1u << __popc(ex);
      const uint32_t pos = x != kNone ? tep_position(x, one, both) : 0u;
      const bool hit = x != kNone && (uint64_t)pos <= (uint64_t)a.cap;
      const uint32_t qn = hit ? pos : (uint32_t)((uint64_t)total < (uint64_t)a.cap ? total : (uint64_t)a.cap);
      a.queries[f] = qn;
      a.abandon[f] = hit ? 0 : 1;
      if (hit) {
        for (uint32_t t = x; t; t &= t - 1u) {
          const uint32_t p = slot_pos(F, __ffs(t) - 1);
          if (p != kNoPos) atomicXor(a.cw + cw_off + (p >> 5), 1u << (p & 31u));
        }
      }
      if (a.scr) {
        // searched: no codeword among the TEPs of the first w0 weights
        const uint32_t done = g_esp.cum[__popc(one)][__popc(both)][min(a.w0, Sp) + 1];
        evaluated = a.solve ? ranked : (unsigned long long)total;
        if (!a.solve && qn > done) {
          hard = 1;
          useful = qn - done;
        }
      }
    }
  }
  if (a.scr) {
    for (int o = 16; o; o >>= 1) {
      evaluated += __shfl_xor_sync(kAll, evaluated, o);
      useful += __shfl_xor_sync(kAll, useful, o);
    }
    hard = __reduce_add_sync(kAll, hard);
    if (lane == 0 && evaluated) {
      atomicAdd(&a.scr->evaluated, evaluated);
      atomicAdd(&a.scr->search_useful, useful);
      atomicAdd(&a.scr->n_hard, hard);
    }
  }
}

size_t decode_smem(bool mixed, int slots, int T, int NWmax) {
  const size_t FT = (size_t)kWarps * T;
  return (mixed ? FT * 20 : 0) + 4 * (32 + 2 * FT + (slots / 2) * FT + NWmax * (FT + 1));
}

template <int kFrom, bool kOne>
const void* pick_slots(int Smax) {
  if (Smax <= 8) return (const void*)k_decode<kFrom, kOne, 16>;
  if (Smax <= 10) return (const void*)k_decode<kFrom, kOne, 20>;
  return (const void*)k_decode<kFrom, kOne, 24>;
}

}  // namespace

int preload_decode_kernels() {
  const void* kernels[] = {(const void*)k_decode<kFromMixed, false, 16>, (const void*)k_decode<kFromMixed, false, 20>,
                           (const void*)k_decode<kFromMixed, false, 24>};
  for (const void* k : kernels) {
    cudaFuncAttributes attr;
    if (cudaFuncGetAttributes(&attr, k) != cudaSuccess) return GRAND_E_CUDA;
  }
  return GRAND_OK;
}

int launch_decode(DecodeArgs a, int Lmax, cudaStream_t st) {
  const int Smax = a.S < Lmax ? a.S : Lmax;
  const int slots = Smax <= 8 ? 16 : (Smax <= 10 ? 20 : 24);
  const bool mixed = a.desc != nullptr, arrays = !mixed && a.symbols == nullptr;
  // frames per warp: as many as keep every SM full (each CTA holds the tile's
  // solve in its first warps, so larger tiles waste fewer lanes there), in
  // equal waves
  const int64_t slots_cta = (int64_t)sm_count() * 7;
  const int64_t waves = (a.n_frames + slots_cta * kWarps * 32 - 1) / (slots_cta * kWarps * 32);
  const int64_t T = (a.n_frames + slots_cta * kWarps * waves - 1) / (slots_cta * kWarps * waves);
  a.T = (int)(T < 1 ? 1 : (T > 32 ? 32 : T));
  const int64_t grid = (a.n_frames + kWarps * a.T - 1) / (kWarps * a.T);
  const size_t smem = decode_smem(mixed, slots, a.T, a.NWmax);
  const void* kern = mixed ? pick_slots<kFromMixed, false>(Smax)
                           : (arrays ? pick_slots<kFromArrays, false>(Smax)
                                     : (Lmax <= 32 ? pick_slots<kFromUniform, true>(Smax)
                                                   : pick_slots<kFromUniform, false>(Smax)));
  if (smem > 48 * 1024) return GRAND_E_CUDA;  // not reachable: 4 x 32 frames of 32 words take 28 KB
  void* args[] = {&a};
  if (cudaLaunchKernel(kern, dim3((unsigned)grid), dim3(32 * kWarps), args, smem, st) != cudaSuccess)
    return GRAND_E_CUDA;
  return GRAND_OK;
}

}  // namespace grand
