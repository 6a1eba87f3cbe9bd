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
// k_decode works on tiles of 4 T frames per CTA:
//   front  (small and demodulated batches) one warp per frame, T frames
//          one after the other: symbols are read coalesced (the next 32 are in
//          flight while 32 are worked on), the hard word is packed by byte
//          stores, the S' least reliable symbols are picked by warp minima.
//          (large batches; uneven ones are first put in order by length) one
//          thread per frame: 8 symbols of each of a
//          warp's 32 frames at a time go through shared memory (asynchronous
//          copies, 64 contiguous bytes a frame, the next 8 under way
//          meanwhile); a thread packs its labels by multiplications and keeps
//          its S' smallest keys sorted by comparator networks. Nothing crosses
//          lanes, where the warp per frame spends 10 warp minima at a quarter
//          of the issue rate and a label reduction a step: 416 warp
//          instructions a frame of 43 symbols (N=256, S=8). 250,000 such
//          frames 137 -> 56 us, N=128 300,000 frames 91 -> 64 us, N=512 S=12
//          80,000 frames 76 -> 41 us, uneven mix of 10^6 frames 904 -> 590 us.
//          What is left of a frame is its hard word and S' symbol records in
//          shared memory.
//   solve  one thread per frame: the base syndrome by the polar transform of
//          the hard word, the slot columns' 32-bit projections, Gaussian
//          elimination with the columns in registers, the check of the
//          solution on the full syndrome, its canonical position in closed
//          form and the outputs. A warp instruction serves 32 frames here,
//          where a warp per frame spent a ballot and a shuffle per slot on one.
#include <type_traits>

#include "axis.cuh"
#include "device_common.cuh"
#include "fused.cuh"
#include "host_util.cuh"

namespace grand {
namespace {

constexpr unsigned kAll = 0xFFFFFFFFu;
constexpr int kCtaWarps = 4;            // warps per CTA
constexpr uint32_t kNone = 0xFFFFFFFFu;
constexpr uint32_t kKeySat = 0x7FFFFEu; // packed selection keys hold 23 bits of the reliability
constexpr uint32_t kOff = 0xFFFFFE00u;     // above every packed key: lane (low bits) without a symbol
constexpr uint32_t kPicked = 0xFFFFFFE0u;  // above those: a key taken as rank (low bits)
constexpr int kLanePick = 4;            // smallest keys kept per lane of a long frame
constexpr int kOwnDim = 3;              // kernels of up to this dimension are walked by the frame's thread
constexpr int kPairDim = 10;            // of larger ones, TEPs of two altered ranks are tested before any walk
constexpr int kPairTeps = 631;          // and where the query cap may lie among those (at most as many)
constexpr int kCutDim = 8;              // frames of larger kernels are cut at the call's deadline
constexpr uint32_t kCut = 0xFFFFFFFEu;  // in the place of a solution: cut at the deadline

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

// Distance of the ordering key (threshold or literal reading), unclamped above.
__device__ __forceinline__ float axis_dist(float e, int literal) {
  const float m = fabsf(e);
  return literal ? fmaxf(0.0f, 256.0f - fabsf(m - 256.0f)) : m;
}

// The alternatives of a selected symbol: the threshold toward each axis's
// neighbour (k) and whether it exists; near: Q's distance is below I's.
struct Alt {
  uint32_t kI, kQ;
  bool exI, exQ, near;
};
__device__ __forceinline__ Alt symbol_alt(float2 v, const AxisRegs& c, int lik) {
  const Axes x = axes_fast(grid2(pack2(v), c), c);
  const float2 e = x.e;
  return Alt{__float_as_uint(x.kb.x) & 63u, __float_as_uint(x.kb.y) & 63u, fabsf(e.x) <= 256.0f, fabsf(e.y) <= 256.0f,
             axis_dist(e.y, lik) < axis_dist(e.x, lik)};
}

// The full ordering key of one symbol (integer arithmetic with the int16
// clamps of the fixed-point definition).
__device__ __forceinline__ uint32_t symbol_key(float2 v, float q, int m, int lik) {
  const AxisDemod I = demod_axis_q(v.x, q, 1 << m, lik), Q = demod_axis_q(v.y, q, 1 << m, lik);
  return (uint32_t)(I.dq * I.dq) + (uint32_t)(Q.dq * Q.dq);
}
__device__ __forceinline__ bool finite2(float2 v) { return isfinite(v.x) && isfinite(v.y); }

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

__device__ __forceinline__ Alt array_alt(const DecodeArgs& a, int64_t o) {
  const uint32_t h = a.hard_idx[o], nm = a.nmask[o];
  // the threshold toward the neighbour (where there is none the value is not used)
  return Alt{(h >> 8) + ((nm >> 3) & 1u) - 1u, (h & 0xFFu) + ((nm >> 4) & 1u) - 1u, (nm & 1u) != 0,
             (nm & 2u) != 0, (nm & 32u) != 0};
}

// How lane `lane` takes part in packing the labels of 32 symbols into bytes
// (m = 1..4): a group of 4, 2, 4, 1 symbols fills 1, 1, 3, 1 bytes; the group
// ORs its labels, each shifted to its place, and some of its lanes store a
// byte. Fields: shift to the place (bits 0..4), shift of the stored byte
// (5..9), partner distances (10: 1, 11: 2), storing lane (12), first byte (13..).
__device__ __forceinline__ uint32_t pack_plan(int m, int lane) {
  if (m == 1) return (2u * (~lane & 3)) | (3u << 10) | ((lane & 3) == 0 ? 1u << 12 : 0u) | ((uint32_t)(lane >> 2) << 13);
  if (m == 2) return (4u * (~lane & 1)) | (1u << 10) | ((lane & 1) == 0 ? 1u << 12 : 0u) | ((uint32_t)(lane >> 1) << 13);
  if (m == 3)
    return (6u * (~lane & 3)) | ((uint32_t)((16 - 8 * (lane & 3)) & 31) << 5) | (3u << 10) |
           ((lane & 3) != 3 ? 1u << 12 : 0u) | ((uint32_t)((lane >> 2) * 3 + (lane & 3)) << 13);
  return (1u << 12) | ((uint32_t)lane << 13);
}

// Exact selection of the S' smallest (key, index) pairs, for frames whose
// packed keys do not settle it (a selected key saturates: a receiver whose gain
// is many times the constellation's, or one lane of a long frame ran out of
// kept keys). Lane r returns the index of rank r. One pass with whole keys,
// each lane keeping its kLanePick smallest; a scan for every rank left when a
// lane runs out of them. (Scans for all ranks computed every key S' times:
// 18,000 frames of 512 symbols, 60 times too large, 581 us, so 212.)
template <int kFrom>
__device__ __noinline__ int select_exact(const DecodeArgs& a, int64_t base, int L, int Sp, int m) {
  const int lane = threadIdx.x & 31;
  auto key_of = [&](int i) {
    if constexpr (kFrom == kFromArrays) return selection_key(a.key[base + i]);
    else return symbol_key(a.symbols[base + i], a.ax[m].q.x, m, a.lik);
  };
  typedef unsigned long long Kept;  // key, index (9 bits)
  constexpr Kept kEmpty = ~0ull;
  Kept b0 = kEmpty, b1 = kEmpty, b2 = kEmpty, b3 = kEmpty;  // ascending
  static_assert(kLanePick == 4, "kept keys");
  for (int i = lane; i < L; i += 32) {
    Kept t = ((Kept)key_of(i) << 9) | (Kept)i, u;
    u = max(b0, t); b0 = min(b0, t);
    t = max(b1, u); b1 = min(b1, u);
    u = max(b2, t); b2 = min(b2, t);
    b3 = min(b3, u);
  }
  uint32_t last_k = 0;
  int last_i = -1, sel = 0, r = 0;
  for (bool out = false; r < Sp && !out; ++r) {
    const uint32_t hi = (uint32_t)(b0 >> 32), hmin = __reduce_min_sync(kAll, hi);
    const uint32_t lo = hi == hmin ? (uint32_t)b0 : kNone, lmin = __reduce_min_sync(kAll, lo);
    if (hi == hmin && lo == lmin) {
      b0 = b1; b1 = b2; b2 = b3; b3 = kEmpty;
    }
    const Kept best = ((Kept)hmin << 32) | lmin;
    last_k = (uint32_t)(best >> 9);
    last_i = (int)(best & 511u);
    if (lane == r) sel = last_i;
    out = __any_sync(kAll, b0 == kEmpty && L > 32 * kLanePick + lane);
  }
  for (; r < Sp; ++r) {
    uint32_t bk = kNone, bi = kNone;
    for (int i = lane; i < L; i += 32) {
      const uint32_t k = key_of(i);
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

// c ^= v when c has a bit of p: a test and a predicated XOR (left to itself the
// compiler selects between both values, twice the instructions).
__device__ __forceinline__ void xor_if(uint32_t& c, uint32_t p, uint32_t v) {
  asm("{\n\t.reg .pred q;\n\t.reg .b32 t;\n\t"
      "and.b32 t, %0, %1;\n\t"
      "setp.ne.b32 q, t, 0;\n\t"
      "@q xor.b32 %0, %0, %2;\n\t}"
      : "+r"(c)
      : "r"(p), "r"(v));
}

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
  const float2* cols;   // rank r: its slots' projections (as bits) at cols[32 r]; NULL: read from the table
};

__device__ __forceinline__ uint32_t slot_pos(const Frame& f, int b) {
  return (f.pos[(b >> 1) * f.pstride] >> (16 * (b & 1))) & 0xFFFFu;
}

// XOR of the slot columns over x (and the base syndrome) is zero everywhere.
// Without the base the packed columns are summed where they have few words (2
// instead of the transform's 32 at 1024 bits and 40 rows); else the
// transform's for polar-form H, whose patterns lie in shared memory (80,000
// frames of 512 bits, 8 words instead of 16: 43 us packed, 40.6 so).
__device__ __noinline__ bool sum_zero(const Frame f, uint32_t x, bool base) {
  const bool packed = !f.polar || (!base && (f.W <= 2 || 4 * f.W <= f.nw));
  for (int w = 0; w < (packed ? f.W : f.nw); ++w) {
    uint32_t acc = base ? f.buf[w * f.stride] : 0u;
    for (uint32_t t = x; t; t &= t - 1u) {
      const uint32_t p = slot_pos(f, __ffs(t) - 1);
      if (p == kNoPos) continue;
      if (packed) acc ^= __ldg(f.hcol + (size_t)p * f.W + w);
      else if (!((uint32_t)w & ~(p >> 5))) acc ^= f.pat[p & 31u] & __ldg(f.fmask + w);
    }
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
    // four subsets a round, so that their loads are in flight together
    for (uint32_t top = sup;;) {
      uint32_t w[4], y[4];
      bool on = true, go[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        w[i] = top;
        go[i] = on;
        on = on && top != 0u;
        top = (top - 1u) & sup;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) y[i] = f.buf[w[i] * f.stride] ^ (pt & __ldg(f.fmask + w[i]));
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (go[i]) f.buf[w[i] * f.stride] = y[i];
      if (!on) break;
    }
  }
  uint32_t orr = 0;
#pragma unroll 4
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

// First solution in canonical order among x0 + span(kv[0..d)), d >= 1, by one
// thread (a Gray-code walk; every solution is a valid TEP). exact: the
// projection decides. Else: when every kernel vector passes the full test the
// projected kernel is the true one, and x0 decides for all; otherwise (the
// projection lost rank on the columns) every candidate is tested.
__device__ __noinline__ uint32_t first_solution(const Frame f, bool exact, uint32_t x0, const uint32_t* kv, int d) {
  bool each = false;
  if (!exact) {
    for (int t = 0; t < d && !each; ++t) each = !sum_zero(f, kv[t], false);
    if (!each && !sum_zero(f, x0, true)) return kNone;
  }
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

// Valid TEPs with at most w altered ranks (ex: existing slots).
__device__ __forceinline__ uint32_t valid_up_to(uint32_t ex, int Sp, int w) {
  const uint32_t h = ex & 0x55555555u, v = (ex >> 1) & 0x55555555u;
  return g_esp.cum[__popc(h ^ v)][__popc(h & v)][min(w, Sp) + 1];
}

// First TEP of weight <= wmax (at most 2) in canonical order whose projection
// equals f0 and which passes the full test, or kNone: by the frame's thread. A
// warp instruction compares a pair of alternatives of 32 frames; by the warp,
// one frame after the other, the pairs waited for each other: 18,000 frames of
// 1024 bits with 10 parity bits, S = 12 and a cap of 300 352 us, so 63. The
// projections are read where the elimination's were put (local arrays would be
// read from L2, as shared memory leaves the first level little room).
__device__ __noinline__ uint32_t light_hit(const Frame f, const Proj proj, uint32_t ex, int Sp, uint32_t f0, bool exact,
                                           int wmax, int64_t cap) {
  auto full = [&](uint32_t x) { return exact || sum_zero(f, x, true); };
  auto columns = [&](int r, uint32_t& a, uint32_t& b) {
    if (f.cols) {
      const float2 v = f.cols[32 * r];
      a = __float_as_uint(v.x);
      b = __float_as_uint(v.y);
    } else {
      a = proj(slot_pos(f, 2 * r));
      b = proj(slot_pos(f, 2 * r + 1));
    }
  };
  if (f0 == 0u && full(0u)) return 0u;
  for (int r = 0; r < Sp; ++r) {
    uint32_t a, b;
    columns(r, a, b);
    const uint32_t e = (ex >> (2 * r)) & 3u;
    if ((e & 1u) && a == f0 && full(1u << (2 * r))) return 1u << (2 * r);
    if ((e & 2u) && b == f0 && full(2u << (2 * r))) return 2u << (2 * r);
    if (e == 3u && (a ^ b) == f0 && full(3u << (2 * r))) return 3u << (2 * r);
  }
  if (cap <= 3 * kSMax && (int64_t)valid_up_to(ex, Sp, 1) >= cap) return kNone;  // the others lie beyond the cap
  for (int hi = 1; wmax >= 2 && hi < Sp; ++hi) {
    uint32_t h0, h1;
    columns(hi, h0, h1);
    const uint32_t t1 = f0 ^ h0, t2 = f0 ^ h1, t3 = t1 ^ h1;
#pragma unroll 2
    for (int lo = 0; lo < hi; ++lo) {
      uint32_t a, b;
      columns(lo, a, b);
      const uint32_t ab = a ^ b;
      if (t1 == a || t1 == b || t1 == ab || t2 == a || t2 == b || t2 == ab || t3 == a || t3 == b || t3 == ab) {
        for (uint32_t c = 0; c < 9; ++c) {  // which of them, in order
          const uint32_t h = c / 3u + 1u, l = c % 3u + 1u, x = (h << (2 * hi)) | (l << (2 * lo));
          const uint32_t z = (l & 1u ? a : 0u) ^ (l & 2u ? b : 0u);
          if ((h == 1u ? t1 : (h == 2u ? t2 : t3)) == z && (ex & x) == x && full(x)) return x;
        }
      }
    }
  }
  return kNone;
}

// The same for weight 3 alone (5,940 TEPs), by one warp (all arguments the same
// in every lane): a lane holds one or two of the 3 S' alternatives as the
// TEP's lowest altered rank and compares their projections with what the two
// higher ranks leave; those are looped over in order.
__device__ __noinline__ uint32_t third_weight_warp(const Frame f, const Proj proj, uint32_t ex, int Sp, uint32_t f0,
                                                   bool exact) {
  const int lane = threadIdx.x & 31;
  uint32_t z[2], own[2];  // own: the alternative at its rank, 0 where it does not exist
  int rank[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int t = lane + 32 * h;
    const uint32_t code = (uint32_t)(t % 3) + 1u;
    rank[h] = t / 3;
    z[h] = own[h] = 0u;
    if (rank[h] < Sp && ((ex >> (2 * rank[h])) & code) == code) {
      own[h] = code << (2 * rank[h]);
      if (code & 1u) z[h] = proj(slot_pos(f, 2 * rank[h]));
      if (code & 2u) z[h] ^= proj(slot_pos(f, 2 * rank[h] + 1));
    }
  }
  auto proj_of = [&](int r, int c) {  // 0 where it does not exist
    const int t = 3 * r + c;
    return t < 32 ? __shfl_sync(kAll, z[0], t) : __shfl_sync(kAll, z[1], t - 32);
  };
  for (int hi = 2; hi < Sp; ++hi) {
    for (int mid = 1; mid < hi; ++mid) {
      uint32_t key = kNone;  // lowest rank, then the alternatives from the largest rank down
#pragma unroll 1
      for (int c = 0; c < 9; ++c) {
        const uint32_t x = ((uint32_t)(c / 3 + 1) << (2 * hi)) | ((uint32_t)(c % 3 + 1) << (2 * mid));
        if ((ex & x) != x) continue;
        const uint32_t want = f0 ^ proj_of(hi, c / 3) ^ proj_of(mid, c % 3);
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (own[h] && rank[h] < mid && z[h] == want && (exact || sum_zero(f, x | own[h], true)))
            key = min(key, (uint32_t)(rank[h] * 27 + 3 * c) + (own[h] >> (2 * rank[h])) - 1u);
      }
      const uint32_t k = __reduce_min_sync(kAll, key);
      if (k != kNone)
        return ((k / 9u % 3u + 1u) << (2 * hi)) | ((k / 3u % 3u + 1u) << (2 * mid)) | ((k % 3u + 1u) << (2 * (k / 27u)));
    }
  }
  return kNone;
}

// first_solution by one warp (all arguments but kv the same in every lane; kv
// is read in lane src). The walk over 2^d solutions takes 2^(d-5) steps; codes
// with few parity bits have large kernels, and then their first hit is light:
// above 2^kPairDim solutions the frame's thread has tested weights <= 2
// (light_hit), above 2^13 weight 3 is tested before the walk. Once the TEPs
// tested are as many as the cap, a solution among the others lies beyond it and
// there is nothing to look for: 20,000 frames of 128 bits, 8 parity bits,
// S = 12 and a cap of 300 348 -> 69 us.
__device__ __noinline__ uint32_t first_solution_warp(const Frame f, const Proj proj, uint32_t ex, int Sp, uint32_t f0,
                                                     bool exact, uint32_t x0, const uint32_t* kv, int d, int src,
                                                     int64_t cap) {
  const int lane = threadIdx.x & 31;
  uint32_t k[2 * kSMax];
  uint32_t mine = 0;
  for (int t = 0; t < d; ++t) {
    k[t] = __shfl_sync(kAll, kv[t], src);
    if (lane == t) mine = k[t];
  }
  bool each = false;
  if (!exact) {
    each = __any_sync(kAll, lane < d && !sum_zero(f, mine, false));
    if (!each && !sum_zero(f, x0, true)) return kNone;
  }
  if (d > 13) {
    const uint32_t x = third_weight_warp(f, proj, ex, Sp, f0, exact || !each);
    if (x != kNone || (int64_t)valid_up_to(ex, Sp, 3) >= cap) return x;
  }
  uint32_t x = x0, bk = kNone, bx = kNone;
  for (int t = 0; t < 5 && t < d; ++t)
    if ((lane >> t) & 1) x ^= k[t];
  const bool on = d >= 5 || lane < 1 << d;
  for (uint32_t i = 0; on;) {
    const uint32_t key = order_key(x);
    if (comes_before(key, x, bk, bx) && (!each || sum_zero(f, x, true))) {
      bk = key;
      bx = x;
    }
    if (d <= 5 || ++i >> (d - 5)) break;
    x ^= k[5 + __ffs(i) - 1];
  }
  const uint32_t kmin = __reduce_min_sync(kAll, bk);
  return __reduce_min_sync(kAll, bk == kmin ? bx : kNone);
}

// The call's deadline has passed and the walk of a frame is not begun.
__device__ __noinline__ bool walk_is_late(const DecodeArgs& a) {
  int late = 0;
  if ((threadIdx.x & 31) == 0) late = past_deadline(a.t0, a.deadline);
  return __shfl_sync(kAll, late, 0) != 0;
}

// ---------------------------------------------------------------------------
// Front helpers (one warp per frame, one symbol per lane and step)
// ---------------------------------------------------------------------------
struct Step {
  uint32_t kp;     // packed (reliability, index) key
  uint32_t label;  // Gray labels, I then Q, most significant bit first
};

// Demodulation of 32 symbols (lane i: symbol i0 + i; off lanes give label 0).
// nf: set when a symbol is not finite (its coordinates are read as 0).
__device__ __forceinline__ Step demod_step(const DecodeArgs& a, const AxisRegs& ax, float2 cur, int m, uint32_t index,
                                           bool on, bool& nf) {
  F2 x = grid2(pack2(cur), ax);
  const float2 xs = unpack2(x);
  const bool plain = fabsf(xs.x) <= ax.lim && fabsf(xs.y) <= ax.lim;
  uint32_t big = 0;  // key of a symbol outside the plain range
  if (__any_sync(kAll, !plain)) {
    float2 v = cur;
    const bool bad = on && !finite2(v);
    if (__any_sync(kAll, bad)) nf = true;
    if (bad) {
      v = make_float2(0.0f, 0.0f);
      x = pack2(0.0f, 0.0f);
    }
    big = min(symbol_key(v, unpack2(ax.q).x, m, a.lik), kKeySat);
  }
  const Axes t = axes_fast(x, ax);
  float2 d = t.e;
  if (a.lik) d = make_float2(axis_dist(d.x, 1), axis_dist(d.y, 1));
  Step s;
  // key < 2^23 in the plain range: 2^23 + key has the key in its mantissa
  const uint32_t key = __float_as_uint(__fadd_rn(__fmaf_rn(d.x, d.x, __fmul_rn(d.y, d.y)), 8388608.0f));
  s.kp = (plain ? key : big) * 512u + index;
  // hard levels: threshold index plus one above it (e >= 0; e is an integer),
  // both axes' in one number on top of 1.5 * 2^23
  const float lI = __fadd_rn(t.k.x, __saturatef(__fadd_rn(t.e.x, 1.0f)));
  const float lQ = __fadd_rn(t.kb.y, __saturatef(__fadd_rn(t.e.y, 1.0f)));
  const uint32_t lv = __float_as_uint(__fmaf_rn(lI, ax.side, lQ)) & (on ? (1u << (2 * m)) - 1u : 0u);
  s.label = lv ^ ((lv >> 1) & ~(1u << (m - 1)));
  return s;
}

// Labels of 32 symbols into the frame's bytes by the lane's plan (m <= 4);
// room: bytes of the frame from the lane's byte of this step on (<= 0: none to
// store). Every lane takes part.
__device__ __forceinline__ void pack_labels(uint32_t label, uint32_t plan, uint8_t* yb, int room) {
  uint32_t v = label << (plan & 31u);
  v |= __shfl_xor_sync(kAll, v, (plan >> 10) & 1u);
  v |= __shfl_xor_sync(kAll, v, (plan >> 10) & 2u);
  if (room > 0) *yb = (uint8_t)(v >> ((plan >> 5) & 31u));
}

// 5 or 6 bits an axis: OR into the words.
__device__ __forceinline__ void or_label(uint32_t label, int i, int m, uint32_t* y, int stride, int NW) {
  const int p0 = 2 * m * i, wd = p0 >> 5, room = 32 - (p0 & 31) - 2 * m;
  if (wd < NW) atomicOr(y + wd * stride, room >= 0 ? label << room : label >> -room);
  if (room < 0 && wd + 1 < NW) atomicOr(y + (wd + 1) * stride, label << (32 + room));
}

// The kRanks smallest of one key per lane, by warp minima: returns the lane's
// rank, 31 or more for none. Always kRanks rounds (straight-line code: a round
// is four instructions); ranks beyond the frame's S' mean nothing.
template <int kRanks>
__device__ __forceinline__ uint32_t pick_ranks(uint32_t kp) {
#pragma unroll
  for (int r = 0; r < kRanks; ++r) {
    const uint32_t kmin = __reduce_min_sync(kAll, kp);
    kp = kp == kmin ? kPicked | (uint32_t)r : kp;
  }
  return kp >= kPicked ? kp & 31u : 32u;
}

// ---------------------------------------------------------------------------
// Front helpers (one thread per frame, kChunk symbols at a time)
// ---------------------------------------------------------------------------
constexpr int kChunk = 8;                      // symbols of a frame per step
constexpr int kRowPad = kChunk + 1;            // odd: the rows' 8-byte reads of half a warp fall into different banks
constexpr int kStageSyms = 32 * kRowPad;       // one chunk of a warp's 32 frames in shared memory
constexpr int kStages = 2;
// CTAs of the thread-per-frame kernels are single warps: nothing is shared
// between warps, and the last wave is finer (against 4 warps: 20,000 frames of
// 128 symbols 34 -> 30 us, 300,000 of 32 70 -> 68 us). 20 of them an SM leave 96
// registers a thread: against 24 (80 registers) 56 for 59 us on 250,000 frames
// of 43 symbols, 41 for 52 us on 80,000 of 86, 64 for 62 us on 300,000 of 32;
// 32 spill and take 74, 53, 75.
constexpr int kThreadCtas = 20;
constexpr int kThreadWarps = 1;
constexpr int kOrderCtas = 16;  // uneven batches: shared memory allows 17 with words of 1024 bits

// 4 or 8 bytes global -> shared without passing the registers; off: zeros.
__device__ __forceinline__ void fetch4(uint32_t dst, const void* src, bool on) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(on ? 4 : 0) : "memory");
}
__device__ __forceinline__ void fetch8(uint32_t dst, const void* src, bool on) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(on ? 8 : 0) : "memory");
}

// max(|a|, |b|, |c|), NaN when one is.
__device__ __forceinline__ float max_abs(float a, float b, float c) {
  float r;
  asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

__device__ __forceinline__ void order2(uint32_t& a, uint32_t& b) {
  const uint32_t lo = min(a, b);
  b = max(a, b);
  a = lo;
}

// Ascending sort of eight keys (odd-even merge sort, 19 comparators).
__device__ __forceinline__ void sort8(uint32_t (&k)[kChunk]) {
  order2(k[0], k[1]); order2(k[2], k[3]); order2(k[4], k[5]); order2(k[6], k[7]);
  order2(k[0], k[2]); order2(k[1], k[3]); order2(k[4], k[6]); order2(k[5], k[7]);
  order2(k[1], k[2]); order2(k[5], k[6]);
  order2(k[0], k[4]); order2(k[1], k[5]); order2(k[2], k[6]); order2(k[3], k[7]);
  order2(k[2], k[4]); order2(k[3], k[5]);
  order2(k[1], k[2]); order2(k[3], k[4]); order2(k[5], k[6]);
}

// The R smallest of best (ascending) and k (ascending), ascending: the minima
// of best against k reversed rise and then fall, and a bitonic merge sorts
// them (for R = 10 and 12 that of 16 numbers of which the first 6 or 4 are
// below all others and stay where they are).
template <int R>
__device__ __forceinline__ void merge_smallest(uint32_t (&best)[R], const uint32_t (&k)[kChunk]) {
  static_assert(R == 8 || R == 10 || R == 12, "ranks");
#pragma unroll
  for (int i = R - kChunk; i < R; ++i) best[i] = min(best[i], k[R - 1 - i]);
#pragma unroll
  for (int i = 0; i < R - 8; ++i) order2(best[i], best[i + 8]);
  if constexpr (R == 12) {
    order2(best[0], best[2]); order2(best[1], best[3]);
    order2(best[2], best[3]);
  }
  if constexpr (R > 8) order2(best[0], best[1]);
  constexpr int o = R - 8;
#pragma unroll
  for (int dist = 4; dist >= 1; dist >>= 1)
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (!(i & dist)) order2(best[o + i], best[o + i + dist]);
}

// Base syndrome of one frame for H not of polar form, by one warp: the sum of
// the columns of its hard word's one-bits (lane w holds word w), four words of
// every column in one load and four columns a lane in flight. Word v goes to
// out[v * stride]; returns the projection. (A word of a column at a time waited
// for each of 16 x 32 scattered loads: 30,000 demodulated frames of 1024 bits and
// 512 rows, cap 30, 334 us, so 162.)
__device__ __noinline__ uint32_t column_syndrome(const uint32_t* __restrict__ hcol, const uint32_t* __restrict__ hf,
                                                 int W, int NW, uint32_t yw, uint32_t* out, int stride) {
  constexpr int kCols = 4, kWords = 4;
  const int lane = threadIdx.x & 31;
  uint32_t f0 = 0;
  for (int v0 = 0; v0 < W; v0 += kWords) {
    uint32_t acc[kWords] = {0u, 0u, 0u, 0u};
#pragma unroll 1
    for (int w0 = 0; w0 < NW; w0 += kCols) {
      uint4 c[kCols];
      uint32_t f[kCols];
#pragma unroll
      for (int i = 0; i < kCols; ++i) {
        const int w = w0 + i;  // (words beyond the last are zero in yw)
        const bool on = (__shfl_sync(kAll, yw, w & 31) >> lane) & 1u;
        c[i] = make_uint4(0u, 0u, 0u, 0u);
        f[i] = 0u;
        if (on) {
          const uint32_t* p = hcol + (size_t)(32 * w + lane) * W + v0;
          if (!(W & 3)) {  // columns start on 16 bytes
            c[i] = __ldg(reinterpret_cast<const uint4*>(p));
          } else {
            c[i].x = __ldg(p);
            if (v0 + 1 < W) c[i].y = __ldg(p + 1);
            if (v0 + 2 < W) c[i].z = __ldg(p + 2);
            if (v0 + 3 < W) c[i].w = __ldg(p + 3);
          }
          if (v0 == 0 && W > 1) f[i] = __ldg(hf + 32 * w + lane);
        }
      }
#pragma unroll
      for (int i = 0; i < kCols; ++i) {
        acc[0] ^= c[i].x;
        acc[1] ^= c[i].y;
        acc[2] ^= c[i].z;
        acc[3] ^= c[i].w;
        f0 ^= f[i];
      }
    }
#pragma unroll
    for (int i = 0; i < kWords; ++i) {
      if (v0 + i >= W) break;
      const uint32_t s = __reduce_xor_sync(kAll, acc[i]);
      if (lane == 0) out[(v0 + i) * stride] = s;
      if (W == 1) return s;  // one word: the syndrome itself
    }
  }
  return __reduce_xor_sync(kAll, f0);
}

// Natural labels of four symbols (m bits an axis, I then Q, the first symbol
// highest) to Gray labels.
template <typename T>
__device__ __forceinline__ T gray4(T v, T below_top) { return v ^ ((v >> 1) & below_top); }

// Base syndrome of this thread's frame for H not of polar form: the parities of
// its hard word under the rows, eight rows at a time (word w of the hard word
// at y[w * stride], of the syndrome at out[32 w]). Returns the projection. A
// row's words are the same in every thread of a code, so they come as
// broadcasts, and the work is one three-input operation per row and word of a
// warp's 32 frames; the sum of the columns of the one-bits, a warp per frame
// and the frames one after the other, waited for its scattered loads: 20,000
// frames of 1024 bits and 512 rows 1165 us, so 144.
__device__ __noinline__ uint32_t row_syndrome(const uint32_t* __restrict__ hrow, const uint32_t* __restrict__ prow, int R,
                                              int NW, const uint32_t* y, int stride, uint32_t* out) {
  constexpr int kRowsAtOnce = 8;  // divides a word
  uint32_t f0 = 0, word = 0;
#pragma unroll 1
  for (int r0 = 0; r0 < R; r0 += kRowsAtOnce) {
    const int last = R - 1 - r0;  // rows beyond the last one repeat it
    const uint32_t* h = hrow + (size_t)r0 * NW;
    uint32_t acc[kRowsAtOnce];
#pragma unroll
    for (int i = 0; i < kRowsAtOnce; ++i) acc[i] = 0u;
    if (NW >= 4) {
#pragma unroll 1
      for (int w = 0; w < NW; w += 4) {
        const uint32_t y0 = y[w * stride], y1 = y[(w + 1) * stride], y2 = y[(w + 2) * stride], y3 = y[(w + 3) * stride];
#pragma unroll
        for (int i = 0; i < kRowsAtOnce; ++i) {
          const uint4 v = __ldg(reinterpret_cast<const uint4*>(h + min(i, last) * NW + w));
          acc[i] ^= v.x & y0;
          acc[i] ^= v.y & y1;
          acc[i] ^= v.z & y2;
          acc[i] ^= v.w & y3;
        }
      }
    } else {
      for (int w = 0; w < NW; ++w) {
        const uint32_t yw = y[w * stride];
#pragma unroll
        for (int i = 0; i < kRowsAtOnce; ++i) acc[i] ^= __ldg(h + min(i, last) * NW + w) & yw;
      }
    }
#pragma unroll
    for (int i = 0; i < kRowsAtOnce; ++i) {
      if (i <= last && (__popc(acc[i]) & 1)) {
        word |= 1u << ((r0 & 31) + i);
        f0 ^= __ldg(prow + r0 + i);
      }
    }
    if ((r0 & 31) == 32 - kRowsAtOnce || last < kRowsAtOnce) {
      out[r0 & ~31] = word;
      if (R <= 32 && last < kRowsAtOnce) return word;  // one word: the syndrome itself
      word = 0;
    }
  }
  return f0;
}

// ---------------------------------------------------------------------------
// The kernel
// ---------------------------------------------------------------------------
// kMap: how the front maps frames to threads. kSlots: 2 x the largest S' (16,
// 20 or 24: the elimination is unrolled over it).
enum {
  kWarpShort = 0,  // a warp per frame of at most 32 symbols (one per lane)
  kWarpLong = 1,   // a warp per frame, 32 symbols at a time
  kThread = 2,     // a thread per frame, kChunk symbols at a time
  kThreadUsual = 3,  // the same without the inner loop for symbols of more than 8 bits and the literal likelihood
};
//
// Words of a hard word are kept bit-reversed in shared memory (the label bits
// of a symbol arrive most significant first) until they are written out or
// transformed.
constexpr int warps_of(int map) { return map >= kThread ? kThreadWarps : kCtaWarps; }

// An uneven batch's frame: symbols | m << 10 | words << 13 | polar << 19;
// kNoFrame (no symbols) for a descriptor that names none.
constexpr uint32_t kNoFrame = 1u << 10;
__device__ __forceinline__ uint32_t frame_par(const DecodeArgs& a, const CodeDev* codes, const grand_frame_desc& d) {
  const int m = (31 - __clz(d.M)) >> 1;
  if (d.code < 0 || d.code >= a.n_codes || m < 1 || m > 6 || d.M != 1 << (2 * m) || d.sym_offset < 0 || d.cw_offset < 0)
    return kNoFrame;
  const CodeDev* code = codes + d.code;
  const int N = code->N, L = (N + 2 * m - 1) / (2 * m);
  if (d.sym_offset > a.n_symbols - L || d.cw_offset > a.n_cw_words - (N >> 5)) return kNoFrame;
  return (uint32_t)L | ((uint32_t)m << 10) | ((uint32_t)(N >> 5) << 13) | (code->polar ? 1u << 19 : 0u);
}

// ---------------------------------------------------------------------------
// Order of an uneven batch: frames of as many steps of kChunk symbols and of
// one constellation together, the longest first, for the thread-per-frame
// front (the lanes of a warp then finish together). A counting sort: counts
// per block, starts by the last block, records by a second pass. A record
// holds what the decode needs of its frame: the way from an index over the
// descriptor and the code to the first symbol was three dependent loads.
// ---------------------------------------------------------------------------
constexpr int kBins = 65 * 8;           // (64 - steps) * 8 + m
constexpr int kSortThreads = 256, kSortEach = 4;
constexpr size_t kSortHeader = 4 * (kBins + 8);  // bins, ticket
static_assert(kSortHeader % 32 == 0 && sizeof(OrderRec) == 32, "records on sectors");

struct SortTile {
  uint32_t count[kBins];
  uint32_t start[kBins];
  CodeDev table[kInlineCodes];
};

// The block's descriptors (loads first, all in flight together) and their bins' counts.
__device__ __forceinline__ void count_bins(const DecodeArgs& a, SortTile& s, grand_frame_desc (&d)[kSortEach],
                                           uint32_t (&par)[kSortEach], int (&bin)[kSortEach]) {
  const int64_t f0 = (int64_t)blockIdx.x * (kSortEach * kSortThreads) + threadIdx.x;
#pragma unroll
  for (int i = 0; i < kSortEach; ++i)
    d[i] = f0 + i * kSortThreads < a.n_frames ? a.desc[f0 + i * kSortThreads] : grand_frame_desc{};
  for (int b = threadIdx.x; b < kBins; b += kSortThreads) s.count[b] = 0u;
  if (!a.codes && (int)threadIdx.x < a.n_codes) s.table[threadIdx.x] = a.code[threadIdx.x];
  __syncthreads();
  const CodeDev* codes = a.codes ? a.codes : s.table;
#pragma unroll
  for (int i = 0; i < kSortEach; ++i) {
    bin[i] = -1;
    par[i] = kNoFrame;
    if (f0 + i * kSortThreads < a.n_frames) {
      par[i] = frame_par(a, codes, d[i]);
      bin[i] = (64 - (int)(((par[i] & 1023u) + kChunk - 1) / kChunk)) * 8 + (int)((par[i] >> 10) & 7u);
      atomicAdd(&s.count[bin[i]], 1u);
    }
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kSortThreads) k_order_count(const __grid_constant__ DecodeArgs a, uint32_t* bins) {
  __shared__ SortTile s;
  __shared__ bool last;
  grand_frame_desc d[kSortEach];
  uint32_t par[kSortEach];
  int bin[kSortEach];
  count_bins(a, s, d, par, bin);
  for (int b = threadIdx.x; b < kBins; b += kSortThreads)
    if (s.count[b]) atomicAdd(bins + b, s.count[b]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(bins + kBins, 1u) == gridDim.x - 1u;
  __syncthreads();
  if (!last || threadIdx.x >= 32) return;
  // starts: one warp, kEach bins a lane
  constexpr int kEach = (kBins + 31) / 32;
  uint32_t v[kEach], sum = 0;
#pragma unroll
  for (int i = 0; i < kEach; ++i) {
    const int b = (int)threadIdx.x * kEach + i;
    v[i] = b < kBins ? __ldcg(bins + b) : 0u;
    sum += v[i];
  }
  uint32_t before = sum;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(kAll, before, o);
    if ((int)threadIdx.x >= o) before += t;
  }
  before -= sum;
#pragma unroll
  for (int i = 0; i < kEach; ++i) {
    const int b = (int)threadIdx.x * kEach + i;
    if (b < kBins) bins[b] = before;
    before += v[i];
  }
}

__global__ void __launch_bounds__(kSortThreads) k_order_index(const __grid_constant__ DecodeArgs a, uint32_t* bins,
                                                              OrderRec* order) {
  __shared__ SortTile s;
  grand_frame_desc d[kSortEach];
  uint32_t par[kSortEach];
  int bin[kSortEach];
  count_bins(a, s, d, par, bin);
  for (int b = threadIdx.x; b < kBins; b += kSortThreads)
    if (s.count[b]) {
      s.start[b] = atomicAdd(bins + b, s.count[b]);
      s.count[b] = 0u;
    }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kSortEach; ++i) {
    if (bin[i] < 0) continue;
    const int64_t f = ((int64_t)blockIdx.x * kSortEach + i) * kSortThreads + threadIdx.x;
    order[s.start[bin[i]] + atomicAdd(&s.count[bin[i]], 1u)] =
        OrderRec{d[i].sym_offset, d[i].cw_offset, par[i], par[i] != kNoFrame ? (uint32_t)d[i].code : 0u, (uint32_t)f, 0u};
  }
}

template <int kFrom, int kMap, int kSlots>
__global__ void __launch_bounds__(32 * (kMap >= kThread ? kThreadWarps : kCtaWarps),
                                  kMap >= kThread ? (kFrom == kFromMixed ? kOrderCtas : kThreadCtas) : 8)
    k_decode(const __grid_constant__ DecodeArgs a) {
  constexpr int kWarps = kMap >= kThread ? kThreadWarps : kCtaWarps;
  constexpr bool kOne = kMap == kWarpShort, kRows = kMap >= kThread;
  extern __shared__ __align__(16) char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int FT = kWarps * a.T;
  const int stride = FT + 1;  // odd: a frame's words fall into different banks
  constexpr int kRanks = kSlots / 2;
  int64_t* s_off = reinterpret_cast<int64_t*>(smem_raw);             // [FT] mixed: first symbol
  int64_t* s_cw = s_off + (kFrom == kFromMixed ? FT : 0);            // [FT] mixed: first output word
  float2* s_sym = reinterpret_cast<float2*>(s_cw + (kFrom == kFromMixed ? FT : 0));  // [kRanks][FT] kOne: the symbol of each rank
  float2* s_stage = s_sym + (kOne ? kRanks * FT : 0);                // [kWarps][kStages][32][kRowPad] kThread: chunks in flight
  uint32_t* s_par = reinterpret_cast<uint32_t*>(s_stage + (kRows ? kWarps * kStages * kStageSyms : 0));  // [FT] mixed: L | m | words | polar
  uint32_t* s_code = s_par + (kFrom == kFromMixed ? FT : 0);         // [FT] mixed: index of the code
  uint32_t* s_plan = s_code + (kFrom == kFromMixed ? FT : 0);        // [4][32] mixed: pack_plan
  uint32_t* pat = s_plan + (kFrom == kFromMixed && !kRows ? 128 : 0);          // [32]
  uint32_t* s_f0 = pat + 32;                                         // [FT] projection of s(y) (H not of polar form)
  uint32_t* s_flag = s_f0 + FT;                                      // [FT] 0, or the abandon flag of an undecodable frame
  uint32_t* rec = s_flag + FT;                                       // [kRanks][FT] symbol index, later slot positions
  uint32_t* buf = rec + kRanks * FT;                                 // [NWmax][stride]
  __shared__ CodeDev s_table[kFrom == kFromMixed ? kInlineCodes : 1];
  const CodeDev* const codes = kFrom == kFromMixed ? (a.codes ? a.codes : s_table) : a.code;
  const int64_t tile = (int64_t)blockIdx.x * FT;
  const int n_here = (int)min((int64_t)FT, a.n_frames - tile);

  if (a.deadline > 0 && threadIdx.x == 0) past_deadline(a.t0, a.deadline);  // start the call's clock
  if (threadIdx.x < 32) pat[threadIdx.x] = subset_pattern(threadIdx.x);
  for (int t = threadIdx.x; t < a.NWmax * stride; t += 32 * kWarps) buf[t] = 0u;
  for (int t = threadIdx.x; t < FT; t += 32 * kWarps) s_flag[t] = 0u;
  if constexpr (kFrom == kFromMixed) {
    if (!a.codes) {
      if ((int)threadIdx.x < a.n_codes) s_table[threadIdx.x] = a.code[threadIdx.x];
      __syncthreads();
    }
    if constexpr (!kRows) s_plan[threadIdx.x] = pack_plan(warp + 1, lane);
    for (int t = threadIdx.x; t < (kRows ? FT : n_here); t += 32 * kWarps) {
      if constexpr (kRows) {
        OrderRec o{0, 0, kNoFrame, 0, 0, 0};
        if (t < n_here) o = a.order[tile + t];
        s_off[t] = o.sym_offset;
        s_cw[t] = o.cw_offset;
        s_par[t] = o.par;
        s_code[t] = o.code;
      } else {
        const grand_frame_desc d = a.desc[tile + t];
        const uint32_t par = frame_par(a, codes, d);
        s_off[t] = d.sym_offset;
        s_cw[t] = d.cw_offset;
        s_par[t] = par;
        s_code[t] = par != kNoFrame ? (uint32_t)d.code : 0u;
      }
    }
  }
  __syncthreads();

  // --- front: one warp per frame ---------------------------------------------
  const int um = kFrom == kFromMixed ? 0 : a.m, uL = kFrom == kFromMixed ? 0 : a.L;
  const bool u_polar = kFrom == kFromMixed ? false : a.code[0].polar != 0;
  const int fr_begin = warp * a.T, fr_end = min(n_here, fr_begin + a.T);
  auto frame_base = [&](int fr) { return kFrom == kFromMixed ? s_off[fr] : (tile + fr) * (int64_t)uL; };
  auto frame_len = [&](int fr) { return kFrom == kFromMixed ? (int)(s_par[fr] & 1023u) : uL; };
  // the rare rest of a frame: exact selection, and for H not of polar form
  // the base syndrome by the columns of y's one-bits
  auto reselect = [&](int fr, int L, int m, int Sp, float2 cur) {
    const int sel = select_exact<kFrom>(a, frame_base(fr), L, Sp, m);
    if constexpr (kOne) {
      const float2 v = make_float2(__shfl_sync(kAll, cur.x, sel), __shfl_sync(kAll, cur.y, sel));
      if (lane < Sp) s_sym[lane * FT + fr] = v;
    }
    __syncwarp();
    if (lane < Sp) rec[lane * FT + fr] = (uint32_t)sel;
  };
  auto general_syndrome = [&](int fr, int NW) {
    __syncwarp();
    uint32_t* y = buf + fr;
    const CodeDev* code = codes + (kFrom == kFromMixed ? s_code[fr] : 0u);
    const uint32_t yw = lane < NW ? __brev(y[lane * stride]) : 0u;
    const int64_t co = kFrom == kFromMixed ? s_cw[fr] : (tile + fr) * (int64_t)NW;
    if (lane < NW) a.cw[co + lane] = yw;
    __syncwarp();  // the hard word makes place for the syndrome
    const uint32_t f0 = column_syndrome(code->hcol, code->hf, code->W, NW, yw, y, stride);
    if (lane == 0) s_f0[fr] = f0;
  };

  if constexpr (kRows) {
    const int rows = n_here - 32 * warp, mine = 32 * warp + lane;
    const bool here = lane < rows;
    // this thread's frame (uneven batch: its own length and constellation)
    const uint32_t par = kFrom == kFromMixed ? s_par[mine] : 0u;
    const int L = kFrom == kFromMixed ? (int)(par & 1023u) : uL;
    const int m = kFrom == kFromMixed ? (int)((par >> 10) & 7u) : um;
    const int NW = kFrom == kFromMixed ? (int)((par >> 13) & 63u) : a.NWmax;
    const int Sp = a.S < L ? a.S : L;
    const AxisRegs ax = axis_regs(a.ax[m], a.ax[1].nz);
    int n_chunks = rows > 0 ? (L + kChunk - 1) / kChunk : 0;
    // the inner loop without the literal likelihood and symbols of more than 8 bits
    bool usual = !a.lik && m <= 4;
    if constexpr (kFrom == kFromMixed) {
      n_chunks = __reduce_max_sync(kAll, n_chunks);
      usual = __all_sync(kAll, usual);
    }
    const uint32_t side2 = 1u << (2 * m);
    // what the fixed exponent bits of four packed labels add up to
    const uint32_t fixed = __float_as_uint(kMagic) * (1u + side2 + side2 * side2 + side2 * side2 * side2);
    const uint64_t below_top = a.ax[m].below_top;
    float2* stage = s_stage + warp * (kStages * kStageSyms);
    // a fetch takes 8 symbols of 4 frames: 64 contiguous bytes of each
    const int frow = lane >> 3, fcol = lane & 7;
    const float2* src = a.symbols + (tile + 32 * warp + frow) * (int64_t)uL + fcol;
    const uint32_t fdst = (uint32_t)__cvta_generic_to_shared(stage + frow * kRowPad + fcol);
    // uneven batch: first symbols of the 8 rows this lane fetches for, and the
    // steps that are complete in every row
    uint32_t first[8];
    int n_full = 0;
    if constexpr (kFrom == kFromMixed) {
      n_full = __reduce_min_sync(kAll, L / kChunk);
#pragma unroll
      for (int k = 0; k < 8; ++k) first[k] = (uint32_t)s_off[32 * warp + frow + 4 * k] + (uint32_t)fcol;
    }
    auto fetch = [&](int c) {
      if (c < n_chunks) {
        const uint32_t dst = fdst + (uint32_t)(c % kStages) * (kStageSyms * 8);
        if constexpr (kFrom == kFromMixed) {
          if (c < n_full) {
#pragma unroll
            for (int k = 0; k < 8; ++k) fetch8(dst + k * (4 * kRowPad * 8), a.symbols + (first[k] + (uint32_t)(c * kChunk)), true);
          } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const bool on = c * kChunk + fcol < (int)(s_par[32 * warp + frow + 4 * k] & 1023u);
              const void* p = on ? (const void*)(a.symbols + (first[k] + (uint32_t)(c * kChunk))) : (const void*)a.desc;
              fetch8(dst + k * (4 * kRowPad * 8), p, on);  // (off: no bytes are read)
            }
          }
        } else {
          const bool in = c * kChunk + fcol < uL;
          const float2* s = in ? src + c * kChunk : a.symbols;
          if (rows >= 32) {
            const int64_t step = in ? 4 * uL : 0;
#pragma unroll
            for (int k = 0; k < 8; ++k, s += step) fetch8(dst + k * (4 * kRowPad * 8), s, in);
          } else {
            for (int k = 0; k < 8; ++k) {
              const bool on = in && frow + 4 * k < rows;
              fetch8(dst + k * (4 * kRowPad * 8), on ? s + (int64_t)(4 * k) * uL : a.symbols, on);
            }
          }
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    uint32_t best[kRanks];
#pragma unroll
    for (int r = 0; r < kRanks; ++r) best[r] = kNone;
    bool nf = false;
    // one step; kUsual: no literal likelihood, at most 8 bits a symbol
    auto step = [&](auto usual_form, int c) {
      constexpr bool kUsual = decltype(usual_form)::value;
      float2* row = stage + (c % kStages) * kStageSyms + lane * kRowPad;
      F2 x[kChunk];
      float top = 0.0f;
#pragma unroll
      for (int j = 0; j < kChunk; ++j) {
        x[j] = grid2(pack2(row[j]), ax);
        const float2 xs = unpack2(x[j]);
        top = max_abs(top, xs.x, xs.y);
      }
      const bool wide = __any_sync(kAll, !(top <= ax.lim));
      if (wide) {  // coordinates that are not finite are read as 0
#pragma unroll
        for (int j = 0; j < kChunk; ++j)
          if (!finite2(row[j])) {
            nf = true;
            x[j] = pack2(0.0f, 0.0f);
            row[j] = make_float2(0.0f, 0.0f);
          }
      }
      uint32_t kp[kChunk], four[2] = {0u, 0u};
      uint32_t pair[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int j = 0; j < kChunk; ++j) {
        const Axes t = axes_fast(x[j], ax);
        float2 d = t.e;
        if (!kUsual && a.lik) d = make_float2(axis_dist(d.x, 1), axis_dist(d.y, 1));
        const uint32_t key = __float_as_uint(__fadd_rn(__fmaf_rn(d.x, d.x, __fmul_rn(d.y, d.y)), 8388608.0f));
        kp[j] = key * 512u + (uint32_t)(c * kChunk + j);
        const float lI = __fadd_rn(t.k.x, __saturatef(__fadd_rn(t.e.x, 1.0f)));
        const float lQ = __fadd_rn(t.kb.y, __saturatef(__fadd_rn(t.e.y, 1.0f)));
        const uint32_t lv = __float_as_uint(__fmaf_rn(lI, ax.side, lQ));
        if constexpr (kUsual) four[j >> 2] = four[j >> 2] * side2 + lv;
        else pair[j >> 1] = (pair[j >> 1] << (2 * m)) | (lv & (side2 - 1u));
      }
      if (wide) {
#pragma unroll
        for (int j = 0; j < kChunk; ++j) {
          const float2 v = row[j], xs = unpack2(grid2(pack2(v), ax));
          if (!(fabsf(xs.x) <= ax.lim && fabsf(xs.y) <= ax.lim))
            kp[j] = (min(symbol_key(v, unpack2(ax.q).x, m, a.lik), kKeySat) << 9) | (uint32_t)(c * kChunk + j);
        }
      }
      if ((c + 1) * kChunk > L) {
#pragma unroll
        for (int j = 0; j < kChunk; ++j)
          if (c * kChunk + j >= L) kp[j] = kNone;
      }
      sort8(kp);
      merge_smallest<kRanks>(best, kp);
      // the labels' 16 m bits, most significant first (N ends with a word:
      // what lies beyond it is not stored)
      if constexpr (kUsual) {
        const uint32_t g0 = gray4(four[0] - fixed, (uint32_t)below_top), g1 = gray4(four[1] - fixed, (uint32_t)below_top);
        uint32_t* y = buf + mine;
        auto half = [&](int h, uint32_t v) {
          if (h < 2 * NW)
            *(reinterpret_cast<uint16_t*>(y + (h >> 1) * stride) + (~h & 1)) = (uint16_t)v;
        };
        if (m == 2) {
          if (c < NW) y[c * stride] = (g0 << 16) | g1;
        } else if (m == 4) {
          if (2 * c < NW) y[2 * c * stride] = g0;
          if (2 * c + 1 < NW) y[(2 * c + 1) * stride] = g1;
        } else if (m == 3) {
          half(3 * c, g0 >> 8);
          half(3 * c + 1, (g0 << 8) | (g1 >> 16));
          half(3 * c + 2, g1);
        } else {
          half(c, (g0 << 8) | g1);
        }
      } else {
        uint8_t* yb = reinterpret_cast<uint8_t*>(buf + mine);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const uint64_t g = gray4(((uint64_t)pair[2 * i] << (4 * m)) | pair[2 * i + 1], below_top);
          for (int t = 0; t < m; ++t) {
            const int b = (2 * c + i) * m + t;
            if (b < 4 * NW) yb[(b >> 2) * (4 * stride) + (~b & 3)] = (uint8_t)(g >> (8 * (m - 1 - t)));
          }
        }
      }
    };
    fetch(0);
    for (int c = 0; c < n_chunks; ++c) {
      fetch(c + 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      __syncwarp();
      if constexpr (kMap == kThreadUsual) step(std::true_type{}, c);
      else if (usual) step(std::true_type{}, c);
      else step(std::false_type{}, c);
      __syncwarp();
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    const bool searched = here && !nf && !(kFrom == kFromMixed && L == 0);
    if (here) {
      if (!searched) s_flag[mine] = L == 0 ? 3u : 2u;  // not a decodable descriptor, or not finite
#pragma unroll
      for (int r = 0; r < kRanks; ++r) rec[r * FT + mine] = best[r] & 511u;
    }
    // a key that does not fit 23 bits was taken
    bool redo = false;
#pragma unroll
    for (int r = 0; r < kRanks; ++r) redo = redo || (r < Sp && best[r] >= kKeySat << 9);
    for (unsigned todo = __ballot_sync(kAll, searched && redo); todo; todo &= todo - 1u) {
      const int of = __ffs(todo) - 1;
      reselect(32 * warp + of, __shfl_sync(kAll, L, of), __shfl_sync(kAll, m, of), __shfl_sync(kAll, Sp, of),
               make_float2(0.0f, 0.0f));
    }
    const bool general = searched && !(kFrom == kFromMixed ? (par >> 19) != 0u : u_polar);
    if (const unsigned todo = __ballot_sync(kAll, general)) {  // H not of polar form: the syndromes now
      const CodeDev* code = codes + (kFrom == kFromMixed && general ? s_code[mine] : 0u);
      uint32_t* y = buf + mine;
      uint32_t* s = reinterpret_cast<uint32_t*>(stage) + lane;
      if (general) {
        for (int w = 0; w < NW; ++w) y[w * stride] = __brev(y[w * stride]);
        s_f0[mine] = row_syndrome(code->hrow, code->prow, code->R, NW, y, stride, s);
      }
      __syncwarp();
      for (unsigned t = todo; t; t &= t - 1u) {  // the hard words out before the syndromes take their place
        const int of = 32 * warp + __ffs(t) - 1, words = __shfl_sync(kAll, NW, __ffs(t) - 1);
        const int64_t co = kFrom == kFromMixed ? s_cw[of] : (tile + of) * (int64_t)words;
        if (lane < words) a.cw[co + lane] = buf[lane * stride + of];
      }
      __syncwarp();
      if (general)
        for (int v = 0; v < code->W; ++v) y[v * stride] = s[32 * v];
    }
    // the selected symbols, rank by rank, on their way to where the chunks were
    __syncwarp();
    if (searched) {
      const float2* own_sym = a.symbols + frame_base(mine);
      const uint32_t sel = (uint32_t)__cvta_generic_to_shared(stage + lane);
#pragma unroll
      for (int r = 0; r < kRanks; ++r)
        if (r < Sp) fetch8(sel + r * 256, own_sym + rec[r * FT + mine], true);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  } else if constexpr (kOne) {
    const AxisRegs ax = axis_regs(a.ax[um], a.ax[1].nz);
    const int NW = a.NWmax, Sp = a.S < uL ? a.S : uL;
    const bool on = lane < uL;
    const uint32_t plan = pack_plan(um, lane);
    const int byte0 = (int)(plan >> 13), room = (plan >> 12) & 1u ? 4 * NW - byte0 : 0;
    uint8_t* yb = reinterpret_cast<uint8_t*>(buf + fr_begin) + (byte0 >> 2) * (4 * stride) + (~byte0 & 3);
    const float2* sym = a.symbols + (tile + fr_begin) * (int64_t)uL + lane;
    float2 nxt = make_float2(0.0f, 0.0f);
    if (on && fr_begin < fr_end) nxt = *sym;
    for (int fr = fr_begin; fr < fr_end; ++fr, yb += 4) {
      const float2 cur = nxt;
      sym += uL;
      if (on && fr + 1 < fr_end) nxt = *sym;  // the next frame's symbols are on their way meanwhile
      bool nf = false;
      const Step st = demod_step(a, ax, cur, um, (uint32_t)lane, on, nf);
      if (um <= 4) pack_labels(st.label, plan, yb, room);
      else if (on) or_label(st.label, lane, um, buf + fr, stride, NW);
      if (nf) {
        if (lane == 0) s_flag[fr] = 2u;
        continue;
      }
      const uint32_t r = pick_ranks<kRanks>(on ? st.kp : kOff + (uint32_t)lane);
      const bool mine = r < (uint32_t)Sp;
      if (mine) {
        s_sym[r * FT + fr] = cur;
        rec[r * FT + fr] = (uint32_t)lane;
      }
      if (__any_sync(kAll, mine && st.kp >= kKeySat << 9)) reselect(fr, uL, um, Sp, cur);
      if (!u_polar) general_syndrome(fr, NW);
    }
  } else {
    float2 nxt = make_float2(0.0f, 0.0f);
    if constexpr (kFrom != kFromArrays) {
      if (fr_begin < fr_end && lane < frame_len(fr_begin)) nxt = a.symbols[frame_base(fr_begin) + lane];
    }
    for (int fr = fr_begin; fr < fr_end; ++fr) {
      const uint32_t par = kFrom == kFromMixed ? s_par[fr] : 0u;
      const int L = kFrom == kFromMixed ? (int)(par & 1023u) : uL;
      const int m = kFrom == kFromMixed ? (int)((par >> 10) & 7u) : um;
      const int NW = kFrom == kFromMixed ? (int)((par >> 13) & 63u) : a.NWmax;
      const bool polar = kFrom == kFromMixed ? (par >> 19) != 0u : u_polar;
      const int Sp = a.S < L ? a.S : L;
      uint32_t* y = buf + fr;
      // this lane's smallest keys, ascending
      uint32_t b0 = kNone, b1 = kNone, b2 = kNone, b3 = kNone;
      static_assert(kLanePick == 4, "kept keys");
      auto keep = [&](uint32_t kp) {
        const uint32_t t0 = max(b0, kp);
        b0 = min(b0, kp);
        const uint32_t t1 = max(b1, t0);
        b1 = min(b1, t0);
        const uint32_t t2 = max(b2, t1);
        b2 = min(b2, t1);
        b3 = min(b3, t2);
      };
      bool nf = false;  // uniform
      if constexpr (kFrom == kFromArrays) {
        const int64_t base = frame_base(fr);
        bool mine = false;
        for (int i = lane; i < L; i += 32) {
          mine |= (a.nmask[base + i] & 128u) != 0;
          keep((min(a.key[base + i], kKeySat) << 9) | (uint32_t)i);
        }
        nf = __any_sync(kAll, mine);
        if (lane < NW) y[lane * stride] = __brev(a.y_in[(tile + fr) * NW + lane]);
      } else {
        const AxisRegs ax = axis_regs(a.ax[m], a.ax[1].nz);
        const uint32_t plan = kFrom == kFromMixed ? s_plan[32 * ((m - 1) & 3) + lane] : pack_plan(um, lane);
        const int byte0 = (int)(plan >> 13);
        uint8_t* yb = reinterpret_cast<uint8_t*>(y) + (byte0 >> 2) * (4 * stride) + (~byte0 & 3);
        int room = (plan >> 12) & 1u ? 4 * NW - byte0 : 0;
        const float2* sym = a.symbols + frame_base(fr) + lane;
        int left = L - lane;  // symbols of this lane's stride from here on: on while positive
        uint32_t index = (uint32_t)lane;
        for (int i0 = 0;;) {
          const float2 cur = nxt;
          const bool on = left > 0, more = i0 + 32 < L;
          // the next 32 symbols, of this frame or the next one, are on their way meanwhile
          if (more) {
            sym += 32;
            if (left > 32) nxt = *sym;
          } else if (fr + 1 < fr_end) {
            if (lane < frame_len(fr + 1)) nxt = a.symbols[frame_base(fr + 1) + lane];
          }
          const Step st = demod_step(a, ax, cur, m, index, on, nf);
          if (m <= 4) {
            pack_labels(st.label, plan, yb, room);
            yb += 8 * m * stride;  // 2 m words on
            room -= 8 * m;
          } else if (on) {
            or_label(st.label, (int)index, m, y, stride, NW);
          }
          keep(on ? st.kp : kNone);
          if (!more) break;
          i0 += 32;
          left -= 32;
          index += 32u;
        }
      }
      if (nf || (kFrom == kFromMixed && L == 0)) {  // not searched, or not a decodable descriptor
        if (lane == 0) s_flag[fr] = L == 0 ? 3u : 2u;
        continue;
      }
      // Steps 2-3: the S' least reliable symbols; the lane that holds a
      // minimum records it
      uint32_t* recf = rec + fr;
      bool redo;
      if (L <= 32) {
        const uint32_t r = pick_ranks<kRanks>(lane < L ? b0 : kOff + (uint32_t)lane);
        const bool mine = r < (uint32_t)Sp;
        if (mine) recf[r * FT] = (uint32_t)lane;
        redo = mine && b0 >= kKeySat << 9;
      } else {
        uint32_t pick = 0;
#pragma unroll
        for (int r = 0; r < kRanks; ++r) {
          const uint32_t kmin = __reduce_min_sync(kAll, b0);
          const bool w = b0 == kmin;
          if (lane == r) pick = kmin;
          b0 = w ? b1 : b0;
          b1 = w ? b2 : b1;
          b2 = w ? b3 : b2;
          b3 = w ? kNone : b3;
        }
        const bool mine = lane < Sp;
        if (mine) recf[lane * FT] = pick & 511u;
        // a saturated key was taken, or a lane ran out of kept keys
        redo = (mine && pick >= kKeySat << 9) || (b0 == kNone && L > 32 * kLanePick + lane);
      }
      if (__any_sync(kAll, redo)) reselect(fr, L, m, Sp, make_float2(0.0f, 0.0f));
      if (!polar) general_syndrome(fr, NW);
    }
  }
  // Where a thread prepared each frame it also solves it; the frames of a warp
  // per frame are solved by the first 4 T threads of the CTA.
  constexpr bool own = kRows;
  auto tile_sync = [&]() {
    if (own) __syncwarp(); else __syncthreads();
  };
  tile_sync();

  // --- hard words out (decoded bits are flipped in place later) ---------------
  {
    const int first = own ? 32 * warp : 0, last = own ? min(n_here, first + 32) : n_here;
    if constexpr (kFrom == kFromMixed) {
      // own: as many lanes a frame as its words at most (32 one-word frames in
      // one step)
      const int per = own ? max(__reduce_max_sync(kAll, (s_par[lane] >> 13) & 63u), 1u) : 32;
      const int w = own ? lane % per : lane;
      for (int fr = own ? first + lane / per : warp; fr < last; fr += own ? 32 / per : kWarps) {
        const uint32_t par = s_par[fr];
        const bool out = (par & 1023u) && ((par >> 19) || s_flag[fr]);  // a general matrix's word is out already
        if (out && w < (int)((par >> 13) & 63u)) a.cw[s_cw[fr] + w] = __brev(buf[w * stride + fr]);
      }
    } else {
      const int NW = a.NWmax, lg = 31 - __clz(NW);
      for (int t = first * NW + (own ? lane : (int)threadIdx.x); t < last * NW; t += own ? 32 : 32 * kWarps) {
        const int fr = t >> lg, w = t & (NW - 1);
        if (u_polar || s_flag[fr]) a.cw[tile * NW + t] = __brev(buf[w * stride + fr]);
      }
    }
  }
  tile_sync();

  // --- solve: one thread per frame ---------------------------------------------
  unsigned long long evaluated = 0, useful = 0;
  unsigned hard = 0;
  // what a thread needs to look at frame fr of the tile
  auto frame_of = [&](int fr, Proj& proj) {
    const CodeDev* code = codes + (kFrom == kFromMixed ? s_code[fr] : 0u);
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
    F.nw = F.polar ? code->N >> 5 : code->W;
    F.cols = kRows ? s_stage + warp * (kStages * kStageSyms) + (fr & 31) : nullptr;
    // one syndrome word: the columns themselves, and the elimination is the full test
    proj.tab = code->W == 1 && !(F.polar && F.nw == 1) ? code->hcol : (F.polar ? code->hx : code->hf);
    return F;
  };
  const int fr = threadIdx.x;
  const uint32_t flag = fr < n_here ? s_flag[fr] : 0u;
  const bool active = fr < n_here && flag == 0u;
  int Sp = 0, d = 0;
  uint32_t ex = 0, f0 = 0, x0 = 0, x = kNone;
  uint32_t kv[kSlots];
  bool solvable = false;  // the projected system has solutions (2^d of them)
  bool shared = false;  // its solutions are walked by the whole warp
  {
    if (active) {
      const int L = frame_len(fr);
      const int m = kFrom == kFromMixed ? (int)((s_par[fr] >> 10) & 7u) : um;
      const CodeDev* code = codes + (kFrom == kFromMixed ? s_code[fr] : 0u);
      const int N = code->N, NW = N >> 5;
      Sp = a.S < L ? a.S : L;
      Proj proj;
      const Frame F = frame_of(fr, proj);
      const bool exact = code->W == 1;

      // base syndrome (polar form: the transform of y on the frozen bits) and its projection
      if (F.polar) {
        uint32_t* b = F.buf;
        auto word = [&](int w) { return transform_word(__brev(b[w * stride])); };
        // four words apart by dw at a time: two levels of the transform
        // with one round of loads in flight together
        auto two_levels = [&](int w, int dw, uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3) {
          x0 ^= x1; x2 ^= x3;
          x0 ^= x2; x1 ^= x3;
          b[w * stride] = x0; b[(w + dw) * stride] = x1; b[(w + 2 * dw) * stride] = x2; b[(w + 3 * dw) * stride] = x3;
        };
        if (NW >= 4) {
          for (int w = 0; w < NW; w += 4) two_levels(w, 1, word(w), word(w + 1), word(w + 2), word(w + 3));
          int dw = 4;
          for (; 2 * dw < NW; dw <<= 2)
            for (int t = 0; t < NW / 4; ++t) {
              const int w = ((t & ~(dw - 1)) << 2) | (t & (dw - 1));
              two_levels(w, dw, b[w * stride], b[(w + dw) * stride], b[(w + 2 * dw) * stride], b[(w + 3 * dw) * stride]);
            }
          if (dw < NW)  // one level left: its words in groups of four (NW >= 8)
            for (int t = 0; t < NW / 2; t += 4) {
              uint32_t lo[4], hi[4];
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const int w = (((t + i) & ~(dw - 1)) << 1) | ((t + i) & (dw - 1));
                lo[i] = b[w * stride];
                hi[i] = b[(w + dw) * stride];
              }
#pragma unroll
              for (int i = 0; i < 4; ++i) b[((((t + i) & ~(dw - 1)) << 1) | ((t + i) & (dw - 1))) * stride] = lo[i] ^ hi[i];
            }
        } else {
          const uint32_t x0 = word(0);
          b[0] = x0;
          if (NW == 2) {
            const uint32_t x1 = word(1);
            b[stride] = x1;
            b[0] = x0 ^ x1;
          }
        }
        f0 = 0;
        if (exact && NW > 1) {  // at most 32 frozen bits: packed as the columns are
          for (int r = 0; r < code->R; ++r) {
            const uint32_t i = __ldg(code->frozen + r);
            f0 |= ((b[(i >> 5) * stride] >> (i & 31u)) & 1u) << r;
          }
        } else {
          for (int w0 = 0; w0 < NW; w0 += 4) {  // (NW is a power of two)
            uint32_t s[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) s[i] = w0 + i < NW ? b[(w0 + i) * stride] & __ldg(F.fmask + w0 + i) : 0u;
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (w0 + i < NW) {
                b[(w0 + i) * stride] = s[i];
                f0 = syndrome_fold(f0, s[i]);
              }
          }
        }
      } else {
        f0 = s_f0[fr];
      }

      // the alternatives of each rank: flip positions, existing slots, and
      // the slots' columns
      uint32_t c[kSlots];
      uint32_t real = 0;  // ex: existing slots; real: those whose flip lies inside the word
      {
        const AxisRegs ax = axis_regs(a.ax[m], a.ax[1].nz);
        // slots of rank r (symbol idx) from its alternatives: their positions,
        // entered in rec, ex and real
        auto enter = [&](int r, uint32_t idx, const Alt& t, uint32_t& p0, uint32_t& p1) {
          // (threshold k lies between the levels k and k + 1)
          const uint32_t pI = flip_pos(2 * m * (int)idx + m, (int)(t.kI + 1u), N);
          const uint32_t pQ = flip_pos(2 * m * (int)idx + 2 * m, (int)(t.kQ + 1u), N);
          uint32_t e0 = r < Sp && t.exI, e1 = r < Sp && t.exQ;
          p0 = e0 ? pI : kNoPos;
          p1 = e1 ? pQ : kNoPos;
          if (a.nearer && t.near) {  // the nearer (vertical) alternative takes the first slot
            const uint32_t tp = p0, te = e0;
            p0 = p1; p1 = tp;
            e0 = e1; e1 = te;
          }
          if (r < Sp) rec[r * FT + fr] = p0 | (p1 << 16);
          ex |= (e0 | (e1 << 1)) << (2 * r);
          real |= ((p0 != kNoPos ? 1u : 0u) | (p1 != kNoPos ? 2u : 0u)) << (2 * r);
        };
        if constexpr (kRows) {
          // a loop of fetches instead of unrolled loads: the columns of a rank
          // replace its symbol in shared memory, so that all of them are under
          // way together, and the code stays small (warps in different parts
          // of the kernel compete for the instruction cache, which is what
          // the solve waits for most): 300,000 frames of 32 symbols 68 -> 62 us
          float2* sel = s_stage + warp * (kStages * kStageSyms) + lane;
          const uint32_t at = (uint32_t)__cvta_generic_to_shared(sel);
          asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll 1
          for (int r = 0; r < Sp; ++r) {
            uint32_t p0, p1;
            enter(r, rec[r * FT + fr], symbol_alt(sel[32 * r], ax, a.lik), p0, p1);
            fetch4(at + r * 256, proj.tab + (p0 != kNoPos ? p0 : 0u), p0 != kNoPos);
            fetch4(at + r * 256 + 4, proj.tab + (p1 != kNoPos ? p1 : 0u), p1 != kNoPos);
          }
          asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
#pragma unroll
          for (int r = 0; r < kRanks; ++r) {
            const float2 v = r < Sp ? sel[32 * r] : make_float2(0.0f, 0.0f);
            c[2 * r] = __float_as_uint(v.x);
            c[2 * r + 1] = __float_as_uint(v.y);
          }
        } else {
          const int64_t base = frame_base(fr);
          float2 v[kRanks];
          uint32_t idx[kRanks];
#pragma unroll
          for (int r = 0; r < kRanks; ++r) {
            v[r] = make_float2(0.0f, 0.0f);
            idx[r] = r < Sp ? rec[r * FT + fr] : 0u;
            if constexpr (kOne) v[r] = s_sym[r * FT + fr];
            else if constexpr (kFrom != kFromArrays) {
              if (r < Sp) v[r] = a.symbols[base + idx[r]];
            }
          }
#pragma unroll
          for (int r = 0; r < kRanks; ++r) {
            Alt t;
            if constexpr (kFrom == kFromArrays) t = array_alt(a, base + idx[r]);
            else t = symbol_alt(v[r], ax, a.lik);
            uint32_t p0, p1;
            enter(r, idx[r], t, p0, p1);
            c[2 * r] = proj(p0);
            c[2 * r + 1] = proj(p1);
          }
        }
      }

      // Gauss-Jordan on the columns: the pivot of column j is its lowest row
      // that no earlier pivot took; the rows of every later column and of the
      // syndrome are reduced by it, so that a pivot row's bit is a coefficient:
      // afterwards the syndrome's bits in the pivot rows are the solution,
      // and a bit elsewhere says there is none. A column without a free row
      // is the sum of the pivot columns named by its bits: a kernel vector.
      uint32_t s = f0, used = 0, free_slots = 0;
      uint32_t piv[kSlots];
#pragma unroll
      for (int j = 0; j < kSlots; ++j) {
        const uint32_t u = c[j] & ~used, p = u & (0u - u);
        const uint32_t clear = c[j] ^ p;
        piv[j] = p;
        used |= p;
#pragma unroll
        for (int k = j + 1; k < kSlots; ++k)
          xor_if(c[k], p, clear);
        xor_if(s, p, clear);
        // a slot that changes nothing (padding) is never part of the first
        // solution: leaving it out lowers the position
        if (p == 0u && ((real >> j) & 1u)) {
          free_slots |= 1u << j;
          kv[d++] = c[j];
        }
      }
      if (!(s & ~used)) {
        auto pivots_of = [&](uint32_t v) {
          uint32_t r = 0;
#pragma unroll
          for (int j = 0; j < kSlots; ++j) r |= (v & piv[j]) ? 1u << j : 0u;
          return r;
        };
        x0 = pivots_of(s);
        solvable = true;
        if (d == 0) {
          if (exact || (F.polar ? consume_zero_polar(F, x0) : sum_zero(F, x0, true))) x = x0;
        } else {
          for (int t = 0; t < d; ++t, free_slots &= free_slots - 1u)
            kv[t] = pivots_of(kv[t]) | (free_slots & (0u - free_slots));
          shared = d > kOwnDim;
          if (!shared) x = first_solution(F, exact, x0, kv, d);
        }
      }
    }
  }
  // frames with many solutions: few parity bits, and then most first hits weigh
  // at most 1 (20,000 frames of 32 bits with 2 parity bits 111 -> 33 us, of 128
  // with 16 54 -> 38); where the query cap lies among the TEPs tested, nothing
  // is left. (Apart from the elimination: among its registers the call spilled.)
  if (shared) {
    Proj proj;
    const Frame F = frame_of(fr, proj);
    const int tested = d > kPairDim || a.cap <= kPairTeps ? 2 : 1;
    x = light_hit(F, proj, ex, Sp, f0, F.W == 1, tested, a.cap);
    shared = x == kNone && (a.cap > kPairTeps || (int64_t)valid_up_to(ex, Sp, tested) < a.cap);
  }
  // the others one after the other
  for (unsigned todo = __ballot_sync(kAll, shared); todo; todo &= todo - 1u) {
    const int src = __ffs(todo) - 1, of = (int)(threadIdx.x & ~31u) + src;
    Proj proj;
    const Frame F = frame_of(of, proj);
    const int sp = __shfl_sync(kAll, Sp, src), dim = __shfl_sync(kAll, d, src);
    const uint32_t e = __shfl_sync(kAll, ex, src), p0 = __shfl_sync(kAll, f0, src), s0 = __shfl_sync(kAll, x0, src);
    const bool late = a.deadline > 0 && dim > kCutDim && walk_is_late(a);
    const uint32_t got = late ? kCut : first_solution_warp(F, proj, e, sp, p0, F.W == 1, s0, kv, dim, src, a.cap);
    if (lane == src) x = got;
  }

  if (fr < n_here) {
    const int64_t f = kFrom == kFromMixed && kRows ? (int64_t)a.order[tile + fr].frame : tile + fr;
    if (flag) {
      a.queries[f] = 0;
      a.abandon[f] = (uint8_t)flag;
    } else {
      const int64_t cw_off = kFrom == kFromMixed ? s_cw[fr] : f * (int64_t)a.NWmax;
      // outputs
      const uint32_t exh = ex & 0x55555555u, exv = (ex >> 1) & 0x55555555u;
      const uint32_t one = exh ^ exv, both = exh & exv;
      const uint32_t total = 1u << __popc(ex);
      const uint32_t pos = x < kCut ? tep_position(x, one, both) : 0u;
      const bool hit = x < kCut && (uint64_t)pos <= (uint64_t)a.cap;
      uint32_t qn = hit ? pos : (uint32_t)((uint64_t)total < (uint64_t)a.cap ? total : (uint64_t)a.cap);
      uint8_t ab = hit ? 0 : 1;
      if (x == kCut) {
        qn = valid_up_to(ex, Sp, 1);
        ab = 5;
        atomicOr(codes[kFrom == kFromMixed ? s_code[fr] : 0u].status, 1u);
      }
      a.queries[f] = qn;
      a.abandon[f] = ab;
      if (hit) {
        for (uint32_t t = x; t; t &= t - 1u) {
          const int b = __ffs(t) - 1;
          const uint32_t p = (rec[(b >> 1) * FT + fr] >> (16 * (b & 1))) & 0xFFFFu;
          if (p != kNoPos) atomicXor(a.cw + cw_off + (p >> 5), 1u << (p & 31u));
        }
      }
      if (a.scr) {
        // searched: no codeword among the TEPs of the first w0 weights
        const uint32_t done = g_esp.cum[__popc(one)][__popc(both)][min(a.w0, Sp) + 1];
        evaluated = !a.solve ? (unsigned long long)total : (solvable && x != kCut ? 1ull << d : 0ull);
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

size_t decode_smem(bool mixed, int map, int slots, int T, int NWmax) {
  const int warps = warps_of(map);
  const size_t FT = (size_t)warps * T;
  return (mixed ? FT * 24 + (map >= kThread ? 0 : 512) : 0) + (map == kWarpShort ? FT * 8 * (slots / 2) : 0) +
         (map >= kThread ? (size_t)warps * kStages * kStageSyms * 8 : 0) +
         4 * (32 + 2 * FT + (slots / 2) * FT + NWmax * (FT + 1));
}

template <int kFrom, int kMap>
const void* pick_slots(int Smax) {
  if (Smax <= 8) return (const void*)k_decode<kFrom, kMap, 16>;
  if (Smax <= 10) return (const void*)k_decode<kFrom, kMap, 20>;
  return (const void*)k_decode<kFrom, kMap, 24>;
}

}  // namespace

int preload_decode_kernels() {
  const void* kernels[] = {(const void*)k_decode<kFromMixed, kWarpLong, 16>, (const void*)k_decode<kFromMixed, kWarpLong, 20>,
                           (const void*)k_decode<kFromMixed, kWarpLong, 24>,
                           (const void*)k_decode<kFromMixed, kThread, 16>, (const void*)k_decode<kFromMixed, kThread, 20>,
                           (const void*)k_decode<kFromMixed, kThread, 24>, (const void*)k_order_count,
                           (const void*)k_order_index};
  for (const void* k : kernels) {
    cudaFuncAttributes attr;
    if (cudaFuncGetAttributes(&attr, k) != cudaSuccess) return GRAND_E_CUDA;
  }
  return GRAND_OK;
}

// Uniform batches from here on are prepared by a thread per frame. Its time
// hardly depends on the batch up to one wave (each lane works through its
// frame's symbols one after the other), the warp's grows from 4,000 frames on:
// both cross near 16,384 frames for every length. Thread against warp per
// frame at 8,192 / 16,384 / 65,536 frames, us: 8 symbols 10.8 / 11.4 / 14.5
// against 10.8 / 13.3 / 25.6; 32: 10.0 / 10.3 / 16.1 against 9.0 / 11.1 / 23.3;
// 86: 22 / 23 / 36 against 18 / 25 / 61; 512: 57 / 57 / 125 against 42 / 60 / 219.
constexpr int64_t kThreadFrames = 16384;

// Uneven batches from here on are put in order first and prepared by a thread
// per frame. A thread takes 40 us for a frame of 512 symbols whatever the
// batch, so the warp per frame (45 us for 16,384 frames of every length, 62
// for 32,768, 85 for 65,536, 160 for 131,072) is left only near 40,000 frames
// (65, 67, 73 and 103 us in order, the sort included).
constexpr int64_t kOrderFrames = 49152;

size_t order_bytes(const DecodeArgs& a) {
  const int64_t wide = (int64_t)1 << 31;  // the records' frame, and symbol offsets, in 32 bits
  return a.desc && a.n_frames >= kOrderFrames && a.n_frames < wide && a.n_symbols < wide
             ? kSortHeader + sizeof(OrderRec) * (size_t)a.n_frames
             : 0;
}

int launch_order(DecodeArgs& a, void* scratch, cudaStream_t st) {
  uint32_t* bins = static_cast<uint32_t*>(scratch);
  OrderRec* order = reinterpret_cast<OrderRec*>(bins + kSortHeader / 4);
  if (cudaMemsetAsync(bins, 0, kSortHeader, st) != cudaSuccess) return GRAND_E_CUDA;
  const unsigned grid = (unsigned)((a.n_frames + kSortThreads * kSortEach - 1) / (kSortThreads * kSortEach));
  k_order_count<<<grid, kSortThreads, 0, st>>>(a, bins);
  k_order_index<<<grid, kSortThreads, 0, st>>>(a, bins, order);
  if (cudaGetLastError() != cudaSuccess) return GRAND_E_CUDA;
  a.order = order;
  return GRAND_OK;
}

int launch_decode(DecodeArgs a, int Lmax, cudaStream_t st) {
  const int Smax = a.S < Lmax ? a.S : Lmax;
  const int slots = Smax <= 8 ? 16 : (Smax <= 10 ? 20 : 24);
  const bool mixed = a.desc != nullptr, arrays = !mixed && a.symbols == nullptr;
  const QamConst qc = make_qam_const();
  for (int m = 1; m <= 6; ++m) a.ax[m] = axis_const(m, qc);
  const bool uniform = !mixed && !arrays, usual = m_of(a.M) <= 4 && !a.lik;
  int map = uniform && Lmax <= 32 ? kWarpShort : kWarpLong;
  if (a.order) map = kThread;
  else if (uniform && a.n_frames >= kThreadFrames) map = usual ? kThreadUsual : kThread;
  // frames per warp: a thread per frame takes 32; else as many as keep every
  // SM full (each CTA holds the tile's solve in its first warps, so larger
  // tiles waste fewer lanes there)
  const int warps = warps_of(map);
  const int64_t slots_cta = (int64_t)sm_count() * 7;
  const int64_t T = map >= kThread ? 32 : (a.n_frames + slots_cta * warps - 1) / (slots_cta * warps);
  a.m = m_of(a.M);
  a.T = (int)(T < 1 ? 1 : (T > 32 ? 32 : T));
  const int64_t grid = (a.n_frames + warps * a.T - 1) / (warps * a.T);
  const size_t smem = decode_smem(mixed, map, slots, a.T, a.NWmax);
  const void* kern = nullptr;
  if (mixed) kern = a.order ? pick_slots<kFromMixed, kThread>(Smax) : pick_slots<kFromMixed, kWarpLong>(Smax);
  else if (arrays) kern = pick_slots<kFromArrays, kWarpLong>(Smax);
  else if (map == kThreadUsual) kern = pick_slots<kFromUniform, kThreadUsual>(Smax);
  else if (map == kThread) kern = pick_slots<kFromUniform, kThread>(Smax);
  else kern = map == kWarpShort ? pick_slots<kFromUniform, kWarpShort>(Smax) : pick_slots<kFromUniform, kWarpLong>(Smax);
  if (smem > 48 * 1024) return GRAND_E_CUDA;  // not reachable: 4 x 32 frames of 32 words take 28 KB, a warp of rows 12 KB
  void* args[] = {&a};
  if (cudaLaunchKernel(kern, dim3((unsigned)grid), dim3(32 * warps), args, smem, st) != cudaSuccess)
    return GRAND_E_CUDA;
  return GRAND_OK;
}

}  // namespace grand
