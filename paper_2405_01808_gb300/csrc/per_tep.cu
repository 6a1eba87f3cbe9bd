// Per-TEP decoding: one warp per frame demodulates it (Def. III.1 / III.2),
// selects the S' least reliable symbols (Alg. 2 Steps 2-3) and walks the
// valid TEPs in canonical order (Step 5), 32 altered-rank sets at a time: lane
// l takes one set of the current weight and steps through that set's
// alternatives in order, so the warp's lowest hitting lane holds the first hit.
//
// It serves what the split search of decode.cu does not: the five-point NNE
// order (up to four alternatives per symbol, no diagonal; the error model the
// paper contrasts with its own in Sec. II), and the two membership tests kept
// for comparison --
//   DELTA       z = s(y) xor the H columns the TEP flips (Alg. 2 Step 4),
//               filtered by a 32-bit projection and confirmed on all rows;
//   ROW_PARITY  the candidate y xor e multiplied by H row by row, each
//               syndrome bit the parity of (row AND word): the product of
//               Alg. 1 (pMult) evaluated for every TEP, stopping at the first
//               odd row.
// Results equal those of the split search (and of the CPU oracle) for every
// order; only the work per TEP differs.
//
// The five-point order with the library's choice of the test (AUTO) walks only
// the lightest weights and then joins the two halves of the ranks (k_per_tep<true>):
// a CTA of four warps prepares four frames, and each frame they leave open is
// decided by all of them -- the partial syndromes of the lower ranks (at most
// 5^5 = 3,125) go into a hash table in shared memory and those of the upper
// ranks are looked up. 6,250 table steps take the place of up to 5^10 =
// 9,765,625 TEPs tested one by one: 6,000 frames (N=128 16-QAM, 6/8/10 dB,
// S=10, cap 2^20) 32 ms -> 0.11 ms. What is left is latency (37 % issue): the
// CTA's warps wait for one another between the preparation and the joins.

#include <stdint.h>

#include "device_common.cuh"
#include "host_util.cuh"

namespace grand {
namespace {

constexpr unsigned kAll = 0xFFFFFFFFu;
constexpr int kAltMax = 4;  // alternatives per symbol (five-point NNE)
constexpr int kTepWarps = 4;
constexpr int kSlotBits = 13;        // hash slots: 2.6 per entry of a full side
constexpr int kSlots = 1 << kSlotBits;
constexpr int kJoinStep = 5;         // table accesses a thread keeps in flight
constexpr int kLowRanks = 3;         // ranks of a side spread over the threads (5^3 <= 128)

struct TepArgs {
  CodeDev code;
  const float2* symbols;
  int64_t n_frames;
  int m, side, L, Sp;
  int walk;                      // weights walked before the join
  int lik, order, rowparity;
  float q;
  uint32_t cap;
  uint32_t* cw;
  uint32_t* queries;
  uint8_t* abandon;
  unsigned int* next;            // frame work queue
  unsigned long long* counters;  // [0] TEPs tested, [1] frames past query 1, [2] their queries
  unsigned long long* t0;        // the call's clock start (deadline)
  long long deadline;            // grand_params.deadline_ns (0: none)
};

// Shared memory of one warp (words):
//   y[32] hard word, s0[kWMax] base syndrome, apos[kSMax][4] the (up to two)
//   bit positions of each alternative, aproj[kSMax][4] their projection,
//   sel[kSMax] selected symbols, kk[16] alternatives per rank (bytes),
//   key[L], info[L], and for the row test xs[N/32][32] (lane l's candidate
//   word in column l).
__host__ __device__ inline size_t tep_warp_bytes(int L, int NW, int rowparity) {
  size_t b = 4 * (32 + kWMax + 2 * kSMax * kAltMax + kSMax) + 16 + 8 * (size_t)L;
  if (rowparity) b += 4 * 32 * (size_t)NW;
  return (b + 15) & ~(size_t)15;
}

__device__ __forceinline__ void flip_lane(uint32_t* xs, int lane, uint32_t ap) {
  const uint32_t p0 = ap & 0xFFFFu, p1 = ap >> 16;
  if (p0 != kNoPos) xs[(p0 >> 5) * 32 + lane] ^= 1u << (p0 & 31);
  if (p1 != kNoPos) xs[(p1 >> 5) * 32 + lane] ^= 1u << (p1 & 31);
}

// H x = 0 for each live lane's candidate x (column `lane` of xs), by rows.
// Warp-collective: every lane calls it; the loop ends when no live lane has
// an all-even prefix of rows left.
__device__ bool row_parity_zero(const uint32_t* __restrict__ hrow, int R, int NW, const uint32_t* xs, int lane,
                                bool live) {
  bool zero = live;
  for (int r = 0; r < R; ++r) {
    if (!__any_sync(kAll, zero)) break;
    if (zero) {
      const uint32_t* h = hrow + (size_t)r * NW;
      uint32_t acc = 0;
      for (int w = 0; w < NW; ++w) acc ^= __ldg(h + w) & xs[w * 32 + lane];
      zero = (__popc(acc) & 1) == 0;
    }
  }
  return zero;
}

// Full syndrome of the TEP is zero: s0 xor the flipped H columns. The TEP is
// held packed: rank of position j in bits [4j, 4j+4) of pp, its alternative
// index in bits [2j, 2j+2) of dg.
__device__ bool delta_zero(const CodeDev& code, const uint32_t* s0, const uint32_t* apos, uint64_t pp, uint32_t dg,
                           int w) {
  for (int k = 0; k < code.W; ++k) {
    uint32_t v = s0[k];
    for (int j = 0; j < w; ++j) {
      const uint32_t ap = apos[(int)((pp >> (4 * j)) & 15u) * kAltMax + ((dg >> (2 * j)) & 3u)];
      const uint32_t p0 = ap & 0xFFFFu, p1 = ap >> 16;
      if (p0 != kNoPos) v ^= __ldg(code.hcol + (size_t)p0 * code.W + k);
      if (p1 != kNoPos) v ^= __ldg(code.hcol + (size_t)p1 * code.W + k);
    }
    if (v) return false;
  }
  return true;
}

// One frame's ranks as the join sees them.
struct JoinFrame {
  const uint32_t* s0;
  const uint32_t* apos;
  const uint32_t* aproj;
  const uint8_t* kk;
  uint32_t f0;
  int Sp;
};

// A vector of digits (3 bits per rank: 0 unchanged, else alternative + 1) and
// its projection.
struct Part {
  uint32_t code, z;
};

// The index-th digit vector of ranks [r0, r0 + n), rank r0 the fastest, radix
// alternatives + 1; `over`: index beyond the last.
__device__ __forceinline__ Part join_part(const JoinFrame& f, int r0, int n, uint32_t index, bool& over) {
  Part p{0u, 0u};
  for (int r = r0; r < r0 + n; ++r) {
    const uint32_t radix = (uint32_t)f.kk[r] + 1u;
    const uint32_t d = index % radix;
    index /= radix;
    p.code |= d << (3 * r);
    if (d) p.z ^= f.aproj[r * kAltMax + d - 1];
  }
  over = index != 0;
  return p;
}

// Order of the TEPs as an integer: weight, altered ranks in colex order (the
// mask as a number), alternatives from the largest rank down (the code).
__device__ __forceinline__ unsigned long long join_key(uint32_t code) {
  uint32_t m = 0;
  for (int r = 0; r < GRAND_S_MAX_NNE5; ++r) m |= (((code >> (3 * r)) & 7u) ? 1u : 0u) << r;
  return ((unsigned long long)__popc(m) << 40) | ((unsigned long long)m << 30) | code;
}

// Ranks and alternative indices of a code, packed as delta_zero takes them.
__device__ __forceinline__ int join_unpack(uint32_t code, uint64_t& pp, uint32_t& dg) {
  int w = 0;
  pp = 0;
  dg = 0;
  for (int r = 0; r < GRAND_S_MAX_NNE5; ++r) {
    const uint32_t d = (code >> (3 * r)) & 7u;
    if (!d) continue;
    pp |= (uint64_t)r << (4 * w);
    dg |= (d - 1u) << (2 * w);
    ++w;
  }
  return w;
}

// Entry n of the lower side's table (its number) and the code c of projection z,
// where projections are syndromes: 0 when they differ, else 1 when the entry
// comes first in the order, 2 when c does.
__device__ __noinline__ int join_alike(const JoinFrame& f, int loA, const uint2* high, uint32_t n, uint32_t c,
                                       uint32_t z) {
  bool none;
  const Part lo = join_part(f, 0, loA, n & 127u, none);
  if ((lo.z ^ high[n >> 7].y) != z) return 0;
  return join_key(lo.code | high[n >> 7].x) < join_key(c) ? 1 : 2;
}

// Hash join of the lower ranks [0, S'/2) with the upper ones, by the whole
// CTA. A thread holds one digit vector of a side's first three ranks and goes
// through those of the other two (at most 25, kept in `high`), kJoinStep table
// accesses in flight at a time. Slots hold 20 bits of the mixed key and the
// entry's number + 1 (low index + 128 x high index); equal ones are confirmed
// on every syndrome word. Where a syndrome has one word (and is its own
// projection) the first in the order of the lower codes that change it alike
// stays alone: with the same upper code the others come after it. (Few parity
// bits leave few syndromes; all of their codes in the table made chains that
// every look-up walked: 300 frames of 128 bits with 6 parity bits 4509 us, so
// 75.) *best: the smallest join_key of a codeword
// (initialised by the caller).
__device__ void join_sides(const CodeDev& code, const JoinFrame& f, uint32_t* table, uint2 (*high)[32],
                           unsigned long long* best) {
  constexpr int kThreads = 32 * kTepWarps;
  const bool exact = code.W == 1;
  const int nA = f.Sp >> 1, nB = f.Sp - nA;
  const int loA = min(nA, kLowRanks), loB = min(nB, kLowRanks);
  const uint32_t t = threadIdx.x;
  uint4* t4 = reinterpret_cast<uint4*>(table);
  for (int i = (int)t; i < kSlots / 4; i += kThreads) t4[i] = make_uint4(0u, 0u, 0u, 0u);
  uint32_t sizeA = 1, sizeB = 1;  // digit vectors of the ranks after the first three
  for (int r = loA; r < nA; ++r) sizeA *= f.kk[r] + 1u;
  for (int r = nA + loB; r < f.Sp; ++r) sizeB *= f.kk[r] + 1u;
  bool over, none;
  if (t < 64) {
    const Part p = t < 32 ? join_part(f, loA, nA - loA, t, over) : join_part(f, nA + loB, nB - loB, t - 32u, over);
    high[t >> 5][t & 31u] = make_uint2(p.code, p.z);
  }
  __syncthreads();
  {
    const Part lo = join_part(f, 0, loA, t, over);
    const uint32_t z0 = f.f0 ^ lo.z;
    for (uint32_t h0 = 0; !over && h0 < sizeA; h0 += kJoinStep) {
      uint32_t k[kJoinStep], was[kJoinStep];
#pragma unroll
      for (int u = 0; u < kJoinStep; ++u) {
        const uint32_t h = h0 + u;
        k[u] = (z0 ^ high[0][h & 31u].y) * 0x9E3779B1u;
        was[u] = h < sizeA ? atomicCAS(table + (k[u] >> (32 - kSlotBits)), 0u, (k[u] << 12) | (t + 128u * h + 1u)) : 0u;
      }
#pragma unroll
      for (int u = 0; u < kJoinStep; ++u) {  // taken: alike, or the next free slot
        const uint32_t entry = (k[u] << 12) | (t + 128u * (h0 + u) + 1u);
        uint32_t slot = k[u] >> (32 - kSlotBits);
        while (was[u] != 0u) {
          if (exact && !((was[u] ^ entry) >> 12)) {
            const uint2 hi = high[0][(h0 + u) & 31u];
            const int alike = join_alike(f, loA, high[0], (was[u] & 4095u) - 1u, lo.code | hi.x, lo.z ^ hi.y);
            if (alike == 1) break;
            if (alike == 2) {
              const uint32_t seen = atomicCAS(table + slot, was[u], entry);
              if (seen == was[u]) break;
              was[u] = seen;  // another thread was here: look again
              continue;
            }
          }
          slot = (slot + 1u) & (kSlots - 1u);
          was[u] = atomicCAS(table + slot, 0u, entry);
        }
      }
    }
  }
  __syncthreads();
  {
    const Part lo = join_part(f, nA, loB, t, over);
    for (uint32_t h0 = 0; !over && h0 < sizeB; h0 += kJoinStep) {
      uint32_t k[kJoinStep], seen[kJoinStep];
#pragma unroll
      for (int u = 0; u < kJoinStep; ++u) {
        const uint32_t h = h0 + u;
        k[u] = (lo.z ^ high[1][h & 31u].y) * 0x9E3779B1u;
        seen[u] = h < sizeB ? table[k[u] >> (32 - kSlotBits)] : 0u;
      }
#pragma unroll
      for (int u = 0; u < kJoinStep; ++u) {
        uint32_t slot = k[u] >> (32 - kSlotBits);
        for (uint32_t e = seen[u]; e != 0u; e = table[slot]) {
          slot = (slot + 1u) & (kSlots - 1u);
          if ((e ^ (k[u] << 12)) >> 12) continue;
          const uint32_t n = (e & 4095u) - 1u;
          const uint32_t c = lo.code | high[1][h0 + u].x | join_part(f, 0, loA, n & 127u, none).code | high[0][n >> 7].x;
          const unsigned long long key = join_key(c);
          if (key >= *(volatile unsigned long long*)best) continue;
          uint64_t pp;
          uint32_t dg;
          const int w = join_unpack(c, pp, dg);
          if (delta_zero(code, f.s0, f.apos, pp, dg, w)) atomicMin(best, key);
        }
      }
    }
  }
  __syncthreads();
}

// Position of a TEP among the valid ones (1-based), by one warp: lane v holds
// the number of valid TEPs altering exactly v of the ranks passed so far.
__device__ uint32_t join_position(const JoinFrame& f, uint32_t code) {
  const int v = threadIdx.x & 31;
  uint32_t e = v == 0 ? 1u : 0u, acc = 0, alt = 0, low = 1;
  int w = 0;
  for (int r = 0; r < f.Sp; ++r) {
    const uint32_t k = f.kk[r], d = (code >> (3 * r)) & 7u;
    if (d) {
      ++w;
      acc = acc * k + __shfl_sync(kAll, e, w);
      alt += (d - 1u) * low;
      low *= k;
    }
    uint32_t up = __shfl_up_sync(kAll, e, 1);
    if (v == 0) up = 0;
    e += k * up;
  }
  return __reduce_add_sync(kAll, v < w ? e : 0u) + acc + alt + 1u;
}

// kJoin: the five-point order with the join (see the head of the file); the
// CTA's warps then take four consecutive frames together.
template <bool kJoin>
__global__ void __launch_bounds__(32 * kTepWarps) k_per_tep(TepArgs a) {
  extern __shared__ __align__(16) char smem_raw[];
  __shared__ unsigned s_first;
  __shared__ uint2 s_high[2][32];
  __shared__ uint32_t s_f0[kTepWarps];
  __shared__ int s_open[kTepWarps];
  __shared__ unsigned long long s_best[kTepWarps];
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const CodeDev& code = a.code;
  const int N = code.N, NW = N >> 5, L = a.L, Sp = a.Sp, m = a.m;
  const uint32_t* proj = kJoin && code.W == 1 ? code.hcol : code.hf;  // one word: the syndrome itself
  const size_t warp_bytes = tep_warp_bytes(L, NW, a.rowparity);
  uint32_t* table = reinterpret_cast<uint32_t*>(smem_raw);  // [kSlots], join only
  char* const bases = smem_raw + (kJoin ? sizeof(uint32_t) * kSlots : 0);
  char* base = bases + (size_t)warp * warp_bytes;
  uint32_t* y = reinterpret_cast<uint32_t*>(base);
  uint32_t* s0 = y + 32;
  uint32_t* apos = s0 + kWMax;
  uint32_t* aproj = apos + kSMax * kAltMax;
  int* sel = reinterpret_cast<int*>(aproj + kSMax * kAltMax);
  uint8_t* kk = reinterpret_cast<uint8_t*>(sel + kSMax);
  uint32_t* key = reinterpret_cast<uint32_t*>(kk + 16);
  uint32_t* info = key + L;
  uint32_t* xs = info + L;
  unsigned long long n_eval = 0, n_hard = 0, n_hard_q = 0;

  for (;;) {
    unsigned int fi = 0;
    bool walk = true;  // this warp has a frame to search
    if constexpr (kJoin) {
      __syncthreads();  // the last round's shared words have been read
      if (threadIdx.x == 0) s_first = atomicAdd(a.next, (unsigned)kTepWarps);
      if (lane == 0) {
        s_open[warp] = 0;
        s_best[warp] = ~0ull;
      }
      __syncthreads();
      if ((int64_t)s_first >= a.n_frames) break;
      fi = s_first + (unsigned)warp;
      walk = (int64_t)fi < a.n_frames;
    } else {
      if (lane == 0) fi = atomicAdd(a.next, 1u);
      fi = __shfl_sync(kAll, fi, 0);
      if ((int64_t)fi >= a.n_frames) break;
    }
    const int64_t f = fi;
    uint32_t f0 = 0;
    const uint32_t cap = a.cap;
    uint32_t cum = 0;  // valid TEPs of the batches already walked
    bool found = false;
    uint32_t hit_rank = 0;
    int hit_lane = -1, w_hit = 0;
    // the lane's TEP, packed: pp = ranks (4 bits per position, ascending),
    // dg = alternative indices (2 bits), km = alternatives - 1 (2 bits)
    uint64_t pp = 0;
    uint32_t dg = 0, km = 0;
    if (walk) {

    // --- Step 1: demodulation and the hard word --------------------------
    if (lane < NW) y[lane] = 0u;
    __syncwarp();
    bool nonfinite = false;
    for (int i = lane; i < L; i += 32) {
      float2 sy = a.symbols[f * L + i];
      const bool nf = !(isfinite(sy.x) && isfinite(sy.y));
      if (nf) sy = make_float2(0.0f, 0.0f);
      nonfinite |= nf;
      const AxisDemod I = demod_axis_q(sy.x, a.q, a.side, a.lik);
      const AxisDemod Q = demod_axis_q(sy.y, a.q, a.side, a.lik);
      key[i] = (uint32_t)I.dq * (uint32_t)I.dq + (uint32_t)Q.dq * (uint32_t)Q.dq;
      info[i] = pack_info(I.level, Q.level, make_nmask(I, Q, nf));
      const uint32_t label = ((uint32_t)gray_code(I.level) << m) | (uint32_t)gray_code(Q.level);
      const uint32_t rl = __brev(label) >> (32 - 2 * m);  // bit k = label bit (2m-1-k)
      const int p0 = 2 * m * i, wd = p0 >> 5, sh = p0 & 31;
      if (wd < NW) atomicOr(&y[wd], rl << sh);
      if (sh && wd + 1 < NW) {
        const uint32_t hi = rl >> (32 - sh);
        if (hi) atomicOr(&y[wd + 1], hi);
      }
    }
    nonfinite = __any_sync(kAll, nonfinite);
    __syncwarp();
    if (nonfinite) {
      if (lane < NW) a.cw[f * NW + lane] = y[lane];
      if (lane == 0) {
        a.queries[f] = 0;
        a.abandon[f] = 2;
      }
      __syncwarp();
      walk = false;
    }
    if (walk && a.deadline > 0) {
      int cut = 0;
      if (lane == 0) cut = past_deadline(a.t0, a.deadline);
      if (__shfl_sync(kAll, cut, 0)) {  // fetched after the deadline: the hard word, marked 5
        if (lane < NW) a.cw[f * NW + lane] = y[lane];
        if (lane == 0) {
          a.queries[f] = 0;
          a.abandon[f] = 5;
          atomicOr(code.status, 1u);
        }
        __syncwarp();
        walk = false;
      }
    }
    }
    if (walk) {

    // --- base syndrome s0 = H y and its projection (delta test) ----------
    if (!a.rowparity) {
      uint32_t s[kWMax];
#pragma unroll
      for (int k = 0; k < kWMax; ++k) s[k] = 0u;
      for (int j = lane; j < N; j += 32) {
        if ((y[j >> 5] >> (j & 31)) & 1u) {
#pragma unroll
          for (int k = 0; k < kWMax; ++k)
            if (k < code.W) s[k] ^= __ldg(code.hcol + (size_t)j * code.W + k);
          f0 ^= __ldg(proj + j);
        }
      }
#pragma unroll
      for (int k = 0; k < kWMax; ++k) {
        if (k < code.W) {  // warp-uniform bound
          uint32_t v = s[k];
          for (int o = 16; o; o >>= 1) v ^= __shfl_xor_sync(kAll, v, o);
          if (lane == 0) s0[k] = v;
        }
      }
      for (int o = 16; o; o >>= 1) f0 ^= __shfl_xor_sync(kAll, f0, o);
    }

    // --- Steps 2-3: the S' least reliable symbols, by (key, index) -------
    for (int r = 0; r < Sp; ++r) {
      uint32_t bk = 0xFFFFFFFFu, bi = 0xFFFFFFFFu;
      for (int i = lane; i < L; i += 32) {
        const uint32_t k = key[i];
        if (k < bk) {
          bk = k;
          bi = (uint32_t)i;
        }
      }
      const uint32_t kmin = __reduce_min_sync(kAll, bk);
      const uint32_t imin = __reduce_min_sync(kAll, bk == kmin ? bi : 0xFFFFFFFFu);
      if (lane == 0) sel[r] = (int)imin;
      if (lane == (int)(imin & 31u)) key[imin] = 0xFFFFFFFFu;  // keys are < 2^31
      __syncwarp();
    }

    // --- Step 4: the alternatives of each rank, in their query order -----
    if (lane < Sp) {
      const int i = sel[lane];
      const uint32_t inf = info[i];
      const int lI = inf & 0xFF, lQ = (inf >> 8) & 0xFF;
      const uint32_t nm = (inf >> 16) & 0xFF;
      const bool exI = nm & 1u, exQ = nm & 2u;
      const int dI = (nm & 8u) ? 1 : -1, dQ = (nm & 16u) ? 1 : -1;
      const uint32_t pI = exI ? flip_pos_I(i, m, lI, dI, N) : kNoPos;
      const uint32_t pQ = exQ ? flip_pos_Q(i, m, lQ, dQ, N) : kNoPos;
      const uint32_t none = (uint32_t)kNoPos << 16;
      uint32_t list[kAltMax];
      int n = 0;
      if (a.order == GRAND_ORDER_QAM_NNE5) {
        // toward the received value on I, on Q; away from it on I, on Q
        if (exI) list[n++] = pI | none;
        if (exQ) list[n++] = pQ | none;
        if (lI - dI >= 0 && lI - dI < a.side) list[n++] = flip_pos_I(i, m, lI, -dI, N) | none;
        if (lQ - dQ >= 0 && lQ - dQ < a.side) list[n++] = flip_pos_Q(i, m, lQ, -dQ, N) | none;
      } else {
        // h, v, diag (Def. III.2); the nearer order puts v first where d_Q < d_I
        const bool swap = a.order == GRAND_ORDER_QAM_NEARER && (nm & 32u);
        const bool e1 = swap ? exQ : exI, e2 = swap ? exI : exQ;
        const uint32_t q1 = swap ? pQ : pI, q2 = swap ? pI : pQ;
        if (e1) list[n++] = q1 | none;
        if (e2) list[n++] = q2 | none;
        if (exI && exQ) list[n++] = pI | (pQ << 16);
      }
      for (int k = 0; k < kAltMax; ++k) {
        const uint32_t ap = k < n ? list[k] : ((uint32_t)kNoPos | none);
        const uint32_t p0 = ap & 0xFFFFu, p1 = ap >> 16;
        apos[lane * kAltMax + k] = ap;
        aproj[lane * kAltMax + k] =
            (p0 != kNoPos ? __ldg(proj + p0) : 0u) ^ (p1 != kNoPos ? __ldg(proj + p1) : 0u);
      }
      kk[lane] = (uint8_t)n;
    }
    __syncwarp();

    // --- Step 5: the canonical walk ----------------------------------------
    const int w_end = kJoin ? min(Sp, a.walk) : Sp;
    for (int w = 0; w <= w_end && !found && cum < cap; ++w) {
      const uint32_t nsets = binom16(Sp, w);
      for (uint32_t b0 = 0; b0 < nsets && !found && cum < cap;) {
        // m sets in this batch, P lanes per set: lane l takes part l % P of
        // set b0 + l / P (parts split the set's alternatives in order, so
        // lane order stays canonical order)
        const uint32_t m = min(32u, nsets - b0);
        const uint32_t P = 32u / m;
        const uint32_t si = b0 + (uint32_t)lane / P;
        const uint32_t part = (uint32_t)lane % P;
        const bool has_set = (uint32_t)lane < m * P;
        b0 += m;
        uint32_t nalpha = 0;
        pp = 0;
        km = 0;
        if (has_set) {
          // colex unranking: the largest rank first
          uint32_t t = si;
          nalpha = 1;
          for (int j = w; j >= 1; --j) {
            int p = j - 1;
            while (binom16(p + 1, j) <= t) ++p;
            t -= binom16(p, j);
            pp |= (uint64_t)p << (4 * (j - 1));
            const uint32_t k = kk[p];
            nalpha *= k;
            km |= ((k ? k : 1u) - 1u) << (2 * (j - 1));
          }
        }
        // this lane's part of the set's alternatives: [a0, a0 + n_lane)
        const uint32_t chunk = (nalpha + P - 1) / P;
        const uint32_t a0 = part * chunk;
        const uint32_t n_lane = a0 < nalpha ? min(chunk, nalpha - a0) : 0u;
        uint32_t incl = n_lane;
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t v = __shfl_up_sync(kAll, incl, o);
          if (lane >= o) incl += v;
        }
        const uint32_t batch = __shfl_sync(kAll, incl, 31);
        const uint32_t first = cum + (incl - n_lane) + 1;  // 1-based position of the lane's first TEP
        uint32_t n_here = 0;
        if (n_lane && first <= cap) n_here = min(n_lane, cap - first + 1);
        // alternative indices of the part's first TEP: a0 in mixed radix,
        // the smallest rank the least significant digit
        uint32_t z = f0;
        dg = 0;
        if (n_here) {
          uint32_t rest = a0;
          for (int j = 0; j < w; ++j) {
            const uint32_t k = ((km >> (2 * j)) & 3u) + 1u;
            const uint32_t d = rest % k;
            rest /= k;
            dg |= d << (2 * j);
            z ^= aproj[(int)((pp >> (4 * j)) & 15u) * kAltMax + d];
          }
        }
        if (a.rowparity) {
          for (int k = 0; k < NW; ++k) xs[k * 32 + lane] = y[k];
          if (n_here)
            for (int j = 0; j < w; ++j)
              flip_lane(xs, lane, apos[(int)((pp >> (4 * j)) & 15u) * kAltMax + ((dg >> (2 * j)) & 3u)]);
        }
        bool live = n_here > 0, hit = false;
        uint32_t ai = 0;
        for (;;) {
          bool h;
          if (a.rowparity)
            h = row_parity_zero(code.hrow, code.R, NW, xs, lane, live);
          else
            h = live && z == 0u && delta_zero(code, s0, apos, pp, dg, w);
          n_eval += live ? 1u : 0u;
          if (h) {
            hit = true;
            live = false;
          }
          if (live) {
            if (++ai >= n_here) {
              live = false;
            } else {
              // next alternative tuple: mixed-radix increment, smallest rank fastest
              for (int j = 0; j < w; ++j) {
                const int sh = 2 * j;
                const int r = (int)((pp >> (4 * j)) & 15u);
                const uint32_t d = (dg >> sh) & 3u;
                const uint32_t nd = d == ((km >> sh) & 3u) ? 0u : d + 1u;
                z ^= aproj[r * kAltMax + d] ^ aproj[r * kAltMax + nd];
                if (a.rowparity) {
                  flip_lane(xs, lane, apos[r * kAltMax + d]);
                  flip_lane(xs, lane, apos[r * kAltMax + nd]);
                }
                dg = (dg & ~(3u << sh)) | (nd << sh);
                if (nd) break;
              }
            }
          }
          const unsigned hm = __ballot_sync(kAll, hit);
          const unsigned lm = __ballot_sync(kAll, live);
          if (hm && !(lm & ((hm & (0u - hm)) - 1u))) break;  // nothing live below the lowest hit
          if (!lm) break;
        }
        const unsigned hm = __ballot_sync(kAll, hit);
        if (hm) {
          hit_lane = __ffs(hm) - 1;
          hit_rank = __shfl_sync(kAll, first + ai, hit_lane);
          w_hit = w;
          found = true;
        }
        cum += batch;
      }
    }

    }

    // --- Step 5, the rest of an open frame by the join -----------------------
    if constexpr (kJoin) {
      if (walk && lane == 0 && !found && cum < cap && Sp > a.walk) {
        s_open[warp] = 1;
        s_f0[warp] = f0;
      }
      __syncthreads();
      for (int q = 0; q < kTepWarps; ++q) {
        if (!s_open[q]) continue;
        const uint32_t* b = reinterpret_cast<const uint32_t*>(bases + (size_t)q * warp_bytes);
        JoinFrame fr;
        fr.s0 = b + 32;
        fr.apos = fr.s0 + kWMax;
        fr.aproj = fr.apos + kSMax * kAltMax;
        fr.kk = reinterpret_cast<const uint8_t*>(fr.aproj + kSMax * kAltMax + kSMax);
        fr.f0 = s_f0[q];
        fr.Sp = Sp;
        join_sides(code, fr, table, s_high, &s_best[q]);
        if (q == warp) {
          uint32_t total = 1;  // valid TEPs: at most 5^10
          for (int r = 0; r < Sp; ++r) total *= kk[r] + 1u;
          if (lane == 0) n_eval += total - cum;
          cum = total;
          const unsigned long long best = s_best[q];
          if (best != ~0ull) {
            const uint32_t c = (uint32_t)best & 0x3FFFFFFFu;
            const uint32_t pos = join_position(fr, c);
            if (pos <= cap) {
              found = true;
              hit_rank = pos;
              hit_lane = 0;
              w_hit = join_unpack(c, pp, dg);
            }
          }
        }
      }
    }
    if (!walk) continue;

    // --- Return: x = y xor e of the first hit, else y ---------------------
    if (found && lane == hit_lane) {
      for (int j = 0; j < w_hit; ++j) {
        const uint32_t ap = apos[(int)((pp >> (4 * j)) & 15u) * kAltMax + ((dg >> (2 * j)) & 3u)];
        const uint32_t p0 = ap & 0xFFFFu, p1 = ap >> 16;
        if (p0 != kNoPos) y[p0 >> 5] ^= 1u << (p0 & 31);
        if (p1 != kNoPos) y[p1 >> 5] ^= 1u << (p1 & 31);
      }
    }
    __syncwarp();
    if (lane < NW) a.cw[f * NW + lane] = y[lane];
    if (lane == 0) {
      const uint32_t qn = found ? hit_rank : min(cum, cap);
      a.queries[f] = qn;
      a.abandon[f] = found ? 0 : 1;
      if (!(found && hit_rank == 1)) {
        n_hard += 1;
        n_hard_q += qn;
      }
    }
    __syncwarp();
  }
  for (int o = 16; o; o >>= 1) n_eval += __shfl_xor_sync(kAll, n_eval, o);
  if (lane == 0) {
    atomicAdd(a.counters + 0, n_eval);
    if (n_hard) {
      atomicAdd(a.counters + 1, n_hard);
      atomicAdd(a.counters + 2, n_hard_q);
    }
  }
}

}  // namespace

int run_per_tep(const grand_code* c, const grand_params* p, const void* symbols, int64_t n_frames, uint32_t* cw,
                uint32_t* queries, uint8_t* abandon, grand_stats* stats, cudaStream_t st) {
  if (n_frames == 0) {
    if (stats) *stats = grand_stats{};
    return GRAND_OK;
  }
  NvtxRange range("grand.per_tep");
  const int m = m_of(p->M);
  TepArgs a{};
  a.code = c->dev;
  a.symbols = static_cast<const float2*>(symbols);
  a.n_frames = n_frames;
  a.m = m;
  a.side = 1 << m;
  a.L = (c->N + 2 * m - 1) / (2 * m);
  a.Sp = p->S < a.L ? p->S : a.L;
  a.lik = p->lik_variant;
  a.order = p->order;
  a.rowparity = p->membership == GRAND_MEMBERSHIP_ROW_PARITY ? 1 : 0;
  a.q = make_qam_const().q[m];
  a.cap = (uint32_t)(p->query_cap < 0xFFFFFFFFll ? p->query_cap : 0xFFFFFFFFll);
  a.cw = cw;
  a.queries = queries;
  a.abandon = abandon;
  // the join decides every TEP at once; DELTA and ROW_PARITY ask for the test
  // of each. Its cost does not depend on the cap (the lower side's table above
  // all), the walk's grows with it: 3,000 frames of 128 bits, S' = 10 (a table
  // of 3,125 entries) 114 - 142 us whatever the cap, the walk 43 us at 300
  // TEPs, 60 at 800, 115 at 3,125; S' = 9, a table of 625 entries, 57 us.
  int64_t table = 1, walked = 0;
  for (int r = 0; r < a.Sp / 2; ++r) table *= 5;
  // Weight 1 (41 TEPs) decides most frames that decode; walking weight 2 (720
  // more) costs more than it saves the join (134 against 125 us for 6,000 N=128
  // frames). With few parity bits, whose space is full of codewords, weights 2
  // and 3 (8,400 TEPs) leave the join little but frames that the walk would
  // search to the cap: 300 frames of 128 bits with 6 parity bits 75 us (137 with
  // weight 2, 92 without the join), 6 frames with 11 parity bits 72 (159, 89).
  a.walk = c->R <= 12 ? 3 : 1;
  int64_t count = 1;  // TEPs of weight w: C(S', w) 4^w
  for (int w = 0; w <= a.walk && w <= a.Sp; ++w) {
    walked += count;
    count = count * 4 * (a.Sp - w) / (w + 1);
  }
  const bool join = p->order == GRAND_ORDER_QAM_NNE5 && p->membership == GRAND_MEMBERSHIP_AUTO &&
                    p->query_cap > (table > walked ? table : walked);
  auto kern = join ? k_per_tep<true> : k_per_tep<false>;
  char* scratch = nullptr;
  if (scratch_alloc((void**)&scratch, 64, st) != cudaSuccess) return GRAND_E_NOMEM;
  a.next = reinterpret_cast<unsigned int*>(scratch);
  a.counters = reinterpret_cast<unsigned long long*>(scratch + 8);
  a.t0 = reinterpret_cast<unsigned long long*>(scratch + 32);
  a.deadline = p->deadline_ns;
  int rc = GRAND_OK;
  cudaEvent_t ev[2] = {nullptr, nullptr};
  do {
    if (cudaMemsetAsync(scratch, 0, 64, st) != cudaSuccess) { rc = GRAND_E_CUDA; break; }
    const size_t smem =
        (join ? sizeof(uint32_t) * kSlots : 0) + kTepWarps * tep_warp_bytes(a.L, c->N / 32, a.rowparity);
    // (a fixed limit for the join: a concurrent call's larger frames are never undercut)
    const size_t limit = join ? 64 * 1024 : smem;
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit) != cudaSuccess) {
      rc = GRAND_E_CUDA;
      break;
    }
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * kTepWarps, smem) != cudaSuccess ||
        per_sm < 1)
      per_sm = 1;
    const int64_t want = (n_frames + kTepWarps - 1) / kTepWarps;
    const int64_t full = (int64_t)sm_count() * per_sm;
    const int grid = (int)(want < full ? want : full);
    if (stats) {
      for (int i = 0; i < 2; ++i)
        if (cudaEventCreate(&ev[i]) != cudaSuccess) { rc = GRAND_E_CUDA; break; }
      if (rc) break;
      cudaEventRecord(ev[0], st);
    }
    kern<<<grid, 32 * kTepWarps, smem, st>>>(a);
    if (cudaGetLastError() != cudaSuccess) { rc = GRAND_E_CUDA; break; }
    if (stats) {
      cudaEventRecord(ev[1], st);
      unsigned long long h[3] = {0, 0, 0};
      if (cudaMemcpyAsync(h, a.counters, sizeof h, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
          cudaStreamSynchronize(st) != cudaSuccess) {
        rc = GRAND_E_CUDA;
        break;
      }
      *stats = grand_stats{};
      stats->evaluated_checks = h[0];
      stats->hard_frames = h[1];
      stats->search_useful = h[2];
      stats->prep_ms = 0.0f;
      cudaEventElapsedTime(&stats->search_ms, ev[0], ev[1]);
    }
  } while (0);
  for (int i = 0; i < 2; ++i)
    if (ev[i]) cudaEventDestroy(ev[i]);
  cudaFreeAsync(scratch, st);
  return rc;
}

}  // namespace grand
