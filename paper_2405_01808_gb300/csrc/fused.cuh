// Launch interface of the fused decode kernel (fused.cu).
#pragma once

#include "axis.cuh"
#include "host_util.cuh"
#include "internal.cuh"

namespace grand {

// Codes passed by value with the launch: the code of a uniform batch, or a
// small table of an uneven one, which then needs no table in device memory.
constexpr int kInlineCodes = 8;

// A frame of an uneven batch in the order of launch_order.
struct alignas(32) OrderRec {
  int64_t sym_offset, cw_offset;
  uint32_t par, code, frame, unused;  // par: frame_par
};

struct DecodeArgs {
  const float2* symbols;         // received symbols, or NULL: the demodulated arrays
  const uint16_t* hard_idx;
  const uint32_t* key;
  const uint8_t* nmask;
  const uint32_t* y_in;
  const grand_frame_desc* desc;  // NULL: uniform batch
  const OrderRec* order;         // uneven batch: its frames by length (launch_order), or NULL
  int64_t n_symbols;             // mixed: length of the flat symbol array
  int64_t n_cw_words;            // mixed: length of the flat output array
  const CodeDev* codes;          // uneven batch: device table, or NULL: code[]
  int n_codes;
  int64_t n_frames;
  int M, L;                      // uniform batch
  int m;                         // log2(M) / 2 (set by launch_decode)
  int S;
  int lik;
  int nearer;                    // GRAND_ORDER_QAM_NEARER: swap h / v where d_Q < d_I
  int solve;                     // statistics of GRAND_MEMBERSHIP_SOLVE (ranked solutions)
  int w0;                        // statistics: weights a searched frame went past
  int NWmax;                     // words of the longest code (uniform batch: of the code)
  int T;                         // frames per warp (set by launch_decode)
  int64_t cap;
  AxisConst ax[7];               // index m = log2(M) / 2
  uint32_t* cw;
  uint32_t* queries;
  uint8_t* abandon;
  Scratch* scr;                  // statistics, or NULL
  unsigned long long* t0;        // the call's clock start (deadline), or NULL
  long long deadline;            // grand_params.deadline_ns of a linear solve (0: none)
  CodeDev code[kInlineCodes];    // uniform batch: [0]
};

// Scratch that launch_order needs for the batch; 0: it is decoded in its own order.
size_t order_bytes(const DecodeArgs& a);
// Frames of an uneven batch by length and constellation (sets a.order).
int launch_order(DecodeArgs& a, void* scratch, cudaStream_t st);

// One launch on `st`; Lmax: the largest frame of the batch in symbols.
int launch_decode(DecodeArgs a, int Lmax, cudaStream_t st);

// Load the kernels an uneven batch can launch (see preload_qam_kernels).
int preload_decode_kernels();

}  // namespace grand
