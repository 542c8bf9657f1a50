// FP64 products on the tensor cores: declarations shared by the FP64 path (sp2_dense_f64.cu), the
// handles (sp2_api.cu) and the allocation-free entry (sp2_noalloc.cu).  The scheme and its error are
// described in sp2_f64_tc.cu.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace sp2 {

struct DevState;

namespace f64tc {

constexpr int ND = 7;              // digits per value
constexpr int MAX_RECS = 32;       // partial records (2 doubles) per upper 64 x 64 tile, at most (Plan::recs)

// The digits of one ld x ld matrix, in the order of the shared-memory stages (see sp2_f64_tc.cu), and one
// power-of-two exponent per row.
struct Digits {
  __half* dig = nullptr;
  int32_t* exp = nullptr;
};

struct Plan {
  Digits X, S;                     // of the iterate; of the McWeeny step's shifted square (dig null: none)
  int ld = 0;
  int bn = 0, ks = 0;              // columns of an output tile (32 or 64); CTAs that share its k range (1, 2, 4, 8)
  int recs = 0;                    // records per 64 x 64 tile: 32 rows x the columns one warp finishes
  bool on = false;
};

// Sizes at which the tensor-core products are used (see emit_product in sp2_dense_f64.cu).
constexpr int kMinN = 129;
// Bytes of the partial records of a problem with T x T tiles of 64 and `recs` records per upper tile (64 for
// N < kMinN).
constexpr size_t part_bytes(int64_t N, int T, int recs) {
  return sizeof(double) * 2 * (size_t)(N < kMinN ? 64 : recs) * ((size_t)T * (T + 1) / 2);
}
inline bool wanted(int64_t N) { return N >= kMinN; }

// Rows are padded to whole tiles of 128; the padding (and the rows past N) stays zero.
constexpr int padded_rows(int ld) { return (ld + 127) / 128 * 128; }
constexpr size_t digit_bytes(int ld) { return (size_t)ND * ld * padded_rows(ld) * sizeof(__half); }
constexpr size_t exp_bytes(int ld) { return (size_t)ld * sizeof(int32_t); }
// Tile shape for matrices with leading dimension ld (bn, ks, recs and ld of the plan).
void choose_tiles(Plan& P, int ld);
// What one product writes.
enum Op : int32_t {
  OP_SP2 = 0,      // X_k from X_{k-1} (Alg. 3, or the scheduled polynomial of Alg. 5)
  OP_MCW_SQ = 1,   // the McWeeny step's shifted square
  OP_MCW_PROD = 2  // the McWeeny step's product of the shifted square and X_{k-1}
};

// Kernels either launched on a stream or appended to a graph as a chain.
struct Sink {
  cudaStream_t s = nullptr;
  cudaGraph_t g = nullptr;
  cudaGraphNode_t last = nullptr;
  cudaError_t put(const void* func, dim3 grid, dim3 block, size_t smem, void** args);
};

// Digits of the newest iterate (buf0 or buf1, st->wrote), or of S when `S` is given.
cudaError_t emit_digits(Sink& sink, const DevState* st, const double* buf0, const double* buf1, const double* S,
                        const Plan& P, int N);
// The product `op` over the upper tiles, with the partial records of the stop test.  hook, wait_ms: of the testing
// entry (0: none, waits of 2 s).
cudaError_t emit_product(Sink& sink, DevState* st, double* buf0, double* buf1, double* S, double* part,
                         const Plan& P, Op op, int hook = 0, int wait_ms = 0);

}  // namespace f64tc
}  // namespace sp2
