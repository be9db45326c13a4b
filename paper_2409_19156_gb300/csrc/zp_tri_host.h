// Host-side interface of the triangle form of the fused float64-accurate series (zp_tri.cu).
#pragma once

#include <cstdint>

#include "zp_fused.h"
#include "zp_internal.h"
#include "zp_tri.h"

namespace zp {

// Bytes of one coefficient group's digits per chunk: 9 blocks of 16 sets x 16 float16.
constexpr uint32_t kTriGroupBytes = (uint32_t)kTriDigits * kFusedMaxSets * kTriChunk * 2u;

// One series instance (device pointers).
struct TriInst {
  int32_t n_max = 0;
  int32_t KC = 0;          // chunks of the contraction
  int32_t seg_chunks = 1;  // chunks per segment
  int64_t kc_base = 0;     // first chunk in the launch's chunk numbering
  int64_t J = 0, P = 0, S = 0;
  const double* r = nullptr;
  const double* theta = nullptr;    // NULL: no mode has an angle
  const double* coeffs = nullptr;   // [J][S]
  const int32_t* perm = nullptr;    // [KC * 16]: mode of every position, -1 for none
  uint8_t* bdig = nullptr;          // [KC][groups] digits (written per call)
  int* cexp = nullptr;              // [groups][16] set scales (written per call)
  double* cpos = nullptr;           // gradients: [2][KC * 16][16] derivative coefficients (per call)
  double* out = nullptr;            // values: [P][S]
  const double* gdot = nullptr;     // gradients: [P][S] upstream
  double* grad_r = nullptr;         // [P], either may be NULL
  double* grad_theta = nullptr;
};

// Launch description: `insts` and `items` in device memory, or (both NULL) one instance passed by
// value whose 128-point tiles are the items in order.
struct TriArgs {
  const TriInst* insts = nullptr;
  const FusedItem* items = nullptr;
  int64_t n_items = 0;
  TriInst single;
};

inline size_t tri_digit_bytes(int64_t chunks, bool gradients) {
  return ((size_t)chunks * kTriGroupBytes * (gradients ? 2 : 1) + 255) / 256 * 256;
}
inline size_t tri_cpos_bytes(int64_t chunks) { return (size_t)chunks * kTriChunk * kFusedMaxSets * 2 * sizeof(double); }

// Coefficient digits of every instance, then the kernel over all items: values into `out`, or (two
// coefficient groups) the point gradients.  n_max: the largest instance's.  Stream-ordered, no
// host synchronisation (capturable).
zp_status tri_launch(const TriArgs& a, int n_max, const int32_t* chunk_inst, int64_t n_chunks, bool gradients,
                     cudaStream_t stream);

// An instance of a plan that has the triangle layout (plan->tri), without buffers and outputs.
TriInst tri_inst(const zp_plan* plan, const double* r, const double* theta, int64_t P, const double* coeffs, int64_t S);

// F = Z C and the point gradients of <G, F> for one plan with plan->tri and S <= kFusedMaxSets.
zp_status tri_series_eval(const zp_plan* plan, const double* r, const double* theta, int64_t P, const double* coeffs,
                          int64_t S, double* out, cudaStream_t stream);
zp_status tri_point_grads(const zp_plan* plan, const double* r, const double* theta, int64_t P, const double* coeffs,
                          int64_t S, const double* G, double* grad_r, double* grad_theta, cudaStream_t stream);

// Reads and optionally clears the kernel's wait-status word (non-zero: a bounded wait gave up).
zp_status tri_error_word(unsigned int* value, bool reset);

}  // namespace zp
