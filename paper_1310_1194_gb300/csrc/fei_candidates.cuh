// fei_candidates.cuh -- what fei_plan_tune times for one degree, as (variant,
// grid cap) pairs; host code without CUDA calls.
#pragma once

#include "fei_internal.cuh"

namespace fei {

struct Candidate {
  int variant;
  int64_t grid_cap;  // blocks, 0 = the kernel's default
};
constexpr int kMaxCandidates = 16;

// kind: the kernel of variant 0; ntc: its tensor-core variants (kind
// KERNEL_TC); sf_too: one variant more, number ntc, is the sum-factorised
// kernel (FEI_AUTO at p >= 3).  Returns the number written to out.
//   tensor-core kernel: every variant (one CTA per SM);
//   sum-factorised kernel: its default, as many blocks as fit, or one per SM;
//   CUDA-core precisions: the default, then 2, 4, 8 and 16 blocks per SM.  The
//     kernels are persistent and their default is the resident grid, which no
//     multiple of the SMs need be (p = 2 FP32: 912 blocks; 100 000 prisms 0.267 ms,
//     the best of the others 0.280); it comes first, so a tie keeps it.
inline int list_candidates(KernelKind kind, int ntc, bool sf_too, Candidate *out) {
  int n = 0;
  if (kind == KERNEL_TC)
    for (int v = 0; v < ntc; ++v) out[n++] = {v, 0};
  if (kind == KERNEL_SF || sf_too) {
    const int v = sf_too ? ntc : 0;
    out[n++] = {v, 0};
    out[n++] = {v, 152};
  }
  if (kind == KERNEL_CC) {
    out[n++] = {0, 0};
    for (int per_sm = 2; per_sm <= 16; per_sm *= 2) out[n++] = {0, 152 * per_sm};
  }
  return n;
}

}  // namespace fei
