// Numbering of the pair form's k-steps (gvm_pair.cuh): which stage and which
// barrier phase a k-step uses. Plain functions, for the kernels and for host
// programs that check them.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define GVM_HD __host__ __device__ __forceinline__
#else
#define GVM_HD inline
#endif

namespace gvm {

constexpr uint32_t kPrStages = 3;           // bf16 stages
constexpr uint32_t kPrBars = 2 * kPrStages; // empty barriers

// K-step q: its stage, the parity of its phase of the stage's full barrier, and
// its empty barrier with the parity of that phase.
GVM_HD uint32_t pr_stage(uint32_t q) { return q % kPrStages; }
GVM_HD uint32_t pr_full_parity(uint32_t q) { return (q / kPrStages) & 1u; }
GVM_HD uint32_t pr_empty_bar(uint32_t q) { return q % kPrBars; }
GVM_HD uint32_t pr_empty_parity(uint32_t q) { return (q / kPrBars) & 1u; }
// The first k-steps of a launch find their stages empty; the others wait for
// k-step q - kPrStages to have been read.
GVM_HD bool pr_stage_used(uint32_t q) { return q >= kPrStages; }

// All of these repeat after kPrPeriod k-steps, and so does the converter group
// (q % 2). 2^32 is no multiple of it: a counter left to run would pass from one
// phase to another at its wrap, which a resident scheduler reaches after about
// an hour of products. So the number of a tile's first k-step is taken back by
// whole periods, to no less than one, once it has reached kPrBack; a product of
// the largest k (32768) adds less than that.
constexpr uint32_t kPrPeriod = 2 * kPrBars;
constexpr uint32_t kPrBack = 128 * kPrPeriod;
GVM_HD uint32_t pr_next_first(uint32_t first, uint32_t ksteps) {
  const uint32_t q = first + ksteps;
  return q < kPrBack ? q : q - (kPrBack - kPrPeriod);
}

}  // namespace gvm
