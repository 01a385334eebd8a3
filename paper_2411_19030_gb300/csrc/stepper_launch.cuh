// stepper_launch.cuh -- kernel table of the cluster stepper.
#pragma once
#include "ptg_internal.h"

namespace ptg {

using StepKernel = void (*)(const StepParams);
using BatchKernel = void (*)(const StepParams*, const int2*, int, int*);
struct StepKernels {
  StepKernel single;
  StepKernel narrow;    // the same for blocks of at most kStepNarrowThreads threads, with more registers each
  BatchKernel batch;
  StepKernel wide;      // grid-wide variant (FP64, single-task kinds, NG <= 3), else null
};

// Groups of 4 nodes per thread (NG) supported by the build; a CTA has up to 512 threads, so
// it holds up to 2048 * NG nodes.  (stepper_inst.cu instantiates the same list.)
constexpr int kStepNG[] = {1, 2, 3, 4, 5, 6};
constexpr int kNumStepNG = sizeof(kStepNG) / sizeof(kStepNG[0]);
constexpr int kStepMaxThreadsHost = 512;
constexpr int kStepNarrowThreads = 384;

// Defined by the per-(precision, kind) translation units.
#define PTG_DECLARE_SELECT(P, K) \
  StepKernels stepper_select_##P##_##K##_lo(int ng); /* ng 1..3 */ \
  StepKernels stepper_select_##P##_##K##_hi(int ng); /* ng 4..6 */
PTG_DECLARE_SELECT(f32, 0) PTG_DECLARE_SELECT(f32, 1) PTG_DECLARE_SELECT(f32, 2)
PTG_DECLARE_SELECT(f32, 3) PTG_DECLARE_SELECT(f32, 4) PTG_DECLARE_SELECT(f32, 5)
PTG_DECLARE_SELECT(f64, 0) PTG_DECLARE_SELECT(f64, 1) PTG_DECLARE_SELECT(f64, 2)
PTG_DECLARE_SELECT(f64, 3) PTG_DECLARE_SELECT(f64, 4) PTG_DECLARE_SELECT(f64, 5)
#undef PTG_DECLARE_SELECT

inline StepKernels stepper_kernels_for(int precision, int kind, int ng) {
  const bool f32 = precision == PTG_FP32_REFINE;
#define PTG_PICK(K)                                                                       \
  case K:                                                                                 \
    return f32 ? (ng <= 3 ? stepper_select_f32_##K##_lo(ng) : stepper_select_f32_##K##_hi(ng)) \
               : (ng <= 3 ? stepper_select_f64_##K##_lo(ng) : stepper_select_f64_##K##_hi(ng))
  switch (kind) {
    PTG_PICK(0); PTG_PICK(1); PTG_PICK(2); PTG_PICK(3); PTG_PICK(4); PTG_PICK(5);
    default: return StepKernels{nullptr, nullptr, nullptr, nullptr};
  }
#undef PTG_PICK
}
inline StepKernel stepper_kernel_for(int precision, int kind, int ng, bool narrow) {
  const StepKernels k = stepper_kernels_for(precision, kind, ng);
  return narrow ? k.narrow : k.single;
}

}  // namespace ptg
