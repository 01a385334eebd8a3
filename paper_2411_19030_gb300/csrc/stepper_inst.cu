// stepper_inst.cu -- instantiates the cluster stepper for one precision and one task kind.
// Compiled once per (PTG_REAL, PTG_KIND, PTG_SET) so the kernels build in parallel:
//   PTG_REAL = float (FP32 CG + FP64 refinement) or double (FP64 CG); PTG_KIND = 0..5.
#include "stepper.cuh"
#include "stepper_launch.cuh"

#ifndef PTG_REAL
#error "define PTG_REAL (float or double)"
#endif
#ifndef PTG_KIND
#error "define PTG_KIND (0..5)"
#endif
#ifndef PTG_TAG
#error "define PTG_TAG (f32 or f64)"
#endif

#if !defined(PTG_SET) || !defined(PTG_FIRST_NG)
#error "define PTG_SET and PTG_FIRST_NG (lo and 1: NG 1..3; hi and 4: NG 4..6)"
#endif

#define PTG_CAT4(a, b, c, d) a##_##b##_##c##_##d
#define PTG_SELECT_NAME(tag, kind, set) PTG_CAT4(stepper_select, tag, kind, set)

namespace ptg {

namespace {   // every unit has its own

// The grid-wide (grouped) variant exists for every kind and precision, for up to 3 groups
// per thread.
template <int NG>
StepKernel wide_kernel() {
  if constexpr (NG <= 3) return &stepper_wide_kernel<PTG_REAL, NG, PTG_KIND>;
  else return nullptr;
}

template <int NG>
StepKernels kernels() {
  if constexpr (NG <= 3)
    return StepKernels{&stepper_kernel<PTG_REAL, NG, PTG_KIND, kStepMaxThreads>,
                       &stepper_kernel<PTG_REAL, NG, PTG_KIND, kStepNarrowThreads>,
                       &stepper_batch_kernel<PTG_REAL, NG, PTG_KIND>, wide_kernel<NG>()};
  else
    return StepKernels{&stepper_kernel<PTG_REAL, NG, PTG_KIND, kStepMaxThreads>, nullptr,
                       &stepper_batch_kernel<PTG_REAL, NG, PTG_KIND>, nullptr};
}

}  // namespace

StepKernels PTG_SELECT_NAME(PTG_TAG, PTG_KIND, PTG_SET)(int ng) {
  switch (ng - PTG_FIRST_NG) {
    case 0: return kernels<PTG_FIRST_NG>();
    case 1: return kernels<PTG_FIRST_NG + 1>();
    case 2: return kernels<PTG_FIRST_NG + 2>();
    default: return StepKernels{nullptr, nullptr, nullptr, nullptr};
  }
}

}  // namespace ptg
