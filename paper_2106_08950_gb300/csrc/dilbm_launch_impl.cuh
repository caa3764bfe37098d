// Bodies of the per-storage launchers (dilbm_launch.cuh), included by the
// translation unit that instantiates them for its storage type.
#pragma once
#include "dilbm_launch.cuh"

namespace dilbm {

template <typename T>
cudaError_t Launch<T>::steps(const SweepArgs<T> &a, const PartArgs &pa, const StepRun &run, bool edges, bool ps, const SweepShape &sh,
                             int num_sms, cudaStream_t st, int *per_sm) {
    if (ps)
        return edges ? step_variant<T, true, PS_WARPS, true>(a, pa, run, SweepShape{PS_WARPS, 0}, num_sms, st, per_sm)
                     : step_variant<T, false, PS_WARPS, true>(a, pa, run, SweepShape{PS_WARPS, 0}, num_sms, st, per_sm);
    switch (sh.warps) {
    case 2: return edges ? step_variant<T, true, 2, false>(a, pa, run, sh, num_sms, st, per_sm)
                         : step_variant<T, false, 2, false>(a, pa, run, sh, num_sms, st, per_sm);
    case 4: return edges ? step_variant<T, true, 4, false>(a, pa, run, sh, num_sms, st, per_sm)
                         : step_variant<T, false, 4, false>(a, pa, run, sh, num_sms, st, per_sm);
    case 8: return edges ? step_variant<T, true, 8, false>(a, pa, run, sh, num_sms, st, per_sm)
                         : step_variant<T, false, 8, false>(a, pa, run, sh, num_sms, st, per_sm);
    default: return cudaErrorInvalidValue;
    }
}

template <typename T>
cudaError_t Launch<T>::batch(const BatchArgs<T> &ba, const StepRun &run, const SweepShape &sh, int num_sms,
                             cudaStream_t st, int *per_sm) {
    switch (sh.warps) {
    case 2: return batch_variant<T, 2>(ba, run, sh, num_sms, st, per_sm);
    case 4: return batch_variant<T, 4>(ba, run, sh, num_sms, st, per_sm);
    case 8: return batch_variant<T, 8>(ba, run, sh, num_sms, st, per_sm);
    default: return cudaErrorInvalidValue;
    }
}

template <typename T>
cudaError_t Launch<T>::sweep(const SweepArgs<T> &a, bool edges, bool ps, const SweepShape &sh, int num_sms,
                             cudaStream_t st, bool chained, int *per_sm) {
    const FieldsOut none{};
    if (ps) return edges ? sweep_variant<T, MODE_STEP, true, true>(a, none, num_sms, st, SWEEP_SHAPE, chained, per_sm)
                         : sweep_variant<T, MODE_STEP, false, true>(a, none, num_sms, st, SWEEP_SHAPE, chained, per_sm);
    switch (sh.warps) {
    case 2: return edges ? sweep_variant<T, MODE_STEP, true, false, 2>(a, none, num_sms, st, sh, chained, per_sm)
                         : sweep_variant<T, MODE_STEP, false, false, 2>(a, none, num_sms, st, sh, chained, per_sm);
    case 4: return edges ? sweep_variant<T, MODE_STEP, true, false, 4>(a, none, num_sms, st, sh, chained, per_sm)
                         : sweep_variant<T, MODE_STEP, false, false, 4>(a, none, num_sms, st, sh, chained, per_sm);
    case 8: return edges ? sweep_variant<T, MODE_STEP, true, false, 8>(a, none, num_sms, st, sh, chained, per_sm)
                         : sweep_variant<T, MODE_STEP, false, false, 8>(a, none, num_sms, st, sh, chained, per_sm);
    default: return cudaErrorInvalidValue;
    }
}

template <typename T>
cudaError_t Launch<T>::fields(const SweepArgs<T> &a, const FieldsOut &fo, bool edges, bool ps, int num_sms,
                              cudaStream_t st) {
    if (ps) return edges ? sweep_variant<T, MODE_FIELDS, true, true>(a, fo, num_sms, st)
                         : sweep_variant<T, MODE_FIELDS, false, true>(a, fo, num_sms, st);
    return edges ? sweep_variant<T, MODE_FIELDS, true, false>(a, fo, num_sms, st)
                 : sweep_variant<T, MODE_FIELDS, false, false>(a, fo, num_sms, st);
}

}  // namespace dilbm
