// Batched sweeps of FP32 levels (work lists), a unit of its own.
#include "instantiate.h"

BIOT_SWEEP_BATCH(float, float)

// A batched launch of storage kind v (SWEEP_V_PAIR set): FP32 levels above FP32 levels.
cudaError_t biot::launch_pair_batch(int v, const biot::BatchParams<float, float> &P, cudaStream_t s)
{
    using namespace biot;
    constexpr int F = KIND_FINE | KIND_NOGHOST, C = KIND_COARSE | KIND_NOGHOST;
    const bool prol = v & SWEEP_V_PROL, zero = v & SWEEP_V_ZERO;
    if (v & SWEEP_V_COARSE) {
        if (v & SWEEP_V_RESTRICT) return launch_pair_batch_fm<float, C, false, true, FETCH_PLAIN>(P, s);
        if (zero) return launch_pair_batch_fm<float, C, false, false, FETCH_ZERO>(P, s);
        if (prol) return launch_pair_batch_fm<float, C, false, false, FETCH_PROL>(P, s);
        return launch_pair_batch_fm<float, C, false, false, FETCH_PLAIN>(P, s);
    }
    if (v & SWEEP_V_RESTRICT) return launch_pair_batch_fm<float, F, true, true, FETCH_PLAIN>(P, s);
    if (v & SWEEP_V_MEAS)
        return prol ? launch_pair_batch_fm<float, F, true, false, FETCH_PROL, true>(P, s)
                    : launch_pair_batch_fm<float, F, true, false, FETCH_PLAIN, true>(P, s);
    if (prol) return launch_pair_batch_fm<float, F, true, false, FETCH_PROL>(P, s);
    return launch_pair_batch_fm<float, F, true, false, FETCH_PLAIN>(P, s);
}
