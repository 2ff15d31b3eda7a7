// Batched sweeps of FP32 levels (work lists), a unit of its own.
#include "instantiate.h"

BIOT_SWEEP_BATCH(float, float)
