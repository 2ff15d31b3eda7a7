// Batched sweeps of FP32 levels above an FP64 level, a unit of its own.
#include "instantiate.h"

BIOT_SWEEP_BATCH(float, double)
