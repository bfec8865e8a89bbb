// FP32-mixed instantiation, part 5: the Heun passes over float4 spins.
#define SS_REAL float
#define SS_PART 5
#include "ss_launch.cuh"
