// Nested passes of quadrature order 6, F32 (a translation unit per order and precision).
#include "nest_launch.cuh"

MOLT_INSTANTIATE_NEST(6, float)
