// Nested passes of quadrature order 2, F32 (a translation unit per order and precision).
#include "nest_launch.cuh"

MOLT_INSTANTIATE_NEST(2, float)
