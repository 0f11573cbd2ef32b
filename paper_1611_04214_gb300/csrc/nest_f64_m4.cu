// Nested passes of quadrature order 4, F64 (a translation unit per order and precision).
#include "nest_launch.cuh"

MOLT_INSTANTIATE_NEST(4, double)
