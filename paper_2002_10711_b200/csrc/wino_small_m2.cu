// Small-layer kernel instantiated for F(2x2, 3x3).
#define WINO_M 2
#include "wino_small_impl.cuh"
