// Small-layer kernel instantiated for F(4x4, 3x3).
#define WINO_M 4
#include "wino_small_impl.cuh"
