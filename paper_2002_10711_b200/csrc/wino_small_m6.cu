// Small-layer kernel instantiated for F(6x6, 3x3).
#define WINO_M 6
#include "wino_small_impl.cuh"
