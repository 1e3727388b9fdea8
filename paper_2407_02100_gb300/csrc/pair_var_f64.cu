// Variable-coefficient patch sweep in double precision.
#define GMG_PAIR_ARITH SoloDF
#include "pair_var.cuh"
