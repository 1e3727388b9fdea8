// Variable-coefficient patch sweep in single precision.
#define GMG_PAIR_ARITH PairF32
#include "pair_var.cuh"
