// Variable-coefficient patch sweep in double precision.
#define GMG_PAIR_ARITH PairDF
#include "pair_var.cuh"
