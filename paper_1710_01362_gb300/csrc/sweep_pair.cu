// The sweep kernel with two CTAs per SM (see sweep.cu).
#define SWEEP_PAIR
#include "sweep.cu"
