// The Verlet list search of the FP32 handles (the kernel sources are in k_verlet.cu).
#define ESPP_STEP_PRECISION 32
#include "k_verlet.cu"
