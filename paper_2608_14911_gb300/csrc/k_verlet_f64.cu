// The Verlet list search of the FP64 handles (the kernel sources are in k_verlet.cu).
#define ESPP_STEP_PRECISION 64
#include "k_verlet.cu"
