// The float32 instances of the solver's box kernels, in a translation unit of their own (parallel compilation).
#define ENS_BOX_F32
#include "solver_box.cu"
