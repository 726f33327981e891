// Element kernels of the variable-coefficient path, N+1 = 9.
#include "gdg_var_ops.cuh"

GDG_VAR_OPS(9)
