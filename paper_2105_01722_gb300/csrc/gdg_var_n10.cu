// Element kernels of the variable-coefficient path, N+1 = 10.
#include "gdg_var_ops.cuh"

GDG_VAR_OPS(10)
