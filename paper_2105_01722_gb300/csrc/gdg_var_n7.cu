// Element kernels of the variable-coefficient path, N+1 = 7.
#include "gdg_var_ops.cuh"

GDG_VAR_OPS(7)
