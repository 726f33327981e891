// Element kernels of the variable-coefficient path, N+1 = 2, 3, 4, 5.
#include "gdg_var_ops.cuh"

GDG_VAR_OPS(2)
GDG_VAR_OPS(3)
GDG_VAR_OPS(4)
GDG_VAR_OPS(5)
