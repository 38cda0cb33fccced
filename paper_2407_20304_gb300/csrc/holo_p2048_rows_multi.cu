// Kernel instantiations for line length P = 2048: passes A and C of several problems.
#include "holo_kernels.cuh"
HOLO_ROWS_MULTI(template, 2048)
