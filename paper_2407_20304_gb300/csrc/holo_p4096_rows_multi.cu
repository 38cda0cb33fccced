// Kernel instantiations for line length P = 4096: passes A and C of several problems.
#include "holo_kernels.cuh"
HOLO_ROWS_MULTI(template, 4096)
