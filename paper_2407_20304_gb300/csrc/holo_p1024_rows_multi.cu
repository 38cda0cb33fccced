// Kernel instantiations for line length P = 1024: passes A and C of several problems.
#include "holo_kernels.cuh"
HOLO_ROWS_MULTI(template, 1024)
