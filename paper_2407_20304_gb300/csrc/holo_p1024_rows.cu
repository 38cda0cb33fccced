// Kernel instantiations for line length P = 1024: passes A and C.
#include "holo_kernels.cuh"
HOLO_ROWS(template, 1024)
