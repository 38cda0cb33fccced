// Kernel instantiations for line length P = 4096: passes A and C.
#include "holo_kernels.cuh"
HOLO_ROWS(template, 4096)
