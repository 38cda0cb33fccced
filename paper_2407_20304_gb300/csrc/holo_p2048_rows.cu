// Kernel instantiations for line length P = 2048: passes A and C.
#include "holo_kernels.cuh"
HOLO_ROWS(template, 2048)
