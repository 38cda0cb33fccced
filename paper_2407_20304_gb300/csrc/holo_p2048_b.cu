// Kernel instantiations for line length P = 2048: pass B.
#include "holo_kernels.cuh"
HOLO_PASS_B(template, 2048)
