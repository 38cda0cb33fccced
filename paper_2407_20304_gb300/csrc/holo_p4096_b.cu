// Kernel instantiations for line length P = 4096: pass B.
#include "holo_kernels.cuh"
HOLO_PASS_B(template, 4096)
