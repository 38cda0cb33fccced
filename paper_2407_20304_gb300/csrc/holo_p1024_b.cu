// Kernel instantiations for line length P = 1024: pass B.
#include "holo_kernels.cuh"
HOLO_PASS_B(template, 1024)
