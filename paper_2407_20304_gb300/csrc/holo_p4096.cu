// Kernel instantiations for line length P = 4096: line and column D-steps (the passes: holo_p4096_*.cu).
#include "holo_kernels.cuh"
HOLO_INSTANTIATE_SPLIT(4096)
