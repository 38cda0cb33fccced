// Kernel instantiations for line length P = 2048: line and column D-steps (the passes: holo_p2048_*.cu).
#include "holo_kernels.cuh"
HOLO_INSTANTIATE_SPLIT(2048)
