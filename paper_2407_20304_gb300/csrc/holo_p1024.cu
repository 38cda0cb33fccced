// Kernel instantiations for line length P = 1024: line and column D-steps (the passes: holo_p1024_*.cu).
#include "holo_kernels.cuh"
HOLO_INSTANTIATE_SPLIT(1024)
