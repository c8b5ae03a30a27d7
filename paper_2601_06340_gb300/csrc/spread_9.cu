#include "spread_launch.cuh"
BPM_INSTANTIATE_SPREAD(9, 2)
