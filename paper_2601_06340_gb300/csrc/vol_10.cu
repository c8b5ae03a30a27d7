#include "vol_launch.cuh"
BPM_INSTANTIATE_VOL(10)
