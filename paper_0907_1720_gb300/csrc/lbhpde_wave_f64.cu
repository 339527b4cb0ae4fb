// k_wave in FP64, and the planning of both precisions.
#define LBH_WAVE_ESZ 8
#include "lbhpde_wave_launch.cuh"
