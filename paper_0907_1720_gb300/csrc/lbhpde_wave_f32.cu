// k_wave in FP32 (a translation unit of its own, so the two precisions compile in parallel).
#define LBH_WAVE_ESZ 4
#include "lbhpde_wave_launch.cuh"
