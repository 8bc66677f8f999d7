// FP16 x3 detection kernels for 32 antennas.
#define APSM_H3_M 32
#include "detect_h3_inst.cuh"
