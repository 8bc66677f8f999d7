// FP16 x3 detection kernels for 64 antennas.
#define APSM_H3_M 64
#include "detect_h3_inst.cuh"
