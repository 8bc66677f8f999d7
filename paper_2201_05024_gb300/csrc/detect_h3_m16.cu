// FP16 x3 detection kernels for 16 antennas.
#define APSM_H3_M 16
#include "detect_h3_inst.cuh"
