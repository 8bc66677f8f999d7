// detect_h3_inst.cuh -- instantiates the FP16 x3 detection kernel for one antenna count (APSM_H3_M)
// and every user-count bucket.
#pragma once

#include "detect_h3.cuh"

#define APSM_H3_CAT2(a, b) a##b
#define APSM_H3_CAT(a, b) APSM_H3_CAT2(a, b)

namespace apsm {

H3Launcher APSM_H3_CAT(detect_h3_launcher_m, APSM_H3_M)(int kb) {
    constexpr int M = APSM_H3_M;
    switch (kb) {
        case 2: return launch_detect_h3<M, 2>;
        case 4: return launch_detect_h3<M, 4>;
        case 6: return launch_detect_h3<M, 6>;
        case 8: return launch_detect_h3<M, 8>;
        case 12: return launch_detect_h3<M, 12>;
        case 16: return launch_detect_h3<M, 16>;
        default: return nullptr;
    }
}

}  // namespace apsm
