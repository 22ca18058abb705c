// The autotuner's settings (flusi_autotune in flusi_capi.cu).
#pragma once

#include "../../include/flusi.h"

namespace flusi {

// A setting and the kernels it changes (names of flusi_profile_step without their
// stage suffix): a candidate is scored by their times.
struct TuneKnob {
    int flusi_tuning::*field;
    const char* kernels[2];
};
constexpr int kTuneKnobs = 6;
extern const TuneKnob tune_knobs[kTuneKnobs];   // in the order of the descent

}  // namespace flusi
