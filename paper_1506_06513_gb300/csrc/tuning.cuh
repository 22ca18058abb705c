// The autotuner's settings (flusi_autotune in flusi_capi.cu).
#pragma once

#include <string>

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

// What a handle's settings run: plans, tiles and the kernel of every pass.  Settings
// of one signature launch the same kernels and are timed once.
std::string tuning_signature(flusi_t h);
// The key of a handle's line in a tuning cache.
std::string tuning_key(flusi_t h);

}  // namespace flusi
