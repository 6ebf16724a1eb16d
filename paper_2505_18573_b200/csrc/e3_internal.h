// What the Python binding takes from the library beyond the C ABI.
#pragma once
#include <stdint.h>

#include "e3.h"

namespace e3 {

// e3_group_advantage that also defines what the C call leaves alone: the advantage of rewards outside every group (n_rewards of
// them in all) and the flags of empty groups become 0, so that outputs need no clearing beforehand.
E3_API e3_status group_advantage_filled(const float *rewards, int64_t n_rewards, const int64_t *group_offsets, int64_t n_groups,
                                        float eps, int unbiased, float *out_adv, uint8_t *out_group_flags, void *stream);

}  // namespace e3
