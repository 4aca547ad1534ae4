// Size of the counting pass's work units (host code only; no CUDA).
#pragma once

#include <algorithm>
#include <cstdint>

namespace rkm {

// User tiles per counting work unit (item tile, group of user tiles): `most`, or fewer where that would
// leave the SMs less than about 8 units each.  2,000 users x 1,000 items made 4 units of 16 tiles
// (counting phase 78 us on 4 SMs; 64 units of one tile: 17 us), and 32 candidates against a million
// users 244 units for 152 SMs.  Smaller units than needed reload the resident item tile more often.
// `fixed`: `most` as it is, for a launch that other problems' units fill as well.  Never below 1: the
// kernels divide by it, and `most` may come from a file of stored choices.
struct UnitRule {
    int most = 32;
    bool fixed = false;

    int tiles(int64_t user_tiles, int64_t item_tiles, int num_sms) const {
        const int64_t share = user_tiles * item_tiles / ((int64_t)num_sms * 8);
        return (int)std::max<int64_t>(1, fixed ? most : std::min<int64_t>(most, share));
    }
};

// The rule of a batch's instance: its tensor-core counting launch holds every instance's units, its FP32
// launches are the instance's own.  The autotuner times the call under this rule too: under the
// single call's, the sizes it compares were one and the same for 10,000 users x 5,000 items, and the
// choice, which the batch then took as it was, was noise.
inline UnitRule batch_units(int group, bool tensor_core) { return UnitRule{group, tensor_core}; }

}  // namespace rkm
