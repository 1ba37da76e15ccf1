// meeting_numbers.hpp -- the numbers that stamp the resident kernel's meetings
// (kernels_resident.cu), handed out launch by launch.  Host code only.
#pragma once
#include <cstdint>

namespace lpgb {

// The `count` numbers after `last` for the next launch: its first one is *seq0 + 1.
// A mailbox keeps the stamps of old launches, and 0 where nothing was written yet, so
// no number is given out twice and 0 never is.  Returns true where the 32-bit
// numbers begin again: the mailboxes must then be zeroed before the launch.
// (209,000 launches away at graph_iters 4096, two minutes of pivots.)
inline bool take_meeting_numbers(uint32_t& last, uint32_t count, uint32_t* seq0) {
    const bool restart = count > UINT32_MAX - last;
    *seq0 = restart ? 0 : last;
    last = *seq0 + count;
    return restart;
}

}  // namespace lpgb
