// once_calls.h -- numbering of the single-launch force calls of one device.
#pragma once

// Calls between two clears of the device words (DSDNA_ONCE_CALLS: a small
// number, to test the clear).
#ifndef DSDNA_ONCE_CALLS
#define DSDNA_ONCE_CALLS (1u << 29)
#endif

namespace dsdna {

// The call number tells this call's agreement words, position records and cell
// lists from those that earlier calls left in the scratch memory: agreement
// number call + 1 (on word (call + 1) mod 3), tag and epoch call + 1.  No two
// calls between clears share a number; after ONCE_CALLS of them, or a call that
// failed, the device words are cleared and the numbers start over.
constexpr unsigned ONCE_CALLS = DSDNA_ONCE_CALLS;
struct OnceCalls {
  unsigned next = 0;
  unsigned take(bool failed, bool* clear) {
    *clear = failed || next >= ONCE_CALLS;
    if (*clear) next = 0;
    return next++;
  }
};

}  // namespace dsdna
