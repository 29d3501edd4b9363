// Error flags in mapped host memory.
//
// Kernels raise a flag when a bounded wait runs out or an input value is bad;
// the host reads it after its stream has been synchronised.  A flag in device
// memory cost every call a clearing memset and a blocking 4-byte copy (about
// 12 us of a 22 us call); a mapped one is written over the bus only when it is
// raised.
#pragma once

namespace tnq {

constexpr int kFlagInput = 0;  // bad bitstring entry
constexpr int kFlagWait = 1;   // a bounded device-side wait ran out

// A zeroed slot of two ints from a process-wide pool of fixed size (thread
// safe; usable from every device), or nullptr when host memory cannot be
// pinned or every slot is taken.  No kernel may still write a slot given back.
int* flags_get();
void flags_put(int* slot);

// Reads a slot after the kernels that write it have completed, and clears it.
struct FlagValues {
  int input, wait;
};
FlagValues flags_take(int* slot);

}  // namespace tnq
