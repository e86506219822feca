// Which way a caller's "device" pointer is read or written.
#pragma once

namespace msgb {

// Kinds of memory, as cudaMemoryType numbers them.
enum { kMemUnregistered = 0, kMemHost = 1, kMemDevice = 2, kMemManaged = 3 };

// A kernel on device `here` may dereference memory of `kind` that lives on device
// `where`: its own, or managed memory.  A buffer on another GPU needs peer access
// for that (a fault without), so it goes through the copy engine, as does what the
// runtime does not know.
inline bool kernel_reaches(int kind, int where, int here) {
  return kind == kMemManaged || (kind == kMemDevice && where == here);
}

}  // namespace msgb
