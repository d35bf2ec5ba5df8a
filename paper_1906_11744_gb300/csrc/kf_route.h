// Who moves a caller's array: a kernel of this library, which reads or writes
// it in place, or a copy of the driver's.  A kernel takes 4-byte words, which
// have to start on 4 bytes (a field of a packed record or a view at an odd
// offset does not), and it reaches the memory of its own GPU and, through the
// host's page tables, of the host; another GPU's memory only where the program
// enabled peer access, while the driver's copy reaches it always.
#ifndef KF_ROUTE_H_
#define KF_ROUTE_H_

#include <cstdint>

namespace kfg {

constexpr int NO_DEVICE = -1;  // host or managed memory

// p: the array; on: the GPU its memory belongs to (or NO_DEVICE); dev: the
// kernel's GPU.
inline bool kernel_reads(const void* p, int on, int dev) {
  return ((std::uintptr_t)p & 3) == 0 && (on == NO_DEVICE || on == dev);
}
// Results are written byte by byte where they do not start on a word.
inline bool kernel_writes(int on, int dev) { return on == NO_DEVICE || on == dev; }

}  // namespace kfg

#endif
