// Which snapshots and restores one kernel may copy (host; no CUDA).
#pragma once

#include <stdint.h>

namespace pflbm {

// Where a snapshot buffer lies, as the runtime and the driver describe it.
struct BufferPlace {
  uintptr_t addr;                 // the buffer
  bool device_memory;             // plain device memory (not managed, not host)
  int device;                     // its device
  uintptr_t range_start;          // the allocation it lies in; range_bytes 0: unknown
  uint64_t range_bytes;
};

// states up to this size are copied by one kernel; above tens of MB one copy
// command per part is as fast
constexpr long long COPY_KERNEL_BYTES = 64LL << 20;

// A copy command finds the devices of both sides by itself and refuses a range
// that its allocation does not hold.  A kernel does neither, so it takes only a
// buffer that holds the state, in 16-byte words, in memory of the handle's
// device, and only while that device is the current one, where it would run (on
// the legacy stream without an error).  parts: the state's own addresses or-ed.
inline bool copy_by_kernel(const BufferPlace& b, uintptr_t parts, long long bytes, int handle_device,
                           int current_device) {
  if (bytes > COPY_KERNEL_BYTES || (b.addr | parts) % 16 != 0) return false;
  if (!b.device_memory || b.device != handle_device || current_device != handle_device) return false;
  return b.addr >= b.range_start && b.addr - b.range_start <= b.range_bytes &&
         b.range_bytes - (b.addr - b.range_start) >= (uint64_t)bytes;
}

}  // namespace pflbm
