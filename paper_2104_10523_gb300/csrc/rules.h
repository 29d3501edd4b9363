// Host-side rules about the buffers a caller hands over (no CUDA in here).
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace tnq {

// Whether the n bytes at p and the m bytes at q share a byte.
inline bool ranges_overlap(const void* p, size_t n, const void* q, size_t m) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(p), b = reinterpret_cast<uintptr_t>(q);
  return a < b ? b - a < n : a - b < m;
}

// Whether kernels on device ctx_device may address caller memory of the given
// kind (device memory of `device`, managed, or neither: host).  Memory of another
// GPU is only copied: peer access may be off.
inline bool kernels_reach(bool device_memory, bool managed, int device, int ctx_device) {
  return managed || (device_memory && device == ctx_device);
}

// Whether every address is a multiple of n.  Complex64 tensors of a caller are
// 8-byte aligned and no more (a slice may start at an odd element): 16-byte
// accesses and tensor maps ask first.
template <typename... P>
bool aligned(size_t n, const P*... p) {
  return (... && (reinterpret_cast<uintptr_t>(p) % n == 0));
}

// A caller's workspace is used from its first multiple of kWorkspaceAlign on (bulk
// copies and 16-byte loads address it); the sizes the library asks for hold the
// bytes in front of it.
constexpr size_t kWorkspaceAlign = 256;
inline char* workspace_base(void* ws) {
  return reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(ws) + kWorkspaceAlign - 1) / kWorkspaceAlign * kWorkspaceAlign);
}

}  // namespace tnq
