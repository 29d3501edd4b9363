// Pool of error flags in mapped host memory (see flags.h).
#include <cuda_runtime.h>

#include <mutex>
#include <vector>

#include "flags.h"

namespace tnq {

namespace {

constexpr int kSlots = 4096, kSlotInts = 16;  // a 64-byte line each, 256 KB in all

struct Pool {
  std::mutex mu;
  int* base = nullptr;
  std::vector<int> free;
};

Pool& pool() {
  static Pool* p = new Pool();  // outlives objects destroyed at exit
  return *p;
}

}  // namespace

int* flags_get() {
  Pool& p = pool();
  std::lock_guard<std::mutex> lock(p.mu);
  if (!p.base) {
    void* m = nullptr;
    if (cudaHostAlloc(&m, size_t(kSlots) * kSlotInts * sizeof(int), cudaHostAllocPortable | cudaHostAllocMapped) !=
        cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    p.base = static_cast<int*>(m);
    p.free.reserve(kSlots);
    for (int i = kSlots - 1; i >= 0; --i) p.free.push_back(i);
  }
  if (p.free.empty()) return nullptr;
  int* slot = p.base + size_t(p.free.back()) * kSlotInts;
  p.free.pop_back();
  slot[kFlagInput] = slot[kFlagWait] = 0;
  return slot;
}

void flags_put(int* slot) {
  if (!slot) return;
  Pool& p = pool();
  std::lock_guard<std::mutex> lock(p.mu);
  p.free.push_back(int((slot - p.base) / kSlotInts));
}

FlagValues flags_take(int* slot) {
  volatile int* v = slot;
  FlagValues f{v[kFlagInput], v[kFlagWait]};
  v[kFlagInput] = 0;
  v[kFlagWait] = 0;
  return f;
}

}  // namespace tnq
