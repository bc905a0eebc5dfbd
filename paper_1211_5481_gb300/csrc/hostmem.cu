// hostmem.cu -- page-locked host memory for the small read-backs (status words, a
// batch's fitness).
//
// Page-locking is paid per process, not per handle: cudaMallocHost and cudaFreeHost
// of the 8 bytes a handle wants took 320 us of its creation and release where the
// process held no other page-locked memory (M = 2000, N = 8: 626 us, 286 so). So one
// block of 256 KB is registered at the first use and handed out in units of 64
// bytes; it stays for the process. Where it is full, or could not be registered (or a
// device reset undid that), the memory is ordinary: copies into it then wait, and
// arrive all the same.
#include <stdlib.h>

#include <mutex>

#include "game_internal.cuh"

namespace game {

namespace {

constexpr size_t kBlock = (size_t)256 << 10, kPage = (size_t)64 << 10, kUnit = 64;
constexpr int kUnits = (int)(kBlock / kUnit);
std::mutex g_lock;
unsigned char* g_block = nullptr;
bool g_used[kUnits];

bool registered() {
  cudaPointerAttributes at{};
  if (cudaPointerGetAttributes(&at, g_block) == cudaSuccess) return at.type == cudaMemoryTypeHost;
  cudaGetLastError();
  return false;
}

int units(size_t bytes) { return bytes > kBlock ? kUnits + 1 : (int)((bytes + kUnit - 1) / kUnit); }

}  // namespace

void* host_take(size_t bytes) {
  {
    std::lock_guard<std::mutex> lock(g_lock);
    if (!g_block) g_block = static_cast<unsigned char*>(aligned_alloc(kPage, kBlock));
    if (g_block && !registered() &&
        cudaHostRegister(g_block, kBlock, cudaHostRegisterPortable) != cudaSuccess)
      cudaGetLastError();
    const int n = units(bytes);
    int run = 0;
    for (int u = 0; g_block && u < kUnits; ++u) {
      run = g_used[u] ? 0 : run + 1;
      if (run < n) continue;
      for (int k = u - n + 1; k <= u; ++k) g_used[k] = true;
      return g_block + (size_t)(u - n + 1) * kUnit;
    }
  }
  return malloc(bytes);
}

void host_give(void* p, size_t bytes) {
  unsigned char* c = static_cast<unsigned char*>(p);
  std::lock_guard<std::mutex> lock(g_lock);
  if (!g_block || c < g_block || c >= g_block + kBlock) {
    free(p);
    return;
  }
  const int u0 = (int)((size_t)(c - g_block) / kUnit);
  for (int k = 0; k < units(bytes); ++k) g_used[u0 + k] = false;
}

}  // namespace game
