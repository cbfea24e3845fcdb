// kpz_host.h -- host helpers shared by the C-ABI layers.
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include <thread>

namespace kpz {

// Writes to every page of a caller's buffer that a kernel is about to fill.
// Pages of a fresh allocation exist only once touched, and a GPU that is the
// first to touch them waits some 55 us for every 64 KiB it stores (heights at L
// = 2048 took 28 ms into a fresh array, 1.2 ms into a touched one). One write to
// each 4096 bytes touches them all, whatever the system's page size is, at 3.5
// us a page that did not exist; large buffers are split over a few threads.
inline void touch_pages(void* p, size_t bytes) {
  constexpr size_t kPage = 4096, kPart = size_t(4) << 20, kThreads = 8;
  auto touch = [](char* a, char* b) {
    for (; a < b; a += kPage) *(volatile char*)a = 0;
  };
  char* base = (char*)p;
  const size_t parts = std::min(kThreads, bytes / kPart);
  size_t done = 0;
  std::thread th[kThreads];
  size_t n = 0;
  try {
    for (; n + 1 < parts; ++n) {
      const size_t end = done + bytes / parts / kPage * kPage;
      th[n] = std::thread(touch, base + done, base + end);
      done = end;
    }
  } catch (...) {   // no thread to be had: the rest is touched here
  }
  touch(base + done, base + bytes);
  for (std::thread& t : th)
    if (t.joinable()) t.join();
  if (bytes) *(volatile char*)(base + bytes - 1) = 0;
}

// Whether the current device reads and writes pageable host memory itself.
inline bool reaches_pageable(int device) {
  int v = 0;
  return cudaDeviceGetAttribute(&v, cudaDevAttrPageableMemoryAccess, device) == cudaSuccess && v != 0;
}

// Whether kernels may use the caller's float arrays in place: `in` (n_in of
// them) read and `out` (may be null) written, sizes in bytes.
// They need the type's alignment, which a copy does not, and an output apart
// from every input: the call may read an input after it has begun to write.
struct HostSpan {
  const void* p;
  size_t bytes;
};
inline bool usable_in_place(const HostSpan* in, int n_in, HostSpan out) {
  const uintptr_t o = (uintptr_t)out.p;
  bool ok = o % alignof(float) == 0;
  for (int i = 0; i < n_in; ++i) {
    const uintptr_t a = (uintptr_t)in[i].p;
    ok = ok && a % alignof(float) == 0 && (!o || a + in[i].bytes <= o || o + out.bytes <= a);
  }
  return ok;
}

}  // namespace kpz
