// Pages of pageable host memory that a device copy is about to write.
#pragma once

#include <sys/mman.h>
#include <unistd.h>

#include <algorithm>
#include <cstdint>
#include <thread>
#include <vector>

namespace lbm {

// Makes the pages of [p, p + bytes) present for writing (their contents stay), several host
// threads at a time. A copy into memory that nothing has touched yet (a fresh numpy array)
// otherwise faults every page in from the GPU's side of the address space: 43 us per 64 KB
// page measured, 70 ms for 103 MB against 0.6 ms into touched memory; the host's own
// faults cost 3 us each. Only a hint: where the kernel does not know the request nothing
// changes, and ranges below a few pages are left alone.
inline void populate_host_pages(void* p, size_t bytes) {
#ifndef MADV_POPULATE_WRITE
  constexpr int kPopulateWrite = 23;
#else
  constexpr int kPopulateWrite = MADV_POPULATE_WRITE;
#endif
  constexpr size_t kPerThread = 2u << 20;
  const size_t page = (size_t)sysconf(_SC_PAGESIZE);
  const uintptr_t lo = (reinterpret_cast<uintptr_t>(p) + page - 1) / page * page;
  const uintptr_t hi = (reinterpret_cast<uintptr_t>(p) + bytes) / page * page;
  if (hi <= lo || hi - lo < 4 * page) return;
  const size_t pages = (hi - lo) / page;
  size_t n = std::max<size_t>(1, std::min<size_t>((hi - lo) / kPerThread, 8));
  const unsigned cores = std::thread::hardware_concurrency();
  if (cores) n = std::min<size_t>(n, cores);
  auto part = [=](size_t j) {
    const uintptr_t a = lo + pages * j / n * page, b = lo + pages * (j + 1) / n * page;
    if (b > a) madvise(reinterpret_cast<void*>(a), b - a, kPopulateWrite);
  };
  std::vector<std::thread> others;
  size_t started = 1;
  try {
    others.reserve(n);
    for (; started < n; ++started) others.emplace_back(part, started);
  } catch (...) {  // no thread to be had: the caller's own takes the rest
  }
  part(0);
  for (size_t j = started; j < n; ++j) part(j);
  for (std::thread& t : others) t.join();
}

}  // namespace lbm
