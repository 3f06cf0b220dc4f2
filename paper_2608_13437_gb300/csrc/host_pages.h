// Pages of pageable host memory that a device copy is about to write.
#pragma once

#include <sys/mman.h>
#include <unistd.h>

#include <algorithm>
#include <cstdint>
#include <thread>
#include <vector>

namespace lbm {

// First page in [lo, hi) that is not present (hi if all are).
inline uintptr_t first_missing_page(uintptr_t lo, uintptr_t hi, size_t page) {
  constexpr size_t kPages = 2048;
  unsigned char present[kPages];
  for (uintptr_t a = lo; a < hi; a += kPages * page) {
    const size_t n = std::min<size_t>(kPages, (hi - a) / page);
    if (mincore(reinterpret_cast<void*>(a), n * page, present) != 0) return a;
    for (size_t j = 0; j < n; ++j)
      if (!(present[j] & 1)) return a + j * page;
  }
  return hi;
}

// Makes the pages of [p, p + bytes) present for writing (their contents stay), several host
// threads at a time, and returns how many it asked for. A copy into memory that nothing has
// touched yet (a fresh numpy array) otherwise faults every page in from the GPU's side of
// the address space: 43 us per 64 KB page measured, 70 ms for 103 MB against 0.6 ms into
// touched memory; the host's own faults cost 3 us each. Memory that has been written before
// (a buffer in use, or one that the allocator hands out again) is left alone after one look:
// the threads alone took longer than the copy (64^3 primitives in FP64, 12.6 MB: 148 us
// without them, 206 with). Only a hint: where the kernel does not know the request nothing
// changes, and ranges below a few pages are left alone.
inline size_t populate_host_pages(void* p, size_t bytes) {
#ifndef MADV_POPULATE_WRITE
  constexpr int kPopulateWrite = 23;
#else
  constexpr int kPopulateWrite = MADV_POPULATE_WRITE;
#endif
  constexpr size_t kPerThread = 2u << 20;
  const size_t page = (size_t)sysconf(_SC_PAGESIZE);
  uintptr_t lo = (reinterpret_cast<uintptr_t>(p) + page - 1) / page * page;
  const uintptr_t hi = (reinterpret_cast<uintptr_t>(p) + bytes) / page * page;
  if (hi <= lo || hi - lo < 4 * page) return 0;
  lo = first_missing_page(lo, hi, page);
  if (lo == hi) return 0;
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
  return pages;
}

}  // namespace lbm
