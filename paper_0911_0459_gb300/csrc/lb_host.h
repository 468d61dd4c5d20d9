// Host memory that results are about to be copied into.
//
// A caller's arrays are often fresh: their pages do not exist until something writes to
// them, and a device-to-host copy into such pages takes a fault for each (16384 x 256
// fields, 134 MB: 9.2 ms, 0.75 ms of it the copy; 2048 x 64, 4 MB: 0.77 ms).
// populate_host asks the system for the pages beforehand, beside the kernels that still
// run and by several threads where there are many (5.4 ms and 0.26 ms).  It changes no
// byte: pages that exist stay as they are, ranges whose pages exist already are left
// alone (asking for 134 MB of them takes 1.4 ms), a range that has some of them is asked for
// whole (predictions of 65536 rows into arrays that a heap hands out again, 33.5 MB: 1443 ->
// 1051 us against looking at four pages only), and where the system does not know the
// request or the address the copy finds what it found before.
#pragma once

#include <stddef.h>
#include <stdint.h>
#include <sys/mman.h>
#include <unistd.h>

#include <exception>
#include <thread>

#ifndef MADV_POPULATE_WRITE
#define MADV_POPULATE_WRITE 23
#endif

namespace lbk {

struct HostRange {
  void* p;
  size_t bytes;
};

// Pages wholly inside the ranges (the first and last partial page hold other data too and
// usually exist; the copy faults them in otherwise).  True if there were any to make.
inline bool populate_host(const HostRange* r, int n) {
  constexpr int kMost = 4;                // ranges looked at
  constexpr size_t kLeast = 1 << 20;      // smaller results: sixteen faults at most, or memory in use already
  constexpr size_t kPerThread = 2 << 20;  // a thread costs about as much to start as 0.5 MB of pages
  constexpr int kThreads = 4;  // more wait for one another in the kernel (134 MB: 3.9, 2.2, 1.5 ms with 1, 2, 4; 2.9 with 8)
  const size_t page = (size_t)sysconf(_SC_PAGESIZE);
  size_t total = 0;
  for (int i = 0; i < n; ++i)
    if (r[i].p) total += r[i].bytes;
  if (page == 0 || total < kLeast) return false;
  // whether a page of the range is not in memory (a heap that shrank and grew again has its
  // first page, and a result that was used in part others)
  auto fresh = [=](const HostRange& x) {
    const uintptr_t a = ((uintptr_t)x.p + page - 1) / page, b = ((uintptr_t)x.p + x.bytes) / page;
    unsigned char in[1024];
    for (uintptr_t k = a; k < b; k += sizeof in) {
      const size_t cnt = b - k < sizeof in ? b - k : sizeof in;
      if (mincore((void*)(k * page), cnt * page, in) != 0) return false;
      for (size_t q = 0; q < cnt; ++q)
        if (!(in[q] & 1)) return true;
    }
    return false;
  };
  HostRange todo[kMost];
  int m = 0;
  total = 0;
  for (int i = 0; i < n && m < kMost; ++i)
    if (r[i].p && fresh(r[i])) {
      todo[m++] = r[i];
      total += r[i].bytes;
    }
  if (total < kLeast) return false;
  // part k of parts: the same share of every range
  auto part = [&todo, m, page](int k, int parts) {
    for (int i = 0; i < m; ++i) {
      const uintptr_t a = ((uintptr_t)todo[i].p + page - 1) / page, b = ((uintptr_t)todo[i].p + todo[i].bytes) / page;
      const uintptr_t lo = a + (b - a) * k / parts, hi = a + (b - a) * (k + 1) / parts;
      if (hi > lo) (void)madvise((void*)(lo * page), (hi - lo) * page, MADV_POPULATE_WRITE);
    }
  };
  int parts = (int)(total / kPerThread);
  parts = parts < 1 ? 1 : (parts > kThreads ? kThreads : parts);
  std::thread t[kThreads];
  int started = 0;
  try {
    for (; started < parts - 1; ++started) t[started] = std::thread(part, started, parts);
  } catch (const std::exception&) {  // no more threads: this one does the rest
  }
  for (int k = started; k < parts; ++k) part(k, parts);
  for (int i = 0; i < started; ++i) t[i].join();
  return true;
}
inline bool populate_host(void* p, size_t bytes) {
  const HostRange r = {p, bytes};
  return populate_host(&r, 1);
}

}  // namespace lbk
