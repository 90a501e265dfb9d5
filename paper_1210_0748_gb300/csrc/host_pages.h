// Pages of the caller's host arrays, mapped before a copy fills them.
#pragma once

#include <stddef.h>
#include <stdint.h>
#include <sys/mman.h>
#include <unistd.h>

#include <initializer_list>

namespace kb {

// Have the kernel map the pages of a large host destination in one call, while
// the device still prepares the copy.  An array just taken from malloc's heap
// (the usual destination of up to 32 MB) may have none, and the copy would
// fault them in one by one: read into arrays that stay, 12.8 MB take 365 us
// with the pages mapped first and 428 without (then with outliers of 7 ms),
// 25.6 MB 950 and 1,061.  Not done where it measured slower: pages that are
// there (12.8 MB 81 us, 87 with a call for nothing), by two of them; memory
// above the program break, which the process maps by itself and whose faults
// the copy overlaps (12.8 MB 659 against 700 us, 64 MB 2,902 against 3,470);
// and arrays of a few MB, which malloc seldom gives back.  Contents stay; where
// the call is not known it fails and the copy does as before.
inline void map_host_pages(void* dst, size_t bytes) {
#ifndef MADV_POPULATE_WRITE
#define MADV_POPULATE_WRITE 23
#endif
  if (bytes < (8u << 20)) return;
  const uintptr_t page = (uintptr_t)sysconf(_SC_PAGESIZE), a = reinterpret_cast<uintptr_t>(dst);
  const uintptr_t lo = (a + page - 1) / page * page, hi = (a + bytes) / page * page;
  if (hi <= lo || hi > reinterpret_cast<uintptr_t>(sbrk(0))) return;
  bool there = true;
  for (uintptr_t p : {lo + (hi - lo) / 2 / page * page, hi - page}) {
    unsigned char in_core = 0;
    there = there && mincore(reinterpret_cast<void*>(p), page, &in_core) == 0 && (in_core & 1);
  }
  if (!there) madvise(reinterpret_cast<void*>(lo), hi - lo, MADV_POPULATE_WRITE);
}

}  // namespace kb
