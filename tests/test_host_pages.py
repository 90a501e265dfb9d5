"""When the pages of a host destination are mapped before the copy (csrc/host_pages.h), compiled for the CPU: the
program counts the calls of madvise."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1210_0748_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <malloc.h>
#include <sys/syscall.h>
#include "host_pages.h"

static int calls = 0;
extern "C" int madvise(void* a, size_t n, int what) noexcept {
  ++calls;
  return (int)syscall(SYS_madvise, a, n, what);
}

int main() {
  mallopt(M_MMAP_THRESHOLD, 1 << 30);  // arrays of this size from the heap
  mallopt(M_TRIM_THRESHOLD, 1 << 30);
  const size_t n = 12u << 20;
  char* heap = static_cast<char*>(malloc(n));
  kb::map_host_pages(heap, n);
  printf("fresh heap %d\n", calls);
  memset(heap, 5, n);
  calls = 0;
  kb::map_host_pages(heap, n);
  printf("written heap %d\n", calls);
  bool kept = true;
  for (size_t i = 0; i < n; ++i) kept = kept && heap[i] == 5;
  char* half = static_cast<char*>(malloc(n));
  memset(half, 5, n / 4);
  calls = 0;
  kb::map_host_pages(half + 3, n - 5);
  printf("partly written heap %d\n", calls);
  for (size_t i = 0; i < n / 4; ++i) kept = kept && half[i] == 5;
  void* own = mmap(nullptr, n, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
  calls = 0;
  kb::map_host_pages(own, n);
  printf("own mapping %d\n", calls);
  char* small = static_cast<char*>(malloc(7u << 20));
  calls = 0;
  kb::map_host_pages(small, 7u << 20);
  kb::map_host_pages(nullptr, 0);
  printf("small %d\n", calls);
  printf("contents %d\n", kept ? 0 : 1);
}
"""


@pytest.fixture(scope="module")
def calls(tmp_path_factory):
    d = tmp_path_factory.mktemp("pages")
    (d / "t.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I" + CSRC, str(d / "t.cpp"), "-o", str(d / "t")], check=True)
    out = subprocess.run([str(d / "t")], check=True, capture_output=True, text=True).stdout
    return {line.rsplit(" ", 1)[0]: int(line.rsplit(" ", 1)[1]) for line in out.splitlines()}


@pytest.mark.parametrize("where,expected", [("fresh heap", 1), ("partly written heap", 1), ("written heap", 0),
                                            ("own mapping", 0), ("small", 0), ("contents", 0)])
def test_pages_are_mapped_only_where_it_saves_time(calls, where, expected):
    assert calls[where] == expected
