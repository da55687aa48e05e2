"""Making the pages of a read-back's destination: every page of a row exists afterwards and none between rows a page
and more apart, only bytes of rows are written, and the work of a single row is divided among the threads too.  Host code: a C++ program with the
library's header."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include <map>
#include <sys/mman.h>
#include "host_pages.h"
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)

// rows of row_bytes, pitch apart, at `off` into fresh memory of which some bytes are in use
static int rows(size_t row_bytes, size_t pitch, size_t n, size_t off) {
  const size_t page = (size_t)sysconf(_SC_PAGESIZE);
  const size_t pages = (off + pitch * n + row_bytes) / page + 2, bytes = pages * page;
  unsigned char* m = (unsigned char*)mmap(nullptr, bytes, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
  CHECK(m != MAP_FAILED);
  madvise(m, bytes, MADV_NOHUGEPAGE);
  std::map<size_t, unsigned char> used;
  for (size_t r = 0; r < n; r += 3) {  // first and last bytes of some rows, and bytes next to them
    for (size_t at : {off + r * pitch, off + r * pitch + row_bytes - 1, off + r * pitch + row_bytes}) used[at] = (unsigned char)(r + 1);
    if (off) used[off - 1] = 200;
  }
  for (auto& u : used) m[u.first] = u.second;
  std::vector<unsigned char> before(pages), after(pages);
  mincore(m, bytes, before.data());
  gs::make_pages(m + off, row_bytes, pitch, n);
  mincore(m, bytes, after.data());
  for (size_t p = 0; p < pages; ++p) {
    bool in_row = false;
    for (size_t r = 0; r < n && !in_row; ++r) {
      const size_t a = off + r * pitch, b = a + row_bytes;
      in_row = a < (p + 1) * page && p * page < b;
    }
    CHECK((after[p] & 1) == (in_row || (before[p] & 1)));
  }
  for (size_t k = 0; k < bytes; ++k) {  // (a row's bytes are the copy's to write)
    auto u = used.find(k);
    const bool in_row = k >= off && (k - off) % pitch < row_bytes && k < off + (n - 1) * pitch + row_bytes;
    CHECK(m[k] == (u == used.end() ? 0 : u->second) || (in_row && m[k] == 0));
  }
  // shares of 1 to 9 threads: together every page of a row, inside the row, none much larger than the others
  const gs::RowPages P(m + off, row_bytes, pitch, n, page);
  for (size_t t = 1; t < 10; ++t) {
    std::vector<size_t> seen(pages), share(t);
    bool inside = true;
    for (size_t k = 0; k < t; ++k)
      P.each(P.count() * k / t, P.count() * (k + 1) / t, [&](uintptr_t a) {
        const size_t at = a - (uintptr_t)m;
        inside = inside && at >= off && (at - off) % pitch < row_bytes && at < off + (n - 1) * pitch + row_bytes;
        ++seen[at / page], ++share[k];
      });
    CHECK(inside);
    for (size_t p = 0; p < pages; ++p) CHECK(seen[p] > 0 || !(after[p] & 1) || (before[p] & 1));
    for (size_t k = 0; k < t; ++k) CHECK(share[k] <= P.count() / t + 1);
  }
  munmap(m, bytes);
  return 0;
}

int main() {
  const size_t page = (size_t)sysconf(_SC_PAGESIZE);
  // single rows, rows next to each other, with small gaps, with gaps of whole pages; off a page's start
  if (rows(1, 1, 1, 0) || rows(page, page, 1, 0) || rows(page + 1, page + 1, 1, page - 1) || rows(2000 * page + 12, 2000 * page + 12, 1, 4)) return 1;
  if (rows(40, 40, 59, 0) || rows(3 * page + 4, 3 * page + 4, 59, 12) || rows(70 * page, 70 * page, 59, 0)) return 1;
  if (rows(4000, 4100, 59, 8) || rows(page, 2 * page - 4, 59, 0) || rows(page, 2 * page, 59, 0) || rows(4, 5 * page, 59, page - 4)) return 1;
  if (rows(2 * page + 8, 7 * page + 40, 59, 16)) return 1;
  std::printf("ok\n");
  return 0;
}
"""


def test_make_pages(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "pages.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "pages"
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", os.path.join(ROOT, "paper_2503_13086_gb300", "csrc"),
                        str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout == "ok\n", (r.returncode, r.stdout, r.stderr)
