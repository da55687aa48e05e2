// host_pages.h -- makes the pages of a host buffer that a device copy is about to fill.  Host code only.
//
// On Grace-Blackwell the copy writes ordinary host memory directly; a page that does not exist yet is then a
// fault of the device, and those take about 50 us per 64 KiB page.  The host makes the pages by writing one
// byte in each, always a byte the copy overwrites: for 1.06 GB read back 46 ms.  (MADV_POPULATE_WRITE from
// the same threads, which writes nothing: 52 ms.  Writing the byte's own value back, by a load and a store or
// by an atomic: 160 ms, the page is first mapped for reading and then copied.)

#pragma once

#include <unistd.h>

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <thread>
#include <vector>

namespace gs {

// The pages of `rows` rows of row_bytes, pitch_bytes apart, numbered row by row.
struct RowPages {
  uintptr_t base;
  size_t row_bytes, pitch_bytes, rows, page;
  size_t per_row;  // page numbers per row: no row has more pages

  RowPages(const void* dst, size_t row_bytes_, size_t pitch_bytes_, size_t rows_, size_t page_)
      : base(reinterpret_cast<uintptr_t>(dst)), row_bytes(row_bytes_), pitch_bytes(pitch_bytes_), rows(rows_), page(page_) {
    if (pitch_bytes == row_bytes) {  // one row from the first to the last
      row_bytes *= rows;
      rows = 1;
    }
    per_row = (row_bytes + page - 1) / page + 1;
  }
  size_t count() const { return rows * per_row; }
  // calls f with an address inside the row and the page, for the existing ones among page numbers [first, last)
  template <class F>
  void each(size_t first, size_t last, F f) const {
    while (first < last) {
      const size_t r = first / per_row, end = std::min(last, (r + 1) * per_row);
      const uintptr_t row = base + r * pitch_bytes, row_end = row + row_bytes;
      uintptr_t at = row / page * page + (first - r * per_row) * page;
      for (; first < end && at < row_end; ++first, at += page) f(std::max(at, row));
      first = end;
    }
  }
};

// 354 MB of fresh memory: the copy alone 284 ms, into pages that exist 1.9 ms; one thread makes them in 11 ms,
// eight in 3.  Pages that exist already cost nothing to speak of.
inline void make_pages(void* dst, size_t row_bytes, size_t pitch_bytes, size_t rows) {
  const RowPages P(dst, row_bytes, pitch_bytes, rows, (size_t)std::max(4096l, sysconf(_SC_PAGESIZE)));
  const size_t total = P.count();
  const auto make = [&P](size_t first, size_t last) {
    P.each(first, last, [](uintptr_t a) { *reinterpret_cast<volatile char*>(a) = 0; });
  };
  // a thread costs about as much as 50 pages
  const size_t n = std::min<size_t>({8, std::max<size_t>(1, std::thread::hardware_concurrency()), total / 200 + 1});
  std::vector<std::thread> threads;
  size_t done = 0;
  try {
    threads.reserve(n);
    for (size_t k = 1; k < n; ++k) {
      threads.emplace_back(make, done, total * k / n);
      done = total * k / n;
    }
  } catch (...) {  // no thread or no memory for one: this thread does the rest
  }
  make(done, total);
  for (std::thread& t : threads) t.join();
}

}  // namespace gs
