// k_sort.cu -- K2 (exclusive scan of tiles touched), K3 (duplication into (tile, depth) keys),
// K4 (stable LSD radix sort, one onesweep pass per 8-bit digit) and K5 (per-tile ranges), sm_103a.
//
// These implement the tile-binning of the 3DGS rasterizer the paper builds on (Sec. III; the
// "original 3DGS" settings of Sec. V-A).  Canonical order: (global tile, fp32 depth bits,
// record index).  Instances are emitted in record order and every sort pass is stable, so the
// record index breaks depth ties.  The key holds only the depth bits that vary within the step
// (their range comes out of the scan), so a step usually needs 5 passes of 8 bits instead of 6; the
// number of passes is decided on the device and the passes always end in buffer 0.  Every count lives in
// device memory: no kernel here needs the host to know how many instances were emitted, so the whole chain
// can be graph-captured.  The inter-CTA waits (decoupled look-back) spin at most kSpinLimit times, then flag
// kErrTimeout; the kernel finishes with what it has and the kernels after it return at once.
#include <atomic>

#include "gs_device.cuh"
#include "gs_engine.h"

namespace gs {

namespace {
constexpr unsigned long long kScanAgg = 1ull << 62;
constexpr unsigned long long kScanPrefix = 2ull << 62;
constexpr unsigned long long kScanValMask = (1ull << 62) - 1;
constexpr unsigned kSortAgg = 1u << 30;
constexpr unsigned kSortPrefix = 2u << 30;
constexpr unsigned kSortValMask = (1u << 30) - 1;

__device__ __forceinline__ unsigned lanemask_lt() {
  unsigned m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}
}  // namespace

// ---------------------------------------------------------------------------------------------
// K2: single-pass exclusive scan with decoupled look-back.  Tiles are taken in launch order via
// an atomic ticket, so every tile a CTA waits on belongs to a CTA that is already running.
// ---------------------------------------------------------------------------------------------
// SCAN_COMPACT also lists the records with instances, (depth bits << 32 | record) in record order, for the
// depth presort of large steps: a second warp runs the same look-back for the number of listed records.
// SCAN_LIST scans the counts of the listed records in list order (n_items = the list's length, device-
// resident) and writes each record's offset to out[record].
enum ScanMode { SCAN_PLAIN, SCAN_COMPACT, SCAN_LIST };

// Decoupled look-back by a whole warp: lane l reads the status of tile j - l, so one round trip covers up
// to 32 predecessors.  Publishes the tile's total, returns the sum before it.
__device__ __forceinline__ unsigned long long scan_lookback(unsigned long long* __restrict__ state, unsigned tile,
                                                            unsigned long long total, int lane,
                                                            Control* __restrict__ ctl, unsigned spin_limit) {
  unsigned long long excl = 0;
  if (tile == 0) {
    if (lane == 0) st_relaxed_u64(&state[0], kScanPrefix | total);
    return 0ull;
  }
  if (lane == 0) st_relaxed_u64(&state[tile], kScanAgg | total);
  long long j = (long long)tile - 1;
  unsigned spins = 0;
  for (;;) {
    const long long idx = j - lane;
    const unsigned long long sv = idx >= 0 ? ld_relaxed_u64(&state[idx]) : kScanPrefix;
    const unsigned long long flag = sv & ~kScanValMask;
    const unsigned notready = __ballot_sync(0xffffffffu, flag == 0ull);
    const unsigned isprefix = __ballot_sync(0xffffffffu, flag == kScanPrefix);
    const unsigned stop = notready | isprefix;
    const int first = stop ? __ffs(stop) - 1 : 32;  // lanes below it hold aggregates
    const bool take = lane < first || (lane == first && ((isprefix >> lane) & 1u));
    unsigned long long v = take ? (sv & kScanValMask) : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    excl += v;
    if (first < 32 && ((isprefix >> first) & 1u)) break;
    j -= first;
    if (first < 32 && ++spins > spin_limit) {
      if (lane == 0) atomicOr(&ctl->error, kErrTimeout);
      break;
    }
  }
  if (lane == 0) st_relaxed_u64(&state[tile], kScanPrefix | (excl + total));
  return excl;
}

// The large steps' scan of all records takes tiles of 8192: the look-back advances 32 tiles per round trip, so
// with 2048 the chain over 4.5M records set the time (49 against 40 us).  The scan of the listed ones keeps
// 2048: its gather wants the CTAs (10 us slower with 8192 at 0.9M).
constexpr int kLargeScanThreads = 512, kLargeScanItems = 16;
constexpr int kLargeScanTile = kLargeScanThreads * kLargeScanItems;

template <int MODE>
__global__ void __launch_bounds__(MODE == SCAN_COMPACT ? kLargeScanThreads : kScanThreads) k_scan(
                                                       const unsigned* __restrict__ in, unsigned* __restrict__ out,
                                                       long long n_items, unsigned long long* __restrict__ state,
                                                       Control* __restrict__ ctl, unsigned long long m_cap,
                                                       Ledger* __restrict__ ledger, const float* __restrict__ depth,
                                                       unsigned spin_limit, unsigned long long* __restrict__ list,
                                                       unsigned long long* __restrict__ list_state) {
  constexpr int kThr = MODE == SCAN_COMPACT ? kLargeScanThreads : kScanThreads;
  constexpr int kItems = MODE == SCAN_COMPACT ? kLargeScanItems : kScanItems;
  constexpr int kTileItems = kThr * kItems;
  dep_wait();
  dep_release();
  __shared__ unsigned s_tile;
  __shared__ unsigned s_warp[kThr / 32], s_lwarp[kThr / 32];
  __shared__ unsigned long long s_excl;
  __shared__ unsigned s_lexcl;
  if (MODE == SCAN_LIST) n_items = (long long)ctl->listed;
  if (threadIdx.x == 0)
    s_tile = MODE == SCAN_LIST ? (step_void(ctl) ? ~0u : atomicAdd(&ctl->list_ticket, 1u)) : atomicAdd(&ctl->scan_ticket, 1u);
  __syncthreads();
  const unsigned tile = s_tile;
  const long long num_tiles = (n_items + kTileItems - 1) / kTileItems;
  if (MODE == SCAN_LIST && (long long)tile >= num_tiles) return;
  const long long base = (long long)tile * kTileItems + (long long)threadIdx.x * kItems;
  unsigned x[kItems], rec[kItems];
  if (MODE == SCAN_LIST) {
#pragma unroll
    for (int k = 0; k < kItems; ++k) rec[k] = base + k < n_items ? (unsigned)list[base + k] : 0u;
#pragma unroll
    for (int k = 0; k < kItems; ++k) x[k] = base + k < n_items ? in[rec[k]] : 0u;
  } else if (base + kItems <= n_items) {
#pragma unroll
    for (int k = 0; k < kItems; k += 4) {
      const uint4 a = *reinterpret_cast<const uint4*>(in + base + k);
      x[k] = a.x;
      x[k + 1] = a.y;
      x[k + 2] = a.z;
      x[k + 3] = a.w;
    }
  } else {
#pragma unroll
    for (int k = 0; k < kItems; ++k) x[k] = (base + k < n_items) ? in[base + k] : 0u;
  }
  unsigned tsum = 0, tlist = 0;
#pragma unroll
  for (int k = 0; k < kItems; ++k) {
    tsum += x[k];
    tlist += x[k] != 0u;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned db[kItems];
  if (MODE != SCAN_LIST && depth) {  // range of the depth bits of the records with instances (the sort key layout)
    unsigned dmax = 0u, dnot = 0u;
#pragma unroll
    for (int k = 0; k < kItems; ++k)
      if (x[k]) {
        const unsigned b = __float_as_uint(depth[base + k]);
        if (MODE == SCAN_COMPACT) db[k] = b;
        dmax = max(dmax, b);
        dnot = max(dnot, ~b);
      }
    dmax = __reduce_max_sync(0xffffffffu, dmax);
    dnot = __reduce_max_sync(0xffffffffu, dnot);
    if (lane == 0 && (dmax | dnot)) {
      atomicMax(&ctl->dmax, dmax);
      atomicMax(&ctl->dnot, dnot);
    }
  }
  // block-wide exclusive scan of the per-thread sums
  unsigned incl = tsum, lincl = tlist;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, incl, d);
    const unsigned z = MODE == SCAN_COMPACT ? __shfl_up_sync(0xffffffffu, lincl, d) : 0u;
    if (lane >= d) {
      incl += y;
      lincl += z;
    }
  }
  if (lane == 31) {
    s_warp[warp] = incl;
    if (MODE == SCAN_COMPACT) s_lwarp[warp] = lincl;
  }
  __syncthreads();
  if (warp == 0 || (MODE == SCAN_COMPACT && warp == 1)) {
    unsigned* sums = warp == 0 ? s_warp : s_lwarp;
    const unsigned w = lane < kThr / 32 ? sums[lane] : 0u;
    unsigned wi = w;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, wi, d);
      if (lane >= d) wi += y;
    }
    if (lane < kThr / 32) sums[lane] = wi - w;  // exclusive warp offsets
    const unsigned total = __shfl_sync(0xffffffffu, wi, kThr / 32 - 1);
    const unsigned long long excl = scan_lookback(warp == 0 ? state : list_state, tile, total, lane, ctl, spin_limit);
    if (lane == 0 && warp == 0) {
      s_excl = excl;
      if (MODE != SCAN_LIST && (long long)tile == num_tiles - 1) {
        const unsigned long long m = excl + total;
        ctl->m_total = m;
        // an overflow skips this step; an earlier skipped or timed-out step of the run skips it too
        if (m > m_cap || (ledger && (ledger->skip || ledger->error))) {
          ctl->overflow = 1u;
          atomicOr(&ctl->error, kErrOverflow);
          if (ledger) {
            ledger->skip = 1u;
            if (m > ledger->m_need) ledger->m_need = m;
          }
        }
      }
    }
    if (MODE == SCAN_COMPACT && lane == 0 && warp == 1) {
      s_lexcl = (unsigned)excl;
      if ((long long)tile == num_tiles - 1) ctl->listed = (unsigned)excl + total;
    }
  }
  __syncthreads();
  unsigned run = (unsigned)s_excl + s_warp[warp] + (incl - tsum);
  if (MODE == SCAN_COMPACT) {
    unsigned pos = s_lexcl + s_lwarp[warp] + (lincl - tlist);
#pragma unroll
    for (int k = 0; k < kItems; ++k)
      if (x[k]) list[pos++] = ((unsigned long long)db[k] << 32) | (unsigned)(base + k);
  }
  if (MODE == SCAN_LIST) {
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
      if (base + k < n_items) out[rec[k]] = run;
      run += x[k];
    }
  } else if (base + kItems <= n_items) {
#pragma unroll
    for (int k = 0; k < kItems; k += 4) {
      uint4 y;
      y.x = run;
      y.y = y.x + x[k];
      y.z = y.y + x[k + 1];
      y.w = y.z + x[k + 2];
      run = y.w + x[k + 3];
      *reinterpret_cast<uint4*>(out + base + k) = y;
    }
  } else {
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
      if (base + k < n_items) out[base + k] = run;
      run += x[k];
    }
  }
}

void launch_scan(const unsigned* in, unsigned* out, long long n_items, unsigned long long* state, Control* ctl,
                 unsigned long long m_cap, Ledger* ledger, cudaStream_t s, const float* depth,
                 unsigned long long* list, unsigned long long* list_state) {
  const int tile = list ? kLargeScanTile : kScanTile;
  launch_dep(list ? k_scan<SCAN_COMPACT> : k_scan<SCAN_PLAIN>, dim3((unsigned)((n_items + tile - 1) / tile)),
      dim3(list ? kLargeScanThreads : kScanThreads), 0, s, in, out, n_items, state, ctl, m_cap, ledger, depth, kSpinLimit,
      list, list_state);
}

// ---------------------------------------------------------------------------------------------
// K3: duplication into (tile, depth) keys, one thread per instance.  First every record writes
// its index over its instances' slots of inst_rec (a record with more than kFillAlone instances is
// written by its whole warp, so one large Gaussian does not serialise a warp); then each instance reads
// its owner from there (one coalesced load) and writes its key.  Also histograms every radix digit
// for the sort (the passes whose digit lies in the depth part of the key once per record, through
// the thread of its first instance).
// ---------------------------------------------------------------------------------------------
constexpr unsigned kFillAlone = 4;  // larger records are written by their whole warp
__global__ void __launch_bounds__(256) k_fill_owner(const unsigned* __restrict__ count,
                                                    const unsigned* __restrict__ offsets, long long n_items,
                                                    unsigned* __restrict__ inst_rec, const Control* __restrict__ ctl) {
  dep_wait();
  dep_release();
  if (step_void(ctl)) return;
  const int lane = threadIdx.x & 31;
  const long long rec = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned cnt = rec < n_items ? count[rec] : 0u;
  const unsigned off = cnt ? offsets[rec] : 0u;
  if (cnt <= kFillAlone) {
    for (unsigned k = 0; k < cnt; ++k) inst_rec[(unsigned long long)off + k] = (unsigned)rec;
  }
  unsigned big = __ballot_sync(0xffffffffu, cnt > kFillAlone);
  while (big) {
    const int l = __ffs(big) - 1;
    big &= big - 1u;
    const unsigned r = __shfl_sync(0xffffffffu, (unsigned)rec, l);
    const unsigned o = __shfl_sync(0xffffffffu, off, l);
    const unsigned c = __shfl_sync(0xffffffffu, cnt, l);
    for (unsigned k = lane; k < c; k += 32u) inst_rec[(unsigned long long)o + k] = r;
  }
}

__global__ void __launch_bounds__(1024) k_emit(const ProjBuffers pb, const ViewDev* __restrict__ views, int stride,
                                              unsigned long long* __restrict__ keys0, unsigned* __restrict__ vals0,
                                              unsigned long long* __restrict__ keys1, unsigned* __restrict__ vals1,
                                              const unsigned* __restrict__ inst_rec, unsigned* __restrict__ hist,
                                              int tile_bits, const Control* __restrict__ ctl) {
  dep_wait();
  dep_release();
  __shared__ unsigned s_hist[kMaxSortPasses][kSortBins];
  for (int k = threadIdx.x; k < kMaxSortPasses * kSortBins; k += blockDim.x) (&s_hist[0][0])[k] = 0u;
  __syncthreads();
  // the passes end in buffer 0: start in buffer (passes & 1)
  const KeyLayout kl = key_layout(ctl, tile_bits);
  const int passes = kl.passes;
  const int depth_passes = min(passes, kl.D / kSortBits);
  unsigned long long* __restrict__ keys = (passes & 1) ? keys1 : keys0;
  unsigned* __restrict__ vals = (passes & 1) ? vals1 : vals0;
  if (!step_void(ctl)) {
    const unsigned long long M = ctl->m_total;
    for (unsigned long long e = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; e < M;
         e += (unsigned long long)gridDim.x * blockDim.x) {
      const unsigned rec = inst_rec[e];
      const unsigned k = (unsigned)(e - pb.offsets[rec]);
      const uint2 rc = pb.rect[rec];
      const unsigned db = __float_as_uint(pb.depth[rec]);
      const ViewDev& V = views[rec / (unsigned)stride];
      const unsigned x0 = rc.x & 0xffffu, x1 = rc.x >> 16, y0 = rc.y & 0xffffu;
      const unsigned w = x1 - x0;
      const unsigned ty = y0 + k / w, tx = x0 + k % w;
      const unsigned long long tile = (unsigned long long)(V.tile_base + (long long)ty * V.gx + tx);
      const unsigned long long key = (tile << kl.D) | (unsigned long long)(db - kl.dmin);
      keys[e] = key;
      vals[e] = rec;
      for (int p = depth_passes; p < passes; ++p)
        atomicAdd(&s_hist[p][(key >> (p * kSortBits)) & (kSortBins - 1)], 1u);
      if (k == 0) {  // every instance of the record has the record's depth digits
        const unsigned cnt = pb.count[rec];
        for (int p = 0; p < depth_passes; ++p)
          atomicAdd(&s_hist[p][((db - kl.dmin) >> (p * kSortBits)) & (kSortBins - 1)], cnt);
      }
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < passes * kSortBins; k += blockDim.x) {
    const unsigned c = (&s_hist[0][0])[k];
    if (c) atomicAdd(hist + k, c);
  }
}

void launch_emit(const ProjBuffers& pb, const ViewDev* views, int stride, long long n_items, unsigned long long* keys0,
                 unsigned* vals0, unsigned long long* keys1, unsigned* vals1, unsigned* inst_rec, unsigned* hist,
                 int tile_bits, long long m_cap, int num_sms, const Control* ctl, cudaStream_t s) {
  if (n_items <= 0) return;
  launch_dep(k_fill_owner, dim3((unsigned)((n_items + 255) / 256)), dim3(256), 0, s, pb.count, pb.offsets, n_items,
      inst_rec, ctl);
  // The same threads per SM either way.  Each CTA adds its shared histograms (up to 8 x 256 bins)
  // into the global ones with one atomic per non-empty bin: with few instances those flushes
  // dominate, so fewer, larger CTAs (0.42M instances: 22.6 -> 14.8 us); with many, the CTA's
  // threads contend on its shared bins instead, so more, smaller CTAs (7M instances: 0.129 ms
  // with 1024-thread CTAs, 0.108 ms with 512).
  const bool small = m_cap <= (1ll << 22);
  launch_dep(k_emit, dim3((unsigned)(num_sms * (small ? 2 : 4))), dim3(small ? 1024 : 512), 0, s, pb, views, stride,
      keys0, vals0, keys1, vals1, inst_rec, hist, tile_bits, ctl);
}

// ---------------------------------------------------------------------------------------------
// K4: one stable counting pass over an 8-bit digit (onesweep: digit offsets from the upfront
// histogram, per-CTA offsets by decoupled look-back per digit).  Within a CTA the keys are
// ranked warp by warp so that the pass is stable, staged in shared memory in digit order, and written
// out as contiguous runs.  The lanes of a warp that hold the same digit find one another through a
// mask per (warp, digit) in shared memory, set by atomicOr and cleared by the first of them: a pass over
// random digits took 35 us with match.any and 24 with one digit alone; with the masks the passes are 11 %
// shorter.
// ---------------------------------------------------------------------------------------------
struct SortSmem {
  unsigned long long keys[kSortTile];
  unsigned vals[kSortTile];
  unsigned cnt[kSortThreads / 32][kSortBins];
  unsigned mask[kSortThreads / 32][kSortBins];
  unsigned bstart[kSortBins];
  unsigned gbase[kSortBins];
  unsigned tile;
};

// Decoupled look-back of one digit: publishes the tile's total and returns the sum over the tiles before.
__device__ __forceinline__ unsigned sort_lookback(unsigned* __restrict__ state, unsigned tile, int d, unsigned total,
                                                  Control* __restrict__ ctl, unsigned spin_limit) {
  unsigned excl = 0u;
  unsigned* st = state + (unsigned long long)tile * kSortBins + d;
  if (tile == 0) {
    st_relaxed_u32(st, kSortPrefix | total);
  } else {
    st_relaxed_u32(st, kSortAgg | total);
    // look-back over windows of kLookBack predecessors (their loads in flight together)
    constexpr int kLookBack = 8;
    long long j = (long long)tile - 1;
    unsigned spins = 0;
    bool done = false;
    while (!done) {
      unsigned sv[kLookBack];
#pragma unroll
      for (int w = 0; w < kLookBack; ++w)
        sv[w] = j - w >= 0 ? ld_relaxed_u32(state + (unsigned long long)(j - w) * kSortBins + d) : kSortPrefix;
      int used = 0;
      bool wait = false;
#pragma unroll
      for (int w = 0; w < kLookBack; ++w) {
        if (done || wait) continue;
        const unsigned flag = sv[w] & ~kSortValMask;
        if (flag == 0u) {
          wait = true;
          continue;
        }
        excl += sv[w] & kSortValMask;
        ++used;
        if (flag == kSortPrefix) done = true;
      }
      j -= used;
      if (wait && ++spins > spin_limit) {
        atomicOr(&ctl->error, kErrTimeout);
        break;
      }
    }
    st_relaxed_u32(st, kSortPrefix | (excl + total));
  }
  return excl;
}

__global__ void __launch_bounds__(kSortThreads, kSortMinBlocks) k_sort_pass(unsigned long long* __restrict__ keys0,
                                                            unsigned* __restrict__ vals0,
                                                            unsigned long long* __restrict__ keys1,
                                                            unsigned* __restrict__ vals1,
                                                            const unsigned* __restrict__ hist,
                                                            unsigned* __restrict__ state, int pass, int tile_bits,
                                                            Control* __restrict__ ctl, unsigned spin_limit) {
  dep_wait();
  dep_release();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SortSmem& S = *reinterpret_cast<SortSmem*>(smem_raw);
  if (ctl->overflow) return;
  // passes beyond the step's key bits do nothing; pass j reads buffer (passes - j) & 1
  const int passes = key_layout(ctl, tile_bits).passes;
  if (pass >= passes) return;
  const bool from1 = ((passes - pass) & 1) != 0;
  const unsigned long long* __restrict__ kin = from1 ? keys1 : keys0;
  const unsigned* __restrict__ vin = from1 ? vals1 : vals0;
  unsigned long long* __restrict__ kout = from1 ? keys0 : keys1;
  unsigned* __restrict__ vout = from1 ? vals0 : vals1;
  const unsigned long long M = ctl->m_total;
  if (threadIdx.x == 0) S.tile = step_void(ctl) ? ~0u : atomicAdd(&ctl->sort_ticket[pass], 1u);
  for (int k = threadIdx.x; k < (kSortThreads / 32) * kSortBins; k += kSortThreads) {
    (&S.cnt[0][0])[k] = 0u;
    (&S.mask[0][0])[k] = 0u;
  }
  __syncthreads();
  const unsigned tile = S.tile;
  const unsigned long long tile0 = (unsigned long long)tile * kSortTile;
  if (tile0 >= M) return;
  const int shift = pass * kSortBits;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = lanemask_lt();

  unsigned long long key[kSortItems];
  unsigned val[kSortItems];
  unsigned rank[kSortItems];
  const unsigned long long wbase = tile0 + (unsigned long long)warp * (kSortItems * 32);
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const unsigned long long idx = wbase + (unsigned)(r * 32 + lane);
    const bool valid = idx < M;
    key[r] = valid ? kin[idx] : ~0ull;
    val[r] = valid ? vin[idx] : 0u;
  }
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const unsigned long long idx = wbase + (unsigned)(r * 32 + lane);
    const bool valid = idx < M;
    const unsigned d = (unsigned)(key[r] >> shift) & (kSortBins - 1);
    if (valid) atomicOr(&S.mask[warp][d], 1u << lane);
    __syncwarp();
    const unsigned peers = valid ? S.mask[warp][d] : 0u;
    const unsigned pre = valid ? S.cnt[warp][d] : 0u;
    __syncwarp();
    if (valid && (peers & lt) == 0u) {
      S.cnt[warp][d] = pre + __popc(peers);
      S.mask[warp][d] = 0u;
    }
    __syncwarp();
    rank[r] = pre + __popc(peers & lt);
  }
  __syncthreads();
  // Per digit (thread d < 256; whole warps): warp-exclusive prefix in place, CTA total, decoupled
  // look-back across CTAs, then the digit bases by a block-wide scan over the 256 digits.
  static_assert(kSortThreads % kSortBins == 0, "the digit threads are whole warps");
  __shared__ unsigned s_wa[kSortBins / 32], s_wb[kSortBins / 32];
  const int d = threadIdx.x;
  const bool digit = d < kSortBins;
  unsigned total = 0u, excl = 0u, h = 0u, a = 0u, b = 0u;
  if (digit) {
    unsigned run = 0;
#pragma unroll
    for (int w = 0; w < kSortThreads / 32; ++w) {
      const unsigned c = S.cnt[w][d];
      S.cnt[w][d] = run;
      run += c;
    }
    total = run;
    excl = sort_lookback(state, tile, d, total, ctl, spin_limit);
    // digit base = exclusive scan of the global histogram; CTA digit start = exclusive scan of
    // the CTA totals
    h = hist[pass * kSortBins + d];
    a = h;
    b = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned ya = __shfl_up_sync(0xffffffffu, a, o);
      const unsigned yb = __shfl_up_sync(0xffffffffu, b, o);
      if (lane >= o) {
        a += ya;
        b += yb;
      }
    }
    if (lane == 31) {
      s_wa[warp] = a;
      s_wb[warp] = b;
    }
  }
  __syncthreads();
  if (digit) {
    unsigned pa = 0, pb = 0;
    for (int w = 0; w < warp; ++w) {
      pa += s_wa[w];
      pb += s_wb[w];
    }
    S.gbase[d] = pa + a - h + excl;
    S.bstart[d] = pb + b - total;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const unsigned long long idx = wbase + (unsigned)(r * 32 + lane);
    if (idx < M) {
      const unsigned d = (unsigned)(key[r] >> shift) & (kSortBins - 1);
      const unsigned pos = S.bstart[d] + S.cnt[warp][d] + rank[r];
      S.keys[pos] = key[r];
      S.vals[pos] = val[r];
    }
  }
  __syncthreads();
  const unsigned tile_count = (unsigned)min((unsigned long long)kSortTile, M - tile0);
  for (unsigned k = threadIdx.x; k < tile_count; k += kSortThreads) {
    const unsigned long long kk = S.keys[k];
    const unsigned d = (unsigned)(kk >> shift) & (kSortBins - 1);
    const unsigned gpos = S.gbase[d] + (k - S.bstart[d]);
    kout[gpos] = kk;
    vout[gpos] = S.vals[k];
  }
}


void launch_sort_pass(unsigned long long* keys0, unsigned* vals0, unsigned long long* keys1, unsigned* vals1,
                      const unsigned* hist, unsigned* state, int pass, int tile_bits, long long m_cap, Control* ctl,
                      cudaStream_t s) {
  const long long tiles = (m_cap + kSortTile - 1) / kSortTile;
  launch_dep(k_sort_pass, dim3((unsigned)(tiles > 0 ? tiles : 1)), dim3(kSortThreads), sizeof(SortSmem), s, keys0,
      vals0, keys1, vals1, hist, state, pass, tile_bits, ctl, kSpinLimit);
}

// ---------------------------------------------------------------------------------------------
// Large steps: depth first, then tiles.  The order of an instance within its tile depends on its record
// alone (depth, then index), and there are two to four instances per listed record.  So the listed
// records are sorted by depth (four 8-bit passes over 8-byte words), their counts scanned in that order,
// the instances emitted to the places that scan gives them, and only the tile digits (one to three
// passes) then run over the instances, on 8-byte words (tile << 32 | record) instead of a 12-byte key and
// value through five or six passes.  The list is the same: both sorts are stable and the records start
// in index order.  The word's own slots, which K9a reads, stay in record order.
// ---------------------------------------------------------------------------------------------
struct WordSmem {
  unsigned long long keys[kSortTile];
  unsigned cnt[kSortThreads / 32][kSortBins];
  unsigned mask[kSortThreads / 32][kSortBins];
  unsigned bstart[kSortBins];
  unsigned gbase[kSortBins];
  unsigned tile;
};

// One stable pass over the digit at `shift` of n 8-byte words; as k_sort_pass, without values.  vout
// (nullable): also the words' low halves.
__global__ void __launch_bounds__(kSortThreads, kWordMinBlocks) k_sort_pass_words(
    const unsigned long long* __restrict__ kin, unsigned long long* __restrict__ kout, unsigned* __restrict__ vout,
    int by_record, const unsigned* __restrict__ hist, unsigned* __restrict__ state, int shift, int ticket,
    Control* __restrict__ ctl, unsigned spin_limit) {
  dep_wait();
  dep_release();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  WordSmem& S = *reinterpret_cast<WordSmem*>(smem_raw);
  if (ctl->overflow) return;
  const unsigned long long M = by_record ? (unsigned long long)ctl->listed : ctl->m_total;
  if (threadIdx.x == 0) S.tile = step_void(ctl) ? ~0u : atomicAdd(&ctl->sort_ticket[ticket], 1u);
  for (int k = threadIdx.x; k < (kSortThreads / 32) * kSortBins; k += kSortThreads) {
    (&S.cnt[0][0])[k] = 0u;
    (&S.mask[0][0])[k] = 0u;
  }
  __syncthreads();
  const unsigned tile = S.tile;
  const unsigned long long tile0 = (unsigned long long)tile * kSortTile;
  if (tile0 >= M) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = lanemask_lt();
  unsigned long long key[kSortItems];
  unsigned rank[kSortItems];
  const unsigned long long wbase = tile0 + (unsigned long long)warp * (kSortItems * 32);
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const unsigned long long idx = wbase + (unsigned)(r * 32 + lane);
    key[r] = idx < M ? kin[idx] : ~0ull;
  }
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const bool valid = wbase + (unsigned)(r * 32 + lane) < M;
    const unsigned d = (unsigned)(key[r] >> shift) & (kSortBins - 1);
    if (valid) atomicOr(&S.mask[warp][d], 1u << lane);
    __syncwarp();
    const unsigned peers = valid ? S.mask[warp][d] : 0u;
    const unsigned pre = valid ? S.cnt[warp][d] : 0u;
    __syncwarp();
    if (valid && (peers & lt) == 0u) {
      S.cnt[warp][d] = pre + __popc(peers);
      S.mask[warp][d] = 0u;
    }
    __syncwarp();
    rank[r] = pre + __popc(peers & lt);
  }
  __syncthreads();
  __shared__ unsigned s_wa[kSortBins / 32], s_wb[kSortBins / 32];
  const int d = threadIdx.x;
  const bool digit = d < kSortBins;
  unsigned total = 0u, excl = 0u, h = 0u, a = 0u, b = 0u;
  if (digit) {
    unsigned run = 0;
#pragma unroll
    for (int w = 0; w < kSortThreads / 32; ++w) {
      const unsigned c = S.cnt[w][d];
      S.cnt[w][d] = run;
      run += c;
    }
    total = run;
    h = hist[d];
    excl = sort_lookback(state, tile, d, total, ctl, spin_limit);
    a = h;
    b = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned ya = __shfl_up_sync(0xffffffffu, a, o);
      const unsigned yb = __shfl_up_sync(0xffffffffu, b, o);
      if (lane >= o) {
        a += ya;
        b += yb;
      }
    }
    if (lane == 31) {
      s_wa[warp] = a;
      s_wb[warp] = b;
    }
  }
  __syncthreads();
  if (digit) {
    unsigned pa = 0, pb = 0;
    for (int w = 0; w < warp; ++w) {
      pa += s_wa[w];
      pb += s_wb[w];
    }
    S.gbase[d] = pa + a - h + excl;
    S.bstart[d] = pb + b - total;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    if (wbase + (unsigned)(r * 32 + lane) < M) {
      const unsigned dd = (unsigned)(key[r] >> shift) & (kSortBins - 1);
      S.keys[S.bstart[dd] + S.cnt[warp][dd] + rank[r]] = key[r];
    }
  }
  __syncthreads();
  const unsigned tile_count = (unsigned)min((unsigned long long)kSortTile, M - tile0);
  for (unsigned k = threadIdx.x; k < tile_count; k += kSortThreads) {
    const unsigned long long kk = S.keys[k];
    const unsigned dd = (unsigned)(kk >> shift) & (kSortBins - 1);
    const unsigned gpos = S.gbase[dd] + (k - S.bstart[dd]);
    kout[gpos] = kk;
    if (vout) vout[gpos] = (unsigned)kk;
  }
}

// The four digit histograms of the listed records' depths.
__global__ void __launch_bounds__(1024) k_depth_hist(const unsigned long long* __restrict__ list,
                                                     unsigned* __restrict__ hist, const Control* __restrict__ ctl) {
  dep_wait();
  dep_release();
  __shared__ unsigned s_hist[kDepthPasses][kSortBins];
  if (step_void(ctl)) return;
  for (int k = threadIdx.x; k < kDepthPasses * kSortBins; k += blockDim.x) (&s_hist[0][0])[k] = 0u;
  __syncthreads();
  const unsigned n = ctl->listed;
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const unsigned db = (unsigned)(list[i] >> 32);
#pragma unroll
    for (int p = 0; p < kDepthPasses; ++p) atomicAdd(&s_hist[p][(db >> (p * kSortBits)) & (kSortBins - 1)], 1u);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < kDepthPasses * kSortBins; k += blockDim.x) {
    const unsigned c = (&s_hist[0][0])[k];
    if (c) atomicAdd(hist + k, c);
  }
}

// K3 of a large step: instance e (record order) of record r goes to place_of[r] + (its index in r).
__global__ void __launch_bounds__(512) k_emit_words(const ProjBuffers pb, const ViewDev* __restrict__ views, int stride,
                                                    const unsigned* __restrict__ place_of,
                                                    unsigned long long* __restrict__ words,
                                                    const unsigned* __restrict__ inst_rec, unsigned* __restrict__ hist,
                                                    int tile_passes, const Control* __restrict__ ctl) {
  dep_wait();
  dep_release();
  __shared__ unsigned s_hist[kMaxSortPasses - kDepthPasses][kSortBins];
  if (step_void(ctl)) return;
  for (int k = threadIdx.x; k < tile_passes * kSortBins; k += blockDim.x) (&s_hist[0][0])[k] = 0u;
  __syncthreads();
  const unsigned long long M = ctl->m_total;
  for (unsigned long long e = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; e < M;
       e += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned rec = inst_rec[e];
    const unsigned k = (unsigned)e - pb.offsets[rec];
    const uint2 rc = pb.rect[rec];
    const unsigned at = place_of[rec] + k;
    const ViewDev& V = views[rec / (unsigned)stride];
    const unsigned x0 = rc.x & 0xffffu, x1 = rc.x >> 16, y0 = rc.y & 0xffffu;
    const unsigned w = x1 - x0;
    const unsigned ty = y0 + k / w, tx = x0 + k % w;
    const unsigned tile = (unsigned)(V.tile_base + (long long)ty * V.gx + tx);
    words[at] = ((unsigned long long)tile << 32) | rec;
    for (int p = 0; p < tile_passes; ++p) atomicAdd(&s_hist[p][(tile >> (p * kSortBits)) & (kSortBins - 1)], 1u);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < tile_passes * kSortBins; k += blockDim.x) {
    const unsigned c = (&s_hist[0][0])[k];
    if (c) atomicAdd(hist + k, c);
  }
}

static void init_small_attributes();

void init_sort_attributes() {
  cudaFuncSetAttribute(k_sort_pass, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortSmem));
  cudaFuncSetAttribute(k_sort_pass_words, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(WordSmem));
  init_small_attributes();
}

int word_tile_passes(int tile_bits) { return tile_bits <= kSortBits ? 1 : (tile_bits + kSortBits - 1) / kSortBits; }

void launch_sort_large(const ProjBuffers& pb, const ViewDev* views, int stride, long long n_items,
                       unsigned long long* list0, unsigned long long* list1, unsigned* place_of,
                       unsigned long long* list_state, unsigned* depth_state, unsigned long long* words0,
                       unsigned long long* words1, unsigned* vals_out, unsigned* inst_rec, unsigned* hist,
                       unsigned* tile_state, int tile_bits, long long m_cap, int num_sms, Control* ctl, cudaStream_t s) {
  const unsigned rec_tiles = (unsigned)((n_items + kSortTile - 1) / kSortTile);
  const unsigned inst_tiles = (unsigned)((m_cap + kSortTile - 1) / kSortTile);
  launch_dep(k_depth_hist, dim3((unsigned)(2 * num_sms)), dim3(1024), 0, s, list0, hist, ctl);
  for (int p = 0; p < kDepthPasses; ++p)
    launch_dep(k_sort_pass_words, dim3(rec_tiles), dim3(kSortThreads), sizeof(WordSmem), s, (p & 1) ? list1 : list0,
        (p & 1) ? list0 : list1, nullptr, 1, hist + p * kSortBins, depth_state + (size_t)p * rec_tiles * kSortBins,
        32 + p * kSortBits, p, ctl, kSpinLimit);
  launch_dep(k_scan<SCAN_LIST>, dim3((unsigned)((n_items + kScanTile - 1) / kScanTile)), dim3(kScanThreads), 0, s,
      pb.count, place_of, 0ll, list_state, ctl, 0ull, nullptr, nullptr, kSpinLimit, list0, nullptr);
  launch_dep(k_fill_owner, dim3((unsigned)((n_items + 255) / 256)), dim3(256), 0, s, pb.count, pb.offsets, n_items,
      inst_rec, ctl);
  const int tp = word_tile_passes(tile_bits);
  // the last pass ends in words0: start in words[tp & 1]
  launch_dep(k_emit_words, dim3((unsigned)(4 * num_sms)), dim3(512), 0, s, pb, views, stride, place_of,
      (tp & 1) ? words1 : words0, inst_rec, hist + kDepthPasses * kSortBins, tp, ctl);
  for (int p = 0; p < tp; ++p) {
    const bool from1 = ((tp - p) & 1) != 0;
    launch_dep(k_sort_pass_words, dim3(inst_tiles), dim3(kSortThreads), sizeof(WordSmem), s, from1 ? words1 : words0,
        from1 ? words0 : words1, p == tp - 1 ? vals_out : nullptr, 0, hist + (kDepthPasses + p) * kSortBins,
        tile_state + (size_t)p * inst_tiles * kSortBins, 32 + p * kSortBits, kDepthPasses + p, ctl, kSpinLimit);
  }
}

// ---------------------------------------------------------------------------------------------
// K5: per-tile [start, end) of the sorted list.  Empty tiles keep the [0, 0) the step's clear
// left them.  Grid-stride over the device-resident instance count.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_ranges(const unsigned long long* __restrict__ keys, uint2* __restrict__ ranges,
                                                int tile_bits, int shift, const Control* __restrict__ ctl) {
  dep_wait();
  dep_release();
  if (step_void(ctl)) return;
  const unsigned long long M = ctl->m_total;
  const int D = shift ? shift : key_layout(ctl, tile_bits).D;  // where the tile starts in the key
  for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < M;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned tile = (unsigned)(keys[i] >> D);
    if (i == 0 || (unsigned)(keys[i - 1] >> D) != tile) ranges[tile].x = (unsigned)i;
    if (i == M - 1 || (unsigned)(keys[i + 1] >> D) != tile) ranges[tile].y = (unsigned)(i + 1);
  }
}

void launch_ranges(const unsigned long long* keys, uint2* ranges, int tile_bits, int shift, long long m_cap,
                   const Control* ctl, cudaStream_t s) {
  long long blocks = (m_cap + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  if (blocks < 1) blocks = 1;
  launch_dep(k_ranges, dim3((unsigned)blocks), dim3(256), 0, s, keys, ranges, tile_bits, shift, ctl);
}

// ---------------------------------------------------------------------------------------------
// Small steps: K3's emission, K4, K5 and the tile order in one launch by one thread-block cluster.
// Up to tens of thousands of instances the separate kernels last as long as their launches and
// chains (5 - 8 us each for emission, every sort pass, ranges and order), whatever the bytes.  Here
// the keys never leave the cluster: CTA r holds positions [r per, (r + 1) per) in shared memory,
// emits them there, and each stable 8-bit pass ranks them in registers (warp by warp, by match.any),
// exchanges the CTAs' digit totals and scatters straight into the owners' shared memory (distributed
// shared memory).  The cluster's barriers are the hardware's; nothing spins.
// K3 - K5 together, event times: 45 -> 28 us at 2.4k instances, 53 -> 30 at 5.2k, 60 -> 38 at 13k, 64 -> 45
// at 29k.  From there the work of sixteen SMs bounds it: with eight keys per thread, 69k instances, it took
// 79 us against 71 (also with each digit's run staged so that it leaves as consecutive words; records
// travelling beside the keys took 45 instead of 30 us at 5.2k), so four keys per thread and sixteen CTAs,
// 65,536 instances, is where it ends.
// ---------------------------------------------------------------------------------------------
namespace {
constexpr int kSmallThreads = 1024;
constexpr int kSmallWarps = kSmallThreads / 32;
constexpr int kSmallItems = 4;                                // keys per thread at most
constexpr int kSmallTile = kSmallThreads * kSmallItems;       // keys per CTA at most
constexpr int kSmallMaxCluster = 16;
constexpr int kSmallIndexBits = 16;                           // an instance's emission index, under its key
constexpr int kSmallMaxTileBits = 14;                         // the order is one CTA's loop over the tiles
static_assert(kSmallMaxTileBits + 32 + kSmallIndexBits <= 64, "tile, depth (at most 32 bits) and index fit a word");
static_assert(kSmallMaxCluster * kSmallTile <= (1 << kSmallIndexBits), "the index holds every instance");

struct SmallSmem {
  unsigned long long keys[kSmallTile];
  unsigned short cnt[kSmallWarps][kSortBins];
  unsigned total[kSortBins];
  unsigned gbase[kSortBins];
  unsigned warp_sum[kSortBins / 32];
  unsigned bucket[32], base[32];
};

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned cluster_size() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}
// Shared-memory address of CTA `rank`'s copy of p.
__device__ __forceinline__ unsigned cluster_addr(const void* p, unsigned rank) {
  unsigned a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ unsigned cluster_ld_u32(unsigned a) {
  unsigned v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long cluster_ld_u64(unsigned a) {
  unsigned long long v;
  asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_st_u64(unsigned a, unsigned long long v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}
}  // namespace

__global__ void __launch_bounds__(kSmallThreads, 1) k_bin_small(const ProjBuffers pb, const ViewDev* __restrict__ views,
                                                                int stride, const unsigned* __restrict__ inst_rec,
                                                                long long n_tiles, unsigned* __restrict__ vals_out,
                                                                uint2* __restrict__ ranges, int* __restrict__ order,
                                                                int tile_bits, const Control* __restrict__ ctl) {
  dep_wait();
  dep_release();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SmallSmem& S = *reinterpret_cast<SmallSmem*>(smem_raw);
  if (step_void(ctl)) return;  // every CTA of the cluster alike
  const unsigned M = (unsigned)ctl->m_total;
  const KeyLayout kl = key_layout(ctl, tile_bits);
  const unsigned r = cluster_rank(), C = cluster_size();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned lt = lanemask_lt();
  // positions per CTA: 1024 << ls, the fewest keys per thread that hold all M (M <= C kSmallTile)
  int ls = 0;
  while (((unsigned)kSmallThreads << ls) * C < M) ++ls;
  const int items = 1 << ls;
  const int per_shift = 10 + ls;
  const unsigned per_mask = (1u << per_shift) - 1u;
  const unsigned first = r << per_shift;          // this CTA's first position
  const int wfirst = warp * items * 32 + lane;    // this thread's first slot: slots wfirst + 32 k

  // (tile, depth) key above the instance's index: one 8-byte word per instance moves in each pass, and
  // the record follows from the index at the end
  unsigned long long key[kSmallItems];
#pragma unroll
  for (int k = 0; k < kSmallItems; ++k) {
    key[k] = 0ull;
    const unsigned e = first + (unsigned)(wfirst + 32 * k);
    if (k < items && e < M) {
      const unsigned rec = inst_rec[e];
      const unsigned q = e - pb.offsets[rec];
      const uint2 rc = pb.rect[rec];
      const unsigned db = __float_as_uint(pb.depth[rec]);
      const ViewDev& V = views[rec / (unsigned)stride];
      const unsigned x0 = rc.x & 0xffffu, x1 = rc.x >> 16, y0 = rc.y & 0xffffu;
      const unsigned w = x1 - x0;
      const unsigned ty = y0 + q / w, tx = x0 + q % w;
      const unsigned long long tile = (unsigned long long)(V.tile_base + (long long)ty * V.gx + tx);
      key[k] = (((tile << kl.D) | (unsigned long long)(db - kl.dmin)) << kSmallIndexBits) | e;
    }
  }

  for (int pass = 0; pass < kl.passes; ++pass) {
    const int shift = kSmallIndexBits + pass * kSortBits;
    for (int k = tid; k < kSmallWarps * kSortBins / 2; k += kSmallThreads) reinterpret_cast<unsigned*>(S.cnt)[k] = 0u;
    __syncthreads();
    // rank within the warp's slots, in slot order (stable)
    unsigned rank[kSmallItems];
#pragma unroll
    for (int k = 0; k < kSmallItems; ++k) {
      rank[k] = 0u;
      if (k < items) {
        const bool valid = first + (unsigned)(wfirst + 32 * k) < M;
        const unsigned d = (unsigned)(key[k] >> shift) & (kSortBins - 1);
        const unsigned peers = __match_any_sync(0xffffffffu, valid ? d : (kSortBins + d));
        const unsigned pre = valid ? S.cnt[warp][d] : 0u;
        __syncwarp();
        if (valid && (peers & lt) == 0u) S.cnt[warp][d] = (unsigned short)(pre + __popc(peers));
        __syncwarp();
        rank[k] = pre + __popc(peers & lt);
      }
    }
    __syncthreads();
    // per digit: exclusive prefix over the warps, and the CTA's total for the cluster
    if (tid < kSortBins) {
      unsigned c[kSmallWarps];
#pragma unroll
      for (int w = 0; w < kSmallWarps; ++w) c[w] = S.cnt[w][tid];
      unsigned run = 0u;
#pragma unroll
      for (int w = 0; w < kSmallWarps; ++w) {
        S.cnt[w][tid] = (unsigned short)run;
        run += c[w];
      }
      S.total[tid] = run;
    }
    cluster_barrier();  // totals published; every CTA's keys of this pass are in registers
    unsigned before = 0u, all = 0u, incl = 0u;
    if (tid < kSortBins) {
      for (unsigned q = 0; q < C; ++q) {
        const unsigned t = cluster_ld_u32(cluster_addr(&S.total[tid], q));
        before += q < r ? t : 0u;
        all += t;
      }
      incl = all;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      if (lane == 31) S.warp_sum[warp] = incl;
    }
    __syncthreads();
    if (tid < kSortBins) {
      unsigned lower = 0u;
      for (int w = 0; w < warp; ++w) lower += S.warp_sum[w];
      S.gbase[tid] = lower + incl - all + before;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kSmallItems; ++k) {
      if (k < items && first + (unsigned)(wfirst + 32 * k) < M) {
        const unsigned d = (unsigned)(key[k] >> shift) & (kSortBins - 1);
        const unsigned pos = S.gbase[d] + S.cnt[warp][d] + rank[k];  // < M
        const unsigned owner = pos >> per_shift, at = pos & per_mask;
        cluster_st_u64(cluster_addr(&S.keys[at], owner), key[k]);
      }
    }
    cluster_barrier();  // every key of this CTA's positions has arrived
#pragma unroll
    for (int k = 0; k < kSmallItems; ++k)
      if (k < items && first + (unsigned)(wfirst + 32 * k) < M) key[k] = S.keys[wfirst + 32 * k];
  }

  // the sorted list, and where each tile's run of it starts and ends
#pragma unroll
  for (int k = 0; k < kSmallItems; ++k) {
    const int at = wfirst + 32 * k;
    const unsigned pos = first + (unsigned)at;
    if (k < items && pos < M) {
      vals_out[pos] = inst_rec[(unsigned)key[k] & ((1u << kSmallIndexBits) - 1u)];
      const int tile_shift = kSmallIndexBits + kl.D;
      const unsigned tile = (unsigned)(key[k] >> tile_shift);
      // neighbours: in this CTA's keys, else the last of the CTA before or the first of the CTA after
      // (passes >= 1 put the keys into shared memory; with none there is one tile)
      bool starts = pos == 0u, ends = pos == M - 1u;
      if (kl.passes > 0) {
        if (!starts) {
          const unsigned long long p =
              at > 0 ? S.keys[at - 1] : cluster_ld_u64(cluster_addr(&S.keys[per_mask], r - 1u));
          starts = (unsigned)(p >> tile_shift) != tile;
        }
        if (!ends) {
          const unsigned long long p =
              (unsigned)at < per_mask ? S.keys[at + 1] : cluster_ld_u64(cluster_addr(&S.keys[0], r + 1u));
          ends = (unsigned)(p >> tile_shift) != tile;
        }
      }
      if (starts) ranges[tile].x = pos;
      if (ends) ranges[tile].y = pos + 1u;
    }
  }
  __threadfence();
  cluster_barrier();  // the ranges are written, and no CTA reads another's shared memory any more
  if (r != 0u) return;
  // K6's tile order (k_tile_order): buckets by floor(log2(list length)), longest first; the ranges come
  // from the other CTAs' SMs, so they are read through L2
  if (tid < 32) S.bucket[tid] = 0u;
  __syncthreads();
  const auto bucket_of = [&](long long t) {
    const unsigned long long rg = ld_relaxed_u64(reinterpret_cast<const unsigned long long*>(ranges + t));
    const unsigned L = (unsigned)(rg >> 32) - (unsigned)rg;
    return min(L ? 32 - __clz(L) : 0, 31);
  };
  for (long long t = tid; t < n_tiles; t += kSmallThreads) atomicAdd(&S.bucket[bucket_of(t)], 1u);
  __syncthreads();
  if (tid == 0) {
    unsigned run = 0u;
    for (int b = 31; b >= 0; --b) {
      S.base[b] = run;
      run += S.bucket[b];
    }
  }
  __syncthreads();
  for (long long t = tid; t < n_tiles; t += kSmallThreads) order[atomicAdd(&S.base[bucket_of(t)], 1u)] = (int)t;
}

// Cluster size for up to m_cap instances, 0 when the step is not small.  Set at start-up: a size the device
// cannot place (16 is beyond the portable 8) is not used.
static std::atomic<int> g_small_max_cluster{0};

int bin_small_cluster(long long m_cap, int tile_bits) {
  const int most = g_small_max_cluster;
  if (tile_bits > kSmallMaxTileBits || m_cap > (long long)most * kSmallTile) return 0;
  int c = 1;
  while (c < most && (long long)c * kSmallThreads < m_cap) c <<= 1;  // as few keys per thread as the cluster allows
  return c;
}

namespace {
cudaLaunchConfig_t small_config(int cluster, cudaLaunchAttribute* attr, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cluster);
  cfg.blockDim = dim3(kSmallThreads);
  cfg.dynamicSmemBytes = sizeof(SmallSmem);
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cfg;
}
}  // namespace

static void init_small_attributes() {
  cudaFuncSetAttribute(k_bin_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallSmem));
  cudaFuncSetAttribute(k_bin_small, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  int best = 0;
  for (int c = 1; c <= kSmallMaxCluster; c <<= 1) {
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = small_config(c, attr, nullptr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_bin_small, &cfg) != cudaSuccess) {
      cudaGetLastError();
      break;
    }
    if (n < 1) break;
    best = c;
  }
  g_small_max_cluster = best;
}

void launch_bin_small(const ProjBuffers& pb, const ViewDev* views, int stride, long long n_items, unsigned* inst_rec,
                      long long n_tiles, unsigned* vals_out, uint2* ranges, int* order, int tile_bits, int cluster,
                      const Control* ctl, cudaStream_t s) {
  if (n_items <= 0) return;
  launch_dep(k_fill_owner, dim3((unsigned)((n_items + 255) / 256)), dim3(256), 0, s, pb.count, pb.offsets, n_items,
      inst_rec, ctl);
  cudaLaunchAttribute attr[2];
  const cudaLaunchConfig_t cfg = small_config(cluster, attr, s);
  cudaLaunchKernelEx(&cfg, k_bin_small, pb, views, stride, (const unsigned*)inst_rec, n_tiles, vals_out, ranges, order,
                     tile_bits, ctl);
}

// ---------------------------------------------------------------------------------------------
// Failure detection for the two inter-CTA waits.  Each wait is run once on a two-tile problem by a
// single CTA that holds ticket 1: tile 0 is never started, so its status word stays 0 and the wait
// can only end by giving up.  The problems are laid out so that the CTA's remaining work after
// giving up (with a partial prefix of 0) stays inside its own buffers.
// ---------------------------------------------------------------------------------------------
gs_status run_wait_probe(unsigned spin_limit, unsigned out_error[2], float out_ms[2]) {
  if (spin_limit == 0u) spin_limit = kSpinLimit;
  init_sort_attributes();
  const size_t n_scan = 2 * (size_t)kScanTile, n_sort = 2 * (size_t)kSortTile;
  const size_t off_ctl_b = kCtlBytes, off_state_a = 2 * kCtlBytes;
  const size_t off_state_b = off_state_a + 2 * sizeof(unsigned long long);
  const size_t off_hist = off_state_b + 2 * kSortBins * sizeof(unsigned);
  const size_t off_in = off_hist + (size_t)kMaxSortPasses * kSortBins * sizeof(unsigned);
  const size_t off_out = off_in + n_scan * sizeof(unsigned);
  const size_t off_k0 = off_out + n_scan * sizeof(unsigned);
  const size_t off_k1 = off_k0 + n_sort * sizeof(unsigned long long);
  const size_t off_v0 = off_k1 + n_sort * sizeof(unsigned long long);
  const size_t off_v1 = off_v0 + n_sort * sizeof(unsigned);
  const size_t bytes = off_v1 + n_sort * sizeof(unsigned);
  char* d = nullptr;
  cudaStream_t st = nullptr;
  cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};
  gs_status status = GS_OK;
  auto check = [&](cudaError_t e, const char* what) {
    if (e != cudaSuccess && status == GS_OK) status = fail(GS_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
    return e == cudaSuccess;
  };
  if (check(cudaMalloc(&d, bytes), "cudaMalloc") && check(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking), "stream") &&
      check(cudaEventCreate(&ev[0]), "event") && check(cudaEventCreate(&ev[1]), "event") &&
      check(cudaEventCreate(&ev[2]), "event") && check(cudaMemsetAsync(d, 0, bytes, st), "cudaMemsetAsync")) {
    Control ca{}, cb{};
    ca.scan_ticket = 1u;       // the CTA takes tile 1 of the scan
    cb.sort_ticket[0] = 1u;    // and tile 1 of pass 0 of the sort
    cb.m_total = n_sort;       // all keys 0: one pass, every key in digit 0
    const unsigned h0 = (unsigned)n_sort;
    Control* ctl_a = reinterpret_cast<Control*>(d);
    Control* ctl_b = reinterpret_cast<Control*>(d + off_ctl_b);
    unsigned* hist = reinterpret_cast<unsigned*>(d + off_hist);
    if (check(cudaMemcpyAsync(ctl_a, &ca, sizeof(Control), cudaMemcpyHostToDevice, st), "cudaMemcpyAsync") &&
        check(cudaMemcpyAsync(ctl_b, &cb, sizeof(Control), cudaMemcpyHostToDevice, st), "cudaMemcpyAsync") &&
        check(cudaMemcpyAsync(hist, &h0, sizeof(unsigned), cudaMemcpyHostToDevice, st), "cudaMemcpyAsync")) {
      cudaEventRecord(ev[0], st);
      k_scan<SCAN_PLAIN><<<1, kScanThreads, 0, st>>>(reinterpret_cast<const unsigned*>(d + off_in),
                                         reinterpret_cast<unsigned*>(d + off_out), (long long)n_scan,
                                         reinterpret_cast<unsigned long long*>(d + off_state_a), ctl_a, ~0ull,
                                         nullptr, nullptr, spin_limit, nullptr, nullptr);
      cudaEventRecord(ev[1], st);
      k_sort_pass<<<1, kSortThreads, sizeof(SortSmem), st>>>(
          reinterpret_cast<unsigned long long*>(d + off_k0), reinterpret_cast<unsigned*>(d + off_v0),
          reinterpret_cast<unsigned long long*>(d + off_k1), reinterpret_cast<unsigned*>(d + off_v1), hist,
          reinterpret_cast<unsigned*>(d + off_state_b), 0, 8, ctl_b, spin_limit);
      cudaEventRecord(ev[2], st);
      check(cudaGetLastError(), "wait probe launch");
      Control ra{}, rb{};
      if (check(cudaMemcpyAsync(&ra, ctl_a, sizeof(Control), cudaMemcpyDeviceToHost, st), "cudaMemcpyAsync") &&
          check(cudaMemcpyAsync(&rb, ctl_b, sizeof(Control), cudaMemcpyDeviceToHost, st), "cudaMemcpyAsync") &&
          check(cudaStreamSynchronize(st), "cudaStreamSynchronize")) {
        out_error[0] = ra.error;
        out_error[1] = rb.error;
        if (out_ms) {
          cudaEventElapsedTime(&out_ms[0], ev[0], ev[1]);
          cudaEventElapsedTime(&out_ms[1], ev[1], ev[2]);
        }
      }
    }
  }
  for (cudaEvent_t e : ev)
    if (e) cudaEventDestroy(e);
  if (st) cudaStreamDestroy(st);
  if (d) cudaFree(d);
  return status;
}

}  // namespace gs
