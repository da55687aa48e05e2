// k_blend.cu -- K6 (front-to-back alpha blending, Eq. 2) and K8 (its splatting-parallel
// backward, Sec. IV-D), sm_103a.
//
// Both are templates over the tile shape TW x TH (a multiple of the 8 x 4 warp block, at most 256
// pixels) and K6 over the staged batch; the autotuner of the session picks the instance.
//
// K6: persistent CTAs of TW x TH threads (one pixel per thread, each warp an 8 x 4 pixel block)
// take tiles longest-list first, so the few very long tiles do not end up as the tail of the
// launch.  A tile's sorted Gaussians come through shared memory as jobs of up to BATCH entries, two
// jobs resident at a time: the warp that finishes a job first stages the next one (the next batch
// of the same tile while a warp of it still blends, else the next tile) with asynchronous copies,
// and publishes it on an mbarrier, so staging overlaps the other warps' walk and a fast warp can run
// a job ahead of the tile's slowest block instead of waiting for it at a CTA barrier.  Jobs are
// walked in chunks of 32.  A warp skips a Gaussian outright when the bounding box of its 1/255 cutoff
// ellipse misses the warp's block (warp-uniform).  The others are taken two at a time (four when the tiles
// are few, see few_tiles) without a branch: every lane evaluates their exponents and alphas, then blends
// them in list order under predicates.  A pixel's walk is one dependent chain, and the longest lists set
// the kernel's duration from a few thousand Gaussians up, so what counts is the chain's length per candidate: with a branch per test
// (cutoff, alpha, stop) it was about 300 cycles, in this form about 210 when a CTA has its SM to itself,
// and about 48 instead of 62 instructions.  A stopped pixel's x becomes NaN, which fails every later
// test by itself; the last index and G_p follow from the chunk's mask.  Measured: 54 -> 32 us on a
// 128 x 97 view of 3,400 Gaussians, 54 -> 39 us at 640 x 361 (20k), 120 -> 108 us at 1297 x 840 (200k,
// 32M blended pairs), 440 -> 345 us at 1.9M, 856 -> 755 us for nine views of 500k.  (A lone last candidate
// is evaluated alone: evaluating it twice cost 4 % on the nine views.)  Measured and not kept: two
// lanes per pixel, each with its own candidate, on 4 x 4 blocks (the blending is then done by both:
// 183 us at 200k); the next pair's records read during the blending (124 us); 80 registers and three
// CTAs per SM (291 us at 1.9M, but 843 us on the nine views); a staging warp of its own (139 us).
// Per (pixel, chunk) K6 stores the transmittance and colour at the chunk start and a 32-bit mask
// of the Gaussians actually blended; a tile gets no more batches once every warp's pixels stopped.
// When the last of a tile's warps leaves it, the tile is flagged complete (a GPU-scope release), so
// the loss that follows can start on the image blocks over finished tiles while K6 still runs.
//
// K8: gradient accumulation per Gaussian (the splatting-based parallelism the paper adopts from
// Taming 3DGS to remove the serialized per-pixel atomics of the original backward).  Work item =
// (tile, 32-entry chunk), one warp each, taken from a global counter.  The warp compacts the
// tile's pixels whose mask for this chunk is non-empty and takes them 128 at a time, four per
// lane held as the halves of two packed FP32x2 values (sm_100's FFMA2 / FMUL2 / FADD2 work on both
// halves at once).  First each lane restarts its pixels from the checkpoint.  The lanes then walk the union
// of their pixels' blended Gaussians in list order, three Gaussians at a time: a lane computes its
// pixels' nine gradient terms for each (a pixel that did not blend it takes G = 0, which leaves
// its state unchanged and its terms zero) and advances transmittance and front colour exactly as
// the forward did (the colour behind a Gaussian is the rendered colour minus the colour
// accumulated in front of it); it adds its pixels' terms, and the 27 terms are summed over the
// lanes through shared memory in a fixed order and added to the Gaussians' running sums.  A round's pixels share
// few Gaussians (about 9 of 32), each blended by many of them, so this keeps more lanes busy than
// one lane per Gaussian.  No atomics: the gradient is deterministic, and each instance's gradient
// is written once, to its own slot.  K8 is bound by issue (66 % at 16 warps per SM; 240 instructions per
// Gaussian and round, of which 1.4 pair bodies are about 95) and, with few items, by one warp's latency
// (5 cycles per instruction).  The load term is a template flag (its test and weights cost 4 registers
// and an instruction per pair), the reciprocal of 1 - alpha is rcp.approx.ftz, the conic terms' factors
// are applied once per row sum, and the tile's position takes 32-bit divisions: 1269 -> 1221 us for nine
// views of 500k Gaussians, 152 -> 144 at 1297 x 840 (200k), 48 -> 45 at 640 x 361 (20k), the same bits.
// Measured and not kept: the records held twice in shared memory for the packed operands (16 bytes more
// per Gaussian through a half-busy pipe: 163 us at 200k), the next item claimed one ahead (63 us at 20k),
// both pairs evaluated without a branch (1323 us on the nine views, no shorter for a lone warp).
#include "gs_device.cuh"
#include "gs_engine.h"

namespace gs {

namespace {

// Pixel layout of a TW x TH tile: warp w covers the 8 x 4 block (w % BX, w / BX) of the tile,
// lane l its pixel (l % 8, l / 8).  K6 and K8 share this mapping.
template <int TW, int TH>
struct Shape {
  static constexpr int kPix = TW * TH;
  static constexpr int kWarps = kPix / 32;
  static constexpr int kBX = TW / 8;
  static constexpr int kBY = TH / 4;
  static_assert(TW % 8 == 0 && TH % 4 == 0 && kPix >= 32 && kPix <= kMaxTilePix, "unsupported tile shape");
  static_assert(kWarps <= 8, "the per-entry warp-block mask is 8 bits");
  __device__ static __forceinline__ void slot_xy(int s, int& ox, int& oy) {
    const int w = s >> 5, l = s & 31;
    ox = ((w % kBX) << 3) + (l & 7);
    oy = ((w / kBX) << 2) + (l >> 3);
  }
};

__device__ __forceinline__ int view_of_tile(const ViewDev* __restrict__ views, int n_views, long long t) {
  int v = 0;
  while (v + 1 < n_views && views[v + 1].tile_base <= t) ++v;
  return v;
}

// Chunk id of a tile's chunk 0: unique over tiles and < (instances / 32) + tiles + 1.
__device__ __forceinline__ long long chunk_base(unsigned start, long long tile) {
  return (long long)(start >> 5) + tile;
}
}  // namespace

// ---------------------------------------------------------------------------------------------
// Tile order for K6: buckets by floor(log2(list length)), longest bucket first (one CTA).
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) k_tile_order(const uint2* __restrict__ ranges, long long n_tiles,
                                                     int* __restrict__ order, const Control* __restrict__ ctl) {
  dep_wait();
  dep_release();
  __shared__ unsigned s_cnt[32];
  __shared__ unsigned s_base[32];
  if (step_void(ctl)) return;
  if (threadIdx.x < 32) s_cnt[threadIdx.x] = 0u;
  __syncthreads();
  for (long long t = threadIdx.x; t < n_tiles; t += blockDim.x) {
    const unsigned L = ranges[t].y - ranges[t].x;
    const int b = L ? 32 - __clz(L) : 0;  // 0 = empty, else 1 + floor(log2 L), at most 31
    atomicAdd(&s_cnt[min(b, 31)], 1u);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned run = 0;
    for (int b = 31; b >= 0; --b) {
      s_base[b] = run;
      run += s_cnt[b];
    }
  }
  __syncthreads();
  for (long long t = threadIdx.x; t < n_tiles; t += blockDim.x) {
    const unsigned L = ranges[t].y - ranges[t].x;
    const int b = L ? 32 - __clz(L) : 0;
    order[atomicAdd(&s_base[min(b, 31)], 1u)] = (int)t;
  }
}

// ---------------------------------------------------------------------------------------------
// K6
// ---------------------------------------------------------------------------------------------
// Work flows through the CTA as jobs: a job is one staged batch (up to BATCH sorted entries) of one
// tile, and kFwdBufs jobs are in shared memory at a time.  Each warp walks every job in order (its 8 x 4
// block of the job's tile); the warp that finishes job j first stages job j + 1 into the other
// buffer of job j + 1 - kFwdBufs once every warp is through that job -- the next batch of the same tile while
// any warp of it still blends, else the first batch of the next tile in the longest-first order -- so staging overlaps the slower warps' walk and a
// warp waits only when it has caught up with the staging, not for the tile's slowest block.  A job
// is published by an mbarrier (`full`, 32 arrivals: the staging warp's lanes) and released by
// another (`empty`, one arrival per warp).  Every wait is bounded: a wait that gives up sets
// kErrTimeout and its warp leaves (the host reports GS_ERR_TIMEOUT; the image is then unspecified).
namespace {
constexpr int kFwdBufs = 2;  // jobs in shared memory at a time (3 measured 112 against 107 us)

struct FwdJob {
  long long t;      // global tile
  unsigned start;   // first entry of the tile's list
  int L;            // list length
  int b0;           // first entry of this batch
  int seq;          // tile sequence number within the CTA
  int end;          // 1: no more work
};

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
// 16-byte asynchronous copy global -> shared (both 16-byte aligned)
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}" ::"r"(smem_u32(bar)) : "memory");
}
// Bounded wait for the phase of the given parity to complete; false when it gave up.
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity, unsigned limit) {
  for (unsigned k = 0; k < limit; ++k) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}
}  // namespace

// DEEP: candidates of a chunk evaluated together in a round of the walk (with 2 a lone last one alone).
template <int TW, int TH, int BATCH, int DEEP>
__device__ __forceinline__ void blend_forward(
    const ViewDev* __restrict__ views, int n_views, long long n_tiles, const uint2* __restrict__ ranges,
    const unsigned* __restrict__ vals, const ProjBuffers& pb, const StepParams* __restrict__ sp,
    Control* __restrict__ ctl, const int* __restrict__ order, float* __restrict__ image, float* __restrict__ Tout,
    unsigned* __restrict__ last_out, unsigned* __restrict__ gp_out, float4* __restrict__ ckpt,
    unsigned* __restrict__ cmask, int* __restrict__ chunk_tile, int* __restrict__ tile_chunks,
    unsigned* __restrict__ tile_done) {
  dep_wait();
  dep_release();
  using S = Shape<TW, TH>;
  constexpr int kPix = S::kPix;
  static_assert(BATCH % kChunk == 0, "batches hold whole chunks");
  __shared__ float4 s_xyo[kFwdBufs][BATCH];
  __shared__ float4 s_con[kFwdBufs][BATCH];
  __shared__ float4 s_rgb[kFwdBufs][BATCH];
  __shared__ unsigned char s_bm[kFwdBufs][BATCH];  // per entry: the warp blocks its cutoff box reaches
  __shared__ FwdJob s_job[kFwdBufs];
  __shared__ __align__(8) unsigned long long s_full[kFwdBufs], s_empty[kFwdBufs];
  __shared__ int s_next;     // the next job to be staged (the stager of job j + 1 is elected on it)
  __shared__ int s_live[kFwdBufs];  // per tile (sequence mod kFwdBufs): warps with pixels still blending
  __shared__ unsigned s_fin[4];     // per tile (sequence mod 4): warps that left it (at most 3 tiles open)
  // the stager's progress through the tiles (only the warp staging the next job reads or writes it;
  // jobs are staged one after another)
  __shared__ long long s_cur_t;
  __shared__ unsigned s_cur_start;
  __shared__ int s_cur_L, s_cur_nb, s_cur_seq;
  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const float bg0 = sp->bg[0], bg1 = sp->bg[1], bg2 = sp->bg[2];
  unsigned my_pairs = 0, my_blend = 0, my_gpn = 0, my_gpsq = 0;  // this thread's pixels (fit 32 bits)

  // Stage job j (one warp): decide what it is, then load its entries into buffer j % kFwdBufs.
  auto stage = [&](int j) -> bool {
    const int buf = j % kFwdBufs;
    if (j >= kFwdBufs && !mbar_wait(&s_empty[buf], ((j - kFwdBufs) / kFwdBufs) & 1, kSpinLimit)) return false;
    if (lane == 0) {
      FwdJob jb;
      jb.end = 0;
      if (s_cur_seq >= 0 && s_cur_nb * BATCH < s_cur_L && s_live[s_cur_seq % kFwdBufs] > 0) {
        jb.t = s_cur_t;  // the tile's next batch
        jb.start = s_cur_start;
        jb.L = s_cur_L;
        jb.b0 = s_cur_nb * BATCH;
        jb.seq = s_cur_seq;
        ++s_cur_nb;
      } else {
        // chunks whose masks every pixel of the finished tile received (the backward reads those)
        if (s_cur_seq >= 0)
          tile_chunks[s_cur_t] = min((s_cur_L + kChunk - 1) / kChunk, s_cur_nb * (BATCH / kChunk));
        const int item = (int)atomicAdd(&ctl->fwd_work, 1u);
        if (item >= n_tiles) {
          jb.end = 1;
          jb.t = 0;
          jb.start = 0;
          jb.L = 0;
          jb.b0 = 0;
          jb.seq = s_cur_seq + 1;
        } else {
          const long long t = order[item];
          const uint2 rg = ranges[t];
          s_cur_t = t;
          s_cur_start = rg.x;
          s_cur_L = (int)(rg.y - rg.x);
          s_cur_nb = 1;
          s_cur_seq += 1;
          s_live[s_cur_seq % kFwdBufs] = S::kWarps;
          jb.t = t;
          jb.start = rg.x;
          jb.L = s_cur_L;
          jb.b0 = 0;
          jb.seq = s_cur_seq;
        }
      }
      s_job[buf] = jb;
    }
    __syncwarp();
    const FwdJob jb = s_job[buf];
    if (!jb.end) {
      if (jb.b0 == 0) {  // a new tile: map its chunks back to it for the backward
        const long long cb = chunk_base(jb.start, jb.t);
        for (int k = lane; k < (jb.L + kChunk - 1) / kChunk; k += 32) chunk_tile[cb + k] = (int)(jb.t + 1);
      }
      const int v = view_of_tile(views, n_views, jb.t);
      const ViewDev& V = views[v];
      const int local = (int)(jb.t - V.tile_base);
      const float tx0 = (float)(local % V.gx * TW), ty0 = (float)(local / V.gx * TH);
      const int nb = min(BATCH, jb.L - jb.b0);
      // all of the lane's record indices in flight at once, then its records copied straight into
      // shared memory by asynchronous 16-byte copies (no registers held), then the block masks
      constexpr int kPer = BATCH / 32;
      unsigned recs[kPer];
#pragma unroll
      for (int k = 0; k < kPer; ++k) {
        const int jj = lane + 32 * k;
        recs[k] = jj < nb ? __ldg(vals + jb.start + jb.b0 + jj) : 0u;
      }
#pragma unroll
      for (int k = 0; k < kPer; ++k) {
        const int jj = lane + 32 * k;
        if (jj < nb) {
          cp_async16(&s_xyo[buf][jj], pb.xyo + recs[k]);
          cp_async16(&s_con[buf][jj], pb.conic + recs[k]);
          cp_async16(&s_rgb[buf][jj], pb.rgb + recs[k]);
        }
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll
      for (int k = 0; k < kPer; ++k) {
        const int jj = lane + 32 * k;
        if (jj >= nb) break;
        const float4 xy = s_xyo[buf][jj];
        // which 8 x 4 warp blocks (warp w at (8 (w % BX), 4 (w / BX))) the cutoff box of this
        // Gaussian reaches; block centres are 3.5 / 1.5 px from their edge pixels
        unsigned xm = 0u, ym = 0u;
#pragma unroll
        for (int bx = 0; bx < S::kBX; ++bx)
          if (fabsf(xy.x - (tx0 + 8.f * bx + 3.5f)) <= xy.z + 3.5f) xm |= 1u << bx;
#pragma unroll
        for (int by = 0; by < S::kBY; ++by)
          if (fabsf(xy.y - (ty0 + 4.f * by + 1.5f)) <= xy.w + 1.5f) ym |= 1u << by;
        unsigned bm = 0u;
#pragma unroll
        for (int by = 0; by < S::kBY; ++by)
          if (ym & (1u << by)) bm |= xm << (S::kBX * by);
        s_bm[buf][jj] = (unsigned char)bm;
      }
    }
    mbar_arrive(&s_full[buf]);  // every lane: its own writes are published with it
    return true;
  };

  if (tid == 0) {
    for (int b = 0; b < kFwdBufs; ++b) {
      mbar_init(&s_full[b], 32);
      mbar_init(&s_empty[b], S::kWarps);
    }
    s_next = 1;
    s_cur_seq = -1;
    s_cur_nb = 0;
    s_cur_L = 0;
    for (int b = 0; b < kFwdBufs; ++b) s_live[b] = 0;
    for (int b = 0; b < 4; ++b) s_fin[b] = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (__syncthreads_or(tid == 0 && step_void(ctl))) return;
  bool ok = warp != 0 || stage(0);

  // this thread's pixel of the current tile
  int my_seq = -1, my_t = 0, my_v = 0;
  long long my_chunk = 0;  // chunk 0's slot of this pixel in the checkpoints and masks
  bool counted = true;
  float T = 1.f, C0 = 0.f, C1 = 0.f, C2 = 0.f;
  unsigned last = 0u, gp = 0u, neval = 0u;
  float pxf = 0.f, pyf = 0.f;  // pxf is NaN where there is no pixel or it has stopped
  auto pixel = [&](int& px, int& py) {
    const ViewDev& V = views[my_v];
    const int local = (int)(my_t - V.tile_base);
    int ox, oy;
    S::slot_xy(tid, ox, oy);
    px = local % V.gx * TW + ox;
    py = local / V.gx * TH + oy;
  };
  // (warp-uniform: every lane of the warp leaves the tile at the same job)
  auto finish_tile = [&]() {
    if (my_seq < 0) return;
    const ViewDev& V = views[my_v];
    int px, py;
    pixel(px, py);
    if (px < V.W && py < V.H) {
      const long long pix = (long long)py * V.W + px, HWv = (long long)V.W * V.H, pix_base = V.pix_base;
      float* img = image + 3 * pix_base;
      img[pix] = C0 + T * bg0;
      img[HWv + pix] = C1 + T * bg1;
      img[2 * HWv + pix] = C2 + T * bg2;
      const long long gpix = pix_base + pix;
      if (Tout) Tout[gpix] = T;
      last_out[gpix] = last;
      if (gp_out) gp_out[gpix] = gp;
      my_pairs += neval;
      my_blend += gp;
      if (gp) {
        my_gpn += 1;
        my_gpsq += gp * gp;
      }
    }
    // this warp's pixels of the tile are final.  The warp barrier orders its lanes' writes before
    // lane 0's CTA-scope release on the tile's arrival count; the last warp to arrive acquires them
    // all and publishes the tile with one GPU-scope release, so a reader that acquires the flag sees
    // every pixel of the tile (the loss forward starts a block once the tiles under it are flagged).
    // Job j + 1 is staged only once every warp is through job j - 1, so the warps that have not left
    // a tile are on the tiles of three consecutive jobs at most: four counters are never shared.
    // (Without tile flags nothing reads this grid's output before it has completed.)
    if (!tile_done) return;
    __syncwarp();
    if (lane == 0) {
      unsigned* fin = &s_fin[my_seq & 3];
      unsigned old;
      asm volatile("atom.acq_rel.cta.shared::cta.add.u32 %0, [%1], 1;" : "=r"(old) : "r"(smem_u32(fin)) : "memory");
      if (old == (unsigned)(S::kWarps - 1)) {
        *fin = 0u;
        red_release_add_u32(tile_done + my_t, 1u);
      }
    }
  };

  struct Cand {
    float alpha, r, g, b;
    bool use;
  };
  // Alpha of entry q of buffer `buf` at this pixel, and whether the pixel takes it (before its stop
  // test).  A pixel that has stopped (or lies outside the image) has pxf = NaN, so that no comparison
  // of its exponent holds.
  auto eval = [&](int buf, int q) -> Cand {
    const float2 xy = *reinterpret_cast<const float2*>(&s_xyo[buf][q]);
    const float4 co = s_con[buf][q];
    const float4 c = s_rgb[buf][q];
    const float power = splat_power(co.x, co.y, co.z, __fsub_rn(xy.x, pxf), __fsub_rn(xy.y, pyf));
    Cand e;
    e.alpha = fminf(kAlphaMax, __fmul_rn(c.w, splat_exp(power)));
    e.use = power <= 0.f && power >= co.w && e.alpha >= kAlphaMin;
    e.r = c.x;
    e.g = c.y;
    e.b = c.z;
    return e;
  };
  // Blends a candidate the pixel takes; true when the pixel stops at it.
  auto blend = [&](const Cand& e, bool use, unsigned bit, int jg, unsigned& mask) -> bool {
    const float testT = __fmul_rn(T, __fsub_rn(1.f, e.alpha));
    const bool stop = use && testT < kTransMin;
    if (stop) {
      pxf = __int_as_float(0x7fffffff);
      neval = (unsigned)jg + 1u;
    }
    if (use && !stop) {
      const float w = __fmul_rn(e.alpha, T);
      C0 = __fmaf_rn(e.r, w, C0);
      C1 = __fmaf_rn(e.g, w, C1);
      C2 = __fmaf_rn(e.b, w, C2);
      T = testT;
      mask |= bit;
    }
    return stop;
  };

  for (int j = 0; ok; ++j) {
    const int buf = j % kFwdBufs;
    if (!mbar_wait(&s_full[buf], (j / kFwdBufs) & 1, kSpinLimit)) {
      ok = false;
      break;
    }
    const FwdJob jb = s_job[buf];
    if (jb.seq != my_seq) {  // a new tile (or the end)
      finish_tile();
      if (jb.end) break;
      my_seq = jb.seq;
      my_t = (int)jb.t;
      my_v = view_of_tile(views, n_views, jb.t);
      int px, py;
      pixel(px, py);
      pxf = px < views[my_v].W && py < views[my_v].H ? (float)px : __int_as_float(0x7fffffff);
      pyf = (float)py;
      my_chunk = chunk_base(jb.start, jb.t) * kPix + tid;
      T = 1.f;
      C0 = C1 = C2 = 0.f;
      last = gp = 0u;
      neval = (unsigned)jb.L;
      counted = false;
    }
    // walk this job's chunks (a warp whose pixels have all stopped still records empty masks)
    const int nb = min(BATCH, jb.L - jb.b0);
    for (int c0 = 0; c0 < nb; c0 += kChunk) {
      const int jg0 = jb.b0 + c0;
      const long long at = my_chunk + (long long)(jg0 >> 5) * kPix;
      const int ce = min(kChunk, nb - c0);
      // entries of this chunk whose cutoff box reaches this warp's block (warp-uniform)
      unsigned cand = __ballot_sync(0xffffffffu, lane < ce && ((s_bm[buf][c0 + lane] >> warp) & 1u));
      const bool done = pxf != pxf;
      if (__all_sync(0xffffffffu, done)) {
        cmask[at] = 0u;
        continue;
      }
      if (jg0 > 0 && !done) ckpt[at] = make_float4(T, C0, C1, C2);
      unsigned mask = 0u;
      // One straight line per candidate, DEEP candidates in flight: every lane evaluates their
      // exponents and alphas, then they are blended in list order under predicates.
      if (DEEP > 2) {
        while (cand) {
          unsigned bit[DEEP];
          int q[DEEP];
#pragma unroll
          for (int u = 0; u < DEEP; ++u) {
            bit[u] = cand & (0u - cand);
            q[u] = bit[u] ? 31 - __clz(bit[u]) : q[u ? u - 1 : 0];
            cand ^= bit[u];
          }
          Cand e[DEEP];
#pragma unroll
          for (int u = 0; u < DEEP; ++u) e[u] = eval(buf, c0 + q[u]);
          bool stop = false;
#pragma unroll
          for (int u = 0; u < DEEP; ++u) stop |= blend(e[u], e[u].use && bit[u] != 0u && !stop, bit[u], jg0 + q[u], mask);
        }
      }
      while (cand) {
        const unsigned bit0 = cand & (0u - cand);
        const int q0 = 31 - __clz(bit0);
        cand ^= bit0;
        if (!cand) {
          const Cand e0 = eval(buf, c0 + q0);
          blend(e0, e0.use, bit0, jg0 + q0, mask);
          break;
        }
        const unsigned bit1 = cand & (0u - cand);
        const int q1 = 31 - __clz(bit1);
        cand ^= bit1;
        const Cand e0 = eval(buf, c0 + q0), e1 = eval(buf, c0 + q1);
        const bool stop = blend(e0, e0.use, bit0, jg0 + q0, mask);
        blend(e1, e1.use && !stop, bit1, jg0 + q1, mask);
      }
      if (mask) {
        last = (unsigned)(jg0 + 32 - __clz(mask));
        gp += __popc(mask);
      }
      cmask[at] = mask;
    }
    // this warp's pixels have all stopped: the stager need not stage more of the tile for it
    if (!counted && __all_sync(0xffffffffu, pxf != pxf)) {
      counted = true;
      if (lane == 0) atomicSub(&s_live[my_seq % kFwdBufs], 1);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&s_empty[buf]);
    // the first warp to finish job j stages job j + 1
    int mine = 0;
    if (lane == 0) mine = atomicCAS(&s_next, j + 1, j + 2) == j + 1;
    if (__shfl_sync(0xffffffffu, mine, 0) && !stage(j + 1)) ok = false;
  }
  if (!ok && lane == 0) atomicOr(&ctl->error, kErrTimeout);
  // Gaussian-pixel pairs by definition: entries evaluated per pixel up to its termination.
  unsigned long long sp_ = my_pairs, sb = my_blend, sn = my_gpn, sq = my_gpsq;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sp_ += __shfl_down_sync(0xffffffffu, sp_, o);
    sb += __shfl_down_sync(0xffffffffu, sb, o);
    sn += __shfl_down_sync(0xffffffffu, sn, o);
    sq += __shfl_down_sync(0xffffffffu, sq, o);
  }
  if (lane == 0) {
    if (sp_) atomicAdd(&ctl->pairs, sp_);
    if (sb) atomicAdd(&ctl->blended, sb);
    if (sn) {
      atomicAdd(&ctl->gp_pixels, sn);
      atomicAdd(&ctl->gp_sq, sq);
    }
    red_release_add_u32(&ctl->fwd_done, 1u);  // after this warp's counters (the loss's last CTA waits)
  }
}

#define GS_FORWARD_PARAMS                                                                                             \
  const ViewDev *__restrict__ views, int n_views, long long n_tiles, const uint2 *__restrict__ ranges,                \
      const unsigned *__restrict__ vals, const ProjBuffers pb, const StepParams *__restrict__ sp,                     \
      Control *__restrict__ ctl, const int *__restrict__ order, float *__restrict__ image, float *__restrict__ Tout,  \
      unsigned *__restrict__ last_out, unsigned *__restrict__ gp_out, float4 *__restrict__ ckpt,                      \
      unsigned *__restrict__ cmask, int *__restrict__ chunk_tile, int *__restrict__ tile_chunks,                      \
      unsigned *__restrict__ tile_done
#define GS_FORWARD_ARGS                                                                                               \
  views, n_views, n_tiles, ranges, vals, pb, sp, ctl, order, image, Tout, last_out, gp_out, ckpt, cmask, chunk_tile, \
      tile_chunks, tile_done

template <int TW, int TH, int BATCH>
__global__ void __launch_bounds__(TW * TH, 1024 / (TW * TH)) k_blend_forward(GS_FORWARD_PARAMS) {
  blend_forward<TW, TH, BATCH, 2>(GS_FORWARD_ARGS);
}

constexpr int kDeep = 4;
template <int TW, int TH, int BATCH>
__global__ void __launch_bounds__(TW * TH, 512 / (TW * TH)) k_blend_forward_few(GS_FORWARD_PARAMS) {
  blend_forward<TW, TH, BATCH, kDeep>(GS_FORWARD_ARGS);
}

void launch_tile_order(const uint2* ranges, long long n_tiles, int* order, const Control* ctl, cudaStream_t s) {
  if (n_tiles <= 0) return;
  launch_dep(k_tile_order, dim3(1), dim3(1024), 0, s, ranges, n_tiles, order, ctl);
}

namespace {
// Resident CTAs per SM of one K6 instance (persistent grid = that x SMs), set at start-up.
template <int TW, int TH, int BATCH, bool FEW>
int& fwd_occupancy() {
  static int occ = 0;
  return occ;
}

template <int TW, int TH, int BATCH, bool FEW>
void init_forward_kernel() {
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
          &occ, FEW ? k_blend_forward_few<TW, TH, BATCH> : k_blend_forward<TW, TH, BATCH>, TW * TH, 0) != cudaSuccess) {
    cudaGetLastError();
    occ = 0;
  }
  fwd_occupancy<TW, TH, BATCH, FEW>() = occ > 0 ? occ : 1;
}

template <int TW, int TH, int BATCH>
void init_forward_instance() {
  init_forward_kernel<TW, TH, BATCH, false>();
  init_forward_kernel<TW, TH, BATCH, true>();
}

// With few tiles the longest lists' chains are the kernel's duration and most of the chip idles, so four
// candidates go into each round of the walk at 108 registers and two 256-thread CTAs per SM (per candidate
// about 130 instead of 210 cycles).  Up to 16 tiles (of 16 x 16) per SM: 616 -> 452 us on a 128 x 96 image of
// 150k Gaussians (48 tiles), 110 -> 84 at 160 x 120 of 30k (80), 164 -> 133 at 300 x 200 of 120k (247), 32 -> 26
// at 128 x 97 of 3k, 70 -> 57 at 640 x 360 of 60k (920), 61 -> 62 at 960 x 540 of 60k (2040), 91 -> 75 at
// 1000 x 600 of 200k (2394).  Smaller tiles have shorter lists for the same count and stay under the line
// only on smaller images.  With 4346 tiles it depends on the lists, which the host does not know (262 against
// 330 us at 1.9M, but 123 against 110 at 200k with large Gaussians over the image), and with 8160 and more
// the lost occupancy shows (148 against 118, 1042 against 751 on nine views).  Eight per round: 471 us on the
// 48 tiles.  Several sessions on one GPU give part of it back: whole steps of one session, ring scenes of 120k
// to 500k Gaussians at 300 x 200 to 640 x 360, take 394 -> 353 down to 624 -> 587 us, a round of eight sessions'
// steps 931 -> 917 and 2911 -> 2906; but where every list is as long as the next (a cube of 120k in the same
// 300 x 200) 284 -> 284 us alone and 1188 -> 1273 by eight.
bool few_tiles(long long n_tiles, int num_sms) { return n_tiles <= 16ll * num_sms; }

// Persistent grid of one K6 instance: every resident CTA, at most one per tile.
template <int TW, int TH, int BATCH>
long long forward_grid(long long n_tiles, int num_sms) {
  const int occ = few_tiles(n_tiles, num_sms) ? fwd_occupancy<TW, TH, BATCH, true>() : fwd_occupancy<TW, TH, BATCH, false>();
  const long long grid = (long long)num_sms * occ;
  return grid > n_tiles ? n_tiles : grid;
}

template <int TW, int TH, int BATCH>
void launch_forward_instance(const ViewDev* views, int n_views, long long n_tiles, const uint2* ranges,
                             const unsigned* vals, const ProjBuffers& pb, const StepParams* sp, Control* ctl,
                             const int* order, float* image, float* T, unsigned* last, unsigned* gp, float4* ckpt,
                             unsigned* cmask, int* chunk_tile, int* tile_chunks, unsigned* tile_done, int num_sms,
                             cudaStream_t s) {
  launch_dep(few_tiles(n_tiles, num_sms) ? k_blend_forward_few<TW, TH, BATCH> : k_blend_forward<TW, TH, BATCH>,
      dim3((unsigned)forward_grid<TW, TH, BATCH>(n_tiles, num_sms)), dim3(TW * TH), 0, s, views, n_views, n_tiles,
      ranges, vals, pb, sp, ctl, order, image, T, last, gp, ckpt, cmask, chunk_tile, tile_chunks, tile_done);
}
}  // namespace

// The compiled (tile shape, batch) instances; the first is the default.
#define GS_TILINGS(X) X(16, 16, 256) X(16, 16, 128) X(16, 8, 256) X(16, 8, 128) X(8, 8, 128) X(8, 8, 64) X(32, 8, 256)

int tiling_candidates(Tiling* out, int cap) {
  int n = 0;
#define GS_LIST(W, H, B)            \
  if (n < cap && out) out[n] = Tiling{W, H, B}; \
  ++n;
  GS_TILINGS(GS_LIST)
#undef GS_LIST
  return n;
}

bool tiling_supported(const Tiling& t) {
#define GS_SUP(W, H, B) \
  if (t.tw == W && t.th == H && t.batch == B) return true;
  GS_TILINGS(GS_SUP)
#undef GS_SUP
  return false;
}

void launch_blend_forward(const Tiling& tl, const ViewDev* views, int n_views, long long n_tiles, const uint2* ranges,
                          const unsigned* vals, const ProjBuffers& pb, const StepParams* sp, Control* ctl,
                          const int* order, float* image, float* T, unsigned* last, unsigned* gp, float4* ckpt,
                          unsigned* cmask, int* chunk_tile, int* tile_chunks, unsigned* tile_done, int num_sms,
                          cudaStream_t s) {
  if (n_tiles <= 0) return;
#define GS_FWD(W, H, B)                                                                                              \
  if (tl.tw == W && tl.th == H && tl.batch == B) {                                                                  \
    launch_forward_instance<W, H, B>(views, n_views, n_tiles, ranges, vals, pb, sp, ctl, order, image, T, last, gp, \
                                     ckpt, cmask, chunk_tile, tile_chunks, tile_done, num_sms, s);                \
    return;                                                                                                        \
  }
  GS_TILINGS(GS_FWD)
#undef GS_FWD
}

long long forward_warps(const Tiling& tl, long long n_tiles, int num_sms) {
  if (n_tiles <= 0) return 0;
#define GS_FWDW(W, H, B) \
  if (tl.tw == W && tl.th == H && tl.batch == B) return forward_grid<W, H, B>(n_tiles, num_sms) * (W * H / 32);
  GS_TILINGS(GS_FWDW)
#undef GS_FWDW
  return 0;
}

// ---------------------------------------------------------------------------------------------
// K8
// ---------------------------------------------------------------------------------------------
// 1 / x for x in [1 - kAlphaMax, 1]: rcp.approx.ftz is within 1 ulp, and neither x nor 1 / x is near the
// denormal range.
__device__ __forceinline__ float fast_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

constexpr int kBwdWarps = 4;
constexpr unsigned kClaimWords = 2;  // per pair of warps that share an item
constexpr int kGroup = 3;  // Gaussians whose gradient terms are summed together (3 x 9 <= 32 lanes)
constexpr int kBwdPairs = 2;  // packed pixel pairs per lane (4 pixels, 128 per round)

template <int PIX>
struct BwdWarp {
  float4 a[kChunk], b[kChunk], c[kChunk];  // the chunk's Gaussians (records A, B, C)
  uint2 act[PIX];                          // compacted (slot, mask) of the pixels to visit
  float red[kGroup * 9][36];               // per term of a group of 3 Gaussians: the 32 lanes' values
                                           // (rows padded to 16-byte multiples for vector reads)
  float acc[kChunk][9];                    // per Gaussian of the chunk: running gradient sums
};

// SPLIT: the two warps of a pair share each item, one taking the even rounds of 128 pixels and one the
// odd ones; the sums of both are added in that order, so the result is the same bits.
template <int TW, int TH, bool LOAD, bool SPLIT>
__global__ void __launch_bounds__(kBwdWarps * 32, 4) k_blend_backward(
    const ViewDev* __restrict__ views, int n_views, long long n_tiles, const uint2* __restrict__ ranges,
    const unsigned* __restrict__ vals, const ProjBuffers pb, Control* __restrict__ ctl,
    const float* __restrict__ image, const float* __restrict__ dimage, const float4* __restrict__ ckpt,
    const unsigned* __restrict__ cmask, const int* __restrict__ chunk_tile, const int* __restrict__ tile_chunks,
    float4* __restrict__ ginst, const unsigned* __restrict__ gp, const StepParams* __restrict__ sp) {
  dep_wait();
  dep_release();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  using Sh = Shape<TW, TH>;
  constexpr int kPix = Sh::kPix;
  BwdWarp<kPix>& S = reinterpret_cast<BwdWarp<kPix>*>(smem_raw)[warp];
  if (step_void(ctl)) return;
  // Eq. 9-10: dL/dG_p = lambda_load (G_p - mean) / (N std) over the N pixels with G_p > 0 (K6's
  // moments of all the step's views); it reaches alpha through the soft count, the sum of the
  // blended Gaussians' alphas.  load_a = lambda_load / (N std), load_mu = mean; off without G_p.
  float load_a = 0.f, load_mu = 0.f;
  if (LOAD && ctl->gp_pixels > 0ull) {
    const double np = (double)ctl->gp_pixels, mean = (double)ctl->blended / np;
    const double var = (double)ctl->gp_sq / np - mean * mean;
    if (var > 0.0) {
      load_a = (float)((double)sp->lambda_load / (np * sqrt(var)));
      load_mu = (float)mean;
    }
  }
  // row sums of the conic's terms (2-4) carry the factors -1/2, -1, -1/2 of their products
  const int row_gi = lane / 9, row_term = lane - 9 * row_gi;
  const float row_scale = row_term == 3 ? -1.f : (row_term == 2 || row_term == 4 ? -0.5f : 1.f);
  const unsigned long long M = ctl->m_total;
  const long long n_ids = (long long)(M >> 5) + n_tiles + 1;
  const unsigned lt = (1u << lane) - 1u;
  const int part = SPLIT ? warp & 1 : 0;
  const auto pair_sync = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(1 + (warp >> 1)) : "memory"); };
  // A pair's claims alternate between two words: an id without a chunk sends both warps straight to the next
  // claim, so the even warp may store that one before the odd warp has read this one.  The store after it,
  // to this word again, lies behind the next turn's barrier, which the odd warp reaches only after its read.
  __shared__ unsigned s_claim[kBwdWarps / 2][kClaimWords];
  for (unsigned turn = 0;; ++turn) {
    long long id = 0;
    if (SPLIT) {
      unsigned* claim = &s_claim[warp >> 1][turn % kClaimWords];
      if (part == 0 && lane == 0) *claim = atomicAdd(&ctl->bwd_work, 1u);
      pair_sync();  // (also: the even warp is through with the odd one's sums)
      id = (long long)*claim;
    } else {
      if (lane == 0) id = (long long)atomicAdd(&ctl->bwd_work, 1u);
      id = __shfl_sync(0xffffffffu, id, 0);
    }
    if (id >= n_ids) break;
    const int tp1 = chunk_tile[id];
    if (tp1 == 0) continue;
    const long long t = tp1 - 1;
    const uint2 rg = ranges[t];
    const unsigned start = rg.x;
    const int L = (int)(rg.y - rg.x);
    const int k = (int)(id - chunk_base(start, t));
    const int base = k * kChunk;
    const int cnt = min(kChunk, L - base);
    const int v = view_of_tile(views, n_views, t);
    const ViewDev& V = views[v];
    const int local = (int)(t - V.tile_base);
    const int tx = local % V.gx, ty = local / V.gx;
    const long long cid = id;

    unsigned long long e = 0;
    if (lane < cnt) {
      const unsigned rec = vals[start + base + lane];
      S.a[lane] = pb.xyo[rec];
      S.b[lane] = pb.conic[rec];
      S.c[lane] = pb.rgb[rec];
      const uint2 rc = pb.rect[rec];
      const unsigned x0 = rc.x & 0xffffu, x1 = rc.x >> 16, y0 = rc.y & 0xffffu;
      e = (unsigned long long)pb.offsets[rec] + (unsigned long long)((ty - (int)y0) * (int)(x1 - x0) + (tx - (int)x0));
    }
#pragma unroll
    for (int c = 0; c < 9; ++c) S.acc[lane][c] = 0.f;
    // Chunks past tile_chunks[t] were never reached by any pixel: all gradients are zero.
    int n_act = 0;
    if (k < tile_chunks[t]) {
      // compact the pixels that blended at least one Gaussian of this chunk
#pragma unroll
      for (int r = 0; r < kPix / 32; ++r) {
        const int slot = r * 32 + lane;
        const unsigned mask = cmask[cid * kPix + slot];
        const unsigned ball = __ballot_sync(0xffffffffu, mask != 0u);
        if (mask) S.act[n_act + __popc(ball & lt)] = make_uint2((unsigned)slot, mask);
        n_act += __popc(ball);
      }
    }
    __syncwarp();
    const long long HW = (long long)V.W * V.H;
    const float* img = image + 3 * V.pix_base;
    const float* dimg = dimage + 3 * V.pix_base;
    for (int r0 = part * 64 * kBwdPairs; r0 < n_act; r0 += (SPLIT ? 2 : 1) * 64 * kBwdPairs) {
      // this lane's pixels act[r0 + 32 h + lane], h = 0 .. 2 kBwdPairs - 1, pair p holding pixels
      // 2p (.x) and 2p + 1 (.y): dL/dC, the rendered colour, the state at the chunk start, minus
      // the pixel coordinates
      unsigned mk[2 * kBwdPairs];
      float2 d0[kBwdPairs], d1[kBwdPairs], d2[kBwdPairs], P0[kBwdPairs], P1[kBwdPairs], P2[kBwdPairs];
      float2 T[kBwdPairs], F0[kBwdPairs], F1[kBwdPairs], F2[kBwdPairs], npx[kBwdPairs], npy[kBwdPairs];
      float2 LW[kBwdPairs];  // dL/dG_p of the load term per pixel (0 without it)
      unsigned any = 0u;
#pragma unroll
      for (int pp = 0; pp < kBwdPairs; ++pp) {
        float st[2][13];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int i = r0 + 32 * (2 * pp + h) + lane;
          const uint2 pm = i < n_act ? S.act[i] : make_uint2(0u, 0u);
          mk[2 * pp + h] = pm.y;
          any |= pm.y;
          float* q = st[h];
          q[0] = q[1] = q[2] = q[3] = q[4] = q[5] = 0.f;
          q[6] = 1.f;
          q[7] = q[8] = q[9] = q[10] = q[11] = q[12] = 0.f;
          if (pm.y) {
            int ox, oy;
            Sh::slot_xy((int)pm.x, ox, oy);
            const int px = tx * TW + ox, py = ty * TH + oy;
            const long long pix = (long long)py * V.W + px;
            q[0] = dimg[pix];
            q[1] = dimg[HW + pix];
            q[2] = dimg[2 * HW + pix];
            q[3] = img[pix];
            q[4] = img[HW + pix];
            q[5] = img[2 * HW + pix];
            if (k > 0) {
              const float4 ck = ckpt[cid * kPix + pm.x];
              q[6] = ck.x;
              q[7] = ck.y;
              q[8] = ck.z;
              q[9] = ck.w;
            }
            q[10] = -(float)px;
            q[11] = -(float)py;
            if (LOAD) q[12] = load_a * ((float)gp[V.pix_base + pix] - load_mu);
          }
        }
        d0[pp] = make_float2(st[0][0], st[1][0]);
        d1[pp] = make_float2(st[0][1], st[1][1]);
        d2[pp] = make_float2(st[0][2], st[1][2]);
        P0[pp] = make_float2(st[0][3], st[1][3]);
        P1[pp] = make_float2(st[0][4], st[1][4]);
        P2[pp] = make_float2(st[0][5], st[1][5]);
        T[pp] = make_float2(st[0][6], st[1][6]);
        F0[pp] = make_float2(st[0][7], st[1][7]);
        F1[pp] = make_float2(st[0][8], st[1][8]);
        F2[pp] = make_float2(st[0][9], st[1][9]);
        npx[pp] = make_float2(st[0][10], st[1][10]);
        npy[pp] = make_float2(st[0][11], st[1][11]);
        LW[pp] = make_float2(st[0][12], st[1][12]);
      }
      const float2 one2 = make_float2(1.f, 1.f), neg2 = make_float2(-1.f, -1.f);
      // The round's pixels walk the union of their Gaussians in list order, three at a time.  A
      // pixel that did not blend a Gaussian takes it with G = 0: alpha = 0 leaves its
      // transmittance and front colour exactly as they were and zeroes its nine terms, so the walk
      // has no per-pixel branch.  Each lane adds its pixels' terms; the 27 terms of a group are
      // then summed over the lanes through shared memory (fixed order).
      unsigned uni = __reduce_or_sync(0xffffffffu, any);
      while (uni) {
        int qs[kGroup];
        int ng = 0;
#pragma unroll
        for (int gi = 0; gi < kGroup; ++gi) {
          qs[gi] = 0;
          // the nine terms summed over this lane's pixel pairs, both halves kept apart until the end
          float2 g2[9];
#pragma unroll
          for (int j = 0; j < 9; ++j) g2[j] = make_float2(0.f, 0.f);
          if (uni) {
            const int q = __ffs(uni) - 1;
            uni &= uni - 1u;
            qs[gi] = q;
            ng = gi + 1;
            const float4 xy = S.a[q], co = S.b[q], c = S.c[q];
            const float2 A2 = make_float2(co.x, co.x), B2 = make_float2(co.y, co.y), C2 = make_float2(co.z, co.z);
            const float2 cx = make_float2(c.x, c.x), cy = make_float2(c.y, c.y), cz = make_float2(c.z, c.z);
            const float2 A2x2 = make_float2(2.f * co.x, 2.f * co.x), C2x2 = make_float2(2.f * co.z, 2.f * co.z);
#pragma unroll
            for (int pp = 0; pp < kBwdPairs; ++pp) {
              const bool ba = (mk[2 * pp] >> q) & 1u, bb = (mk[2 * pp + 1] >> q) & 1u;
              if (!(ba || bb)) continue;
              const float2 dx = __fadd2_rn(make_float2(xy.x, xy.x), npx[pp]);
              const float2 dy = __fadd2_rn(make_float2(xy.y, xy.y), npy[pp]);
              // the forward's exponent, rounding step for rounding step (splat_power)
              const float2 pw =
                  __ffma2_rn(dx, __ffma2_rn(A2, dx, __fmul2_rn(B2, dy)), __fmul2_rn(__fmul2_rn(C2, dy), dy));
              const float2 G = make_float2(ba ? splat_exp(pw.x) : 0.f, bb ? splat_exp(pw.y) : 0.f);
              const float2 oG = __fmul2_rn(make_float2(c.w, c.w), G);
              const float2 alpha = make_float2(fminf(kAlphaMax, oG.x), fminf(kAlphaMax, oG.y));
              const float2 w = __fmul2_rn(alpha, T[pp]);
              const float2 n0 = __ffma2_rn(cx, w, F0[pp]);
              const float2 n1 = __ffma2_rn(cy, w, F1[pp]);
              const float2 n2 = __ffma2_rn(cz, w, F2[pp]);
              // colour behind = rendered colour (incl. background) - colour in front incl. this one
              const float2 behind2 = __fmul2_rn(d2[pp], __ffma2_rn(n2, neg2, P2[pp]));
              const float2 DS = __ffma2_rn(d0[pp], __ffma2_rn(n0, neg2, P0[pp]),
                                           __ffma2_rn(d1[pp], __ffma2_rn(n1, neg2, P1[pp]), behind2));
              // dL/dalpha = sum_ch dL/dC_ch (c_ch T - behind_ch / (1 - alpha)); no gradient to the
              // opacity and footprint where alpha was clamped
              const float2 cd = __ffma2_rn(cx, d0[pp], __ffma2_rn(cy, d1[pp], __fmul2_rn(cz, d2[pp])));
              const float2 ninv = make_float2(-fast_rcp(1.f - alpha.x), -fast_rcp(1.f - alpha.y));
              float2 dal = __ffma2_rn(DS, ninv, __fmul2_rn(T[pp], cd));
              if (LOAD) dal = __fadd2_rn(dal, LW[pp]);  // + dL/dG_p x d alpha / d alpha
              dal.x = oG.x > kAlphaMax ? 0.f : dal.x;
              dal.y = oG.y > kAlphaMax ? 0.f : dal.y;
              const float2 dpow = __fmul2_rn(dal, alpha);
              const float2 ex = __ffma2_rn(A2x2, dx, __fmul2_rn(B2, dy));
              const float2 ey = __ffma2_rn(B2, dx, __fmul2_rn(C2x2, dy));
              const float2 pdx = __fmul2_rn(dpow, dx), pdy = __fmul2_rn(dpow, dy);
              g2[0] = __ffma2_rn(dpow, ex, g2[0]);
              g2[1] = __ffma2_rn(dpow, ey, g2[1]);
              g2[2] = __ffma2_rn(pdx, dx, g2[2]);
              g2[3] = __ffma2_rn(pdx, dy, g2[3]);
              g2[4] = __ffma2_rn(pdy, dy, g2[4]);
              g2[5] = __ffma2_rn(dal, G, g2[5]);
              g2[6] = __ffma2_rn(w, d0[pp], g2[6]);
              g2[7] = __ffma2_rn(w, d1[pp], g2[7]);
              g2[8] = __ffma2_rn(w, d2[pp], g2[8]);
              T[pp] = __fmul2_rn(T[pp], __ffma2_rn(alpha, neg2, one2));
              F0[pp] = n0;
              F1[pp] = n1;
              F2[pp] = n2;
            }
          }
#pragma unroll
          for (int j = 0; j < 9; ++j) S.red[9 * gi + j][lane] = g2[j].x + g2[j].y;
        }
        __syncwarp();
        if (lane < 9 * ng) {
          // the term's 32 values: eight 16-byte reads, four running sums (fixed order)
          const float4* row = reinterpret_cast<const float4*>(S.red[lane]);
          float2 sa = make_float2(row[0].x, row[0].y), sb = make_float2(row[0].z, row[0].w);
#pragma unroll
          for (int k = 1; k < 8; ++k) {
            const float4 x = row[k];
            sa = __fadd2_rn(sa, make_float2(x.x, x.y));
            sb = __fadd2_rn(sb, make_float2(x.z, x.w));
          }
          const float sum = row_scale * ((sa.x + sa.y) + (sb.x + sb.y));
          const int q = row_gi == 0 ? qs[0] : (row_gi == 1 ? qs[1] : qs[2]);
          S.acc[q][row_term] += sum;
        }
        __syncwarp();
      }
    }
    __syncwarp();
    if (SPLIT) {
      pair_sync();
      if (part != 0) continue;
      const BwdWarp<kPix>& O = reinterpret_cast<BwdWarp<kPix>*>(smem_raw)[warp + 1];
#pragma unroll
      for (int c = 0; c < 9; ++c) S.acc[lane][c] += O.acc[lane][c];
    }
    if (lane < cnt) {
      const float* a = S.acc[lane];
      ginst[3 * e] = make_float4(a[0], a[1], a[2], a[3]);
      ginst[3 * e + 1] = make_float4(a[4], a[5], a[6], a[7]);
      ginst[3 * e + 2] = make_float4(a[8], 0.f, 0.f, 0.f);
    }
    __syncwarp();
  }
}

namespace {
template <int TW, int TH, bool LOAD, bool SPLIT>
int& bwd_occupancy() {
  static int occ = 0;
  return occ;
}

template <int TW, int TH, bool LOAD, bool SPLIT>
void init_backward_instance() {
  const int smem = (int)(sizeof(BwdWarp<TW * TH>) * kBwdWarps);
  cudaFuncSetAttribute(k_blend_backward<TW, TH, LOAD, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_blend_backward<TW, TH, LOAD, SPLIT>, kBwdWarps * 32, smem) !=
      cudaSuccess) {
    cudaGetLastError();
    occ = 0;
  }
  bwd_occupancy<TW, TH, LOAD, SPLIT>() = occ > 0 ? occ : 1;
}

template <int TW, int TH, bool LOAD, bool SPLIT>
void launch_backward_kernel(const ViewDev* views, int n_views, long long n_tiles, const uint2* ranges,
                            const unsigned* vals, const ProjBuffers& pb, Control* ctl, const float* image,
                            const float* dimage, const float4* ckpt, const unsigned* cmask, const int* chunk_tile,
                            const int* tile_chunks, float4* ginst, const unsigned* gp, const StepParams* sp,
                            int num_sms, cudaStream_t s) {
  launch_dep(k_blend_backward<TW, TH, LOAD, SPLIT>, dim3(num_sms * bwd_occupancy<TW, TH, LOAD, SPLIT>()),
      dim3(kBwdWarps * 32), sizeof(BwdWarp<TW * TH>) * kBwdWarps, s, views, n_views, n_tiles, ranges, vals, pb, ctl,
      image, dimage, ckpt, cmask, chunk_tile, tile_chunks, ginst, gp, sp);
}

// A warp works on an item for 25 - 45 us (about 40 Gaussians in its two rounds, 0.6 - 1 us each), so with few
// items the kernel lasts as long as the slowest of them: two warps share each up to one item per pair of warps
// on the chip, and up to eight where the lists are short (about 300 entries each, 380 of capacity).  One warp
// against two: 33 -> 25 us at 220 items (at most, by the buffers), 39 -> 26 at 1.6k, 36 -> 33 at 2.8k (297 entries
// per list), 45 -> 43 at 3.6k (75), 60 -> 56 at 5.9k (78), 81 -> 80 at 9.0k (84); with 14k and more the second head
// per item shows.  In longer lists most items lie behind the depth where the pixels stop, and the second
// head is all there is: 40 and 40 us at 3.2k items (377 per list), a whole step 271 -> 283 us at 11k (1500), and
// with several sessions on the chip more: a round of eight sessions' steps 338 -> 387 us (30k Gaussians at 160
// x 120) without and with sharing there.
template <int TW, int TH, bool LOAD>
void launch_backward_instance(const ViewDev* views, int n_views, long long n_tiles, const uint2* ranges,
                              const unsigned* vals, const ProjBuffers& pb, Control* ctl, const float* image,
                              const float* dimage, const float4* ckpt, const unsigned* cmask, const int* chunk_tile,
                              const int* tile_chunks, float4* ginst, const unsigned* gp, const StepParams* sp,
                              long long m_cap, int num_sms, cudaStream_t s) {
  if constexpr (TW * TH > 64 * kBwdPairs) {
    const long long items = (m_cap >> 5) + n_tiles + 1;  // at most
    const long long per_pair = m_cap <= 380 * n_tiles ? 8 : 1;
    if (items <= per_pair * num_sms * bwd_occupancy<TW, TH, LOAD, true>() * (kBwdWarps / 2)) {
      launch_backward_kernel<TW, TH, LOAD, true>(views, n_views, n_tiles, ranges, vals, pb, ctl, image, dimage, ckpt,
                                                 cmask, chunk_tile, tile_chunks, ginst, gp, sp, num_sms, s);
      return;
    }
  }
  launch_backward_kernel<TW, TH, LOAD, false>(views, n_views, n_tiles, ranges, vals, pb, ctl, image, dimage, ckpt,
                                              cmask, chunk_tile, tile_chunks, ginst, gp, sp, num_sms, s);
}

template <int TW, int TH, bool LOAD>
void init_backward_instances() {
  init_backward_instance<TW, TH, LOAD, false>();
  if constexpr (TW * TH > 64 * kBwdPairs) init_backward_instance<TW, TH, LOAD, true>();
}
}  // namespace

void init_blend_attributes() {
#define GS_INIT(W, H, B)              \
  init_forward_instance<W, H, B>();   \
  init_backward_instances<W, H, false>(); \
  init_backward_instances<W, H, true>();
  GS_TILINGS(GS_INIT)
#undef GS_INIT
}

void launch_blend_backward(const Tiling& tl, const ViewDev* views, int n_views, long long n_tiles, const uint2* ranges,
                           const unsigned* vals, const ProjBuffers& pb, Control* ctl, const float* image,
                           const float* dimage, const float4* ckpt, const unsigned* cmask, const int* chunk_tile,
                           const int* tile_chunks, float4* ginst, const unsigned* gp, bool load, const StepParams* sp,
                           long long m_cap, int num_sms, cudaStream_t s) {
  // the backward depends on the tile shape only
#define GS_BWD(W, H, B)                                                                                          \
  if (tl.tw == W && tl.th == H) {                                                                               \
    (load ? launch_backward_instance<W, H, true> : launch_backward_instance<W, H, false>)(                     \
        views, n_views, n_tiles, ranges, vals, pb, ctl, image, dimage, ckpt, cmask, chunk_tile, tile_chunks,    \
        ginst, gp, sp, m_cap, num_sms, s);                                                                     \
    return;                                                                                                    \
  }
  GS_TILINGS(GS_BWD)
#undef GS_BWD
}

}  // namespace gs
