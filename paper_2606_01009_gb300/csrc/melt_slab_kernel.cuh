// Device side of the slab kernel, included by melt_slab.cu.
#pragma once
// The FP32 form of the projection (Eq. 6) on the tensor cores.
//
// Every FP32 sample and every basis value is split exactly into three BF16
// parts (hi = rn(v), mid = rn(v - hi), lo = rn(v - hi - mid): 3 x 8 bits), and
// the six products of parts whose weight is at least 2^-16 of the leading one
// are formed: hi hi, hi mid, mid hi, mid mid, hi lo, lo hi.  What is dropped
// is below 2^-24 of each product, the size of an FP32 rounding.
//
// Accumulation.  The tensor core truncates its FP32 accumulator at every MMA,
// a bias that grows with the number of MMAs (25 of them put -3.0e-6 dB on the
// bins near the frame maximum, where the FFMA kernel's error is 2.7e-6 dB
// RMS).  So K is cut into chunks of at most kps K-steps; each chunk starts
// from zero, adds its five small products first (they are 2^-8 of the sum, so
// their truncation does not count) and its hi hi products last, and the epilogue
// adds the chunks up in FP32 registers with round-to-nearest.
//
// Bound.  Six products make 6 x 128,000 flops a frame at (N, M) = (400, 80):
// 147 TFLOP for the 64 x 30 s batch, tensor-bound (its 184 MB of samples and
// features take a third of that time).  So everything else has to stay out of
// the MMAs' way: the basis (384 KB in three parts) does not fit shared memory
// and neither do two converted tiles (125 KB each), but one K slab of both
// does.  A slab is 16 columns of the polyphase rows Z[u][r] = x[(t0+u) H + r]
// (all rows of the tile) and, for each slice j, the K-step n = j H + r of the
// basis; the slices of a slab read the same A slab at row offset j, so every
// sample is converted once.  Slabs and K-steps flow through two rings.
//
// Clusters of two CTAs share each MMA (cta_group::2, M = 256: two tiles): the
// even CTA holds the W_r rows of a K-step, the odd one the W_i rows, so each
// streams half of the basis.  More than 80 Mel bins run as blocks of at most
// 80 (the epilogue's accumulators live in registers); a short batch is cut
// into more blocks to use more SMs.
//
// Warps: 0-7 epilogue (two per TMEM lane quarter, each half of the block's
// bins), 8-10 and 12-14 converters (each takes whole slabs by itself: its samples
// arrive by asynchronous copies in a staging area of its own, one arrival per
// slab), 11 MMA issue (odd CTA: forwards its basis fills to the even one), 15
// basis producer and L2 prefetch.
//
// Code size counts here: the issue thread's few hundred instructions per chunk
// run once per 1200 clocks between three other warps on its scheduler, and it
// fetches them anew each time.  With converters unrolled over 17 register
// quads the 64 x 30 s batch took 132 us, of which two thirds of the MMAs could
// be left out for 11 us.
//
// Samples the split cannot hold.  An infinity or NaN (whose parts would also
// turn the sums of frames that only meet it at a zero basis row into NaN), or
// sums that overflow: a frame whose power is not finite is recomputed by its
// epilogue thread with FP32 FFMAs.
#include <cuda_bf16.h>

#include "melt_slab.h"
#include "melt_tc.h"
#include "sm100_ptx.cuh"

namespace melt {
namespace slab {

using namespace ptx;

constexpr int kF = kTileFrames;
// Warps 0-7 epilogue; 8-10 and 12-14 converters; 11 and 15, on the scheduler
// that no converter shares, MMA issue and basis producer.
constexpr int kEpiWarps = 8, kCvtWarps = 6, kCvtWarp0 = 8, kMmaWarp = 11, kBWarp = 15;
constexpr int kThreads = 512;  // 128 registers a thread
constexpr int kBlockBins = 80;  // Mel bins of a block: 2 x 40 accumulators per epilogue thread
constexpr int kGroupsPerWarp = kBlockBins / 16;  // groups of 8 bins per epilogue warp
constexpr int kNacc = 3;        // TMEM accumulators of 2 x kBlockBins columns
constexpr int kStageRows = 136; // rows of a slab that a converter warp stages at a time
constexpr uint32_t kStageBytes = kStageRows * 64u;
constexpr int kMaxSlots = 8;    // slots of either ring

struct SlabParams {
  const float* wave;
  const TileDesc* tiles;
  const uint8_t* img;  // [half][K-step][group of 8 bins][part][core column][8 rows x 16 B]
  const float* dct;
  const float* w32;
  float* out;
  int* err;
  float eps;
  int n_tiles, n_pairs, mp;
  int N, H, M, J, n_slab, ksteps, groups;
  int zrows;           // Z rows of a tile: 128 + J - 1
  int n_last;          // samples of the last slice: N - (J - 1) H
  int nblk, wbg;       // blocks of wbg groups of 8 bins (the last may have fewer)
  int inner;           // blocks a unit takes in turn (MFCC: all of them, else 1)
  int n_units;
  int kps;             // K-steps per basis slot (one accumulation chunk)
  int NA, NB;          // slots of the A and basis rings
  int ncv;             // converter warps at work: at most NA (a warp that took slab g waits for the slot of
                       // slab g + ncv by one parity bit, which tells only neighbouring phases apart)
  uint32_t lbo_a, a_part, a_slot, b_slot, step_bytes;
  uint32_t off_a, off_b, off_st, off_bar, off_misc, off_dct, off_part;
  int n_mfcc, n_out;
};

struct SlabBars {
  int a_full, a_empty, b_full, b_empty, t_full, t_empty, half, drain, total;
  __host__ __device__ SlabBars(int NA, int NB) {
    a_full = 0;               // both CTAs' converters (even CTA's copy is used)
    a_empty = a_full + NA;    // MMA commit, both CTAs
    b_full = a_empty + NA;    // this CTA's basis copies; even CTA: and the odd one's signal that its own are in
    b_empty = b_full + NB;    // MMA commit, both CTAs
    t_full = b_empty + NB;    // MMA commit, both CTAs
    t_empty = t_full + kNacc; // both CTAs' epilogues (even CTA's copy is used)
    half = t_empty + kNacc;   // MFCC, per lane quarter: part buffers 0, 1 filled; [16 B on] taken
    drain = half + 16;
    total = drain + 1;
  }
};

struct Ctx {
  uint32_t sbase, rank;
  int cluster, n_clusters;
  volatile int* abort;
};

// Ring position: slot and the parity its next completion has.
struct Ring {
  int slot = 0;
  uint32_t phase = 0;
  __device__ __forceinline__ void next(int n) {
    if (++slot == n) {
      slot = 0;
      phase ^= 1;
    }
  }
};

static __device__ __forceinline__ uint32_t bar_at(const SlabParams& p, const Ctx& c, int i) {
  return c.sbase + p.off_bar + 8 * i;
}

// Bounded wait, short where the phase has completed or is about to: the clock
// and the abort flag are looked at every 16 polls, out of line.
static __device__ __noinline__ bool wait_gives_up(uint64_t& t0, volatile int* abort, int* err) {
  if (*abort) return true;
  const uint64_t t = globaltimer();
  if (t0 == 0) t0 = t;
  if (t - t0 <= kWaitLimitNs) return false;
  atomicOr(err, kErrTimeout);
  *abort = 1;
  return true;
}
static __device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity, volatile int* abort, int* err) {
  uint64_t t0 = 0;
  for (uint32_t it = 1; !mbar_try_wait(bar, parity); ++it)
    if ((it & 15) == 0 && wait_gives_up(t0, abort, err)) return false;
  return true;
}
// The same for a whole warp: every lane polls, all leave together.
static __device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int* abort, int* err) {
  uint64_t t0 = 0;
  for (uint32_t it = 1; !__all_sync(0xffffffffu, mbar_try_wait(bar, parity)); ++it)
    if ((it & 15) == 0 && __any_sync(0xffffffffu, wait_gives_up(t0, abort, err))) return false;
  return true;
}

static __device__ __forceinline__ void warp_arrive_leader(uint32_t local_bar) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive_cluster(mapa_shared(local_bar, 0));
}

static __device__ __forceinline__ void warp_arrive_local(uint32_t bar) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(bar);
}

// Unit of ordinal i of this cluster: tile pair q and block b; false past the end.
static __device__ __forceinline__ bool unit_at(const SlabParams& p, const Ctx& c, int i, int& q, int& b) {
  const int u = c.cluster + (i / p.inner) * c.n_clusters;
  if (u >= p.n_units) return false;
  if (p.inner > 1) {
    q = u;
    b = i % p.inner;
  } else {
    q = u / p.nblk;
    b = u - q * p.nblk;
  }
  return true;
}

static __device__ __forceinline__ TileDesc tile_of(const SlabParams& p, const Ctx& c, int q) {
  const int t = 2 * q + (int)c.rank;
  if (t < p.n_tiles) return p.tiles[t];
  TileDesc td;
  td.in_off = 0;
  td.out_row = 0;
  td.n_frames = 0;
  td.n_samples = 0;
  td.group = 0;
  td.clip = -1;
  return td;
}

static __device__ __forceinline__ int blk_groups(const SlabParams& p, int b) { return min(p.wbg, p.groups - b * p.wbg); }

// Slices with samples in slab kk (the last slice may be shorter than H).
static __device__ __forceinline__ int slab_steps(const SlabParams& p, int kk) {
  return 16 * kk < p.n_last ? p.J : p.J - 1;
}

// Bulk prefetch of a tile's samples into L2 (pieces of <= 32 KB).
static __device__ __forceinline__ void prefetch_span(const SlabParams& p, const TileDesc& td) {
  if (td.n_frames == 0) return;
  const int avail = min((td.n_samples & 3) ? (td.n_samples | 3) + 1 : td.n_samples, (td.n_frames + p.J - 1) * p.H);
  for (int o = 0; o < avail; o += 8192) prefetch_l2(p.wave + td.in_off + o, (uint32_t)min(8192, avail - o) * 4u);
}

// ---- basis producer: each unit's K-steps of this CTA's half, a slot per chunk
template <int P>
static __device__ void basis_producer(const SlabParams& p, const Ctx& c, const SlabBars& B) {
  const uint64_t pol = policy_evict_last();
  const uint8_t* half = p.img + (size_t)c.rank * p.ksteps * p.step_bytes;
  Ring r;
  int issued = 0, q, b;
  bool ok = true;
  for (int i = 0; ok && unit_at(p, c, i, q, b); ++i) {
    const int ng = blk_groups(p, b);
    const uint32_t blk = (uint32_t)ng * P * 256u;
    const uint8_t* src = half + (size_t)b * p.wbg * P * 256u;
    bool ahead = false;  // the next unit's span has been sent for
    for (int kk = 0; ok && kk < p.n_slab; ++kk) {
      const int js = slab_steps(p, kk);
      for (int j0 = 0; j0 < js; j0 += p.kps) {
        if (!bar_wait(bar_at(p, c, B.b_empty + r.slot), r.phase ^ 1, c.abort, p.err)) {
          ok = false;
          break;
        }
        const int n = min(p.kps, js - j0);
        const uint32_t full = bar_at(p, c, B.b_full + r.slot);
        const uint32_t dst = c.sbase + p.off_b + r.slot * p.b_slot;
        mbar_arrive_expect_tx(full, blk * n);
        if (blk == p.step_bytes) {
          bulk_g2s_hint(dst, src, blk * n, full, pol);
        } else {
          for (int k = 0; k < n; ++k) bulk_g2s_hint(dst + k * blk, src + (size_t)k * p.step_bytes, blk, full, pol);
        }
        src += (size_t)n * p.step_bytes;
        ++issued;
        r.next(p.NB);
        if (!ahead) {
          // L2 prefetch of the samples, one unit ahead of the converters' copies
          ahead = true;
          if (i == 0) pdl_wait();
          int qn, bn;
          if (unit_at(p, c, i + 1, qn, bn) && (qn != q || i == 0)) prefetch_span(p, tile_of(p, c, qn));
        }
      }
    }
  }
  // every issued copy has landed before the CTA can exit
  volatile int never = 0;
  for (int k = max(0, issued - p.NB); k < issued; ++k)
    mbar_wait(bar_at(p, c, B.b_full + k % p.NB), (k / p.NB) & 1, &never, p.err, kErrTimeout);
}

// ---- odd CTA: one arrival on the even CTA's b_full per filled slot
static __device__ void basis_signal(const SlabParams& p, const Ctx& c, const SlabBars& B) {
  Ring r;
  int q, b;
  for (int i = 0; unit_at(p, c, i, q, b); ++i)
    for (int kk = 0; kk < p.n_slab; ++kk) {
      const int js = slab_steps(p, kk);
      for (int j0 = 0; j0 < js; j0 += p.kps) {
        if (!bar_wait(bar_at(p, c, B.b_full + r.slot), r.phase, c.abort, p.err)) return;
        mbar_arrive_cluster(mapa_shared(bar_at(p, c, B.b_full + r.slot), 0));
        r.next(p.NB);
      }
    }
}

// One MMA of the pair; ACC (accumulate or overwrite) is a constant, so that an
// MMA is a handful of instructions.  (The issue loop is latency bound: with
// the accumulate flag, the part offsets and the K-steps of a chunk computed
// per MMA it took about 200 clocks an MMA; straight-line code under
// elect.sync, whose operands stay in uniform registers, takes 39, below the
// 80 clocks that the MMA itself takes at 80 bins.)
template <bool ACC>
static __device__ __forceinline__ void mma_pair(uint32_t d, uint32_t a, uint32_t a_hi, uint32_t b, uint32_t b_hi,
                                                uint32_t idesc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 x, y;\n\t"
      "mov.b64 x, {%1, %2};\n\tmov.b64 y, {%3, %4};\n\t"
      "setp.ne.u32 p, %6, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], x, y, %5, p;\n\t}\n" ::"r"(d),
      "r"(a), "r"(a_hi), "r"(b), "r"(b_hi), "r"(idesc), "n"(ACC ? 1 : 0));
}

static __device__ __forceinline__ bool elect_one() {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
  return r != 0;
}

// The products of a chunk of NK K-steps into accumulator d.  a, w: descriptors
// (low words) of the first K-step's hi parts (parts 0 hi, 1 mid, 2 lo are ap
// and 16 apart, K-steps 1 row of A and `step` of the basis, in 16-byte units).
// The small products of every K-step first, then the hi hi products.
template <int NK>
static __device__ __forceinline__ void chunk_mmas(uint32_t d, uint32_t a, uint32_t ah, uint32_t w, uint32_t wh,
                                                  uint32_t ap, uint32_t step, uint32_t idesc) {
  const uint32_t am = a + ap, al = am + ap;
#pragma unroll
  for (int k = 0; k < NK; ++k) {
    const uint32_t wk = w + k * step;
    if (k == 0) mma_pair<false>(d, al + k, ah, wk, wh, idesc);
    else mma_pair<true>(d, al + k, ah, wk, wh, idesc);
    mma_pair<true>(d, a + k, ah, wk + 32, wh, idesc);
    mma_pair<true>(d, am + k, ah, wk + 16, wh, idesc);
    mma_pair<true>(d, am + k, ah, wk, wh, idesc);
    mma_pair<true>(d, a + k, ah, wk + 16, wh, idesc);
  }
#pragma unroll
  for (int k = 0; k < NK; ++k) mma_pair<true>(d, a + k, ah, w + k * step, wh, idesc);
}

static __device__ __forceinline__ bool bar_done(uint32_t bar, uint32_t parity) { return mbar_test_wait(bar, parity); }

// ---- even CTA: every MMA of the pair.
// A chunk's 15 to 24 MMAs take 1200 to 1900 clocks at 80 bins.  With its waits,
// ring arithmetic, MMAs and commits one after another this thread took about
// 1650 clocks a chunk and so bounded the kernel; it now looks at the next
// chunk's barriers (all at once) before it issues the MMAs of this one.
template <int P>
static __device__ void mma_issue(const SlabParams& p, const Ctx& c, const SlabBars& B, uint32_t tmem) {
  constexpr uint32_t ah = (128u >> 4) | (1u << 14);         // SBO 128 B
  constexpr uint32_t wh = ((P * 256u) >> 4) | (1u << 14);   // SBO: the next group of 8 bins
  const uint32_t a0 = ((c.sbase + p.off_a) >> 4) | ((p.lbo_a >> 4) << 16);
  const uint32_t b0 = ((c.sbase + p.off_b) >> 4) | ((128u >> 4) << 16);    // LBO 128 B
  const uint32_t ap = p.a_part >> 4, as = p.a_slot >> 4, bs = p.b_slot >> 4;
  const uint32_t a_full = bar_at(p, c, B.a_full), a_empty = bar_at(p, c, B.a_empty);
  const uint32_t b_full = bar_at(p, c, B.b_full), b_empty = bar_at(p, c, B.b_empty);
  const uint32_t t_full = bar_at(p, c, B.t_full), t_empty = bar_at(p, c, B.t_empty);
  const int kps = p.kps, J = p.J, n_last = p.n_last, n_slab = p.n_slab, NA = p.NA, NB = p.NB;
  volatile int* abort = c.abort;
  int* err = p.err;
  Ring ra, rb, rt;
  uint32_t al = a0, bl = b0, d = tmem;
  int i = 0, q, b, kk = 0, j0 = 0, js = slab_steps(p, 0);
  bool more = unit_at(p, c, 0, q, b), ready = false;
  uint32_t ng = more ? (uint32_t)blk_groups(p, b) : 0u;
  while (more) {
    const uint32_t bar_a = a_full + 8 * ra.slot, bar_b = b_full + 8 * rb.slot, bar_t = t_empty + 8 * rt.slot;
    if (!ready && !(bar_wait(bar_a, ra.phase, abort, err) && bar_wait(bar_b, rb.phase, abort, err) &&
                    bar_wait(bar_t, rt.phase ^ 1, abort, err)))
      break;
    tc_fence_after();
    // this chunk, and the step to the next one
    const uint32_t a = al + (uint32_t)j0, w = bl, acc = d, idesc = idesc_f32acc(1u, 2 * kF, 16u * ng);
    const uint32_t step = ng * ((P * 256u) >> 4);
    const uint32_t done_a = a_empty + 8 * ra.slot, done_b = b_empty + 8 * rb.slot, done_t = t_full + 8 * rt.slot;
    const int n = min(kps, js - j0);
    bl += bs;
    rb.next(NB);
    if (rb.slot == 0) bl = b0;
    d += 2 * kBlockBins;
    rt.next(kNacc);
    if (rt.slot == 0) d = tmem;
    j0 += kps;
    const bool slab_end = j0 >= js;
    if (slab_end) {
      j0 = 0;
      al += as;
      ra.next(NA);
      if (ra.slot == 0) al = a0;
      if (++kk == n_slab) {
        kk = 0;
        more = unit_at(p, c, ++i, q, b);
        if (more) ng = (uint32_t)blk_groups(p, b);
      }
      js = 16 * kk < n_last ? J : J - 1;
    }
    const bool ok_a = bar_done(a_full + 8 * ra.slot, ra.phase), ok_b = bar_done(b_full + 8 * rb.slot, rb.phase),
               ok_t = bar_done(t_empty + 8 * rt.slot, rt.phase ^ 1);
    switch (n) {
      case 1: chunk_mmas<1>(acc, a, ah, w, wh, ap, step, idesc); break;
      case 2: chunk_mmas<2>(acc, a, ah, w, wh, ap, step, idesc); break;
      case 3: chunk_mmas<3>(acc, a, ah, w, wh, ap, step, idesc); break;
      default: chunk_mmas<4>(acc, a, ah, w, wh, ap, step, idesc); break;
    }
    mma_commit_pair_mc(done_b, 3);
    mma_commit_pair_mc(done_t, 3);
    if (slab_end) mma_commit_pair_mc(done_a, 3);
    ready = ok_a && ok_b && ok_t;
  }
  // no pair MMA may still be running when either CTA releases TMEM
  mma_commit_pair_mc(bar_at(p, c, B.drain), 3);
}

static __device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);  // a -> low half
  return *reinterpret_cast<const uint32_t*>(&h);
}
static __device__ __forceinline__ float lo_f(uint32_t h) { return __uint_as_float(h << 16); }
static __device__ __forceinline__ float hi_f(uint32_t h) { return __uint_as_float(h & 0xffff0000u); }

// 16 bytes global -> shared through L2; the bytes past `valid` are zero.
static __device__ __forceinline__ void copy_quad(uint32_t dst, const float* src, int valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid) : "memory");
}

// Rows [r0, r0 + kStageRows) of a slab (column r of lane quad qd, row u0 + 8 k)
// into the warp's staging area.  Four lanes take the 16 samples of a row (64
// contiguous bytes), so a warp's copies read whole sectors of 8 rows.
static __device__ __forceinline__ void stage_rows(const SlabParams& p, const float* src, int nsamp, int rows, int r,
                                                  uint32_t st, int r0, int u0) {
  int s = (r0 + u0) * p.H + r;
  const int n = min(rows - r0, kStageRows);
#pragma unroll 4
  for (int u = u0; u < n; u += 8, s += 8 * p.H, st += 512) {
    const int left = r < p.H ? min(max(nsamp - s, 0), 4) : 0;  // samples of the quad before the clip's end
    copy_quad(st, src + (left ? s : 0), 4 * left);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// ---- converters: warp w takes slabs w, w + ncv, ... of the CTA's stream.  Its
// copies of the next slab are in flight while it waits for that slab's slot;
// every lane converts what it copied itself.  Quad qd of row u goes, four BF16
// values of each part, as 8 bytes to core column qd / 2, row u.
template <int P>
static __device__ void convert(const SlabParams& p, const Ctx& c, const SlabBars& B) {
  const int w = (int)(threadIdx.x >> 5) - kCvtWarp0 - (threadIdx.x >= 32 * kMmaWarp ? 1 : 0),
            lane = threadIdx.x & 31;
  const int qd = lane & 3, u0 = lane >> 2;
  const uint32_t to = c.sbase + p.off_a + (uint32_t)(qd >> 1) * p.lbo_a + (uint32_t)(qd & 1) * 8u + 16u * u0;
  const uint32_t st = c.sbase + p.off_st + w * kStageBytes + 16u * lane;
  const uint32_t part = p.a_part;
  if (w >= p.ncv) return;
  int q, b, i = 0, kk = w;  // unit ordinal and slab of it
  Ring ra;
  for (int k = 0; k < w; ++k) ra.next(p.NA);
  while (kk >= p.n_slab) {
    kk -= p.n_slab;
    ++i;
  }
  if (!unit_at(p, c, i, q, b)) return;
  TileDesc td = tile_of(p, c, q);
  int rows = td.n_frames > 0 ? td.n_frames + p.J - 1 : 0;
  stage_rows(p, p.wave + td.in_off, td.n_samples, rows, 16 * kk + 4 * qd, st, 0, u0);
  for (;;) {
    if (!warp_wait(bar_at(p, c, B.a_empty + ra.slot), ra.phase ^ 1, c.abort, p.err)) break;
    const uint32_t slot = to + ra.slot * p.a_slot;
    for (int r0 = 0; r0 < rows; r0 += kStageRows) {
      if (r0 > 0) stage_rows(p, p.wave + td.in_off, td.n_samples, rows, 16 * kk + 4 * qd, st, r0, u0);
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      const int n = min(rows - r0, kStageRows);
      uint32_t at = slot + 16u * r0, from = st;
#pragma unroll 2
      for (int u = u0; u < n; u += 8, at += 128, from += 512) {
        float a0, a1, a2, a3;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(a0), "=f"(a1), "=f"(a2), "=f"(a3) : "r"(from));
#pragma unroll
        for (int t = 0; t < P; ++t) {
          const uint32_t h0 = pack2(a0, a1), h1 = pack2(a2, a3);
          asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(at + t * part), "r"(h0), "r"(h1) : "memory");
          if (t + 1 < P) {
            a0 -= lo_f(h0);
            a1 -= hi_f(h0);
            a2 -= lo_f(h1);
            a3 -= hi_f(h1);
          }
        }
      }
    }
    fence_proxy_async();
    warp_arrive_leader(bar_at(p, c, B.a_full + ra.slot));
    // the warp's next slab
    for (int k = 0; k < p.ncv; ++k) ra.next(p.NA);
    const int before = i;
    kk += p.ncv;
    while (kk >= p.n_slab) {
      kk -= p.n_slab;
      ++i;
    }
    if (i != before) {
      if (!unit_at(p, c, i, q, b)) break;
      td = tile_of(p, c, q);
      rows = td.n_frames > 0 ? td.n_frames + p.J - 1 : 0;
    }
    stage_rows(p, p.wave + td.in_off, td.n_samples, rows, 16 * kk + 4 * qd, st, 0, u0);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");  // no copy is in flight when the CTA exits
}

// ln(S + eps) of one frame (its samples at x) as FP32 FFMAs form it, by a whole
// warp: lane l gets bins m0 + l and m0 + 32 + l (those below `end`).  Where a
// sample is an infinity or a NaN, the finite ones cannot change either sum any
// more (each is an infinity or a NaN), so only the others are added, until
// every power is a NaN.
static __device__ __noinline__ float2 redo_row(const SlabParams& p, const float* x, int m0, int end) {
  const int lane = threadIdx.x & 31;
  const float inf = __int_as_float(0x7f800000);
  bool odd = false;
#pragma unroll 4
  for (int n = lane; n < p.N; n += 32) odd |= !(fabsf(x[n]) < inf);
  const bool only = __any_sync(0xffffffffu, odd);
  const int a = min(m0 + lane, end - 1), b = min(m0 + 32 + lane, end - 1);
  const float2* w = reinterpret_cast<const float2*>(p.w32);  // [sample][bin] of (R, I)
  float ra = 0.f, ia = 0.f, rb = 0.f, ib = 0.f;
  auto add = [&](int n, float v) {
    const float2 wa = w[(size_t)n * p.mp + a], wb = w[(size_t)n * p.mp + b];
    ra = fmaf(v, wa.x, ra);
    ia = fmaf(v, wa.y, ia);
    rb = fmaf(v, wb.x, rb);
    ib = fmaf(v, wb.y, ib);
  };
  if (!only) {
#pragma unroll 4
    for (int n = 0; n < p.N; ++n) add(n, x[n]);
  } else {
    for (int n0 = 0; n0 < p.N; n0 += 32) {
      const float v = n0 + lane < p.N ? x[n0 + lane] : 0.f;
      if (__any_sync(0xffffffffu, v != v)) {
        ra = rb = __int_as_float(0x7fffffff);
        break;
      }
      for (unsigned left = __ballot_sync(0xffffffffu, !(fabsf(v) < inf)); left; left &= left - 1) {
        const int k = __ffs(left) - 1;
        add(n0 + k, __shfl_sync(0xffffffffu, v, k));
      }
      if (__all_sync(0xffffffffu, (ra != ra || ia != ia) && (rb != rb || ib != ib))) break;
    }
  }
  return make_float2(__logf(fmaf(ra, ra, ia * ia) + p.eps), __logf(fmaf(rb, rb, ib * ib) + p.eps));
}

static __device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
               : "r"(taddr));
}
static __device__ __forceinline__ void ld_wait8(float (&a)[8], float (&b)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+f"(a[0]), "+f"(a[1]), "+f"(a[2]), "+f"(a[3]), "+f"(a[4]), "+f"(a[5]), "+f"(a[6]), "+f"(a[7]),
                 "+f"(b[0]), "+f"(b[1]), "+f"(b[2]), "+f"(b[3]), "+f"(b[4]), "+f"(b[5]), "+f"(b[6]), "+f"(b[7])
               :
               : "memory");
}

// ---- epilogue: adds the chunks of each unit, then power, log, (DCT) and store
template <int P, bool MFCC>
static __device__ void epilogue(const SlabParams& p, uint8_t* gbase, const Ctx& c, const SlabBars& B, uint32_t tmem) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int quarter = warp & 3, half = warp >> 2;
  const int row = 32 * quarter + lane;
  const uint32_t tl = tmem + ((uint32_t)(32 * quarter) << 16);
  const bool vec8 = ((p.n_out & 7) == 0) && ((reinterpret_cast<uintptr_t>(p.out) & 31) == 0);
  const float* dct = reinterpret_cast<const float*>(gbase + p.off_dct);
  Ring rt, rp;
  int q, b;
  for (int i = 0; unit_at(p, c, i, q, b); ++i) {
    const TileDesc td = tile_of(p, c, q);
    const int ng = blk_groups(p, b);
    const int g_n = ng / 2, g_lo = half * g_n;  // (blocks hold an even number of groups)
    float acc[kGroupsPerWarp][2][8];
#pragma unroll
    for (int g = 0; g < kGroupsPerWarp; ++g)
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[g][0][e] = acc[g][1][e] = 0.f;
    bool ok = true;
    for (int kk = 0; ok && kk < p.n_slab; ++kk) {
      const int js = slab_steps(p, kk);
      for (int j0 = 0; j0 < js; j0 += p.kps) {
        if (!warp_wait(bar_at(p, c, B.t_full + rt.slot), rt.phase, c.abort, p.err)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t t0 = tl + rt.slot * 2 * kBlockBins + 8 * g_lo;
#pragma unroll
        for (int g = 0; g < kGroupsPerWarp; ++g)
          if (g < g_n) {
            float re[8], im[8];
            tmem_ld8(t0 + 8 * g, re);
            tmem_ld8(t0 + 8 * ng + 8 * g, im);
            ld_wait8(re, im);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              acc[g][0][e] += re[e];
              acc[g][1][e] += im[e];
            }
          }
        tc_fence_before();
        warp_arrive_leader(bar_at(p, c, B.t_empty + rt.slot));
        rt.next(kNacc);
      }
    }
    if (!ok) break;
    const bool valid = row < td.n_frames;
    const int m_lo = 8 * (b * p.wbg + g_lo);  // first bin of this warp
    bool finite = true;
#pragma unroll
    for (int g = 0; g < kGroupsPerWarp; ++g)
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float s = fmaf(acc[g][0][e], acc[g][0][e], acc[g][1][e] * acc[g][1][e]);
        finite = finite && s < __int_as_float(0x7f800000);
        acc[g][0][e] = __logf(s + p.eps);
      }
    const float* x = p.wave + td.in_off + (long long)row * p.H;
    if constexpr (!MFCC) {
      float* orow = p.out + (size_t)(td.out_row + row) * p.n_out;
      if (valid) {
#pragma unroll
        for (int g = 0; g < kGroupsPerWarp; ++g)
          if (g < g_n) {
            const int m = m_lo + 8 * g;
            if (vec8 && m + 8 <= p.M) {
              asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(orow + m),
                           "f"(acc[g][0][0]), "f"(acc[g][0][1]), "f"(acc[g][0][2]), "f"(acc[g][0][3]),
                           "f"(acc[g][0][4]), "f"(acc[g][0][5]), "f"(acc[g][0][6]), "f"(acc[g][0][7])
                           : "memory");
            } else {
#pragma unroll
              for (int e = 0; e < 8; ++e)
                if (m + e < p.M) orow[m + e] = acc[g][0][e];
            }
          }
      }
      for (unsigned left = __ballot_sync(0xffffffffu, !finite && valid); left; left &= left - 1) {
        const int l = __ffs(left) - 1, end = min(m_lo + 8 * g_n, p.M);
        const float2 v = redo_row(p, x + (long long)(l - lane) * p.H, m_lo, end);
        float* o = orow + (long long)(l - lane) * p.n_out + m_lo;
        if (m_lo + lane < end) o[lane] = v.x;
        if (m_lo + 32 + lane < end) o[32 + lane] = v.y;
      }
    } else {
      for (unsigned left = __ballot_sync(0xffffffffu, !finite && valid); left; left &= left - 1) {
        const int l = __ffs(left) - 1;
        const float2 v = redo_row(p, x + (long long)(l - lane) * p.H, m_lo, min(m_lo + 8 * g_n, p.M));
#pragma unroll
        for (int g = 0; g < kGroupsPerWarp; ++g)
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const float t = __shfl_sync(0xffffffffu, 8 * g + e < 32 ? v.x : v.y, (8 * g + e) & 31);
            if (lane == l) acc[g][0][e] = t;
          }
      }
      // bins past M (zero basis rows) take no part, whatever their log is
#pragma unroll
      for (int g = 0; g < kGroupsPerWarp; ++g)
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (m_lo + 8 * g + e >= p.M) acc[g][0][e] = 0.f;
      // C = ln(S + eps) D^T over this warp's bins, eight coefficients at a time.
      // The second warp of a lane quarter hands its part to the first through
      // one of two buffers; the first adds both (and, above 80 bins, what the
      // blocks before left in the row) and stores.
      float* orow = p.out + (size_t)(td.out_row + row) * p.n_mfcc;
      const bool add = b > 0 && valid && !half;
      float prev[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) prev[k] = add && k < p.n_mfcc ? orow[k] : 0.f;
      for (int k0 = 0; k0 < p.n_mfcc; k0 += 8) {
        float v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          v[k] = prev[k];
          prev[k] = add && k0 + 8 + k < p.n_mfcc ? orow[k0 + 8 + k] : 0.f;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const float* d = dct + (size_t)min(k0 + k, p.n_mfcc - 1) * (8 * p.groups) + m_lo;
#pragma unroll
          for (int g = 0; g < kGroupsPerWarp; ++g)
            if (g < g_n) {
              const float4 d0 = *reinterpret_cast<const float4*>(d + 8 * g);
              const float4 d1 = *reinterpret_cast<const float4*>(d + 8 * g + 4);
              const float* l = acc[g][0];
              v[k] = fmaf(l[0], d0.x, v[k]);
              v[k] = fmaf(l[1], d0.y, v[k]);
              v[k] = fmaf(l[2], d0.z, v[k]);
              v[k] = fmaf(l[3], d0.w, v[k]);
              v[k] = fmaf(l[4], d1.x, v[k]);
              v[k] = fmaf(l[5], d1.y, v[k]);
              v[k] = fmaf(l[6], d1.z, v[k]);
              v[k] = fmaf(l[7], d1.w, v[k]);
            }
        }
        float* buf = reinterpret_cast<float*>(gbase + p.off_part) + rp.slot * 8 * kF + row;
        const uint32_t full = bar_at(p, c, B.half + 4 * quarter + rp.slot), empty = full + 16;
        if (half) {
          if (!warp_wait(empty, rp.phase ^ 1, c.abort, p.err)) return;
#pragma unroll
          for (int k = 0; k < 8; ++k) buf[k * kF] = v[k];
          warp_arrive_local(full);
        } else {
          if (!warp_wait(full, rp.phase, c.abort, p.err)) return;
#pragma unroll
          for (int k = 0; k < 8; ++k) v[k] += buf[k * kF];
          warp_arrive_local(empty);
          if (valid) {
#pragma unroll
            for (int k = 0; k < 8; ++k)
              if (k0 + k < p.n_mfcc) orow[k0 + k] = v[k];
          }
        }
        rp.next(2);
      }
    }
  }
}

template <int P, bool MFCC>
__global__ void __launch_bounds__(kThreads, 1) melt_slab_kernel(const __grid_constant__ SlabParams p) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  Ctx c;
  c.sbase = (raw + 127u) & ~127u;
  uint8_t* gbase = smem_raw + (c.sbase - raw);
  c.rank = cluster_ctarank();
  c.cluster = (int)(blockIdx.x >> 1);
  c.n_clusters = (int)(gridDim.x >> 1);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gbase + p.off_misc);
  c.abort = reinterpret_cast<volatile int*>(gbase + p.off_misc + 4);
  const SlabBars B(p.NA, p.NB);
  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    auto bar = [&](int i) { return bar_at(p, c, i); };
    for (int i = 0; i < p.NA; ++i) {
      mbar_init(bar(B.a_full + i), 2);  // one converter warp of each CTA
      mbar_init(bar(B.a_empty + i), 1);
    }
    for (int i = 0; i < p.NB; ++i) {
      mbar_init(bar(B.b_full + i), c.rank == 0 ? 2 : 1);
      mbar_init(bar(B.b_empty + i), 1);
    }
    for (int i = 0; i < kNacc; ++i) {
      mbar_init(bar(B.t_full + i), 1);
      mbar_init(bar(B.t_empty + i), 2 * kEpiWarps);
    }
    for (int i = 0; i < 16; ++i) mbar_init(bar(B.half + i), 1);
    mbar_init(bar(B.drain), 1);
    *c.abort = 0;
    fence_mbar_init();
  }
  if (warp == kMmaWarp) {
    tmem_alloc_pair(smem_u32(tmem_slot), 512);
    tmem_relinquish_pair();
  }
  if constexpr (MFCC) {
    // D as [n_mfcc][8 groups] rows, zero past M
    float* d = reinterpret_cast<float*>(gbase + p.off_dct);
    const int ld = 8 * p.groups;
    for (int i = threadIdx.x; i < p.n_mfcc * ld; i += kThreads) {
      const int k = i / ld, m = i - k * ld;
      d[i] = m < p.M ? p.dct[k * p.M + m] : 0.f;
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // both CTAs' barriers exist before either arrives on the other's
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  if (threadIdx.x == 0) pdl_launch_dependents();
  // the basis and the MMAs touch the library's own data only; what reads
  // tiles or samples or writes features waits for the stream's previous kernel
  if (warp == kMmaWarp) {
    if (elect_one()) {
      if (c.rank == 0) mma_issue<P>(p, c, B, tmem);
      else basis_signal(p, c, B);
      volatile int never = 0;
      mbar_wait(bar_at(p, c, B.drain), 0, &never, p.err, kErrTimeout);
    }
    __syncwarp();
  } else if (warp == kBWarp) {
    if (elect_one()) basis_producer<P>(p, c, B);
    __syncwarp();
  } else if (warp >= kCvtWarp0) {
    pdl_wait();
    convert<P>(p, c, B);
    __syncwarp();
  } else {
    pdl_wait();
    epilogue<P, MFCC>(p, gbase, c, B, tmem);
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // neither CTA leaves (or frees TMEM) while its peer may still use it
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, 512);
  }
}

}  // namespace slab
}  // namespace melt
