// Device side of the slab kernel, included by melt_slab.cu.
#pragma once
// The projection (Eq. 6) on the tensor cores with both operands streamed in K
// slabs: the FP32 form (P 3), and log-Mel of split BF16 (P 2) and of BF16 bases
// that do not stay resident (P 1).
//
// FP32.  Every FP32 sample and every basis value is split exactly into three BF16
// parts (hi = rn(v), mid = rn(v - hi), lo = rn(v - hi - mid): 3 x 8 bits), and
// the six products of parts whose weight is at least 2^-16 of the leading one
// are formed: hi hi, hi mid, mid hi, mid mid, hi lo, lo hi.  What is dropped
// is below 2^-24 of each product, the size of an FP32 rounding.
//
// Accumulation.  The tensor core truncates its FP32 accumulator at every MMA,
// a bias that grows with the number of MMAs (25 of them put -3.0e-6 dB on the
// bins near the frame maximum, where the FFMA kernel's error is 2.7e-6 dB
// RMS).  So K is cut into stages of at most kps K-steps; each starts from zero,
// adds its small products first (they are 2^-8 of the sum, so their truncation
// does not count) and its hi hi products last, and the epilogue adds the stages
// up in FP32 registers with round-to-nearest.  (Two stages to an accumulator
// measured 96 against 98 us on the 64 x 30 s batch, with errors up to 1.3 times
// larger: not kept.)
//
// Bound.  Six products make 6 x 128,000 flops a frame at (N, M) = (400, 80):
// 147 GFLOP for the 64 x 30 s batch, tensor-bound (its 184 MB of samples and
// features take a third of that time).  So everything else has to stay out of
// the MMAs' way: the basis (384 KB in three parts) does not fit shared memory
// and neither do two converted tiles (125 KB each), but one K slab of both
// does.  A slab is 16 columns of the polyphase rows Z[u][r] = x[(t0+u) H + r]
// and, for each slice j, the K-step n = j H + r of the basis; the slices of a
// slab read the same rows at row offset j, so a sample is converted once for
// all of them.  A stage holds up to kps slices of a slab: the 128 + kps - 1 rows
// that they read, converted, and their basis blocks.  Stages flow through one
// ring (shared memory has 4 to 8), each with one barrier that both operands of
// both CTAs complete.  With more slices than kps (short hops) a slab's rows are
// converted once per stage.
//
// Clusters of two CTAs share each MMA (cta_group::2, M = 256: two tiles): the
// even CTA holds the W_r rows of a K-step, the odd one the W_i rows, so each
// streams half of the basis.  More than 80 Mel bins run as blocks of at most
// 80 (the epilogue's accumulators live in registers); a short batch is cut
// into more blocks to use more SMs.
//
// Split BF16 and BF16 (P 2 and P 1).  The same pieces serve the log-Mel of split
// BF16 (three products, two parts) and of BF16 bases whose half does not fit
// resident (the 22.05 kHz geometry).  Their sums are those of their other
// layouts, bit for bit: one accumulator per unit, K-steps slice by slice.  So a
// tile's slabs stay in a ring of their own (A) until their last slice is
// done, a third to a whole tile more than a tile has, and the basis flows beside them (B),
// slots of up to 3 or 8 K-steps.  (Samples loaded straight into registers leave room
// for more slots of both, but not enough loads in flight: 256 x 10 s split BF16 90
// us for 73, BF16 at 22.05 kHz 64 for 41.)
//
// Warps: 0-7 epilogue (two per TMEM lane quarter, each half of the block's
// bins), 8-10 and 12-14 converters (each takes whole slabs by itself: its samples
// arrive by asynchronous copies in a staging area of its own, one arrival per
// slab), 11 MMA issue (odd CTA: forwards its basis fills to the even one), 15
// basis producer.
//
// Code size counts here: the issue thread's few hundred instructions per chunk
// run once per 1200 clocks between three other warps on its scheduler, and it
// fetches them anew each time.  With converters unrolled over 17 register
// quads the 64 x 30 s batch took 132 us, of which two thirds of the MMAs could
// be left out for 11 us.
//
// Samples the split cannot hold.  An infinity or NaN (whose parts would also
// turn the sums of frames that only meet it at a zero basis row into NaN), or
// sums that overflow: a frame whose power is not finite is looked at again by its
// epilogue warp, sample by sample, and recomputed with FP32 FFMAs unless its samples
// are finite and its powers only overflow.  64 x 30 s, where the FFMA kernel took
// 507 us throughout: 90 us clean, 96 with one clip of NaN, 132 with a NaN every
// quarter of a second, 237 with an infinity, 234 all NaN, 435 all powers overflowing,
// 580 all infinite; 6.3 ms where all sums overflow (samples of 1e37 and more).
#include <cuda_bf16.h>

#include "melt_slab.h"
#include "melt_tc.h"
#include "sm100_ptx.cuh"

namespace melt {
namespace slab {

using namespace ptx;

constexpr int kF = kTileFrames;
// Warps 0-7 epilogue; 11 and 15, on one scheduler, MMA issue and basis
// producer; the others from 8 on converters: six in the FP32 form, twelve where
// there are fewer MMAs to a slab (a slab took a warp 6000 clocks, 1000 with six
// at work, where P 2's MMAs take 480 to 720).
constexpr int kEpiWarps = 8, kMmaWarp = 11, kBWarp = 15;
constexpr int kMaxTeams = 6;  // slabs in conversion at once, each by a team of tw warps
__host__ __device__ constexpr int cvt_warps(int P) { return P == 3 ? 6 : 12; }
__host__ __device__ constexpr int slab_threads(int P) { return 32 * (kEpiWarps + 2 + cvt_warps(P)); }
// Groups of 8 Mel bins of a block at most: the FP32 form's sums live in the
// epilogue's registers (80 per thread); split BF16's 128 bins in one block
// leave its rings too few slots.
__host__ __device__ constexpr int max_groups(int P) { return P == 1 ? 16 : 10; }
constexpr int kMaxAcc = 3;      // TMEM accumulators of the widest block's columns: 3 up to 80 bins, else 2
constexpr int kMaxKps = 8;
// K-steps at most of a stage (P 3: its truncations grow with them, its drains
// with their number) or of a basis slot.
__host__ __device__ constexpr int max_kps(int P) { return P == 3 ? 4 : P == 2 ? 3 : kMaxKps; }
constexpr int kRowsA = 132;     // rows of a stage's A operand: 128 + kps - 1 and up to 4 mod 8, so that the two core
                                // columns of a converter store fall on other banks (kMaxKps - 1 more at most)
constexpr int kStageRows = kF + kMaxKps;  // sample rows a converter warp copies for a stage
constexpr uint32_t kRawBytes = kStageRows * 64u;
constexpr int kMaxStages = 8;   // P 3
constexpr int kMaxA = 48, kMaxB = 8;  // P 1, 2: slots of the two rings

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
  int n_last;          // samples of the last slice: N - (J - 1) H
  int nblk, wbg;       // blocks of wbg groups of 8 bins (the last may have fewer)
  int inner;           // blocks a unit takes in turn (MFCC: all of them, else 1)
  int n_units;
  int kps;             // K-steps per stage (slices of a slab); P 1, 2: per basis slot (slabs of a slice)
  int NS, NB;          // stages of the ring (NB 0); P 1, 2: slots of the A and basis rings
  int nacc;            // TMEM accumulators, acc_cols columns apart
  uint32_t acc_cols;
  int ncv, tw;         // converter teams at work (at most NS: a team that took slab g waits for the place of slab
                       // g + ncv by a parity, which tells only neighbouring phases apart; P 3's stages are
                       // freed in order, by commits a stage's MMAs apart, P 1, 2: freed_bar), warps of a team
  uint32_t lbo_a, a_part, a_bytes, stage, step_bytes;  // a stage: A (a_bytes: P parts of two core columns), then B;
                                                       // P 1, 2: an A slot
  uint32_t off_b, b_slot;  // P 1, 2: the basis ring
  uint32_t off_raw, off_bar, off_misc, off_dct, off_part;
  int n_mfcc, n_out;
  int early_inputs;    // the waveform's readers need not wait for the stream's previous kernel
};

// P 1, 2: the `empty` barrier that the MMAs of slot `slot`'s turn `turn` (0, 1,
// ...) complete, and the one and its phase parity that a converter waits for
// before it fills a slot.
// Two barriers a slot, one for its even turns and one for the odd ones.  A team
// waits only for its own slabs' places, and the slabs of a tile are freed out of
// order (those past the last slice's end a slice early), so when a team comes to
// slab g even slab g - 2 NS may not be freed, and the parity of one barrier cannot
// tell that from g - NS being freed.  Slab g - 3 NS is: the team took the place of
// slab h = g - ncv - NS >= g - 2 NS; the MMAs begin slabs in order, so all up to h
// had been filled when h was freed, g - 2 NS into the place of g - 3 NS.
__host__ __device__ constexpr int freed_bar(int NS, int slot, uint32_t turn) { return slot + (turn & 1 ? NS : 0); }
// `pos`: the slab's place among two turns of the slots (slot + NS in odd turns),
// `phase`: how often these have come round.  The barrier is the turn before's (at
// the start the parity is that of the phase before its first, which passes).
__host__ __device__ constexpr int place_bar(int NS, int pos) { return pos >= NS ? pos - NS : pos + NS; }
__host__ __device__ constexpr uint32_t place_parity(int NS, int pos, uint32_t phase) {
  return (phase ^ (pos >= NS ? 0u : 1u)) & 1u;
}

struct SlabBars {
  int full, empty, b_full, b_empty, t_full, t_empty, part, drain, total;
  // P 3: NS stages, NB = 0.  P 1, 2: NS A slots and NB basis slots.
  __host__ __device__ SlabBars(int NS, int NB) {
    full = 0;                 // converters of both CTAs (even CTA's copy is used); P 3: and the basis, as b_full
    empty = full + NS;        // MMA commit, both CTAs; P 1, 2: two a slot (freed_bar)
    b_full = empty + (NB > 0 ? 2 : 1) * NS;  // this CTA's basis copies; even CTA: and the odd one's signal that its own
                                             // are in
    b_empty = b_full + NB;    // MMA commit, both CTAs
    t_full = b_empty + NB;    // MMA commit, both CTAs
    t_empty = t_full + kMaxAcc;  // both CTAs' epilogues (even CTA's copy is used)
    part = t_empty + kMaxAcc; // MFCC, per lane quarter: part buffers 0, 1 filled; [16 B on] taken
    drain = part + 16;
    total = drain + 1;
  }
};

struct Ctx {
  uint32_t sbase, rank;
  int cluster, n_clusters;
  volatile int* abort;
};

// P 3: stages of a unit (an accumulator each; the epilogue adds them up).
static __device__ __forceinline__ int unit_stages(const SlabParams& p) {
  const int last = (p.n_last + 15) / 16;  // slabs that all slices reach
  return last * ((p.J + p.kps - 1) / p.kps) + (p.n_slab - last) * ((p.J - 1 + p.kps - 1) / p.kps);
}

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
  // (the divisions only where there are several blocks)
  const int u = c.cluster + (p.inner > 1 ? i / p.inner : i) * c.n_clusters;
  if (u >= p.n_units) return false;
  if (p.inner > 1) {
    q = u;
    b = i % p.inner;
  } else if (p.nblk == 1) {
    q = u;
    b = 0;
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

// ---- basis producer: each unit's K-steps of this CTA's half, stage by stage
// (A bulk prefetch of the next tile's samples into L2 from here, a unit ahead of the
// converters, cost more than it gave: 64 x 30 s FP32 91.6 us with, 90.2 without; 256
// x 10 s split BF16 76.2, 73.5; BF16 at 22.05 kHz, 64 x 20 s 42.1, 40.8, all in one
// process on a fixed input; over changing inputs the calls take 95 to 98, 77 to 80 and
// 43.)
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
    for (int kk = 0; ok && kk < p.n_slab; ++kk) {
      const int js = slab_steps(p, kk);
      for (int j0 = 0; j0 < js; j0 += p.kps) {
        if (!bar_wait(bar_at(p, c, B.empty + r.slot), r.phase ^ 1, c.abort, p.err)) {
          ok = false;
          break;
        }
        const int n = min(p.kps, js - j0);
        const uint32_t full = bar_at(p, c, B.full + r.slot);
        const uint32_t dst = c.sbase + r.slot * p.stage + p.a_bytes;
        mbar_arrive_expect_tx(full, blk * n);
        if (blk == p.step_bytes) {
          bulk_g2s_hint(dst, src, blk * n, full, pol);
        } else {
          for (int k = 0; k < n; ++k) bulk_g2s_hint(dst + k * blk, src + (size_t)k * p.step_bytes, blk, full, pol);
        }
        src += (size_t)n * p.step_bytes;
        ++issued;
        r.next(p.NS);
      }
    }
  }
  // every issued copy has landed before the CTA can exit
  volatile int never = 0;
  for (int k = max(0, issued - p.NS); k < issued; ++k)
    mbar_wait(bar_at(p, c, B.full + k % p.NS), (k / p.NS) & 1, &never, p.err, kErrTimeout);
}

// The same for P 1, 2: slice by slice, up to kps slabs to a slot.
template <int P>
static __device__ void basis_producer_slices(const SlabParams& p, const Ctx& c, const SlabBars& B) {
  const uint64_t pol = policy_evict_last();
  const uint8_t* half = p.img + (size_t)c.rank * p.ksteps * p.step_bytes;
  const int last = (p.n_last + 15) / 16;
  Ring r;
  int issued = 0, q, b;
  bool ok = true;
  for (int i = 0; ok && unit_at(p, c, i, q, b); ++i) {
    const uint32_t blk = (uint32_t)blk_groups(p, b) * P * 256u;
    const uint8_t* src = half + (size_t)b * p.wbg * P * 256u;
    for (int j = 0; ok && j < p.J; ++j) {
      const int nk = j + 1 < p.J ? p.n_slab : last;
      for (int k0 = 0; k0 < nk; k0 += p.kps) {
        if (!bar_wait(bar_at(p, c, B.b_empty + r.slot), r.phase ^ 1, c.abort, p.err)) {
          ok = false;
          break;
        }
        const int n = min(p.kps, nk - k0);
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
      }
    }
  }
  // every issued copy has landed before the CTA can exit
  volatile int never = 0;
  for (int k = max(0, issued - p.NB); k < issued; ++k)
    mbar_wait(bar_at(p, c, B.b_full + k % p.NB), (k / p.NB) & 1, &never, p.err, kErrTimeout);
}

// ---- odd CTA, P 1, 2: one arrival on the even CTA's b_full per filled slot
static __device__ void basis_signal_slices(const SlabParams& p, const Ctx& c, const SlabBars& B) {
  const int last = (p.n_last + 15) / 16;
  Ring r;
  int q, b;
  for (int i = 0; unit_at(p, c, i, q, b); ++i)
    for (int j = 0; j < p.J; ++j)
      for (int k0 = 0; k0 < (j + 1 < p.J ? p.n_slab : last); k0 += p.kps) {
        if (!bar_wait(bar_at(p, c, B.b_full + r.slot), r.phase, c.abort, p.err)) return;
        mbar_arrive_cluster(mapa_shared(bar_at(p, c, B.b_full + r.slot), 0));
        r.next(p.NB);
      }
}

// ---- odd CTA: one arrival on the even CTA's barrier per stage whose basis is in
static __device__ void basis_signal(const SlabParams& p, const Ctx& c, const SlabBars& B) {
  Ring r;
  int q, b;
  for (int i = 0; unit_at(p, c, i, q, b); ++i)
    for (int kk = 0; kk < p.n_slab; ++kk) {
      const int js = slab_steps(p, kk);
      for (int j0 = 0; j0 < js; j0 += p.kps) {
        if (!bar_wait(bar_at(p, c, B.full + r.slot), r.phase, c.abort, p.err)) return;
        mbar_arrive_cluster(mapa_shared(bar_at(p, c, B.full + r.slot), 0));
        r.next(p.NS);
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

static __device__ __forceinline__ void mma_pair_if(uint32_t d, uint32_t a, uint32_t a_hi, uint32_t b, uint32_t b_hi,
                                                   uint32_t idesc, bool acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 x, y;\n\t"
      "mov.b64 x, {%1, %2};\n\tmov.b64 y, {%3, %4};\n\t"
      "setp.ne.u32 p, %6, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], x, y, %5, p;\n\t}\n" ::"r"(d),
      "r"(a), "r"(a_hi), "r"(b), "r"(b_hi), "r"(idesc), "r"((uint32_t)acc));
}

// Products of a stage's n K-steps into accumulator d (P 3).  a, w: descriptors
// (low words) of the first K-step's hi parts (parts 0 hi, 1 mid, 2 lo are ap and
// 16 apart, K-steps 1 row of A and `step` of the basis, in 16-byte units).
// SMALL: the products with a mid or lo part, else hi hi.  Straight-line code
// with one predicate per K-step: a switch over n cost 150 to 200 clocks a stage.
template <bool SMALL>
static __device__ __forceinline__ void stage_mmas(int n, uint32_t d, uint32_t a, uint32_t ah, uint32_t w, uint32_t wh,
                                                  uint32_t ap, uint32_t step, uint32_t idesc) {
  const uint32_t am = a + ap, al = am + ap;
#pragma unroll
  for (int k = 0; k < max_kps(3); ++k) {
    if (k >= n) break;
    const uint32_t wk = w + k * step;
    if constexpr (!SMALL) {
      mma_pair<true>(d, a + k, ah, wk, wh, idesc);
    } else {
      if (k == 0) mma_pair<false>(d, al, ah, wk, wh, idesc);
      else mma_pair<true>(d, al + k, ah, wk, wh, idesc);
      mma_pair<true>(d, a + k, ah, wk + 32, wh, idesc);
      mma_pair<true>(d, am + k, ah, wk + 16, wh, idesc);
      mma_pair<true>(d, am + k, ah, wk, wh, idesc);
      mma_pair<true>(d, a + k, ah, wk + 16, wh, idesc);
    }
  }
}

// Both phases complete?  The two tests are in flight together.
static __device__ __forceinline__ bool warp_wait2(uint32_t b0, uint32_t p0, uint32_t b1, uint32_t p1,
                                                  volatile int* abort, int* err) {
  const bool x = mbar_test_wait(b0, p0), y = mbar_test_wait(b1, p1);
  return (__all_sync(0xffffffffu, x) || warp_wait(b0, p0, abort, err)) &&
         (__all_sync(0xffffffffu, y) || warp_wait(b1, p1, abort, err));
}

// ---- even CTA: every MMA of the pair (P 3).
// What this warp does besides its MMAs has to stay below the time they take
// (960 to 1900 clocks a stage at 80 bins), and it runs at ten and more clocks an
// instruction beside the SM's other warps: with rings of their own for A and the
// basis (three waits, three commits and three ring steps a slab), acquires at
// cluster scope and one lane at work it took 1650 clocks and bounded the kernel.
static __device__ void mma_issue(const SlabParams& p, const Ctx& c, const SlabBars& B, uint32_t tmem) {
  constexpr uint32_t ah = (128u >> 4) | (1u << 14);         // SBO 128 B
  constexpr uint32_t wh = ((3 * 256u) >> 4) | (1u << 14);   // SBO: the next group of 8 bins
  const uint32_t a0 = (c.sbase >> 4) | ((p.lbo_a >> 4) << 16);
  const uint32_t b0 = ((c.sbase + p.a_bytes) >> 4) | ((128u >> 4) << 16);  // LBO 128 B
  const uint32_t ap = p.a_part >> 4, stage = p.stage >> 4;
  const uint32_t full = bar_at(p, c, B.full), empty = bar_at(p, c, B.empty);
  const uint32_t t_full = bar_at(p, c, B.t_full), t_empty = bar_at(p, c, B.t_empty);
  const int kps = p.kps, J = p.J, n_last = p.n_last, n_slab = p.n_slab, NS = p.NS;
  Ring r, rt;
  uint32_t at = 0, d = tmem;  // the stage's offset in 16-byte units, the accumulator
  int q, b;
  bool ok = true;
  for (int i = 0; ok && unit_at(p, c, i, q, b); ++i) {
    const uint32_t ng = (uint32_t)blk_groups(p, b);
    const uint32_t idesc = idesc_f32acc(1u, 2 * kF, 16u * ng), step = ng * ((3 * 256u) >> 4);
    int kk = 0, left = J;  // slab, its slices to come (n_last > 0: the first slab has them all)
    while (kk < n_slab) {
      ok = warp_wait2(full + 8 * r.slot, r.phase, t_empty + 8 * rt.slot, rt.phase ^ 1, c.abort, p.err);
      if (!ok) break;
      tc_fence_after();
      const int n = min(kps, left);
      if (elect_one()) {
        stage_mmas<true>(n, d, a0 + at, ah, b0 + at, wh, ap, step, idesc);
        stage_mmas<false>(n, d, a0 + at, ah, b0 + at, wh, ap, step, idesc);
        mma_commit_pair_mc(empty + 8 * r.slot, 3);
        mma_commit_pair_mc(t_full + 8 * rt.slot, 3);
      }
      __syncwarp();
      at += stage;
      r.next(NS);
      if (r.slot == 0) at = 0;
      left -= n;
      if (left == 0) {
        ++kk;
        left = 16 * kk < n_last ? J : J - 1;
      }
      d += p.acc_cols;
      rt.next(p.nacc);
      if (rt.slot == 0) d = tmem;
    }
  }
  // no pair MMA may still be running when either CTA releases TMEM
  if (elect_one()) mma_commit_pair_mc(bar_at(p, c, B.drain), 3);
}

// The same for P 1, 2: slice by slice over the unit's slabs, a basis slot at a
// time, each K-step's hi hi (hi lo, lo hi) into the unit's one accumulator, the
// order of the other layouts' sums.  The first slice waits for each slab; a
// slab's last one frees its place.
template <int P>
static __device__ void mma_issue_slices(const SlabParams& p, const Ctx& c, const SlabBars& B, uint32_t tmem) {
  constexpr uint32_t ah = (128u >> 4) | (1u << 14);         // SBO 128 B
  constexpr uint32_t wh = ((P * 256u) >> 4) | (1u << 14);   // SBO: the next group of 8 bins
  const uint32_t a0 = (c.sbase >> 4) | ((p.lbo_a >> 4) << 16);
  const uint32_t b0 = ((c.sbase + p.off_b) >> 4) | ((128u >> 4) << 16);  // LBO 128 B
  const uint32_t ap = p.a_part >> 4, as = p.stage >> 4, a_end = as * (uint32_t)p.NS, bs = p.b_slot >> 4;
  const uint32_t full = bar_at(p, c, B.full), empty = bar_at(p, c, B.empty);
  const uint32_t b_full = bar_at(p, c, B.b_full), b_empty = bar_at(p, c, B.b_empty);
  const int kps = p.kps, J = p.J, n_slab = p.n_slab, NS = p.NS, NB = p.NB, last = (p.n_last + 15) / 16;
  Ring ra, rb, rt;
  uint32_t bl = b0, d = tmem;
  int q, b;
  bool ok = true;
  for (int i = 0; ok && unit_at(p, c, i, q, b); ++i) {
    const uint32_t ng = (uint32_t)blk_groups(p, b);
    const uint32_t idesc = idesc_f32acc(1u, 2 * kF, 16u * ng), step = ng * ((P * 256u) >> 4);
    const int slot0 = ra.slot, free0 = freed_bar(NS, ra.slot, ra.phase);  // the unit's first slab
    ok = warp_wait(bar_at(p, c, B.t_empty + rt.slot), rt.phase ^ 1, c.abort, p.err);
    for (int j = 0; ok && j < J; ++j) {
      const int nk = j + 1 < J ? n_slab : last;
      const int free_from = j + 1 == J ? 0 : j + 2 == J ? last : n_slab;  // slabs this slice is the last of
      int fr = free0;  // (slabs in order take these barriers round and round)
      uint32_t at = (uint32_t)slot0 * as;
      for (int k0 = 0; k0 < nk; k0 += kps) {
        const int n = min(kps, nk - k0);
        ok = warp_wait(b_full + 8 * rb.slot, rb.phase, c.abort, p.err);
        if (j == 0)
          for (int k = 0; ok && k < n; ++k) {
            ok = warp_wait(full + 8 * ra.slot, ra.phase, c.abort, p.err);
            ra.next(NS);
          }
        if (!ok) break;
        tc_fence_after();
        const uint32_t a = a0 + (uint32_t)j;
        if (elect_one()) {
          uint32_t o = at, w = bl;
#pragma unroll
          for (int k = 0; k < max_kps(P); ++k) {
            if (k >= n) break;
            if (k == 0) mma_pair_if(d, a + o, ah, w, wh, idesc, j + k0 > 0);
            else mma_pair<true>(d, a + o, ah, w, wh, idesc);
            if constexpr (P == 2) {
              mma_pair<true>(d, a + o, ah, w + 16, wh, idesc);
              mma_pair<true>(d, a + o + ap, ah, w, wh, idesc);
            }
            w += step;
            o += as;
            if (o == a_end) o = 0;
          }
          mma_commit_pair_mc(b_empty + 8 * rb.slot, 3);
          for (int k = max(0, free_from - k0); k < n; ++k) {
            const int f = fr + k < 2 * NS ? fr + k : fr + k - 2 * NS;
            mma_commit_pair_mc(empty + 8 * f, 3);
          }
        }
        __syncwarp();
        fr += n;
        if (fr >= 2 * NS) fr -= 2 * NS;
        at += (uint32_t)n * as;
        if (at >= a_end) at -= a_end;
        bl += bs;
        rb.next(NB);
        if (rb.slot == 0) bl = b0;
      }
    }
    if (!ok) break;
    if (elect_one()) mma_commit_pair_mc(bar_at(p, c, B.t_full + rt.slot), 3);
    __syncwarp();
    d += p.acc_cols;
    rt.next(p.nacc);
    if (rt.slot == 0) d = tmem;
  }
  // no pair MMA may still be running when either CTA releases TMEM
  if (elect_one()) mma_commit_pair_mc(bar_at(p, c, B.drain), 3);
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

// A stage's sample rows [0, rows) (column r of lane quad qd, row u0 + 8 k; s0:
// sample of row 0, column r) into the warp's own area.  Four lanes take the 16
// samples of a row (64 contiguous bytes), so a warp's copies read whole sectors
// of 8 rows.
static __device__ __forceinline__ void stage_rows(const SlabParams& p, const float* src, int nsamp, int rows, bool live,
                                                  int s0, uint32_t to, int u0, int tw) {
  int s = s0 + u0 * p.H;
  if (s0 + rows * p.H <= nsamp && p.H % 16 == 0) {  // no sample of this lane's past the clip's end
    const float* from = src + s;
#pragma unroll 4
    for (int u = u0; u < rows; u += 8 * tw, from += 8 * tw * p.H, to += 512 * tw) copy_quad(to, from, 16);
  } else {
#pragma unroll 2
    for (int u = u0; u < rows; u += 8 * tw, s += 8 * tw * p.H, to += 512 * tw) {
      const int left = live ? min(max(nsamp - s, 0), 4) : 0;  // samples of the quad before the clip's end
      copy_quad(to, src + (left ? s : 0), 4 * left);
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// ---- converters: team w takes stages w, w + ncv, ... of the CTA's stream (its
// warps every other group of 8 rows).  The copies of the next one are in flight
// while a warp waits for that stage's place; every lane converts what it copied itself.  Quad qd of row u goes, four BF16
// values of each part, as 8 bytes to core column qd / 2, row u.
template <int P>
static __device__ void convert(const SlabParams& p, const Ctx& c, const SlabBars& B) {
  const int TW = P == 3 ? 1 : p.tw;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cw = warp - kEpiWarps - (warp > kMmaWarp ? 1 : 0) - (warp > kBWarp ? 1 : 0);  // converter warp
  const int w = cw / TW;
  const int qd = lane & 3, u0 = (lane >> 2) + 8 * (cw % TW);
  const uint32_t to = c.sbase + (uint32_t)(qd >> 1) * p.lbo_a + (uint32_t)(qd & 1) * 8u + 16u * u0;
  const uint32_t raw = c.sbase + p.off_raw + w * kRawBytes + 64u * u0 + 16u * qd;
  const uint32_t part = p.a_part;
  if (w >= p.ncv) return;
  // unit ordinal and stage of it; the slab and first slice of that stage.  The
  // descriptor of the unit after is loaded one unit early.
  const int U = P == 3 ? unit_stages(p) : p.n_slab, last = (p.n_last + 15) / 16;
  const int per = P == 3 ? (p.J + p.kps - 1) / p.kps : 1, per2 = max(1, (p.J - 1 + p.kps - 1) / p.kps);  // stages of a slab
  int i = 0, st = 0, kk = 0, j0 = 0, q, b;
  const int round = P < 3 ? 2 * p.NS : p.NS;  // P 1, 2: two turns of the slots (place_bar)
  Ring r;
  TileDesc td, nxt;
  bool more = unit_at(p, c, 0, q, b);
  if (more) td = tile_of(p, c, q);
  bool more_n = more && unit_at(p, c, 1, q, b);
  if (more_n) nxt = tile_of(p, c, q);
  auto step = [&](int n) {  // n stages on
    r.slot += n;  // (n <= ncv <= NS)
    if (r.slot >= round) {
      r.slot -= round;
      r.phase ^= 1;
    }
    st += n;
    while (st >= U && more) {
      st -= U;
      ++i;
      more = more_n;
      td = nxt;
      more_n = more && unit_at(p, c, i + 1, q, b);
      if (more_n) nxt = tile_of(p, c, q);
    }
    if (per == 1) {
      kk = st;
    } else if (st < last * per) {
      kk = st / per;
      j0 = (st - kk * per) * p.kps;
    } else {
      const int s2 = st - last * per;
      kk = last + s2 / per2;
      j0 = (s2 % per2) * p.kps;
    }
  };
  int rows = 0;
  auto copy = [&] {
    rows = td.n_frames > 0 ? td.n_frames + (P == 3 ? min(p.kps, slab_steps(p, kk) - j0) : p.J) - 1 : 0;
    const int col = 16 * kk + 4 * qd;
    stage_rows(p, p.wave + td.in_off, td.n_samples, rows, col < p.H, j0 * p.H + col, raw, u0, TW);
  };
  step(w);
  if (more) copy();
  while (more) {
    const int slot = P < 3 && r.slot >= p.NS ? r.slot - p.NS : r.slot;
    if (!warp_wait(bar_at(p, c, B.empty + (P < 3 ? place_bar(p.NS, r.slot) : slot)),
                   P < 3 ? place_parity(p.NS, r.slot, r.phase) : r.phase ^ 1, c.abort, p.err))
      break;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    uint32_t at = to + slot * p.stage, from = raw;
#pragma unroll 4
    for (int u = u0; u < rows; u += 8 * TW, at += 128 * TW, from += 512 * TW) {
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
    fence_proxy_async();
    warp_arrive_leader(bar_at(p, c, B.full + slot));
    step(p.ncv);
    if (more) copy();
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");  // no copy is in flight when the CTA exits
}

// What a frame's N samples at x hold, by a whole warp: 1 a NaN (then it stops
// there), else 2 an infinity, else 0.
static __device__ __noinline__ int scan_row(const float* x, int N) {
  const int lane = threadIdx.x & 31;
  bool odd = false;
  for (int n0 = lane; n0 < N + lane; n0 += 128) {
    float v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = x[min(n0 + 32 * k, N - 1)];
    bool nan = false;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      odd |= !(fabsf(v[k]) < __int_as_float(0x7f800000));
      nan |= v[k] != v[k];
    }
    if (__any_sync(0xffffffffu, nan)) return 1;
  }
  return __any_sync(0xffffffffu, odd) ? 2 : 0;
}

// ln(S + eps) of one frame (its samples at x, no NaN) as FP32 FFMAs form it, by a
// whole warp: lane l gets bins m0 + l and m0 + 32 + l (those below `end`).  Where a
// sample is an infinity (`only`), the finite ones cannot change either sum any
// more (each is an infinity or a NaN), so only the others are added, until
// every power is a NaN.
static __device__ __noinline__ float2 redo_row(const SlabParams& p, const float* x, int m0, int end, bool only) {
  const int lane = threadIdx.x & 31;
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
#pragma unroll 8
    for (int n = 0; n < p.N; ++n) add(n, x[n]);
  } else {
    bool more = true;
    for (int n0 = 0; more && n0 < p.N; n0 += 32) {
      const float v = n0 + lane < p.N ? x[n0 + lane] : 0.f;
      unsigned left = __ballot_sync(0xffffffffu, !(fabsf(v) < __int_as_float(0x7f800000)));
      for (; more && left; left &= left - 1) {
        const int k = __ffs(left) - 1;
        add(n0 + k, __shfl_sync(0xffffffffu, v, k));
        more = __any_sync(0xffffffffu, (ra == ra && ia == ia) || (rb == rb && ib == ib));
      }
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

// 32 bytes, one sector (address 32-byte aligned).
static __device__ __forceinline__ void store8(float* p, const float (&v)[8]) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
               "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}

// ---- epilogue: adds the chunks of each unit, then power, log, (DCT) and store
template <int P, bool MFCC>
static __device__ void epilogue(const SlabParams& p, uint8_t* gbase, const Ctx& c, const SlabBars& B, uint32_t tmem) {
  constexpr int kG = max_groups(P) / 2;  // groups of 8 bins per epilogue warp at most
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
    const bool valid = row < td.n_frames;
    const int m_lo = 8 * (b * p.wbg + g_lo);  // first bin of this warp
    if constexpr (P < 3) {
      // the unit's accumulator, group by group straight to the log and the row
      // (as the other kernels of these forms evaluate it)
      const uint32_t slot0 = rt.slot, t0 = tl + slot0 * p.acc_cols + 8 * g_lo;
      if (!warp_wait(bar_at(p, c, B.t_full + rt.slot), rt.phase, c.abort, p.err)) break;
      rt.next(p.nacc);
      tc_fence_after();
      float* orow = p.out + (size_t)(td.out_row + row) * p.n_out;
#pragma unroll 1
      for (int g = 0; g < g_n; ++g) {
        float v[8], im[8];
        tmem_ld8(t0 + 8 * g, v);
        tmem_ld8(t0 + 8 * ng + 8 * g, im);
        ld_wait8(v, im);
        if (g + 1 == g_n) {
          tc_fence_before();
          warp_arrive_leader(bar_at(p, c, B.t_empty + slot0));
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = fast_ln(fmaf(v[e], v[e], fmaf(im[e], im[e], p.eps)));
        if (valid) {
          const int m = m_lo + 8 * g;
          if (vec8 && m + 8 <= p.M) {
            store8(orow + m, v);
          } else {
#pragma unroll
            for (int e = 0; e < 8; ++e)
              if (m + e < p.M) orow[m + e] = v[e];
          }
        }
      }
    } else {
      float acc[kG][2][8];
      bool ok = true;
#pragma unroll
        for (int g = 0; g < kG; ++g)
#pragma unroll
          for (int e = 0; e < 8; ++e) acc[g][0][e] = acc[g][1][e] = 0.f;
        for (int left = unit_stages(p); left > 0; --left) {
          if (!warp_wait(bar_at(p, c, B.t_full + rt.slot), rt.phase, c.abort, p.err)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t t0 = tl + rt.slot * p.acc_cols + 8 * g_lo;
#pragma unroll
          for (int g = 0; g < kG; ++g)
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
          rt.next(p.nacc);
        }
      if (!ok) break;
      bool finite = true;
#pragma unroll
      for (int g = 0; g < kG; ++g)
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float s = fmaf(acc[g][0][e], acc[g][0][e], acc[g][1][e] * acc[g][1][e]);
          finite = finite && s < __int_as_float(0x7f800000);
          acc[g][0][e] = __logf(s + p.eps);
        }
      // Rows to look at again: those with a power that is not finite.  With finite
      // samples a power that overflows is the FFMA sum's too, a NaN is not.
      const float* x = p.wave + td.in_off + (long long)row * p.H;
      const int end = min(m_lo + 8 * g_n, p.M);
      const unsigned odd = __ballot_sync(0xffffffffu, !finite && valid);
      unsigned nans = 0;
      if (odd) {
        bool nan = false;
#pragma unroll
        for (int g = 0; g < kG; ++g)
#pragma unroll
          for (int e = 0; e < 8; ++e) nan |= acc[g][0][e] != acc[g][0][e];
        nans = __ballot_sync(0xffffffffu, nan);
      }
      const auto redo = [&](int l, float2& v) {  // false: row l stands
        const float* xl = x + (long long)(l - lane) * p.H;
        const int f = scan_row(xl, p.N);
        if (f == 0 && !(nans >> l & 1)) return false;
        v = f == 1 ? make_float2(__int_as_float(0x7fffffff), __int_as_float(0x7fffffff))
                   : redo_row(p, xl, m_lo, end, f == 2);
        return true;
      };
      if constexpr (!MFCC) {
        float* orow = p.out + (size_t)(td.out_row + row) * p.n_out;
        if (valid) {
#pragma unroll
          for (int g = 0; g < kG; ++g)
            if (g < g_n) {
              const int m = m_lo + 8 * g;
              if (vec8 && m + 8 <= p.M) {
                store8(orow + m, acc[g][0]);
              } else {
#pragma unroll
                for (int e = 0; e < 8; ++e)
                  if (m + e < p.M) orow[m + e] = acc[g][0][e];
              }
            }
        }
        __syncwarp();  // (the rows' own stores come before the recomputed ones)
        for (unsigned left = odd; left; left &= left - 1) {
          const int l = __ffs(left) - 1;
          float2 v;
          if (!redo(l, v)) continue;
          float* o = orow + (long long)(l - lane) * p.n_out + m_lo;
          if (m_lo + lane < end) o[lane] = v.x;
          if (m_lo + 32 + lane < end) o[32 + lane] = v.y;
        }
      } else {
        for (unsigned left = odd; left; left &= left - 1) {
          const int l = __ffs(left) - 1;
          float2 v;
          if (!redo(l, v)) continue;
#pragma unroll
          for (int g = 0; g < kG; ++g)
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const float t = __shfl_sync(0xffffffffu, 8 * g + e < 32 ? v.x : v.y, (8 * g + e) & 31);
              if (lane == l) acc[g][0][e] = t;
            }
        }
        // bins past M (zero basis rows) take no part, whatever their log is
#pragma unroll
        for (int g = 0; g < kG; ++g)
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
            for (int g = 0; g < kG; ++g)
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
          const uint32_t full = bar_at(p, c, B.part + 4 * quarter + rp.slot), empty = full + 16;
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
}

template <int P, bool MFCC>
__global__ void __launch_bounds__(slab_threads(P), 1) melt_slab_kernel(const __grid_constant__ SlabParams p) {
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
  const SlabBars B(p.NS, p.NB);
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  if (threadIdx.x == 0) {
    auto bar = [&](int i) { return bar_at(p, c, i); };
    for (int i = 0; i < p.NS; ++i) {
      mbar_init(bar(B.full + i), P < 3 ? 2 * p.tw : c.rank == 0 ? 4 : 1);
      mbar_init(bar(B.empty + i), 1);
      if constexpr (P < 3) mbar_init(bar(B.empty + p.NS + i), 1);
    }
    for (int i = 0; i < p.NB; ++i) {
      mbar_init(bar(B.b_full + i), c.rank == 0 ? 2 : 1);
      mbar_init(bar(B.b_empty + i), 1);
    }
    for (int i = 0; i < kMaxAcc; ++i) {
      mbar_init(bar(B.t_full + i), 1);
      mbar_init(bar(B.t_empty + i), 2 * kEpiWarps);
    }
    for (int i = 0; i < 16; ++i) mbar_init(bar(B.part + i), 1);
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
    for (int i = threadIdx.x; i < p.n_mfcc * ld; i += slab_threads(P)) {
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
    // (the whole warp walks the stages, so that descriptors and ring state can
    // stay in uniform registers; one elected lane issues)
    if constexpr (P == 3) {
      if (c.rank == 0) mma_issue(p, c, B, __shfl_sync(0xffffffffu, tmem, 0));
      else if (elect_one()) basis_signal(p, c, B);
    } else {
      if (c.rank == 0) mma_issue_slices<P>(p, c, B, __shfl_sync(0xffffffffu, tmem, 0));
      else if (elect_one()) basis_signal_slices(p, c, B);
    }
    __syncwarp();
    volatile int never = 0;
    mbar_wait(bar_at(p, c, B.drain), 0, &never, p.err, kErrTimeout);
    __syncwarp();
  } else if (warp == kBWarp) {
    if (elect_one()) {
      if constexpr (P == 3) basis_producer<P>(p, c, B);
      else basis_producer_slices<P>(p, c, B);
    }
    __syncwarp();
  } else if (warp >= kEpiWarps) {
    if (!p.early_inputs) pdl_wait();
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
