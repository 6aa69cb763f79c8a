// Host side of the slab kernel: the operand image, the shared-memory plan and
// the launch (device code in melt_slab_kernel.cuh).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <utility>
#include <vector>

#include "melt_slab_kernel.cuh"

namespace melt {

using namespace slab;

namespace {

constexpr uint32_t kSmemMax = 227 * 1024;

uint32_t up(uint32_t v, uint32_t a) { return (v + a - 1) / a * a; }

// BF16 (round to nearest even; zero below 2^-126) nearest to v, which becomes
// the exact remainder.
uint16_t take_bf16(double* v) {
  uint64_t d;
  std::memcpy(&d, v, 8);
  d = (d + ((uint64_t)1 << 44) - 1 + ((d >> 45) & 1)) & ~(((uint64_t)1 << 45) - 1);  // 8 significant bits
  double r;
  std::memcpy(&r, &d, 8);
  if (!(std::fabs(r) >= 1.1754943508222875e-38)) r = 0.0;
  const float f = (float)r;  // exact
  uint32_t bits;
  std::memcpy(&bits, &f, 4);
  *v -= r;
  return (uint16_t)(bits >> 16);
}

// MFCC: the DCT matrix and two buffers of eight coefficients of every row.
uint32_t mfcc_bytes(const SlabParams& p, int n_mfcc) {
  return n_mfcc > 0 ? up(4u * n_mfcc * 8u * p.groups, 128) + 2u * 8u * kF * 4u : 0u;
}

// Geometry and shared-memory plan.  P 3: false where two stages do not fit (three
// or more do for every basis that can be created).  P 1, 2: false where a tile
// has more rows than a converter copies at once, or its slabs and a few more do
// not fit beside the basis ring; P 1 also where hops above 416 leave two teams,
// which are slower than the single-CTA layouts (64 x 7.8 s, 41 geometries: 1.13
// times their time; at 944 / 656 / 64 27.6 us for 21.2; three teams 0.92 times).
bool plan(const SlabBasis* sb, int n_mfcc, SlabParams& p) {
  const int P = sb->parts;
  p.N = sb->n_fft;
  p.H = sb->hop;
  p.M = sb->n_mels;
  p.J = sb->J;
  p.n_slab = sb->n_slab;
  p.ksteps = sb->ksteps;
  p.groups = sb->groups;
  p.n_last = p.N - (p.J - 1) * p.H;
  // K-steps in equal stages of a slab's slices (P 3) or slots of a slice's slabs
  const int total = P == 3 ? p.J : p.n_slab, runs = (total + max_kps(P) - 1) / max_kps(P);
  p.kps = (total + runs - 1) / runs;
  p.step_bytes = (uint32_t)p.groups * P * 256u;
  const int rows = kF + (P == 3 ? p.kps : p.J) - 1;
  if (rows > kStageRows) return false;
  p.lbo_a = (uint32_t)(rows <= kRowsA ? kRowsA : kRowsA + 8) * 16u;
  p.a_part = 2 * p.lbo_a;
  p.a_bytes = up(P * p.a_part, 128);
  const int least = (p.groups + max_groups(P) - 1) / max_groups(P);  // blocks, and groups of the widest one
  const int wbg = 2 * ((p.groups / 2 + least - 1) / least);
  p.nacc = wbg <= 10 ? 3 : 2;
  p.acc_cols = wbg <= 10 ? 160 : 256;
  const uint32_t basis = up((uint32_t)wbg * P * 256u * p.kps, 128);
  const auto bars = [](int ns, int nb) { return up(8u * SlabBars(ns, nb).total, 128); };
  const uint32_t fixed = mfcc_bytes(p, n_mfcc) + 256u;
  uint32_t end = 0;  // of the rings
  if (P == 3) {
    p.stage = p.a_bytes + basis;
    // as many stages as fit, each of the first kMaxTeams with a converter warp's raw samples
    for (int ns = kMaxStages; ns >= 2 && !end; --ns) {
      p.NS = ns;
      p.ncv = std::min(ns, kMaxTeams);
      p.tw = 1;
      if (fixed + bars(kMaxStages, 0) + p.ncv * kRawBytes + ns * p.stage <= kSmemMax) end = p.stage * ns;
    }
  } else {
    p.stage = p.a_bytes;
    p.b_slot = basis;
    // As many converter teams and slabs beside the tile in use (up to another
    // tile of them) as leave three basis slots; then more of those.  Measured in
    // one process on a fixed input, split BF16 256 x 10 s: 6 / 4 / 3 teams 76 / 77 / 81 us with 5 slabs, 2 / 8
    // slabs (fewer teams) 82 / 78; BF16 at 22.05 kHz, 64 x 20 s: 10 / 7 / 4 slabs
    // 42.4 / 43.8 / 45.2.  (Never more teams than slots: see SlabParams::ncv.)
    for (int least_nb = 3; least_nb >= 2; --least_nb)
      for (int teams : {6, 4, 3, 2}) {
        const uint32_t other = fixed + teams * kRawBytes;
        const auto left = [&](int na, int nb) { return (int)(kSmemMax - other - bars(na, nb)) - (int)p.stage * na; };
        if (end || left(0, least_nb) < (int)(least_nb * basis)) continue;
        int na = std::min({(left(0, least_nb) - (int)(least_nb * basis)) / (int)p.stage, 2 * p.n_slab, kMaxA});
        if (left(na, least_nb) < (int)(least_nb * basis)) --na;  // (its own barriers)
        if (teams > na || (P == 1 && teams == 2 && p.n_slab > 26)) continue;
        if (na < p.n_slab + std::max(2, least_nb == 3 ? p.n_slab / 3 : 2)) continue;
        p.NS = na;
        p.NB = std::max(least_nb, std::min(kMaxB, left(na, kMaxB) / (int)basis));
        p.ncv = teams;
        p.tw = cvt_warps(P) / teams;
        p.off_b = p.stage * na;
        end = p.off_b + basis * p.NB;
      }
  }
  if (!end) return false;
  p.off_raw = end;
  p.off_bar = p.off_raw + p.ncv * kRawBytes;
  p.off_misc = p.off_bar + bars(p.NS, p.NB);
  p.off_dct = p.off_misc + 128u;
  p.off_part = p.off_dct + up(4u * n_mfcc * 8u * p.groups, 128);
  return true;
}

uint32_t smem_bytes(const SlabParams& p, int n_mfcc) { return p.off_dct + mfcc_bytes(p, n_mfcc) + 128u; }

}  // namespace

melt_status slab_build(SlabBasis* sb, int n_fft, int hop, int n_mels, int n_mfcc, int parts, const double* w64) {
  sb->parts = parts;
  sb->n_fft = n_fft;
  sb->hop = hop;
  sb->n_mels = n_mels;
  sb->J = (n_fft + hop - 1) / hop;
  sb->n_slab = (hop + 15) / 16;
  sb->groups = (n_mels + 15) / 16 * 2;
  const int n_last = n_fft - (sb->J - 1) * hop;
  sb->ksteps = sb->n_slab * (sb->J - 1) + (n_last + 15) / 16;
  SlabParams p;
  std::memset(&p, 0, sizeof(p));
  if (!plan(sb, n_mfcc, p)) return MELT_ERR_UNSUPPORTED;
  sb->layout = new (std::nothrow) SlabParams(p);
  if (!sb->layout) return MELT_ERR_OOM;
  const size_t half = (size_t)sb->ksteps * p.step_bytes;
  std::vector<uint16_t> img(half);  // two halves of half / 2 values each
  // K-steps slab by slab over the slices (P 3), or slice by slice over the slabs
  std::vector<std::pair<int, int>> steps;  // (slab, slice)
  if (parts == 3) {
    for (int kk = 0; kk < sb->n_slab; ++kk)
      for (int j = 0; j < (16 * kk < n_last ? sb->J : sb->J - 1); ++j) steps.push_back({kk, j});
  } else {
    for (int j = 0; j < sb->J; ++j)
      for (int kk = 0; kk < sb->n_slab && (j + 1 < sb->J || 16 * kk < n_last); ++kk) steps.push_back({kk, j});
  }
  for (int h = 0; h < 2; ++h) {
    uint16_t* step = img.data() + (size_t)h * (half / 2);
    for (const auto& sj : steps) {
      for (int m = 0; m < n_mels; ++m) {
        const double* w = w64 + ((size_t)h * n_mels + m) * n_fft;
        uint16_t* grp = step + (size_t)(m >> 3) * parts * 128 + (m & 7) * 8;
        for (int e = 0; e < 16; ++e) {
          const int r = 16 * sj.first + e, n = sj.second * hop + r;
          double v = r < hop && n < n_fft ? w[n] : 0.0;
          for (int t = 0; t < parts; ++t) grp[t * 128 + (e >> 3) * 64 + (e & 7)] = take_bf16(&v);
        }
      }
      step += p.step_bytes / 2;
    }
  }
  if (melt::dev_alloc(&sb->d_img, 2 * half) != cudaSuccess) return MELT_ERR_OOM;
  if (cudaMemcpy(sb->d_img, img.data(), 2 * half, cudaMemcpyHostToDevice) != cudaSuccess) return MELT_ERR_CUDA;
  return MELT_OK;
}

void slab_free(SlabBasis* sb) {
  cudaFree(sb->d_img);
  sb->d_img = nullptr;
  delete sb->layout;
  sb->layout = nullptr;
}

cudaError_t slab_launch(SlabBasis* sb, const SlabLaunch& L, cudaStream_t stream) {
  if (!sb->d_img || !sb->layout) return cudaErrorInvalidConfiguration;
  SlabParams p = *sb->layout;
  p.wave = L.wave;
  p.tiles = L.tiles;
  p.img = static_cast<const uint8_t*>(sb->d_img);
  p.dct = L.dct;
  p.w32 = L.w32;
  p.mp = L.mp;
  p.out = L.out;
  p.err = L.err;
  p.eps = L.eps;
  p.n_tiles = L.n_tiles;
  p.n_pairs = (L.n_tiles + 1) / 2;
  p.n_mfcc = L.n_mfcc;
  p.n_out = L.n_mfcc ? L.n_mfcc : sb->n_mels;
  p.early_inputs = L.early_inputs ? 1 : 0;
  void (*fn)(SlabParams) = sb->parts == 1   ? melt_slab_kernel<1, false>
                           : sb->parts == 2 ? melt_slab_kernel<2, false>
                           : L.n_mfcc       ? melt_slab_kernel<3, true>
                                            : melt_slab_kernel<3, false>;
  const int smem = (int)smem_bytes(p, L.n_mfcc);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  cfg.blockDim = dim3(slab_threads(sb->parts), 1, 1);
  if (sb->clusters < 0 || sb->clusters_smem != smem) {
    // (always the same limit, so that bases of different sizes do not lower each other's)
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
    if (e != cudaSuccess) return e;
    cfg.gridDim = dim3(2 * (L.sm_count / 2), 1, 1);
    int n = 0;
    e = cudaOccupancyMaxActiveClusters(&n, fn, &cfg);
    if (e != cudaSuccess) return e;
    sb->clusters = n;
    sb->clusters_smem = smem;
  }
  const int C = sb->clusters;
  if (C < 1) return cudaErrorInvalidConfiguration;
  // Blocks of Mel bins: as few as fit the epilogue's registers, or more where
  // the pairs leave clusters idle (a block below about 44 bins takes no less
  // time: reading A from shared memory bounds its MMAs).  MFCC sums over all
  // bins, so its blocks stay in one cluster.
  const int pairs16 = p.groups / 2;
  const int most = max_groups(sb->parts) / 2;
  int best = (pairs16 + most - 1) / most;
  if (L.n_mfcc == 0) {
    long long cost = -1;
    for (int nb = best, first = best; nb <= std::max(first, (pairs16 + 1) / 2); ++nb) {
      const int w = (pairs16 + nb - 1) / nb, n = (pairs16 + w - 1) / w;
      const long long rounds = ((long long)p.n_pairs * n + C - 1) / C;
      const long long t = rounds * (std::max(16 * w, 44) + 6);
      if (cost < 0 || t < cost) {
        cost = t;
        best = nb;
      }
    }
  }
  p.wbg = 2 * ((pairs16 + best - 1) / best);
  p.nblk = (p.groups + p.wbg - 1) / p.wbg;
  p.inner = L.n_mfcc ? p.nblk : 1;
  p.n_units = L.n_mfcc ? p.n_pairs : p.n_pairs * p.nblk;
  cfg.gridDim = dim3(2 * std::min(p.n_units, C), 1, 1);
  return cudaLaunchKernelEx(&cfg, fn, p);
}

}  // namespace melt
