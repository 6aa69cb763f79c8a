// Host check of the FP8 converters' waits for staged chunks, from the planner's own
// code (no GPU), over frame lengths, hops, bin and coefficient counts.  Where two
// groups of converter warps take the chunks in turn, a group sees only some of the
// completions of a slot's barrier, copies may complete in any order, and a parity
// wait cannot tell a phase from the one two before it.  The check replays every
// wait of a group against every count of completions that the barrier may have by
// then, given only what is proven by the time: the group's own chunks before had
// landed, so they had been issued; the producer issues in order, each chunk into a
// slot that had been released, so every chunk a ring before the group's last one
// had landed; and all warps meet between tiles, so earlier tiles' chunks had.
#include <cstdio>
#include <map>

#include "melt_tc.cu"

namespace melt {
cudaError_t dev_alloc_bytes(void**, size_t) { return cudaErrorMemoryAllocation; }
melt_status mlp_fused_image(const melt_mlp*, void*, cudaStream_t) { return MELT_ERR_CUDA; }
cudaError_t slab_launch(SlabBasis*, const SlabLaunch&, cudaStream_t) { return cudaErrorInvalidValue; }
namespace tc {
KernelFn kernel_for_plain(int, int, bool) { return nullptr; }
KernelFn kernel_for_mfcc(int, int) { return nullptr; }
KernelFn kernel_for_pair(bool, int, bool, int) { return nullptr; }
KernelFn kernel_for_pair_mlp(int) { return nullptr; }
KernelFn kernel_for_pair_fp8(bool, int, bool, int) { return nullptr; }
KernelFn kernel_for_pair_x3() { return nullptr; }
GroupKernelFn kernel_for_pair_group() { return nullptr; }
}  // namespace tc
}  // namespace melt

using namespace melt;
using namespace melt::tc;

// First chunk whose wait may pass before it has landed; -1 if there is none.
static int unsound(int slots, int chunks, int groups) {
  for (int w = 0; w < groups; ++w)
    for (int c = w; c < 12 * slots * chunks; c += groups) {
      const auto landed = [&](int d) {  // known to this group
        return (d < c && d % groups == w) || d <= c - groups - slots || d / chunks < c / chunks;
      };
      const int round = c / slots;  // completions of the barrier by earlier rounds: all `round`, known:
      int least = 0;
      while (least < round && landed(least * slots + c % slots)) ++least;
      for (int n = least; n <= round + 1; ++n)  // round: chunk c has not landed, round + 1: it has
        if (((n & 1) != (round & 1)) != (n > round)) return c;
    }
  return -1;
}

int main() {
  long plans = 0, two = 0, bad = 0;
  std::map<int, int> seen;
  char image = 0;
  for (int n_fft = 16; n_fft <= 4096; n_fft += n_fft < 512 ? 4 : 20)
    for (int hop = 4; hop <= 256 && hop <= n_fft; hop += 4)
      for (int mels : {13, 40, 80, 100, 128})
        for (int mfcc : {0, 13, 40}) {
          if (mfcc > mels) continue;
          TcBasis tb;
          tb.precision = MELT_FP8E4M3;
          tb.n_fft = n_fft;
          tb.hop = hop;
          tb.n_mels = mels;
          tb.n_mfcc = mfcc;
          tb.J = (n_fft + hop - 1) / hop;
          tb.n_cols = 2 * ((mels + 15) / 16 * 16);
          tb.kstep_k = 32;
          tb.kstep_bytes = (size_t)tb.n_cols * 32;
          for (int j = 0; j < tb.J; ++j) tb.ksteps += (std::min(hop, n_fft - j * hop) + 31) / 32;
          tb.d_b2 = reinterpret_cast<decltype(tb.d_b2)>(&image);  // (never read)
          TcParams p;
          std::memset(&p, 0, sizeof(p));
          if (!plan_smem(&tb, p, mfcc)) continue;
          ++plans;
          two += p.cvt_groups == 2;
          const auto it = seen.emplace((p.NS * 1024 + p.NCHUNK) * 4 + p.cvt_groups, 0);
          if (it.second) it.first->second = unsound(p.NS, p.NCHUNK, p.cvt_groups);
          if (it.first->second >= 0 && bad++ < 20)
            std::printf("%d / %d / %d / %d: %d groups, %d slots, %d chunks: chunk %d\n", n_fft, hop, mels, mfcc,
                        p.cvt_groups, p.NS, p.NCHUNK, it.first->second);
        }
  std::printf("plans %ld two groups %ld bad %ld\n", plans, two, bad);
  return two > 0 && two < plans && bad == 0 ? 0 : 1;
}
