// Host check of the slab kernel's shared-memory plans and ring waits, from the
// planner's and the kernel's own code (no GPU), over every frame length, hop and
// bin count that the forms of one and two parts accept.  (Of the three-part form,
// whose stages are freed in order, only the rule that there are no more teams than
// stages is checked, over every hop and every 20th length.)  Converter teams take
// slabs in turn, so a team sees only some of the completions of a slot's
// barriers, and a parity wait cannot tell a phase from the one two before it.
// The check replays every wait of a team against every count of completions that
// the barrier may have by then, given only what the team's earlier waits prove:
//   - the slabs whose places it took itself had been freed;
//   - the MMAs take slabs in order, so if slab h was freed, every slab up to h
//     had been filled, hence the previous holder of each of their places freed.
// (Slabs are not freed in order: those past the last slice's end go first.)
#include <algorithm>
#include <cstdio>
#include <vector>

#include "melt_slab.cu"

namespace melt {
cudaError_t dev_alloc_bytes(void**, size_t) { return cudaErrorMemoryAllocation; }
}  // namespace melt

using namespace melt;
using namespace melt::slab;

// First slab whose wait may pass before its place is free; -1 if there is none.
static long unsound(int NS, int ncv) {
  if (ncv < 1 || ncv > NS) return 0;
  for (int w = 0; w < ncv; ++w) {
    long known = -1, filled = -1;  // the latest slab this team knows to be freed; all up to `filled` were filled
    for (long g = w; g < 4L * NS + (long)NS * ncv; g += ncv) {
      const int slot = (int)(g % NS), turn = (int)(g / NS);
      if (turn > 0) {
        const int bar = freed_bar(NS, slot, turn - 1);
        const int pos = (int)(g % (2 * NS));
        const uint32_t parity = place_parity(NS, pos, (uint32_t)(g / (2 * NS)));
        if (place_bar(NS, pos) != bar) return g;
        // completions of that barrier: by earlier turns of its slot, those the team knows of and all
        long least = 0, need = 0;
        bool sure = true;
        for (int t = 0; t < turn - 1; ++t)
          if (freed_bar(NS, slot, t) == bar) {
            const long s = (long)t * NS + slot;
            // s is known to be freed: its place was filled again, or this team took its place
            sure = sure && (s + NS <= filled || (s + NS < g && (s + NS) % ncv == w));
            if (sure) ++least;
            ++need;
          }
        for (long c = least; c <= need + 1; ++c) {  // need: the turn before has not freed the slot, need + 1: it has
          const bool passes = ((uint32_t)c & 1u) != parity;
          if (passes != (c > need)) return g;
        }
        known = std::max(known, g - NS);
        filled = std::max(filled, known);
      }
    }
  }
  return -1;
}

int main() {
  long plans = 0, bad = 0;
  std::vector<int> seen(64 * 64, -2);
  for (int parts = 1; parts <= 2; ++parts)
    for (int n_fft = 16; n_fft <= 4096; n_fft += 4)
      for (int hop = 16; hop <= n_fft; hop += 16)
        for (int mels = 16; mels <= 128; mels += 16) {
          SlabBasis sb;
          sb.parts = parts;
          sb.n_fft = n_fft;
          sb.hop = hop;
          sb.n_mels = mels;
          sb.J = (n_fft + hop - 1) / hop;
          sb.n_slab = (hop + 15) / 16;
          sb.groups = (mels + 15) / 16 * 2;
          sb.ksteps = sb.n_slab * (sb.J - 1) + (n_fft - (sb.J - 1) * hop + 15) / 16;
          SlabParams p;
          std::memset(&p, 0, sizeof(p));
          if (!plan(&sb, 0, p)) continue;
          ++plans;
          int& s = seen[p.NS * 64 + p.ncv];
          if (s == -2) s = (int)unsound(p.NS, p.ncv);
          if (smem_bytes(p, 0) > 227u * 1024u && bad++ < 20)
            std::printf("parts %d, %d / %d / %d: %u bytes of shared memory\n", parts, n_fft, hop, mels, smem_bytes(p, 0));
          if (s >= 0 && bad++ < 20)
            std::printf("parts %d, %d / %d / %d: %d teams, %d slots, slab %d\n", parts, n_fft, hop, mels, p.ncv, p.NS, s);
        }
  for (int n_fft = 16; n_fft <= 4096; n_fft += n_fft < 256 ? 4 : 20)
    for (int hop = 4; hop <= n_fft; hop += 4)
      for (int mels : {1, 17, 80, 81, 128})
        for (int mfcc : {0, 13}) {
          if (mfcc > mels) continue;
          SlabBasis sb;
          sb.parts = 3;
          sb.n_fft = n_fft;
          sb.hop = hop;
          sb.n_mels = mels;
          sb.J = (n_fft + hop - 1) / hop;
          sb.n_slab = (hop + 15) / 16;
          sb.groups = (mels + 15) / 16 * 2;
          SlabParams p;
          std::memset(&p, 0, sizeof(p));
          const bool ok = plan(&sb, mfcc, p);
          ++plans;
          if (!ok || p.ncv < 1 || p.ncv > p.NS || smem_bytes(p, mfcc) > 227u * 1024u) ++bad;
        }
  std::printf("plans %ld bad %ld\n", plans, bad);
  return plans > 0 && bad == 0 ? 0 : 1;
}
