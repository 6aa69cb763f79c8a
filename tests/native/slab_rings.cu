// Host check of the slab kernel's shared-memory plans, from the planner's own
// code (no GPU): over every frame length, hop and bin count that the forms of
// one and two parts accept, a converter team is never more than a ring ahead of
// the place it waits for.  (A team that has converted slab g waits for the place
// of slab g + ncv by one parity bit, which cannot tell a phase from the one two
// before it: with more teams than slots the wait passes while slabs of the
// previous turn are still in use.)
#include <cstdio>

#include "melt_slab.cu"

namespace melt {
cudaError_t dev_alloc_bytes(void**, size_t) { return cudaErrorMemoryAllocation; }
}  // namespace melt

using namespace melt;
using namespace melt::slab;

int main() {
  long plans = 0, bad = 0;
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
          if (p.ncv < 1 || p.ncv > p.NS) {
            if (bad++ < 20)
              std::printf("parts %d, %d / %d / %d: %d teams, %d slots\n", parts, n_fft, hop, mels, p.ncv, p.NS);
          }
        }
  std::printf("plans %ld bad %ld\n", plans, bad);
  return plans > 0 && bad == 0 ? 0 : 1;
}
