// Host interface of the slab kernel (melt_slab_kernel.cuh): the projection in
// CTA pairs with both operands streamed through shared memory in K slabs.
#pragma once

#include "melt_internal.h"

namespace melt {

namespace slab {
struct SlabParams;
}

// Device-resident operands of one basis for the slab kernel.
struct SlabBasis {
  int parts = 0;                       // BF16 parts per operand: 3 for the FP32 form, 2 for split BF16, 1 for BF16
  int n_fft = 0, hop = 0, n_mels = 0;
  int J = 0, n_slab = 0, ksteps = 0;   // polyphase slices, 16-sample slabs, MMA K-steps
  int groups = 0;                      // groups of 8 Mel bins
  void* d_img = nullptr;               // two halves (W_r rows, W_i rows) of K-step blocks
  slab::SlabParams* layout = nullptr;  // geometry and shared-memory plan (the launch's other fields are zero)
  int clusters = -1, clusters_smem = 0;  // co-resident clusters of the kernel at that shared-memory size
};

struct SlabLaunch {
  const float* wave;
  const TileDesc* tiles;
  int n_tiles;
  float* out;
  const float* dct;    // [n_mfcc][n_mels] or nullptr
  const float* w32;    // [n_fft][2 mp] FP32 basis (the tiles the split operands cannot hold)
  int mp;
  int n_mfcc;
  float eps;
  int* err;
  int sm_count;
  bool early_inputs;   // MELT_FWD_INPUT_READY: the waveform readers need not wait for the kernel before
};

// Builds the operand image for `parts` BF16 parts; MELT_ERR_UNSUPPORTED (with
// nothing allocated) where the rings of 1 or 2 parts do not fit shared memory.
melt_status slab_build(SlabBasis* sb, int n_fft, int hop, int n_mels, int n_mfcc, int parts, const double* w64);
void slab_free(SlabBasis* sb);
cudaError_t slab_launch(SlabBasis* sb, const SlabLaunch& L, cudaStream_t stream);

}  // namespace melt
