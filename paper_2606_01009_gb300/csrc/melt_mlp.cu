// Learned per-frame correction of MelT features (a residual MLP) and its
// training step.  The paper does not evaluate such a layer: Sec. VI-C names a
// calibration layer as future work, and Sec. IV-H / Sec. V describe the
// MelT-to-STFT+Mel gap as mostly a per-band affine map.  The model:
//
//   xh = (x - mu) / sd                  per-band standardisation (fixed stats)
//   h  = xh W1^T + b1                   W1 [Hd x M]
//   a  = GELU(h) = 0.5 h (1 + erf(h / sqrt 2))
//   y  = x + a W2^T + b2                W2 [M x Hd], residual output
//   L  = mean over the batch and the M bands of (y - target)^2
//
// and AdamW with decoupled weight decay on every parameter.  Everything runs
// in FP32 on CUDA cores: one training step is a few hundred MFLOP, far too
// small to be worth tensor-core tiles, and FP32 keeps the gradients close
// enough to the FP64 definition to check them element by element.
//
// Kernels of one step (B = batch rows gathered through `rows`), three launches:
//   rows_kernel   8 rows per block: Xh, H = Xh W1^T + b1, A = GELU(H),
//                 Y = X + A W2^T + b2, dY = 2 (Y - T) / (B M), the loss, and
//                 dH = (dY W2) * GELU'(H); Xh, A, dY and dH go to memory
//   wgrad_kernel  dW1 = dH^T Xh, dW2 = dY^T A and the column sums db1, db2 over
//                 a slice of the batch, partial sums to memory
//   reduce_kernel sums the slices in order; in a training step also AdamW
// Each may start while the one before drains (programmatic dependent launch).
//
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include <cuda_bf16.h>

#include "melt_internal.h"

namespace {

constexpr int kMaxSmem = 227 * 1024;
constexpr int kMaxIn = 128;       // M (bands) limit of the fused apply kernel
constexpr int kApplyFrames = 64;  // frames per CTA of the fused apply kernel
constexpr int kApplyChunk = 64;   // hidden units per chunk of the fused apply kernel

__device__ __forceinline__ float gelu_f(float h) {
  return 0.5f * h * (1.0f + erff(h * 0.70710678118654752f));
}

__device__ __forceinline__ float gelu_grad_f(float h) {
  return 0.5f * (1.0f + erff(h * 0.70710678118654752f)) +
         h * 0.39894228040143268f * expf(-0.5f * h * h);
}

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void copy16(float* dst, const float* src, int bytes) {  // zeros past `bytes`
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void copy4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT>
__device__ __forceinline__ void copies_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
}

// ---- rows_kernel: forward and backward of 8 rows per block.
//
// Bound: a step of 1024 rows at 80 -> 256 -> 80 is 0.1 GFMA of FP32, about 3 us
// of the chip's FFMAs, so what counts is to have every SM at work and few
// launches.  8 rows per block make 128 blocks; the block holds UC hidden units
// of both weight matrices in shared memory (all of them up to 256 at 80 bands:
// one copy of 160 KB from L2, kept for the block's further rows), and its
// three products read shared memory about as long as they multiply:
//   H   thread = unit, its rows: one 16-byte read of W1 and one broadcast per
//       row for 4 FFMAs a row (W1 rows an odd number of 16-byte steps apart)
//   Y   warp = a run of units, lanes = bands: per four units one 16-byte read
//       per band and 8 broadcasts; the 8 warps' sums meet in shared memory
//   dH  thread = unit: one read of W2 and broadcasts of dY per band
// With more hidden units than UC, the block walks chunks of UC (weights copied
// per chunk, GELU' and A through memory).
// It replaces three 64 x 64-tile GEMM launches; with wgrad_kernel and
// reduce_kernel a gradient of 1024 rows went from 478 to 22 us on the GPU (4096
// rows: 1430 to 57), of which the serial column sums over the batch and the
// weight gradients on 8 blocks had taken most.
constexpr int kRows = 8, kRowThreads = 256, kRowWarps = kRowThreads / 32;

__host__ __device__ constexpr int rows_ld1(int M) { return 4 * (((M + 3) / 4) | 1); }
int rows_smem_bytes(int M, int UC) {
  const int M4 = (M + 3) / 4 * 4;
  return 4 * (UC * rows_ld1(M) + M * (UC + 4) + kRows * M4 + kRows * UC + kRows * M + kRowWarps * kRows * M);
}

struct RowsParams {
  const float *x, *t;
  const int64_t* rows;
  const float *W1, *b1, *W2, *b2, *mu, *sd;
  float *xh, *A, *dY, *dH, *loss;
  int B, M, Hd;
  float scale;  // 2 / (B M)
};

template <int UC, int MQ>
__global__ void __launch_bounds__(kRowThreads, 1) rows_kernel(RowsParams p) {
  extern __shared__ __align__(16) float sm[];
  constexpr int RPT = kRows * UC / kRowThreads;  // rows per thread in the H and dH products
  constexpr int ld2 = UC + 4;
  const int M = p.M, M4 = (M + 3) / 4 * 4, ld1 = rows_ld1(M), Hd = p.Hd;
  float* w1s = sm;                   // [UC][ld1]
  float* w2s = w1s + UC * ld1;       // [M][ld2]
  float* xs = w2s + M * ld2;         // [kRows][M4]
  float* as = xs + kRows * M4;       // [kRows][UC]
  float* dys = as + kRows * UC;      // [M][kRows]
  float* red = dys + kRows * M;      // [kRowWarps][kRows][M]
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int unit = t % UC, r0 = t / UC * RPT;  // H and dH products: this thread's unit and rows
  const int chunks = Hd / UC;
  pdl_next();
  pdl_wait();
  auto load_w1 = [&](int h0) {
    if ((M & 3) == 0) {
      const int q = M >> 2;
      for (int e = t; e < UC * q; e += kRowThreads) copy16(w1s + e / q * ld1 + e % q * 4, p.W1 + (size_t)h0 * M + 4 * e, 16);
    } else {
      for (int e = t; e < UC * M; e += kRowThreads) copy4(w1s + e / M * ld1 + e % M, p.W1 + (size_t)h0 * M + e);
    }
    copies_commit();
  };
  auto load_w2 = [&](int h0) {
    for (int e = t; e < M * (UC / 4); e += kRowThreads)
      copy16(w2s + e / (UC / 4) * ld2 + e % (UC / 4) * 4, p.W2 + (size_t)(e / (UC / 4)) * Hd + h0 + e % (UC / 4) * 4, 16);
    copies_commit();
  };
  if (M4 != M) {  // the columns that pad a row to 16 bytes
    for (int e = t; e < UC * (M4 - M); e += kRowThreads) w1s[e / (M4 - M) * ld1 + M + e % (M4 - M)] = 0.f;
    for (int e = t; e < kRows * (M4 - M); e += kRowThreads) xs[e / (M4 - M) * M4 + M + e % (M4 - M)] = 0.f;
  }
  if (chunks == 1) {
    load_w1(0);
    load_w2(0);
  }
  // this thread's elements (t, t + 256, ...) of the rows' bands: x and target are
  // fetched one block of rows ahead, so that the gathers' latency hides
  // behind the products of the rows before
  constexpr int kOwn = (kRows * kMaxIn + kRowThreads - 1) / kRowThreads;
  float xv[kOwn], tv[kOwn];
  auto gather = [&](int b0) {
#pragma unroll
    for (int k = 0; k < kOwn; ++k) {
      const int e = t + k * kRowThreads, r = e / M, m = e - r * M;
      xv[k] = tv[k] = 0.f;
      if (e < kRows * M && b0 + r < p.B) {
        const long long src = p.rows ? p.rows[b0 + r] : b0 + r;
        xv[k] = p.x[src * M + m];
        tv[k] = p.t[src * M + m];
      }
    }
  };
  gather(blockIdx.x * kRows);
  float loss = 0.f;
  bool first = true;
  for (int b0 = blockIdx.x * kRows; b0 < p.B; b0 += gridDim.x * kRows) {
    if (!first) __syncthreads();  // the previous rows' readers of xs, as, dys are done
    float xc[kOwn], tc[kOwn];
#pragma unroll
    for (int k = 0; k < kOwn; ++k) {
      const int e = t + k * kRowThreads, r = e / M, m = e - r * M;
      xc[k] = xv[k];
      tc[k] = tv[k];
      if (e < kRows * M) {
        float v = 0.f;
        if (b0 + r < p.B) {
          v = (xc[k] - p.mu[m]) / p.sd[m];
          p.xh[(size_t)(b0 + r) * M + m] = v;
        }
        xs[r * M4 + m] = v;
      }
    }
    if (b0 + (int)gridDim.x * kRows < p.B) gather(b0 + gridDim.x * kRows);
    float y[kRows][MQ];
#pragma unroll
    for (int r = 0; r < kRows; ++r)
#pragma unroll
      for (int q = 0; q < MQ; ++q) y[r][q] = 0.f;
    float gp[RPT];  // GELU'(H) of this thread's unit and rows (one chunk)
    for (int c = 0; c < chunks; ++c) {
      const int h0 = c * UC;
      if (chunks > 1) {
        __syncthreads();  // the previous chunk's readers of w1s, w2s and as are done
        load_w1(h0);
        load_w2(h0);
      }
      if (chunks > 1 || first) copies_wait<1>();
      __syncthreads();  // W1 and xs are in
      float h[RPT];
#pragma unroll
      for (int r = 0; r < RPT; ++r) h[r] = 0.f;
#pragma unroll 4
      for (int m = 0; m < M4; m += 4) {
        const float4 w = *reinterpret_cast<const float4*>(w1s + unit * ld1 + m);
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
          const float4 v = *reinterpret_cast<const float4*>(xs + (r0 + r) * M4 + m);
          h[r] = fmaf(v.x, w.x, h[r]);
          h[r] = fmaf(v.y, w.y, h[r]);
          h[r] = fmaf(v.z, w.z, h[r]);
          h[r] = fmaf(v.w, w.w, h[r]);
        }
      }
      const float bias = p.b1[h0 + unit];
#pragma unroll
      for (int r = 0; r < RPT; ++r) {
        const float v = h[r] + bias, a = gelu_f(v);
        gp[r] = gelu_grad_f(v);
        as[(r0 + r) * UC + unit] = a;
        if (b0 + r0 + r < p.B) {
          p.A[(size_t)(b0 + r0 + r) * Hd + h0 + unit] = a;
          if (chunks > 1) p.dH[(size_t)(b0 + r0 + r) * Hd + h0 + unit] = gp[r];
        }
      }
      if (chunks > 1 || first) copies_wait<0>();
      __syncthreads();  // W2 and this chunk's A are in
      const int j0 = warp * (UC / kRowWarps);
#pragma unroll 2
      for (int j = j0; j < j0 + UC / kRowWarps; j += 4) {
        float4 w[MQ];
#pragma unroll
        for (int q = 0; q < MQ; ++q) w[q] = *reinterpret_cast<const float4*>(w2s + min(lane + 32 * q, M - 1) * ld2 + j);
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
          const float4 a = *reinterpret_cast<const float4*>(as + r * UC + j);
#pragma unroll
          for (int q = 0; q < MQ; ++q) {
            y[r][q] = fmaf(a.x, w[q].x, y[r][q]);
            y[r][q] = fmaf(a.y, w[q].y, y[r][q]);
            y[r][q] = fmaf(a.z, w[q].z, y[r][q]);
            y[r][q] = fmaf(a.w, w[q].w, y[r][q]);
          }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < kRows; ++r)
#pragma unroll
      for (int q = 0; q < MQ; ++q)
        if (lane + 32 * q < M) red[(warp * kRows + r) * M + lane + 32 * q] = y[r][q];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kOwn; ++k) {
      const int e = t + k * kRowThreads, r = e / M, m = e - r * M;
      if (e >= kRows * M) continue;
      float d = 0.f;
      if (b0 + r < p.B) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < kRowWarps; ++w) s += red[w * kRows * M + e];
        d = xc[k] + s + p.b2[m] - tc[k];
        loss = fmaf(d, d, loss);
        d *= p.scale;
        p.dY[(size_t)(b0 + r) * M + m] = d;
      }
      dys[m * kRows + r] = d;
    }
    for (int c = 0; c < chunks; ++c) {
      const int h0 = c * UC;
      if (chunks > 1) {
        __syncthreads();  // the readers of w2s are done
        load_w2(h0);
        copies_wait<0>();
      }
      __syncthreads();  // dys (and W2) are in
      float g[RPT];
#pragma unroll
      for (int r = 0; r < RPT; ++r) g[r] = 0.f;
#pragma unroll 8
      for (int m = 0; m < M; ++m) {
        const float w = w2s[m * ld2 + unit];
        float d[RPT];
        if constexpr (RPT == 1) {
          d[0] = dys[m * kRows + r0];
        } else if constexpr (RPT == 2) {
          const float2 v = *reinterpret_cast<const float2*>(dys + m * kRows + r0);
          d[0] = v.x;
          d[1] = v.y;
        } else {
#pragma unroll
          for (int r = 0; r < RPT; r += 4) {
            const float4 v = *reinterpret_cast<const float4*>(dys + m * kRows + r0 + r);
            d[r] = v.x;
            d[r + 1] = v.y;
            d[r + 2] = v.z;
            d[r + 3] = v.w;
          }
        }
#pragma unroll
        for (int r = 0; r < RPT; ++r) g[r] = fmaf(d[r], w, g[r]);
      }
#pragma unroll
      for (int r = 0; r < RPT; ++r)
        if (b0 + r0 + r < p.B) {
          float* d = p.dH + (size_t)(b0 + r0 + r) * Hd + h0 + unit;
          *d = g[r] * (chunks > 1 ? *d : gp[r]);
        }
    }
    first = false;
  }
  if (first) copies_wait<0>();
  if (p.loss) {
#pragma unroll
    for (int o = 16; o; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    __syncthreads();
    if (lane == 0) red[warp] = loss;
    __syncthreads();
    if (t == 0) {
      float s = 0.f;
      for (int w = 0; w < kRowWarps; ++w) s += red[w];
      atomicAdd(p.loss, s);
    }
  }
}

// ---- wgrad_kernel: a 64-unit tile of dW1 (blockIdx.y 0: dH^T Xh, and db1) or
// dW2 (1: A^T dY, and db2 by tile 0) over one slice of the batch (blockIdx.z).
// Stages of 32 rows of both operands arrive by asynchronous copies while the
// previous stage multiplies; thread (ty, tx) owns units 4 ty .. 4 ty + 3 and
// bands tx + 16 q.  The batch is cut into enough slices to fill the chip (the
// 64 x 64 tiles over the whole batch before ran on 8 blocks); their partial
// sums are added in order by reduce_kernel.
constexpr int kStage = 32;

struct WgradParams {
  const float *xh, *A, *dY, *dH;
  float* part;        // [slices][n_params], packed like the parameters
  long long n_params;
  int B, M, Hd, slice;  // rows per slice
};

// Asks for more than half of an SM's shared memory, so that an SM takes one
// block: the blocks are scheduled while rows_kernel's still fill most SMs, and
// four or five of them would gather on the few free ones (1024 rows: 38.7 us
// a gradient that way, 22.1 with one to an SM).
int wgrad_smem_bytes(int M) { return std::max(4 * (2 * kStage * 64 + 2 * (kStage * M + 128)), 116 * 1024); }

template <int NQ>
__global__ void __launch_bounds__(256) wgrad_kernel(WgradParams p) {
  extern __shared__ __align__(16) float sm[];
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int M = p.M, Hd = p.Hd, j0 = blockIdx.x * 64;
  const bool second = blockIdx.y != 0;
  const float* P = second ? p.A : p.dH;   // [B][Hd]
  const float* Q = second ? p.dY : p.xh;  // [B][M]
  const int qs = kStage * M + 128;        // (a band lane past M reads on past its row)
  float* Ps = sm;                         // [2][kStage][64]
  float* Qs = sm + 2 * kStage * 64;       // [2][kStage][M]
  const int first = blockIdx.z * p.slice, end = min(first + p.slice, p.B);
  pdl_next();
  pdl_wait();
  auto load = [&](int k0, int s) {
    for (int e = t; e < kStage * 16; e += 256) {
      const int k = e >> 4, c = e & 15;
      const bool ok = k0 + k < end;
      copy16(Ps + (s * kStage + k) * 64 + 4 * c, P + (size_t)(ok ? k0 + k : first) * Hd + j0 + 4 * c, ok ? 16 : 0);
    }
    const long long from = (long long)k0 * M, left = (long long)(end - k0) * M;  // floats of this slice
    for (int e = 4 * t; e < kStage * M; e += 1024) {
      const int n = (int)min(4ll, max(0ll, left - e));
      copy16(Qs + s * qs + e, Q + (n ? from + e : 0), 4 * n);
    }
    copies_commit();
  };
  float acc[4][NQ];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc[i][q] = 0.f;
  float col = 0.f;  // column sum: unit j0 + t of dH, or band t of dY
  const bool sums = second ? blockIdx.x == 0 && t < M : t < 64;
  load(first, 0);
  int s = 0;
  for (int k0 = first; k0 < end; k0 += kStage, s ^= 1) {
    if (k0 + kStage < end) {
      load(k0 + kStage, s ^ 1);
      copies_wait<1>();
    } else {
      copies_wait<0>();
    }
    __syncthreads();
    const float* a = Ps + s * kStage * 64 + 4 * ty;
    const float* b = Qs + s * qs + tx;
#pragma unroll 8
    for (int k = 0; k < kStage; ++k) {
      const float4 v = *reinterpret_cast<const float4*>(a + k * 64);
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const float w = b[k * M + 16 * q];
        acc[0][q] = fmaf(v.x, w, acc[0][q]);
        acc[1][q] = fmaf(v.y, w, acc[1][q]);
        acc[2][q] = fmaf(v.z, w, acc[2][q]);
        acc[3][q] = fmaf(v.w, w, acc[3][q]);
      }
    }
    if (sums) {
      const float* cs = second ? Qs + s * qs + t : Ps + s * kStage * 64 + t;
      const int ld = second ? M : 64;
      float s0 = 0.f, s1 = 0.f;
#pragma unroll 8
      for (int k = 0; k < kStage; k += 2) {
        s0 += cs[k * ld];
        s1 += cs[(k + 1) * ld];
      }
      col += s0 + s1;
    }
    __syncthreads();  // this stage's readers are done before it is refilled
  }
  float* g = p.part + (size_t)blockIdx.z * p.n_params;
  const size_t w1 = (size_t)Hd * M;
  if (!second) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int q = 0; q < NQ; ++q)
        if (tx + 16 * q < M) g[(size_t)(j0 + 4 * ty + i) * M + tx + 16 * q] = acc[i][q];
    if (sums) g[w1 + j0 + t] = col;
  } else {
    g += w1 + Hd;
#pragma unroll
    for (int q = 0; q < NQ; ++q)
      if (tx + 16 * q < M) {
        float* row = g + (size_t)(tx + 16 * q) * Hd + j0 + 4 * ty;
#pragma unroll
        for (int i = 0; i < 4; ++i) row[i] = acc[i][q];
      }
    if (sums) g[w1 + t] = col;
  }
}

struct AdamW {
  float lr, b1, b2, eps, wd, c1, c2;
};

__device__ __forceinline__ void adamw_update(float* p, float* m, float* v, long long i, float gi, const AdamW& a) {
  const float mi = a.b1 * m[i] + (1.f - a.b1) * gi;
  const float vi = a.b2 * v[i] + (1.f - a.b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] = p[i] * (1.f - a.lr * a.wd) - a.lr * (mi * a.c1) / (sqrtf(vi * a.c2) + a.eps);
}

// Gradients from the slices' partial sums, added in order: to `grads`, or
// (grads null) straight into the AdamW update.
__global__ void reduce_kernel(const float* part, int slices, long long n, float* grads, float* prm, float* m, float* v,
                              AdamW a) {
  pdl_next();
  pdl_wait();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float g = 0.f;
#pragma unroll 8
  for (int s = 0; s < slices; ++s) g += part[s * n + i];
  if (grads) grads[i] = g;
  else adamw_update(prm, m, v, i, g, a);
}

__global__ void adamw_kernel(float* p, const float* g, float* m, float* v, long long n, AdamW a) {
  pdl_next();
  pdl_wait();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) adamw_update(p, m, v, i, g[i], a);
}

// Launch that may start while the stream's previous kernel drains (the kernels
// above touch memory only after griddepcontrol.wait).
template <class... A>
cudaError_t launch_pdl(void (*fn)(A...), dim3 grid, int threads, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fn, args...);
}

using RowsFn = void (*)(RowsParams);
template <int UC>
RowsFn rows_fn(int M) {
  switch ((M + 31) / 32) {
    case 1: return rows_kernel<UC, 1>;
    case 2: return rows_kernel<UC, 2>;
    case 3: return rows_kernel<UC, 3>;
    default: return rows_kernel<UC, 4>;
  }
}

RowsFn rows_fn(int M, int uc) { return uc == 256 ? rows_fn<256>(M) : uc == 128 ? rows_fn<128>(M) : rows_fn<64>(M); }

using WgradFn = void (*)(WgradParams);
WgradFn wgrad_fn(int M) {
  switch ((M + 15) / 16) {
    case 1: return wgrad_kernel<1>;
    case 2: return wgrad_kernel<2>;
    case 3: return wgrad_kernel<3>;
    case 4: return wgrad_kernel<4>;
    case 5: return wgrad_kernel<5>;
    case 6: return wgrad_kernel<6>;
    case 7: return wgrad_kernel<7>;
    default: return wgrad_kernel<8>;
  }
}

// Batch slices of the weight gradients: about 152 blocks over the tiles, at
// least 32 rows each (a stage), at most 32 slices.
int wgrad_slices(int Hd, int B) {
  const int want = std::max(1, 152 / (2 * (Hd / 64)));
  return std::max(1, std::min(std::min(want, 32), (B + kStage - 1) / kStage));
}

// Per-band population mean and standard deviation (two passes, one thread per band).
__global__ void stats_kernel(const float* x, long long n, int M, float* mu, float* sd) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= M) return;
  double s = 0.0;
  for (long long r = 0; r < n; ++r) s += x[r * M + m];
  const double mean = n > 0 ? s / (double)n : 0.0;
  double q = 0.0;
  for (long long r = 0; r < n; ++r) {
    const double d = x[r * M + m] - mean;
    q += d * d;
  }
  mu[m] = (float)mean;
  sd[m] = (float)fmax(sqrt(n > 0 ? q / (double)n : 0.0), 1e-6);
}

// Fused forward for inference: y = x + W2 GELU(W1 xh + b1) + b2 over kApplyFrames
// frames per CTA; the hidden layer is formed kApplyChunk units at a time in
// shared memory and never leaves the SM.  In place (y == x) is allowed: each
// output element is read and then written by the same thread.
// Dynamic shared memory: xs [F][M+1], w1c [C][M+1], w2c [M][C+1], ac [F][C+1].
int apply_smem_bytes(int M) {
  return 4 * (kApplyFrames * (M + 1) + kApplyChunk * (M + 1) + M * (kApplyChunk + 1) +
              kApplyFrames * (kApplyChunk + 1));
}

__global__ void __launch_bounds__(256) apply_kernel(const float* x, float* y, long long n,
                                                    const float* W1, const float* b1,
                                                    const float* W2, const float* b2,
                                                    const float* mu, const float* sd, int M,
                                                    int Hd) {
  extern __shared__ float sm[];
  const int ldx = M + 1, ldc = kApplyChunk + 1;
  float* xs = sm;                              // [kApplyFrames][ldx]
  float* w1c = xs + kApplyFrames * ldx;        // [kApplyChunk][ldx]
  float* w2c = w1c + kApplyChunk * ldx;        // [M][ldc]
  float* ac = w2c + M * ldc;                   // [kApplyFrames][ldc]
  const int t = threadIdx.x;
  const long long f0 = (long long)blockIdx.x * kApplyFrames;
  for (int e = t; e < kApplyFrames * M; e += 256) {
    const int f = e / M, m = e - f * M;
    xs[f * ldx + m] = (f0 + f < n) ? (x[(f0 + f) * M + m] - mu[m]) / sd[m] : 0.f;
  }
  // output accumulators: frames fy*4 .. +3, bands ox + 16 q
  const int fy = t >> 4, ox = t & 15;
  const int nq = (M + 15) >> 4;
  float acc[4][kMaxIn / 16];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int q = 0; q < kMaxIn / 16; ++q) acc[r][q] = 0.f;
  for (int h0 = 0; h0 < Hd; h0 += kApplyChunk) {
    __syncthreads();  // previous chunk fully consumed (and xs written, first time)
    for (int e = t; e < kApplyChunk * M; e += 256) {
      const int j = e / M, m = e - j * M;
      w1c[j * ldx + m] = W1[(long long)(h0 + j) * M + m];
    }
    for (int e = t; e < M * kApplyChunk; e += 256) {
      const int o = e / kApplyChunk, j = e - o * kApplyChunk;
      w2c[o * ldc + j] = W2[(long long)o * Hd + h0 + j];
    }
    __syncthreads();
    // hidden chunk: ac[f][j] = GELU(b1 + xs[f] . w1c[j]); thread: frames fy*4.., units ox*4..
    {
      float hacc[4][4];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) hacc[r][c] = 0.f;
      for (int m = 0; m < M; ++m) {
        float a[4], b[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) a[r] = xs[(fy * 4 + r) * ldx + m];
#pragma unroll
        for (int c = 0; c < 4; ++c) b[c] = w1c[(ox * 4 + c) * ldx + m];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) hacc[r][c] = fmaf(a[r], b[c], hacc[r][c]);
      }
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c)
          ac[(fy * 4 + r) * ldc + ox * 4 + c] = gelu_f(hacc[r][c] + b1[h0 + ox * 4 + c]);
    }
    __syncthreads();
    for (int j = 0; j < kApplyChunk; ++j) {
      float a[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) a[r] = ac[(fy * 4 + r) * ldc + j];
#pragma unroll
      for (int q = 0; q < kMaxIn / 16; ++q) {
        const int o = ox + 16 * q;
        if (q < nq && o < M) {
          const float w = w2c[o * ldc + j];
#pragma unroll
          for (int r = 0; r < 4; ++r) acc[r][q] = fmaf(a[r], w, acc[r][q]);
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const long long f = f0 + fy * 4 + r;
    if (f >= n) continue;
#pragma unroll
    for (int q = 0; q < kMaxIn / 16; ++q) {
      const int o = ox + 16 * q;
      if (q < nq && o < M) y[f * M + o] = x[f * M + o] + acc[r][q] + b2[o];
    }
  }
}

}  // namespace

struct melt_mlp {
  int device = 0;
  int M = 0, Hd = 0;
  long long n_params = 0;
  float* d_params = nullptr;  // [W1 | b1 | W2 | b2]
  float* d_grads = nullptr;   // same packing
  float* d_m = nullptr;
  float* d_v = nullptr;
  float* d_mu = nullptr;
  float* d_sd = nullptr;
  long long t = 0;            // AdamW steps taken
  double lr = 1e-3, beta1 = 0.9, beta2 = 0.999, eps = 1e-8, wd = 0.01;
  int cap = 0;                // batch rows the workspace holds
  float* d_xh = nullptr;
  float* d_A = nullptr;
  float* d_dY = nullptr;
  float* d_dH = nullptr;
  float* d_part = nullptr;    // partial weight gradients, one packed vector per batch slice
  int uc = 0;                 // hidden units a block of rows_kernel holds
  int sms = 0;
};

namespace {

long long param_count(int M, int Hd) { return 2LL * M * Hd + Hd + M; }

void free_ws(melt_mlp* p) {
  cudaFree(p->d_xh);
  cudaFree(p->d_A);
  cudaFree(p->d_dY);
  cudaFree(p->d_dH);
  cudaFree(p->d_part);
  p->d_xh = p->d_A = p->d_dY = p->d_dH = p->d_part = nullptr;
  p->cap = 0;
}

melt_status ensure_ws(melt_mlp* p, int batch) {
  if (batch <= p->cap) return MELT_OK;
  free_ws(p);
  const size_t h = (size_t)batch * p->Hd * sizeof(float), o = (size_t)batch * p->M * sizeof(float);
  const size_t g = (size_t)wgrad_slices(p->Hd, batch) * p->n_params * sizeof(float);
  if (melt::dev_alloc(&p->d_xh, o) != cudaSuccess || melt::dev_alloc(&p->d_A, h) != cudaSuccess ||
      melt::dev_alloc(&p->d_dY, o) != cudaSuccess || melt::dev_alloc(&p->d_dH, h) != cudaSuccess ||
      melt::dev_alloc(&p->d_part, g) != cudaSuccess) {
    free_ws(p);
    return MELT_ERR_OOM;
  }
  p->cap = batch;
  return MELT_OK;
}

AdamW adamw_of(const melt_mlp* p) {  // of step p->t
  AdamW a;
  a.lr = (float)p->lr;
  a.b1 = (float)p->beta1;
  a.b2 = (float)p->beta2;
  a.eps = (float)p->eps;
  a.wd = (float)p->wd;
  a.c1 = (float)(1.0 / (1.0 - std::pow(p->beta1, (double)p->t)));
  a.c2 = (float)(1.0 / (1.0 - std::pow(p->beta2, (double)p->t)));
  return a;
}

// Gradient of one batch to `grads`, or (null) an AdamW update from it.
melt_status grad_impl(melt_mlp* p, const float* X, const float* T, const int64_t* rows, int B,
                      float* grads, float* loss, cudaStream_t s) {
  const int M = p->M, Hd = p->Hd;
  RowsParams r;
  r.x = X;
  r.t = T;
  r.rows = rows;
  r.W1 = p->d_params;
  r.b1 = r.W1 + (long long)Hd * M;
  r.W2 = r.b1 + Hd;
  r.b2 = r.W2 + (long long)M * Hd;
  r.mu = p->d_mu;
  r.sd = p->d_sd;
  r.xh = p->d_xh;
  r.A = p->d_A;
  r.dY = p->d_dY;
  r.dH = p->d_dH;
  r.loss = loss;
  r.B = B;
  r.M = M;
  r.Hd = Hd;
  r.scale = 2.f / ((float)B * (float)M);
  const int blocks = std::min((B + kRows - 1) / kRows, p->sms);
  if (launch_pdl(rows_fn(M, p->uc), dim3(blocks), kRowThreads, rows_smem_bytes(M, p->uc), s, r) != cudaSuccess)
    return MELT_ERR_CUDA;
  WgradParams w;
  w.xh = p->d_xh;
  w.A = p->d_A;
  w.dY = p->d_dY;
  w.dH = p->d_dH;
  w.part = p->d_part;
  w.n_params = p->n_params;
  w.B = B;
  w.M = M;
  w.Hd = Hd;
  const int want = wgrad_slices(Hd, B);
  w.slice = ((B + want - 1) / want + kStage - 1) / kStage * kStage;
  const int slices = (B + w.slice - 1) / w.slice;
  if (launch_pdl(wgrad_fn(M), dim3(Hd / 64, 2, slices), 256, wgrad_smem_bytes(M), s, w) != cudaSuccess)
    return MELT_ERR_CUDA;
  const long long n = p->n_params;
  if (launch_pdl(reduce_kernel, dim3((unsigned)((n + 255) / 256)), 256, 0, s, (const float*)p->d_part, slices, n, grads,
                 p->d_params, p->d_m, p->d_v, grads ? AdamW{} : adamw_of(p)) != cudaSuccess)
    return MELT_ERR_CUDA;
  return MELT_OK;
}

melt_status check_batch(const melt_mlp* p, const float* X, const float* T, int batch) {
  if (!p || !X || !T || batch < 1) return MELT_ERR_ARG;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return MELT_ERR_CUDA;
  return dev == p->device ? MELT_OK : MELT_ERR_ARG;
}

}  // namespace

namespace melt {

// ---- image of the MLP for the CTA-pair kernel's fused epilogue
// Two halves, one per CTA of a pair; each half is
//   W1 blocks  MP/16 K-steps x [2 core columns][Hd/2 rows][8 bf16]   rows n of W1
//              from r*Hd/2 (hidden units), K = bands (zero past M)
//   W2 blocks  Hd/16 K-steps x [2 core columns][MP/2 rows][8 bf16]   rows o of W2
//              from r*MP/2 (bands, zero past M), K = hidden units
//   vectors    FP32 b1[Hd], b2[MP], mu[MP], 1/sd[MP] (zero past M), padded to 128 B
// The blocks are the no-swizzle K-major core-matrix layout of the tcgen05
// B operand (rows 16 B apart, the two core columns of a K-step Hd/2*16 or
// MP/2*16 bytes apart).
bool mlp_fused_shape_ok(int M, int Hd) {
  const int MP = (M + 15) / 16 * 16;
  return M >= 1 && MP <= 80 && Hd >= 64 && Hd <= 256 && Hd % 32 == 0 && MP <= Hd / 2 &&
         (MP / 2) % 8 == 0;
}

long long mlp_fused_half_bytes(int M, int Hd) {
  const int MP = (M + 15) / 16 * 16;
  const long long w1 = (long long)(MP / 16) * 2 * (Hd / 2) * 16;
  const long long w2 = (long long)(Hd / 16) * 2 * (MP / 2) * 16;
  const long long vec = ((long long)(Hd + 3 * MP) * 4 + 127) / 128 * 128;
  return w1 + w2 + vec;
}

__global__ void fused_image_kernel(const float* prm, const float* mu, const float* sd, int M, int Hd,
                                   uint8_t* img, long long half) {
  const int MP = (M + 15) / 16 * 16;
  const long long w1b = (long long)(MP / 16) * 2 * (Hd / 2) * 8;  // bf16 elements
  const long long w2b = (long long)(Hd / 16) * 2 * (MP / 2) * 8;
  const int nvec = Hd + 3 * MP;
  const long long per_half = w1b + w2b + nvec;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * per_half) return;
  const int r = (int)(i / per_half);
  long long e = i - (long long)r * per_half;
  uint8_t* base = img + (long long)r * half;
  const float* W1 = prm;
  const float* b1 = W1 + (long long)Hd * M;
  const float* W2 = b1 + Hd;
  const float* b2 = W2 + (long long)M * Hd;
  if (e < w1b) {
    const int rows = Hd / 2;
    const int s = (int)(e / (2 * rows * 8));
    const int rem = (int)(e - (long long)s * 2 * rows * 8);
    const int cc = rem / (rows * 8), row = (rem / 8) % rows, q = rem % 8;
    const int n = r * rows + row, k = 16 * s + 8 * cc + q;
    const float v = k < M ? W1[(long long)n * M + k] : 0.f;
    reinterpret_cast<__nv_bfloat16*>(base)[e] = __float2bfloat16_rn(v);
    return;
  }
  e -= w1b;
  if (e < w2b) {
    const int rows = MP / 2;
    const int s = (int)(e / (2 * rows * 8));
    const int rem = (int)(e - (long long)s * 2 * rows * 8);
    const int cc = rem / (rows * 8), row = (rem / 8) % rows, q = rem % 8;
    const int o = r * rows + row, k = 16 * s + 8 * cc + q;
    const float v = o < M ? W2[(long long)o * Hd + k] : 0.f;
    reinterpret_cast<__nv_bfloat16*>(base + w1b * 2)[e] = __float2bfloat16_rn(v);
    return;
  }
  e -= w2b;
  float* vec = reinterpret_cast<float*>(base + (w1b + w2b) * 2);
  const int j = (int)e;
  float v;
  if (j < Hd) v = b1[j];
  else if (j < Hd + MP) v = (j - Hd < M) ? b2[j - Hd] : 0.f;
  else if (j < Hd + 2 * MP) v = (j - Hd - MP < M) ? mu[j - Hd - MP] : 0.f;
  else v = (j - Hd - 2 * MP < M) ? 1.f / sd[j - Hd - 2 * MP] : 0.f;
  vec[j] = v;
}

melt_status mlp_apply(const melt_mlp* p, const float* x, float* y, long long n, cudaStream_t s) {
  if (n <= 0) return MELT_OK;
  const float* W1 = p->d_params;
  const float* b1 = W1 + (long long)p->Hd * p->M;
  const float* W2 = b1 + p->Hd;
  const float* b2 = W2 + (long long)p->M * p->Hd;
  const long long blocks = (n + kApplyFrames - 1) / kApplyFrames;
  if (blocks > 0x7fffffffLL) return MELT_ERR_ARG;
  const int smem = apply_smem_bytes(p->M);
  if (cudaFuncSetAttribute(apply_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
      cudaSuccess)
    return MELT_ERR_CUDA;
  apply_kernel<<<(unsigned)blocks, 256, smem, s>>>(x, y, n, W1, b1, W2, b2, p->d_mu, p->d_sd, p->M,
                                                   p->Hd);
  return cudaGetLastError() == cudaSuccess ? MELT_OK : MELT_ERR_CUDA;
}

int mlp_inputs(const melt_mlp* p) { return p->M; }

melt_status mlp_fused_image(const melt_mlp* p, void* d_img, cudaStream_t s) {
  const int MP = (p->M + 15) / 16 * 16;
  const long long per_half = (long long)(MP / 16) * 2 * (p->Hd / 2) * 8 +
                             (long long)(p->Hd / 16) * 2 * (MP / 2) * 8 + p->Hd + 3 * MP;
  const long long n = 2 * per_half;
  fused_image_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(
      p->d_params, p->d_mu, p->d_sd, p->M, p->Hd, static_cast<uint8_t*>(d_img),
      mlp_fused_half_bytes(p->M, p->Hd));
  return cudaGetLastError() == cudaSuccess ? MELT_OK : MELT_ERR_CUDA;
}

int mlp_hidden(const melt_mlp* p) { return p->Hd; }

int mlp_device(const melt_mlp* p) { return p->device; }

}  // namespace melt

extern "C" {

int64_t melt_mlp_num_params(int n_in, int n_hidden) {
  if (n_in < 1 || n_hidden < 1) return 0;
  return param_count(n_in, n_hidden);
}

melt_status melt_mlp_create(int n_in, int n_hidden, const float* params, const float* mu,
                            const float* sd, melt_mlp** out) {
  if (!out || !params || n_in < 1 || n_in > kMaxIn || n_hidden < kApplyChunk ||
      n_hidden % kApplyChunk != 0 || n_hidden > 4096)
    return MELT_ERR_ARG;
  *out = nullptr;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return MELT_ERR_NO_DEVICE;
  melt_mlp* p = new (std::nothrow) melt_mlp;
  if (!p) return MELT_ERR_OOM;
  p->device = dev;
  p->M = n_in;
  p->Hd = n_hidden;
  p->n_params = param_count(n_in, n_hidden);
  // the most hidden units (256, 128 or 64, dividing Hd) whose weights fit a block's shared memory
  p->uc = 256;
  while (p->uc > 64 && (n_hidden % p->uc != 0 || rows_smem_bytes(n_in, p->uc) > kMaxSmem)) p->uc /= 2;
  // (the limit is set to the same value whatever the sizes, for every MLP of the process)
  if (cudaDeviceGetAttribute(&p->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaFuncSetAttribute(rows_fn(n_in, p->uc), cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem) != cudaSuccess ||
      cudaFuncSetAttribute(wgrad_fn(n_in), cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem) != cudaSuccess) {
    delete p;
    return MELT_ERR_NO_DEVICE;
  }
  const size_t pb = (size_t)p->n_params * sizeof(float);
  bool ok = melt::dev_alloc(&p->d_params, pb) == cudaSuccess && melt::dev_alloc(&p->d_grads, pb) == cudaSuccess &&
            melt::dev_alloc(&p->d_m, pb) == cudaSuccess && melt::dev_alloc(&p->d_v, pb) == cudaSuccess &&
            melt::dev_alloc(&p->d_mu, n_in * sizeof(float)) == cudaSuccess &&
            melt::dev_alloc(&p->d_sd, n_in * sizeof(float)) == cudaSuccess;
  if (ok) {
    std::vector<float> m0(n_in, 0.f), s0(n_in, 1.f);
    ok = cudaMemcpy(p->d_params, params, pb, cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemset(p->d_grads, 0, pb) == cudaSuccess && cudaMemset(p->d_m, 0, pb) == cudaSuccess &&
         cudaMemset(p->d_v, 0, pb) == cudaSuccess &&
         cudaMemcpy(p->d_mu, mu ? mu : m0.data(), n_in * sizeof(float), cudaMemcpyHostToDevice) ==
             cudaSuccess &&
         cudaMemcpy(p->d_sd, sd ? sd : s0.data(), n_in * sizeof(float), cudaMemcpyHostToDevice) ==
             cudaSuccess;
  }
  if (!ok) {
    melt_mlp_destroy(p);
    return MELT_ERR_OOM;
  }
  *out = p;
  return MELT_OK;
}

melt_status melt_mlp_fit_stats(melt_mlp* p, const float* X, int64_t n, void* stream) {
  if (!p || !X || n < 1) return MELT_ERR_ARG;
  stats_kernel<<<(p->M + 63) / 64, 64, 0, (cudaStream_t)stream>>>(X, n, p->M, p->d_mu, p->d_sd);
  return cudaGetLastError() == cudaSuccess ? MELT_OK : MELT_ERR_CUDA;
}

melt_status melt_mlp_set_adamw(melt_mlp* p, double lr, double beta1, double beta2, double eps,
                               double wd) {
  if (!p || !(lr >= 0) || !(beta1 >= 0 && beta1 < 1) || !(beta2 >= 0 && beta2 < 1) || !(eps > 0) ||
      !(wd >= 0))
    return MELT_ERR_ARG;
  p->lr = lr;
  p->beta1 = beta1;
  p->beta2 = beta2;
  p->eps = eps;
  p->wd = wd;
  return MELT_OK;
}

melt_status melt_mlp_grad(melt_mlp* p, const float* X, const float* target, const int64_t* rows,
                          int batch, float* grads, float* loss, void* stream) {
  melt_status st = check_batch(p, X, target, batch);
  if (st != MELT_OK) return st;
  if ((st = ensure_ws(p, batch)) != MELT_OK) return st;
  return grad_impl(p, X, target, rows, batch, grads ? grads : p->d_grads, loss, (cudaStream_t)stream);
}

melt_status melt_mlp_train_step(melt_mlp* p, const float* X, const float* target,
                                const int64_t* rows, int batch, float* loss, void* stream) {
  melt_status st = check_batch(p, X, target, batch);
  if (st != MELT_OK) return st;
  if ((st = ensure_ws(p, batch)) != MELT_OK) return st;
  cudaStream_t s = (cudaStream_t)stream;
  p->t += 1;
  if ((st = grad_impl(p, X, target, rows, batch, nullptr, loss, s)) != MELT_OK) p->t -= 1;
  return st;
}

melt_status melt_mlp_adamw_apply(melt_mlp* p, const float* grads, void* stream) {
  if (!p || !grads) return MELT_ERR_ARG;
  p->t += 1;
  const long long n = p->n_params;
  return launch_pdl(adamw_kernel, dim3((unsigned)((n + 255) / 256)), 256, 0, (cudaStream_t)stream, p->d_params, grads,
                    p->d_m, p->d_v, n, adamw_of(p)) == cudaSuccess
             ? MELT_OK
             : MELT_ERR_CUDA;
}

melt_status melt_mlp_forward(const melt_mlp* p, const float* X, float* Y, int64_t n, void* stream) {
  if (!p || n < 0 || (n > 0 && (!X || !Y))) return MELT_ERR_ARG;
  return melt::mlp_apply(p, X, Y, n, (cudaStream_t)stream);
}

melt_status melt_mlp_get_params(const melt_mlp* p, float* params, float* mu, float* sd) {
  if (!p) return MELT_ERR_ARG;
  if (cudaDeviceSynchronize() != cudaSuccess) return MELT_ERR_CUDA;
  if (params && cudaMemcpy(params, p->d_params, (size_t)p->n_params * sizeof(float),
                           cudaMemcpyDeviceToHost) != cudaSuccess)
    return MELT_ERR_CUDA;
  if (mu && cudaMemcpy(mu, p->d_mu, p->M * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess)
    return MELT_ERR_CUDA;
  if (sd && cudaMemcpy(sd, p->d_sd, p->M * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess)
    return MELT_ERR_CUDA;
  return MELT_OK;
}

melt_status melt_mlp_destroy(melt_mlp* p) {
  if (!p) return MELT_OK;
  cudaDeviceSynchronize();
  free_ws(p);
  cudaFree(p->d_params);
  cudaFree(p->d_grads);
  cudaFree(p->d_m);
  cudaFree(p->d_v);
  cudaFree(p->d_mu);
  cudaFree(p->d_sd);
  delete p;
  return MELT_OK;
}

}  // extern "C"
