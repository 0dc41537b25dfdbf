// Folded full-grid likelihood (fold.cuh): the weights of an event and the
// batched evaluation.
#include <cuda_runtime.h>

#include "fold.cuh"
#include "kernels.h"

namespace swig {

// ---------------------------------------------------------------------------
// Node weights.  Moments M_m = sum_k D'(k) T_m(x_k) of each folded chunk (m <
// 64; T_m by the three-term recurrence), then W_j = (2 / 64) (M_0 / 2 + sum_m
// T_m(x_j) M_m), the discrete orthogonality of the Chebyshev nodes.  FP64
// throughout; about seven FP64 multiply-adds per (bin, m) for three detectors.
// ---------------------------------------------------------------------------
constexpr int kMomThreads = 128, kMomParts = 8;

__device__ __forceinline__ double2 fold_rotated(const FoldTables& F, const FoldChunk& ck, int det, int n_bins, int k,
                                                double x) {
  // D(k) exp(-2 pi i s (f_k - f_c)), s (f_k - f_c) = slope_h x
  double ph = ck.slope_h * x;
  ph -= rint(ph);
  double s, c;
  sincospi(2.0 * ph, &s, &c);
  const float2 d = F.data[(size_t)det * n_bins + k];
  return make_double2((double)d.x * c + (double)d.y * s, (double)d.y * c - (double)d.x * s);
}

template <int NDET>
__global__ void __launch_bounds__(kMomThreads)
    k_fold_moments(FoldTables F, const FoldChunk* __restrict__ chunks, int n_bins, double* __restrict__ mom) {
  extern __shared__ double sm[];
  double(*T)[kMomThreads + 1] = reinterpret_cast<double(*)[kMomThreads + 1]>(sm);  // [64][129]
  double(*Dr)[kMomThreads] = reinterpret_cast<double(*)[kMomThreads]>(sm + kFoldNodes * (kMomThreads + 1));
  const FoldChunk ck = chunks[blockIdx.x];
  const int tid = threadIdx.x, m = tid & (kFoldNodes - 1), half = tid / kFoldNodes;
  double acc[2 * NDET];
#pragma unroll
  for (int j = 0; j < 2 * NDET; ++j) acc[j] = 0.0;
  if (!ck.kind)
    for (int b = blockIdx.y * kMomThreads; b < ck.nbins; b += kMomParts * kMomThreads) {
      const int o = b + tid;
      const bool in = o < ck.nbins;
      const double x = in ? (double)(2 * o - (ck.nbins - 1)) / (double)(ck.nbins - 1) : 0.0;
      __syncthreads();
      double t0 = 1.0, t1 = x;
      for (int q = 0; q < kFoldNodes; ++q) {
        T[q][tid] = t0;
        const double t2 = 2.0 * x * t1 - t0;
        t0 = t1;
        t1 = t2;
      }
#pragma unroll
      for (int i = 0; i < NDET; ++i) {
        const double2 d = in ? fold_rotated(F, ck, i, n_bins, ck.k0 + o, x) : make_double2(0.0, 0.0);
        Dr[2 * i][tid] = d.x;
        Dr[2 * i + 1][tid] = d.y;
      }
      __syncthreads();
      constexpr int kPer = kMomThreads / 2;
      for (int q = half * kPer; q < (half + 1) * kPer; ++q) {
        const double t = T[m][q];
#pragma unroll
        for (int j = 0; j < 2 * NDET; ++j) acc[j] += t * Dr[j][q];
      }
    }
  __syncthreads();
  double* s2 = sm;  // [2 NDET][64]: the second half's sums
  if (half == 1)
#pragma unroll
    for (int j = 0; j < 2 * NDET; ++j) s2[j * kFoldNodes + m] = acc[j];
  __syncthreads();
  if (half == 0)
#pragma unroll
    for (int j = 0; j < 2 * NDET; ++j)
      mom[(((size_t)blockIdx.x * kMomParts + blockIdx.y) * 2 * NDET + j) * kFoldNodes + m] =
          acc[j] + s2[j * kFoldNodes + m];
}

// One warp per (chunk, detector): lane l forms the weights of nodes +x_l, -x_l.
template <int NDET>
__global__ void k_fold_weights(FoldTables F, const FoldChunk* __restrict__ chunks, int n_bins,
                               const double* __restrict__ mom, float4* __restrict__ w) {
  const int lane = threadIdx.x, i = blockIdx.y;
  const FoldChunk ck = chunks[blockIdx.x];
  double pr = 0.0, pi = 0.0, nr = 0.0, ni = 0.0;  // node +x, node -x
  if (ck.kind) {
    const int bw = 2 * kFoldNodes >> ck.kind;  // the block's bins
    const int kp = bw / 2 + lane, kn = bw / 2 - 1 - lane;
    const double x = (double)(2 * lane + 1) / (double)bw;
    if (lane < bw / 2 && kp < ck.nbins) {
      const double2 d = fold_rotated(F, ck, i, n_bins, ck.k0 + kp, x);
      pr = d.x, pi = d.y;
    }
    if (lane < bw / 2 && kn < ck.nbins) {
      const double2 d = fold_rotated(F, ck, i, n_bins, ck.k0 + kn, -x);
      nr = d.x, ni = d.y;
    }
  } else {
    const double x = cospi((2.0 * lane + 1.0) / (2.0 * kFoldNodes));
    double t0 = 1.0, t1 = x, er = 0.0, ei = 0.0, orr = 0.0, oi = 0.0;
    for (int m = 0; m < kFoldNodes; ++m) {
      double mr = 0.0, mi = 0.0;
      for (int p = 0; p < kMomParts; ++p) {
        const double* q = mom + (((size_t)blockIdx.x * kMomParts + p) * 2 * NDET + 2 * i) * kFoldNodes + m;
        mr += q[0];
        mi += q[kFoldNodes];
      }
      const double g = (m ? 2.0 : 1.0) / kFoldNodes * t0;
      if (m & 1) {
        orr += g * mr;
        oi += g * mi;
      } else {
        er += g * mr;
        ei += g * mi;
      }
      const double t2 = 2.0 * x * t1 - t0;
      t0 = t1;
      t1 = t2;
    }
    pr = er + orr, pi = ei + oi, nr = er - orr, ni = ei - oi;
  }
  w[((size_t)blockIdx.x * NDET + i) * 32 + lane] = make_float4((float)pr, (float)nr, (float)pi, (float)ni);
}

namespace {

template <int NDET>
cudaError_t weights_launch(const FoldTables& F, const FoldChunk* chunks, int n_bins, float4* w, cudaStream_t st) {
  double* mom = nullptr;
  cudaError_t e = cudaMalloc(&mom, sizeof(double) * (size_t)F.nc * kMomParts * 2 * NDET * kFoldNodes);
  if (e != cudaSuccess) return e;
  const size_t smem = sizeof(double) * (kFoldNodes * (kMomThreads + 1) + 2 * NDET * kMomThreads);
  e = cudaFuncSetAttribute(k_fold_moments<NDET>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) {
    k_fold_moments<NDET><<<dim3(F.nc, kMomParts), kMomThreads, smem, st>>>(F, chunks, n_bins, mom);
    k_fold_weights<NDET><<<dim3(F.nc, NDET), 32, 0, st>>>(F, chunks, n_bins, mom, w);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(mom);
  return e;
}

}  // namespace

cudaError_t launch_fold_weights(const LikeConst& L, const DeviceBuffers& B, const FoldChunk* chunks, cudaStream_t st) {
  const FoldTables F = fold_tables(B);
  switch (L.n_det) {
    case 1: return weights_launch<1>(F, chunks, L.n_bins, B.fold_w, st);
    case 2: return weights_launch<2>(F, chunks, L.n_bins, B.fold_w, st);
    case 3: return weights_launch<3>(F, chunks, L.n_bins, B.fold_w, st);
    default: return weights_launch<4>(F, chunks, L.n_bins, B.fold_w, st);
  }
}

// ---------------------------------------------------------------------------
// Batched evaluation: a CTA of 16 warps per parameter vector (grid-stride).
// ---------------------------------------------------------------------------
template <int NDET>
__global__ void __launch_bounds__(32 * kFoldWarps, 2)
    k_fold(LikeConst L, FoldTables F, const EvalRecord* __restrict__ rec, int n, double* __restrict__ out,
           double* __restrict__ kappa_out) {
  __shared__ __align__(16) float s_an[kFoldPanel * kFoldAnchor];
  __shared__ FoldIn s_in;
  __shared__ float s_sum[2 * NDET][kFoldWarps];
  __shared__ double s_dir[2 * NDET][kFoldWarps];
  __shared__ int s_bad;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int th = blockIdx.x; th < n; th += gridDim.x) {
    const EvalRecord& r = rec[th];
    __syncthreads();  // the previous vector's shared memory has been read
    if (tid < (int)(sizeof(FoldIn) / sizeof(float))) reinterpret_cast<float*>(&s_in)[tid] = fold_in_word(r, tid);
    if (tid == 0) s_bad = 0;
    const bool valid = r.valid != 0;  // block-uniform
    __syncthreads();
    FoldAcc<NDET> acc;
    acc.clear();
    if (valid)
      for (int base = 0; base < F.nc; base += kFoldPanel) {
        const int np = min(kFoldPanel, F.nc - base);
        const int npw = (np + 31) & ~31;  // a warp's lanes share one quarter
        for (int it = tid; it < 4 * npw; it += blockDim.x) {
          const int sub = it / npw, q = it - sub * npw;
          if (q < np && !fold_anchor<NDET>(F, s_in, sub, base + q, s_an + q * kFoldAnchor)) s_bad = 1;
        }
        __syncthreads();
        if (tid < np && !fold_in_band<NDET>(F, s_an + tid * kFoldAnchor, base + tid)) s_bad = 1;
        for (int q = warp; q < np; q += kFoldWarps)
          fold_chunk<NDET>(F, s_an + q * kFoldAnchor, base + q, lane, acc);
        if (base + kFoldPanel < F.nc) __syncthreads();
      }
#pragma unroll
    for (int i = 0; i < NDET; ++i) {
      float re, im;
      acc.total(i, re, im);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
      }
      if (lane == 0) {
        s_sum[2 * i][warp] = re;
        s_sum[2 * i + 1][warp] = im;
      }
    }
    __syncthreads();
    const bool bad = valid && s_bad;  // block-uniform
    if (bad) {
      double v[2 * NDET];
      fold_direct<NDET>(L, F, r, warp, kFoldWarps, lane, s_an + warp * kAnchorStride, v);
      if (lane == 0)
#pragma unroll
        for (int j = 0; j < 2 * NDET; ++j) s_dir[j][warp] = v[j];
      __syncthreads();
    }
    if (warp == 0) {
      // the warps' sums in FP64 by a fixed tree, component j on lane j
      double kapc = 0.0;
#pragma unroll
      for (int j = 0; j < 2 * NDET; ++j) {
        double v;
        if (bad) {
          v = lane < kFoldWarps ? s_dir[j][lane] : 0.0;
#pragma unroll
          for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        } else {
          dfl t = {lane < kFoldWarps ? s_sum[j][lane] : 0.0f, 0.0f};
#pragma unroll
          for (int o = 8; o > 0; o >>= 1)
            t = df_add(t, dfl{__shfl_xor_sync(0xffffffffu, t.hi, o), __shfl_xor_sync(0xffffffffu, t.lo, o)});
          v = (double)t.hi + (double)t.lo;
        }
        v = __shfl_sync(0xffffffffu, v, 0);
        if (lane == j) kapc = v;
      }
      const double ll = loglike_epilogue_warp<NDET>(L, r, kapc, lane);
      if (lane == 0) out[th] = ll;
      if (kappa_out && lane < 2 * SWIG_MAX_DET) kappa_out[(size_t)th * 2 * SWIG_MAX_DET + lane] = kapc;
    }
  }
}

namespace {

template <int NDET>
cudaError_t fold_launch(const LikeConst& L, const DeviceBuffers& B, int n, double* out, cudaStream_t st,
                        double* kappa_out) {
  const int grid = n < 2 * L.sm_count ? n : 2 * L.sm_count;
  k_fold<NDET><<<grid, 32 * kFoldWarps, 0, st>>>(L, fold_tables(B), B.rec, n, out, kappa_out);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_fold(const LikeConst& L, const DeviceBuffers& B, int n, double* out, cudaStream_t st,
                        double* kappa_out) {
  switch (L.n_det) {
    case 1: return fold_launch<1>(L, B, n, out, st, kappa_out);
    case 2: return fold_launch<2>(L, B, n, out, st, kappa_out);
    case 3: return fold_launch<3>(L, B, n, out, st, kappa_out);
    default: return fold_launch<4>(L, B, n, out, st, kappa_out);
  }
}

}  // namespace swig
