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
  e = allow_shared((const void*)k_fold_moments<NDET>);
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
// Batched evaluation.  A team of T warps (T a power of two up to 16, a CTA
// holds 16 / T teams) takes one parameter vector at a time: anchors of a panel
// of chunks into shared memory, a warp per chunk over its nodes, the warps'
// sums and the FP64 epilogue on the team's first warp.  An evaluation is a
// chain of latencies (table loads, the double-float sums, the epilogue's FP64),
// so a team waits more than it works: small batches take T = 16 for the
// shortest chain, large ones one warp per vector and as many vectors in flight
// as there are warps (32 per SM), without block barriers.
// ---------------------------------------------------------------------------
constexpr int kFoldSlots = 512;  // anchors in shared memory, all teams together

// Dynamic shared memory: anchors, abscissae and, RES, the weights and table.
inline __host__ __device__ size_t fold_fixed_bytes() {
  return sizeof(float) * kFoldSlots * kFoldAnchor + sizeof(float2) * 32 * kFoldKinds;
}
__device__ __forceinline__ void team_sync(int team, int T) {
  if (T == 1)
    __syncwarp();
  else
    named_barrier(1 + team, 32 * T);
}

template <int NDET, bool RES>
__global__ void __launch_bounds__(32 * kFoldWarps, 1)
    k_fold(LikeConst L, FoldTables F, const EvalRecord* __restrict__ rec, int n, int T, double* __restrict__ out,
           double* __restrict__ kappa_out) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ FoldIn s_in[kFoldWarps];
  __shared__ float2 s_sum[2 * NDET][kFoldWarps];
  __shared__ double s_dir[2 * NDET][kFoldWarps];
  __shared__ int s_bad[kFoldWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int team = warp / T, tw = warp - team * T, tid = 32 * tw + lane;  // within the team
  const int teams = kFoldWarps / T, panel = min(128, kFoldSlots / teams);
  float* s_anchor = reinterpret_cast<float*>(smem);
  float2* s_x = reinterpret_cast<float2*>(s_anchor + kFoldSlots * kFoldAnchor);
  const float4* w = F.w;
  const float* tab = F.tab;
  const int ld = F.ld;
  if (RES) {
    float4* s_w = reinterpret_cast<float4*>(s_x + 32 * kFoldKinds);
    float4* s_t = s_w + F.nc * NDET * 32;
    const float4* g_t = reinterpret_cast<const float4*>(F.tab);
    for (int k = threadIdx.x; k < FR_ROWS * ld / 4; k += blockDim.x) cp_async16(s_t + k, g_t + k);
    for (int k = threadIdx.x; k < F.nc * NDET * 32; k += blockDim.x) cp_async16(s_w + k, F.w + k);
    w = s_w;
    tab = reinterpret_cast<const float*>(s_t);
  }
  for (int k = threadIdx.x; k < 32 * kFoldKinds; k += blockDim.x) s_x[k] = F.x[k];
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  // the set-up kernel's records, while this one's start overlapped its end
  asm volatile("griddepcontrol.wait;" ::: "memory");
  float* an = s_anchor + team * panel * kFoldAnchor;
  const float2 x0 = s_x[lane];
  for (int th = blockIdx.x * teams + team; th < n; th += gridDim.x * teams) {
    const EvalRecord& r = rec[th];
    team_sync(team, T);  // the previous vector's shared memory has been read
    if (tid < (int)(sizeof(FoldIn) / sizeof(float)))
      reinterpret_cast<float*>(&s_in[team])[tid] = fold_in_word(r, tid);
    if (tid == 0) s_bad[team] = 0;
    const bool valid = r.valid != 0;  // team-uniform
    team_sync(team, T);
    FoldAcc<NDET> acc;
    FoldSum<NDET> sum;
    acc.clear();
    sum.hi.clear();
    if (valid)
      for (int base = 0; base < F.nc; base += panel) {
        const int np = min(panel, F.nc - base);
        // two nodes' data in turn, one in flight while the other is summed
        // (the first during the anchors)
        FoldNode<NDET> v0, v1;
        const float4* wq = w + (base + tw) * NDET * 32 + lane;
        auto kind = [&](int q) { return __float_as_int(tab[FR_KIND * ld + base + q]); };
        if (tw < np) fold_load<NDET>(wq, kind(tw), x0, s_x, lane, v0);
        // quarter sub of 32 chunks per warp and turn
        const int np32 = (np + 31) >> 5;
        for (int it = tw, sub = 0, blk = tw; it < 4 * np32; it += T, blk += T) {
          while (blk >= np32) blk -= np32, ++sub;
          const int q = 32 * blk + lane;
          if (q < np && !fold_anchor<NDET>(tab, ld, s_in[team], sub, base + q, q, an + q * kFoldAnchor)) s_bad[team] = 1;
        }
        team_sync(team, T);
        for (int q = tid; q < np; q += 32 * T)
          if (!fold_in_band<NDET>(tab, ld, an + q * kFoldAnchor, q, base + q)) s_bad[team] = 1;
        const float* aq = an + tw * kFoldAnchor;
        for (int q = tw; q < np;) {
          const int end = min(np, q + kFoldBlock * T);
          for (; q < end; q += 2 * T, wq += 2 * T * NDET * 32, aq += 2 * T * kFoldAnchor) {
            if (q + T < np) fold_load<NDET>(wq + T * NDET * 32, kind(q + T), x0, s_x, lane, v1);
            fold_chunk<NDET>(aq, q, v0, acc);
            if (q + T < np) {
              if (q + 2 * T < np) fold_load<NDET>(wq + 2 * T * NDET * 32, kind(q + 2 * T), x0, s_x, lane, v0);
              fold_chunk<NDET>(aq + T * kFoldAnchor, q + T, v1, acc);
            }
          }
          if (F.nc > kFoldBlock * T) sum.take(acc);
        }
        team_sync(team, T);
      }
    fold_warp_sums<NDET, 1, 1>(&acc, F.nc > kFoldBlock * T, &sum.hi, lane,
                               [&](int j, dfl v) { s_sum[j][warp] = make_float2(v.hi, v.lo); });
    team_sync(team, T);
    const bool bad = valid && s_bad[team];  // team-uniform
    if (bad) {
      double v[2 * NDET];
      fold_direct<NDET>(L, F, r, tw, T, lane, an + tw * kAnchorStride, v);
      if (lane == 0)
#pragma unroll
        for (int j = 0; j < 2 * NDET; ++j) s_dir[j][warp] = v[j];
      team_sync(team, T);
    }
    if (tw == 0) {
      // the warps' sums (double-float, four lanes a component), component j on lane j
      const int j = lane & 7;
      dfl t = {0.0f, 0.0f};
      if (j < 2 * NDET)
        for (int w = lane >> 3; w < T; w += 4)
          t = df_accumulate(t, dfl{s_sum[j][warp + w].x, s_sum[j][warp + w].y});
#pragma unroll
      for (int o = 8; o < 32; o <<= 1)
        t = df_accumulate(t, dfl{__shfl_xor_sync(0xffffffffu, t.hi, o), __shfl_xor_sync(0xffffffffu, t.lo, o)});
      double kapc = lane < 2 * NDET ? (double)t.hi + (double)t.lo : 0.0;
      if (bad) {
        kapc = 0.0;
        if (lane < 2 * NDET)
          for (int w = 0; w < T; ++w) kapc += s_dir[lane][warp + w];
        __syncwarp();
      }
      const double ll = loglike_epilogue_warp<NDET>(L, r, kapc, lane);
      if (lane == 0) out[th] = ll;
      if (kappa_out && lane < 2 * SWIG_MAX_DET) kappa_out[(size_t)th * 2 * SWIG_MAX_DET + lane] = kapc;
    }
  }
}

namespace {

template <int NDET, bool RES>
cudaError_t fold_launch_as(const LikeConst& L, const FoldTables& F, const EvalRecord* rec, int n, double* out,
                           cudaStream_t st, double* kappa_out, size_t smem) {
  cudaError_t e = allow_shared((const void*)k_fold<NDET, RES>);
  if (e != cudaSuccess) return e;
  // the widest team that leaves no vector waiting for a second turn
  const int ctas = L.sm_count;
  int T = kFoldWarps;
  while (T > 1 && (long long)n * T > (long long)ctas * kFoldWarps) T /= 2;
  const int teams = kFoldWarps / T, need = (n + teams - 1) / teams;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(need < ctas ? need : ctas);
  cfg.blockDim = dim3(32 * kFoldWarps);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_fold<NDET, RES>, L, F, rec, n, T, out, kappa_out);
}

template <int NDET>
cudaError_t fold_launch(const LikeConst& L, const DeviceBuffers& B, int n, double* out, cudaStream_t st,
                        double* kappa_out) {
  const FoldTables F = fold_tables(B);
  const size_t fixed = fold_fixed_bytes(), res = fixed + fold_resident_bytes(F.nc, NDET);
  if (n > L.sm_count && res <= 220 * 1024)
    return fold_launch_as<NDET, true>(L, F, B.rec, n, out, st, kappa_out, res);
  return fold_launch_as<NDET, false>(L, F, B.rec, n, out, st, kappa_out, fixed);
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
