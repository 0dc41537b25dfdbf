// Folded full-grid likelihood (fold.cuh): the weights of an event and the
// batched evaluation.
#include <cuda_runtime.h>

#include <algorithm>

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

// The strays of a batch, vectors far from the prior box that the node weights do
// not serve, are summed bin by bin by the CTAs that are left: a slice of the grid for
// two strays per warp, on packed FP32.  Few strays: units by ticket, a warp each.  32
// or more: a slice and up to 128 strays per CTA, the slice's tables in shared memory
// for all.  The warp that finishes a stray's last slice adds its partial sums in FP64
// and writes the result.
//
// Every stray is summed whatever the others do: the CTA that is the last to have
// decided its vectors knows how many there are and takes units until none is left.
// The others wait for that only to help, where they know of a stray when they are
// done, so that a batch without strays waits for nothing: a CTA asks with its last
// decision, ahead of that vector's epilogue.
//
// A pair over a slice of 1,700 bins and three detectors is bound by the sines (a
// quarter of a warp per clock) and the issue slots about alike.  One GB300, 128 s
// grid, three detectors: one stray among 1000 vectors 31 -> 63 us (by the team that met
// it, one or two warps, 965; any 1000 vectors summed over all bins 667), a stray by
// itself 47 us (174; 66), 100 strays 136 us (177; 135), 1000 strays 877 us (1440;
// 667), 4099 on the 256 s grid 4.32 ms (10.3; 4.74).
constexpr int kStrayCtas = 16;   // CTAs of a small batch at least: a warp per slice of one stray
constexpr int kStrayTiles = 18;  // tiles whose anchors, of two strays, a warp holds
constexpr int kStrayGroup = 128;

// The strays once all CTAs with vectors have decided them, or -1 after so many polls
// (0.7 us each).
__device__ __forceinline__ int strays_known(const FoldStrays& S, int ctas, int polls, int polls_stray) {
  for (int p = 0;; ++p) {
    const unsigned long long c = *(const volatile unsigned long long*)S.ctl;
    if ((int)(unsigned)c >= ctas) return (int)(c >> 32);
    if (p >= (c >> 32 ? polls_stray : polls)) return -1;
    __nanosleep(100);
  }
}

// sweep_warp_mixed for two vectors: bins lo .. hi - 1 of a slice that starts at bin b0,
// row: StrayRow of the tiles from tile0 on.  re, im - jm: the lane's sums.
struct StrayRow {
  f2 an[kAnchorStride];  // the anchors (compute_anchor)
  int k0, end;           // the tile's bins
  float inv_T, pad;
};
static_assert(kStrayTiles * sizeof(StrayRow) <= kFoldSlots * kFoldAnchor * sizeof(float) / kFoldWarps,
              "a warp's share of the anchors");

template <int NDET>
__device__ __forceinline__ void sweep_warp_pair(const float2* data, int stride, const int* tile, int b0, int lo, int hi,
                                                const StrayRow* row, int tile0, const f2* shift, int lane, f2* re,
                                                f2* im, f2* jm) {
  using O = PkOps<2>;
  const f2 magic = O::all(12582912.0f), nmagic = O::all(-12582912.0f), none = O::all(-1.0f);
  const auto off = [&](f2 v) { return f2_fma(f2_add(f2_add(v, magic), nmagic), none, v); };  // (see round_nearest)
  StrayRow a;
  a.end = -1;
  const auto phase = [&](float x) {
    const float u = x * a.inv_T;
    const f2 u2 = O::all(u), x2 = O::all(x);
    f2 p = a.an[2 + kNumPoly];
#pragma unroll
    for (int m = kNumPoly - 2; m >= 0; --m) p = f2_fma(p, u2, a.an[3 + m]);
    p = f2_mul(p, O::all(u * u));
    return f2_add(off(f2_mul(x2, a.an[1])), f2_add(a.an[0], f2_fma(x2, a.an[2], p)));
  };
  const auto add = [&](float x, f2 p, int k) {
    const f2 x2 = O::all(x);
#pragma unroll
    for (int i = 0; i < NDET; ++i) {
      const f2 ph = f2_mul(off(f2_add(p, f2_fma(x2, shift[i], a.an[3 + kNumPoly + i]))), O::all(6.283185307179586f));
      float pa, pb, sa, ca, sb, cb;
      f2_split(ph, pa, pb);
      __sincosf(pa, &sa, &ca);
      __sincosf(pb, &sb, &cb);
      const f2 c2 = f2_make(ca, cb), s2 = f2_make(sa, sb);
      const float2 d = data[i * stride + k];
      const f2 dx = O::all(d.x), dy = O::all(d.y);
      re[i] = f2_fma(dx, c2, f2_fma(dy, s2, re[i]));
      im[i] = f2_fma(dy, c2, im[i]);
      jm[i] = f2_fma(dx, s2, jm[i]);
    }
  };
  for (int k = lo + lane; k < hi;) {
    if (k >= a.end) {
      a = row[tile[k] - tile0];
      a.k0 -= b0;
      a.end -= b0;
    }
    const float x = (float)(k - a.k0);
    const f2 p = phase(x);
    if (k + 32 < min(hi, a.end)) {  // two bins of a tile at a time
      const f2 q = phase(x + 32.0f);
      add(x, p, k);
      add(x + 32.0f, q, k + 32);
      k += 64;
    } else {
      add(x, p, k);
      k += 32;
    }
  }
}

// A slice's tables where a warp reads them: data and tile indices of the bins from b0
// on, tiles from t0 on.
struct StraySlice {
  const float2* data;
  int stride;
  const int* tile;
  int b0;
  const TileInfo* tiles;
  const TileBasis* basis;
  int t0;
};
inline __host__ __device__ size_t stray_slice_bytes(int n_det, int bins, int tiles) {
  return (sizeof(float2) * n_det + sizeof(int)) * (size_t)bins + (sizeof(TileInfo) + sizeof(TileBasis)) * (size_t)tiles;
}

// Strays i and i + 1 over one slice by a warp; row: the warp's share of the anchors.
template <int NDET>
__device__ __forceinline__ void stray_unit(const LikeConst& L, const FoldTables& F, const EvalRecord* rec,
                                           const FoldStrays& S, int strays, int slice, int i, const StraySlice& T,
                                           StrayRow* row, int lane, double* out, double* kappa_out) {
  const bool two = i + 1 < strays;
  const EvalRecord* r = &rec[__ldcg(&S.list[two ? i + (lane & 1) : i])];  // even lanes', odd lanes'
  const int k0 = F.slice_begin[slice], k1 = F.slice_begin[slice + 1];
  const int t1 = T.tile[k1 - 1 - T.b0] + 1;
  const float sh = lane < 2 * NDET ? (float)(L.df * r->tau[lane >> 1]) : 0.0f;
  f2 shift[NDET], re[NDET], im[NDET], jm[NDET];
#pragma unroll
  for (int d = 0; d < NDET; ++d) {
    shift[d] = f2_make(__shfl_sync(0xffffffffu, sh, 2 * d), __shfl_sync(0xffffffffu, sh, 2 * d + 1));
    re[d] = im[d] = jm[d] = 0ull;
  }
  for (int t = T.tile[k0 - T.b0]; t < t1; t += kStrayTiles) {
    const int nt = min(kStrayTiles, t1 - t);
    __syncwarp();
    for (int q = lane; q < 2 * nt; q += 32) {
      const int at = t - T.t0 + (q >> 1);
      const TileInfo ti = T.tiles[at];
      float an[kAnchorStride];
      compute_anchor(NDET, ti, T.basis[at], *r, an);
      StrayRow& w = row[q >> 1];
#pragma unroll
      for (int m = 0; m < kAnchorStride; ++m) reinterpret_cast<float*>(&w.an[m])[q & 1] = an[m];
      if (!(q & 1)) w.k0 = ti.k0, w.end = ti.k0 + ti.nbins, w.inv_T = ti.inv_T;
    }
    __syncwarp();
    const int lo = max(k0, row[0].k0), hi = min(k1, row[nt - 1].end);
    sweep_warp_pair<NDET>(T.data, T.stride, T.tile, T.b0, lo - T.b0, hi - T.b0, row, t, shift, lane, re, im, jm);
  }
#pragma unroll
  for (int d = 0; d < NDET; ++d) im[d] = pk_sub<2>(im[d], jm[d]);
#pragma unroll
  for (int d = 0; d < NDET; ++d)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      re[d] = f2_add(re[d], __shfl_xor_sync(0xffffffffu, re[d], o));
      im[d] = f2_add(im[d], __shfl_xor_sync(0xffffffffu, im[d], o));
    }
  float* p[2] = {S.part + (size_t)i * L.n_slices * kPartialStride, S.part + (size_t)(i + 1) * L.n_slices * kPartialStride};
#pragma unroll
  for (int j = 0; j < 2 * NDET; ++j) {
    float a, b;
    f2_split(j & 1 ? im[j / 2] : re[j / 2], a, b);
    if (lane == j) __stcg(&p[0][slice * kPartialStride + j], a);
    if (lane == j && two) __stcg(&p[1][slice * kPartialStride + j], b);
  }
  __threadfence();
  __syncwarp();
  int last = 0;
  if (lane < 2 && i + lane < strays) last = atomicAdd(&S.done[i + lane], 1) == L.n_slices - 1;
  const unsigned done = __ballot_sync(0xffffffffu, last);
  if (!done) return;
  __threadfence();
#pragma unroll 1
  for (int e = 0; e < 2; ++e) {
    if (!((done >> e) & 1u)) continue;
    double acc[2 * NDET];
#pragma unroll
    for (int j = 0; j < 2 * NDET; ++j) acc[j] = 0.0;
    const float* q = S.part + (size_t)(i + e) * L.n_slices * kPartialStride;
    for (int s = lane; s < L.n_slices; s += 32)
#pragma unroll
      for (int j = 0; j < 2 * NDET; ++j) acc[j] += (double)__ldcg(&q[s * kPartialStride + j]);
    double kapc = 0.0;
#pragma unroll
    for (int j = 0; j < 2 * NDET; ++j) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], o);
      if (lane == j) kapc = acc[j];
    }
    const int th = __ldcg(&S.list[i + e]);
    const double ll = loglike_epilogue_warp<NDET>(L, rec[th], kapc, lane);
    if (lane == 0) out[th] = ll;
    if (kappa_out && lane < 2 * SWIG_MAX_DET) kappa_out[(size_t)th * 2 * SWIG_MAX_DET + lane] = kapc;
  }
}

// s_slice: room for the tables of a slice of cap bins and tiles (cap.x 0: none).
template <int NDET>
__device__ __noinline__ void fold_strays(const LikeConst& L, const FoldTables& F, const EvalRecord* rec,
                                         const FoldStrays& S, int strays, StrayRow* row, float2* s_slice, int2 cap,
                                         int lane, double* out, double* kappa_out) {
  __shared__ int s_unit;
  const int warp = threadIdx.x >> 5, pairs = (strays + 1) / 2;
  StraySlice T = {F.data, L.n_bins, F.bin_tile, 0, F.tiles, F.basis, 0};
  if (pairs < kFoldWarps || cap.x == 0) {
    for (;;) {
      int u = 0;
      if (lane == 0) u = atomicAdd(&S.ctl[2], 1);
      u = __shfl_sync(0xffffffffu, u, 0);
      if (u >= pairs * L.n_slices) return;
      stray_unit<NDET>(L, F, rec, S, strays, u / pairs, 2 * (u % pairs), T, row, lane, out, kappa_out);
    }
  }
  int* s_tile = reinterpret_cast<int*>(s_slice + (size_t)NDET * cap.x);
  TileBasis* s_basis = reinterpret_cast<TileBasis*>(s_tile + cap.x);
  TileInfo* s_info = reinterpret_cast<TileInfo*>(s_basis + cap.y);
  T.data = s_slice, T.stride = cap.x, T.tile = s_tile, T.tiles = s_info, T.basis = s_basis;
  const int groups = (strays + kStrayGroup - 1) / kStrayGroup;
  for (int held = -1;;) {
    __syncthreads();  // the previous unit's tables have been read
    if (threadIdx.x == 0) s_unit = atomicAdd(&S.ctl[2], 1);
    __syncthreads();
    const int slice = s_unit / groups, first = (s_unit - slice * groups) * kStrayGroup;
    if (slice >= L.n_slices) return;
    if (slice != held) {
      T.b0 = F.slice_begin[slice];
      const int nb = F.slice_begin[slice + 1] - T.b0;
      T.t0 = F.bin_tile[T.b0];
      const int nt = F.bin_tile[T.b0 + nb - 1] + 1 - T.t0;
      for (int d = 0; d < NDET; ++d)
        for (int k = threadIdx.x; k < nb; k += blockDim.x) s_slice[d * cap.x + k] = F.data[(size_t)d * L.n_bins + T.b0 + k];
      for (int k = threadIdx.x; k < nb; k += blockDim.x) s_tile[k] = F.bin_tile[T.b0 + k];
      const float* from = reinterpret_cast<const float*>(F.basis + T.t0);
      for (int k = threadIdx.x; k < nt * (int)(sizeof(TileBasis) / sizeof(float)); k += blockDim.x)
        reinterpret_cast<float*>(s_basis)[k] = from[k];
      for (int k = threadIdx.x; k < nt; k += blockDim.x) s_info[k] = F.tiles[T.t0 + k];
      __syncthreads();
      held = slice;
    }
    const int end = min(strays, first + kStrayGroup);
    for (int i = first + 2 * warp; i < end; i += 2 * kFoldWarps)
      stray_unit<NDET>(L, F, rec, S, strays, slice, i, T, row, lane, out, kappa_out);
  }
}

template <int NDET, bool RES>
__global__ void __launch_bounds__(32 * kFoldWarps, 1)
    k_fold(LikeConst L, FoldTables F, const EvalRecord* __restrict__ rec, int n, int T, double* __restrict__ out,
           double* __restrict__ kappa_out, FoldStrays S, int2 slice_cap) {
  // (16 bytes off a line, as the static arrays left it, 1000 vectors took 31.0 us for 27.5)
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ FoldIn s_in[kFoldWarps];
  __shared__ float2 s_sum[2 * NDET][kFoldWarps];
  __shared__ int s_bad[kFoldWarps], s_left, s_met, s_strays;  // (strays: teams at work, strays met, all known)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int team = warp / T, tw = warp - team * T, tid = 32 * tw + lane;  // within the team
  const int teams = kFoldWarps / T, panel = min(128, kFoldSlots / teams);
  float* s_anchor = reinterpret_cast<float*>(smem);
  float2* s_x = reinterpret_cast<float2*>(s_anchor + kFoldSlots * kFoldAnchor);
  const float4* w = F.w;
  const float* tab = F.tab;
  const int ld = F.ld;
  const bool idle = blockIdx.x * teams >= n;  // here to help with strays
  if (RES) {
    float4* s_w = reinterpret_cast<float4*>(s_x + 32 * kFoldKinds);
    float4* s_t = s_w + F.nc * NDET * 32;
    const float4* g_t = reinterpret_cast<const float4*>(F.tab);
    if (!idle) {
      for (int k = threadIdx.x; k < FR_ROWS * ld / 4; k += blockDim.x) cp_async16(s_t + k, g_t + k);
      for (int k = threadIdx.x; k < F.nc * NDET * 32; k += blockDim.x) cp_async16(s_w + k, F.w + k);
    }
    w = s_w;
    tab = reinterpret_cast<const float*>(s_t);
  }
  for (int k = threadIdx.x; k < 32 * kFoldKinds; k += blockDim.x) s_x[k] = F.x[k];
  if (threadIdx.x == 0) {
    s_left = min(teams, n - (int)blockIdx.x * teams);
    s_met = 0;
    s_strays = 0;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  // the set-up kernel's records, while this one's start overlapped its end
  asm volatile("griddepcontrol.wait;" ::: "memory");
  float* an = s_anchor + team * panel * kFoldAnchor;
  const float2 x0 = s_x[lane];
  unsigned long long seen = 0;  // CTAs done deciding, strays << 32, with this one: of the thread that reported it
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
    const bool stray = valid && s_bad[team];  // team-uniform
    if (tid == 0) {
      if (stray) {
        S.list[atomicAdd(&S.ctl[3], 1)] = th;
        __threadfence();
        atomicAdd(&s_met, 1);
      }
      if (th + gridDim.x * teams >= n && (teams == 1 || atomicSub(&s_left, 1) == 1)) {
        const unsigned long long mine = 1 + ((unsigned long long)*(volatile int*)&s_met << 32);
        seen = atomicAdd(reinterpret_cast<unsigned long long*>(S.ctl), mine) + mine;
      }
    }
    if (tw == 0 && !stray) {
      // the warps' sums (double-float, four lanes a component), component j on lane j
      const int j = lane & 7;
      dfl t = {0.0f, 0.0f};
      if (j < 2 * NDET)
        for (int w = lane >> 3; w < T; w += 4)
          t = df_accumulate(t, dfl{s_sum[j][warp + w].x, s_sum[j][warp + w].y});
#pragma unroll
      for (int o = 8; o < 32; o <<= 1)
        t = df_accumulate(t, dfl{__shfl_xor_sync(0xffffffffu, t.hi, o), __shfl_xor_sync(0xffffffffu, t.lo, o)});
      const double kapc = lane < 2 * NDET ? (double)t.hi + (double)t.lo : 0.0;
      const double ll = loglike_epilogue_warp<NDET>(L, r, kapc, lane);
      if (lane == 0) out[th] = ll;
      if (kappa_out && lane < 2 * SWIG_MAX_DET) kappa_out[(size_t)th * 2 * SWIG_MAX_DET + lane] = kapc;
    }
  }
  // all strays if this CTA was the last to decide, -1 if there are some so far
  const int ctas = min((int)gridDim.x, (n + teams - 1) / teams);
  if (seen) s_strays = (int)(unsigned)seen == ctas ? (int)(seen >> 32) : seen >> 32 ? -1 : 0;
  __syncthreads();
  int strays = s_strays;
  if (strays < 0 || idle) {  // block-uniform
    __syncthreads();
    if (threadIdx.x == 0) s_strays = strays_known(S, ctas, idle ? 40 : 0, 200);
    __syncthreads();
    strays = s_strays;
  }
  if (strays > 0) {
    __threadfence();  // the list, behind the count
    fold_strays<NDET>(L, F, rec, S, strays,
                      reinterpret_cast<StrayRow*>(s_anchor + warp * (kFoldSlots * kFoldAnchor / kFoldWarps)),
                      reinterpret_cast<float2*>(smem + fold_fixed_bytes()), slice_cap, lane, out, kappa_out);
  }
}

namespace {

template <int NDET, bool RES>
cudaError_t fold_launch_as(const LikeConst& L, const FoldTables& F, const EvalRecord* rec, int n, double* out,
                           cudaStream_t st, double* kappa_out, const FoldStrays& S, int2 slice_cap, size_t smem) {
  cudaError_t e = allow_shared((const void*)k_fold<NDET, RES>);
  if (e != cudaSuccess) return e;
  // the widest team that leaves no vector waiting for a second turn
  const int ctas = L.sm_count;
  int T = kFoldWarps;
  while (T > 1 && (long long)n * T > (long long)ctas * kFoldWarps) T /= 2;
  // a small batch gets CTAs to help with strays (one among up to 100: 47 us, 227
  // without them; without strays they change nothing)
  const int teams = kFoldWarps / T, need = std::max(3 * ((n + teams - 1) / teams), kStrayCtas);
  // room for a slice's tables, over the weights or beside the anchors
  const size_t slice = fold_fixed_bytes() + stray_slice_bytes(NDET, slice_cap.x, slice_cap.y);
  if (slice <= 220 * 1024)
    smem = std::max(smem, slice);
  else
    slice_cap = make_int2(0, 0);
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
  return cudaLaunchKernelEx(&cfg, k_fold<NDET, RES>, L, F, rec, n, T, out, kappa_out, S, slice_cap);
}

template <int NDET>
cudaError_t fold_launch(const LikeConst& L, const DeviceBuffers& B, int n, double* out, cudaStream_t st,
                        double* kappa_out) {
  const FoldTables F = fold_tables(B);
  const FoldStrays S = fold_strays_at(B.strays, n);
  const int2 slice = make_int2(B.max_slice_bins, B.max_slice_tiles);
  const size_t fixed = fold_fixed_bytes(), res = fixed + fold_resident_bytes(F.nc, NDET);
  if (n > L.sm_count && res <= 220 * 1024)
    return fold_launch_as<NDET, true>(L, F, B.rec, n, out, st, kappa_out, S, slice, res);
  return fold_launch_as<NDET, false>(L, F, B.rec, n, out, st, kappa_out, S, slice, fixed);
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
