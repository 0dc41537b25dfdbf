// The chain sampler: persistent nested-sampling kernel of the mixed-precision
// full grid (folded sums) and of the heterodyned likelihood, with t_c sampled or
// marginalised (chain.cuh has a chain's control).
//
// One cooperative launch runs up to max_iters iterations.  Between boundaries a
// CTA takes one chain at a time and runs it to its end; the grid meets around
// the boundaries alone.  Several events (a campaign) share a launch: the chains
// of all are dealt to the CTAs as these come free, CTA e runs event e's boundary,
// and the launch returns before any event starts new chains once one has left
// the running state.  Which CTA runs a chain does not enter its arithmetic.
#include <cuda_runtime.h>

#include "chain.cuh"

namespace swig {

// Fixed shared memory: the chain, the event's constants, and the inputs and
// sums of a round's evaluation (only what the mode uses, so that the folded
// weights fit beside it).
template <int NDET, int MODE>
struct ChainEval;
template <int NDET>
struct ChainEval<NDET, CHAIN_FOLD> {
  float2 x[32 * kFoldKinds];  // node abscissae
  FoldPair in[kCand / 2];
  FoldPair cur;               // the chain's current point
  int base_ok;                // its partial sums are formed
  float2 sum[kChainWarps][4 * NDET];  // of a warp's pair of candidates, double-float
  double tot[kCand][2 * NDET];
  double dir[kChainWarps][2 * NDET];  // bin by bin, per warp
};
template <int NDET>
struct ChainEval<NDET, CHAIN_HET> {
  double fc[NBASIS], ft[SWIG_MAX_DET];  // the fiducial's coefficients and delays
  HetPrep<NDET> prep[kCand], cur_prep;
  HetIn<NDET, 1> cur;         // the chain's current point
  int base_ok;                // its partial sums are formed
  HetIn<NDET, 2> in[kCand / 2];
  float part[kChainWarps][NDET][3 * kCand];  // per warp: value 8 kind + slot
  double tot[NDET][3 * kCand];
};
template <int NDET>
struct ChainEval<NDET, CHAIN_HET_TM> {
  HetPrep<NDET> prep;
  HetIn<NDET, 1> in;
  float hh[kChainWarps][NDET];
  float tm[kChainWarps][2];
};
template <int NDET, int MODE>
struct ChainShared {
  ChainWork w;
  LikeConst L;
  SamplerConst S;
  ChainEval<NDET, MODE> e;
  unsigned long long prof[8], cta[4];
  int task, event;
};

namespace {
template <int NDET>
size_t shared_bytes(int mode) {
  return mode == CHAIN_FOLD  ? sizeof(ChainShared<NDET, CHAIN_FOLD>)
         : mode == CHAIN_HET ? sizeof(ChainShared<NDET, CHAIN_HET>)
                             : sizeof(ChainShared<NDET, CHAIN_HET_TM>);
}
}  // namespace

size_t chain_fixed_bytes(int n_det, int mode) {
  const size_t b = n_det == 1   ? shared_bytes<1>(mode)
                   : n_det == 2 ? shared_bytes<2>(mode)
                   : n_det == 3 ? shared_bytes<3>(mode)
                                : shared_bytes<4>(mode);
  return (b + 15) & ~(size_t)15;
}

// Chunks that a lane adds in FP32 (fold.cuh kFoldBlock): a round's groups share the
// chunks, so that blocks of 32 are beyond what the 128 s grid's 78 come to (20 for
// each of four groups) and their sums stay out of the way of the chunks' loop (blocks
// of 8, in registers: 12.77 -> 13.17 ms for 4 iterations).
constexpr int kChainFoldBlock = 32;
// A warp's sums over its pair of candidates to sum, or added to what is there.
template <int NDET>
__device__ __forceinline__ void fold_take_sums(const FoldAcc<NDET>* acc, bool add, float2* sum, int lane) {
  fold_warp_sums<NDET, 2, 2>(acc, false, nullptr, lane, [&](int j, dfl v) {
    if (add) v = df_add(v, dfl{sum[j].x, sum[j].y});
    sum[j] = make_float2(v.hi, v.lo);
  });
}
// The same out of the chunks' loop (by value: the accumulators stay in registers).
template <int NDET>
__device__ __noinline__ void fold_block_sums(FoldAcc<NDET> a, FoldAcc<NDET> b, bool add, float2* sum, int lane) {
  const FoldAcc<NDET> acc[2] = {a, b};
  fold_take_sums<NDET>(acc, add, sum, lane);
}

// Folded full-grid sums of the round's candidates, two at a time: anchors of a
// panel of chunks (packed over the pair, quarter by quarter), then a (pair, group
// of chunks) per warp, the chunks q = group, group + G, ..., the weights loaded
// once for both.  The groups' sums go to s.e.sum.  A block that leaves the masses
// and tides alone takes the sums over their basis functions from base (the
// current point's) and adds the spin terms only.
template <int NDET>
__device__ __forceinline__ void eval_fold(ChainShared<NDET, CHAIN_FOLD>& s, const FoldTables& F, const float4* W,
                                         const float* tab, float* base, float* s_an, int slots, int warp, int lane) {
  ChainWork& w = s.w;
  const int na = w.n_act, pairs = (na + 1) / 2, ld = F.ld;
  const int G = kChainWarps / pairs;
  const bool use = base != nullptr && !(w.fl & (BF_INTR | BF_TIDE));  // uniform
  if (threadIdx.x < pairs * 16) {
    const int p = threadIdx.x >> 4, j = threadIdx.x & 15;
    const EvalRecord& a = w.rec[w.list[2 * p]];
    const EvalRecord& b = w.rec[w.list[min(2 * p + 1, na - 1)]];
    fold_pair_set(s.e.in[p], j, a, b);
  } else if (use && !s.e.base_ok && threadIdx.x >= 256 && threadIdx.x < 272) {
    fold_pair_set(s.e.cur, threadIdx.x & 15, w.rx, w.rx);
  }
  __syncthreads();
  if (use && !s.e.base_ok) {
    const int nb = (F.nc + 31) >> 5;
    for (int it = warp; it < 4 * nb; it += kChainWarps) {
      const int q = 32 * (it % nb) + lane;
      if (q < F.nc) fold_base(tab, ld, s.e.cur, it / nb, q, base, F.ld);
    }
    __syncthreads();
    if (threadIdx.x == 0) s.e.base_ok = 1;
  }
  int panel = slots / na & ~31;  // whole turns
  if (slots / na >= F.nc) panel = F.nc;
  FoldAcc<NDET> acc[2];
  acc[0].clear();
  acc[1].clear();
  int held = 0;           // chunks in the accumulators
  bool blocks = false;    // earlier blocks' sums in s.e.sum
  const float2 x0 = s.e.x[lane];
  const int p = warp / G, g = warp - p * G;  // this warp's pair and group
  for (int q0 = 0; q0 < F.nc; q0 += panel) {
    const int np = min(panel, F.nc - q0), nb = (np + 31) >> 5, per = pairs * nb;
    for (int it = warp, sub = 0, t = warp; it < 4 * per; it += kChainWarps, t += kChainWarps) {
      while (t >= per) t -= per, ++sub;
      const int a = t / nb, q = 32 * (t - a * nb) + lane;
      if (q < np) {
        const int k0 = 2 * a, k1 = min(2 * a + 1, na - 1);
        const int bad = fold_anchor_pair<NDET>(tab, ld, s.e.in[a], use ? base : nullptr, sub, q0 + q, q,
                                               s_an + (k0 * panel + q) * kFoldAnchor,
                                               s_an + (k1 * panel + q) * kFoldAnchor);
        if (bad & 1) w.bad[w.list[k0]] = 1;
        if (bad & 2) w.bad[w.list[k1]] = 1;
      }
    }
    __syncthreads();
    for (int it = threadIdx.x; it < na * np; it += kChainBlock) {
      const int a = it / np, q = it - a * np;
      if (!fold_in_band<NDET>(tab, ld, s_an + (a * panel + q) * kFoldAnchor, q, q0 + q)) w.bad[w.list[a]] = 1;
    }
    if (p < pairs) {
      const bool two = 2 * p + 1 < na;
      // the group takes the chunks whose number is g modulo G, whatever the panels
      // (their length follows the launch's scratch; five groups do not divide it)
      int g0 = g;
      if (q0 > 0) g0 += (G - q0 % G) % G;
      if (g0 >= G) g0 -= G;
      const float* an0 = s_an + (2 * p * panel + g0) * kFoldAnchor;
      const float* an1 = an0 + panel * kFoldAnchor;
      const float4* wq = W + (q0 + g0) * NDET * 32 + lane;
      auto kind = [&](int q) { return __float_as_int(tab[FR_KIND * ld + q0 + q]); };
      for (int q = g0; q < np; q += G, wq += G * NDET * 32, an0 += G * kFoldAnchor, an1 += G * kFoldAnchor) {
        FoldNode<NDET> v;
        fold_load<NDET>(wq, kind(q), x0, s.e.x, lane, v);
        fold_chunk<NDET>(an0, q, v, acc[0]);
        if (two) fold_chunk<NDET>(an1, q, v, acc[1]);
        if (++held == kChainFoldBlock) {  // warp-uniform; many chunks
          fold_block_sums<NDET>(acc[0], acc[1], blocks, s.e.sum[warp], lane);
          acc[0].clear();
          acc[1].clear();
          held = 0;
          blocks = true;
        }
      }
    }
    __syncthreads();
  }
  if (p < pairs) fold_take_sums<NDET>(acc, blocks, s.e.sum[warp], lane);
  __syncthreads();
  {  // the groups' sums (double-float, four threads a value), rounded once to FP64
    const int v = threadIdx.x >> 2, a = v / (2 * NDET), j = v - a * (2 * NDET), g0 = threadIdx.x & 3;
    const int k = a < na ? w.list[a] : 0;
    dfl t = {0.0f, 0.0f};
    for (int r = g0; r < G; r += 4) {
      const float2 x = a < na ? s.e.sum[(a >> 1) * G + r][(a & 1) * 2 * NDET + j] : make_float2(0.0f, 0.0f);
      t = df_accumulate(t, dfl{x.x, x.y});
    }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1)
      t = df_accumulate(t, dfl{__shfl_xor_sync(0xffffffffu, t.hi, o), __shfl_xor_sync(0xffffffffu, t.lo, o)});
    if (a < na && g0 == 0) s.e.tot[k][j] = (double)t.hi + (double)t.lo;
  }
  for (int a = 0; a < na; ++a) {
    const int k = w.list[a];
    if (!w.bad[k]) continue;  // block-uniform, rare: bin by bin
    __syncthreads();
    double v[2 * NDET];
    fold_direct<NDET>(s.L, F, w.rec[k], warp, kChainWarps, lane, s_an + warp * kAnchorStride, v);
    if (lane == 0)
#pragma unroll
      for (int j = 0; j < 2 * NDET; ++j) s.e.dir[warp][j] = v[j];
    __syncthreads();
    if (threadIdx.x < 2 * NDET) {
      double t = 0.0;
      for (int q = 0; q < kChainWarps; ++q) t += s.e.dir[q][threadIdx.x];
      s.e.tot[k][threadIdx.x] = t;
    }
    __syncthreads();
  }
}

// logL of the round's candidates from their sums, by warp 0: candidate
// lane / 4, detector lane % 4.
template <int NDET>
__device__ __forceinline__ void finish_fold(ChainShared<NDET, CHAIN_FOLD>& s, int lane) {
  ChainWork& w = s.w;
  const LikeConst& L = s.L;
  const int k = lane >> 2, i = lane & 3;
  const bool on = (w.act >> k) & 1u;
  double kre = 0.0, kim = 0.0, tr = 0.0, ti = 0.0;
  if (on) {
    if (i < NDET) {
      kre = s.e.tot[k][2 * i];
      kim = s.e.tot[k][2 * i + 1];
      const EvalRecord& r = w.rec[k];
      const double a = kre * L.inv_scale[i], b = kim * L.inv_scale[i];
      tr = r.cre[i] * a - r.cim[i] * b;
      ti = r.cre[i] * b + r.cim[i] * a;
    }
    w.kap[k][2 * i] = kre;
    w.kap[k][2 * i + 1] = kim;
  }
  const int l0 = lane & ~3;
  double zr = __shfl_sync(0xffffffffu, tr, l0), zi = __shfl_sync(0xffffffffu, ti, l0);
#pragma unroll
  for (int d = 1; d < NDET; ++d) {
    zr += __shfl_sync(0xffffffffu, tr, l0 + d);
    zi += __shfl_sync(0xffffffffu, ti, l0 + d);
  }
  if (L.dist_marg) {  // a candidate after another, the quadrature across the warp
    for (int a = 0; a < w.n_act; ++a) {
      const int kk = w.list[a];
      const double ll = distance_marg_logl_warp(L, __shfl_sync(0xffffffffu, zr, 4 * kk),
                                                __shfl_sync(0xffffffffu, zi, 4 * kk), w.rec[kk].hh, lane);
      if (lane == 0) w.ly[kk] = ll;
    }
  } else if (on && i == 0) {
    const double base = -0.5 * w.rec[k].hh - 0.5 * L.DD;
    double out = zr + base;
    if (L.phase_marg) {
      const double x = sqrt(zr * zr + zi * zi);
      out = (L.fast_epilogue ? x + (double)log_i0e_f32((float)x) : log_bessel_i0(x)) + base;
    }
    w.ly[k] = out;
  }
  __syncwarp();
}

// Heterodyned sums of the round's candidates: pairs of candidates per packed
// instruction, a warp per chunk over all pairs (see k_het); a warp per candidate
// forms its result.
template <int NDET>
__device__ __forceinline__ void eval_het(ChainShared<NDET, CHAIN_HET>& s, const HetTables& H, const float* tab,
                                         float* base, float* s_an, int bytes, int warp, int lane) {
  ChainWork& w = s.w;
  const int na = w.n_act, pairs = (na + 1) / 2;
  const bool use = base != nullptr && !(w.fl & (BF_INTR | BF_TIDE)), form = use && !s.e.base_ok;  // uniform
  if (warp < 2 * pairs) {  // (an odd round's last pair holds its candidate twice)
    het_differences<NDET>(s.e.fc, s.e.ft, w.rec[w.list[min(warp, na - 1)]], s.e.prep[warp], lane);
    het_in_set<NDET, 2>(s.e.in[warp >> 1], warp & 1, s.e.prep[warp], lane);
  } else if (form && warp == kChainWarps - 1) {
    het_differences<NDET>(s.e.fc, s.e.ft, w.rx, s.e.cur_prep, lane);
    het_in_set<NDET, 1>(s.e.cur, 0, s.e.cur_prep, lane);
  }
  if (form) {
    __syncthreads();
    const int nb = (H.n_chunks + 31) >> 5;
    for (int t = warp; t < 4 * nb; t += kChainWarps) {
      const int q = 32 * (t % nb) + lane;
      if (q < H.n_chunks) het_anchor_part<NDET, 1, -1>(tab, H.n_chunks, s.e.cur, t / nb, q, nullptr, base + q);
    }
    if (threadIdx.x == 0) s.e.base_ok = 1;
  }
  const int fit = bytes / (pairs * kHetAncPair * (int)sizeof(float));
  const int panel = fit >= H.n_chunks ? H.n_chunks : fit & ~31;
  HetAcc<NDET, 2> acc[kCand / 2];
#pragma unroll
  for (int p = 0; p < kCand / 2; ++p) acc[p].clear();
  for (int q0 = 0; q0 < H.n_chunks; q0 += panel) {
    const int np = min(panel, H.n_chunks - q0);
    __syncthreads();
    // the first chunk's weights, then always the next one's: in flight meanwhile
    float4 nx[NDET];
    const float4* ew = H.ew + (size_t)q0 * NDET * 32 + lane;
    if (warp < np)
#pragma unroll
      for (int i = 0; i < NDET; ++i) nx[i] = __ldg(ew + (warp * NDET + i) * 32);
    if (use)
      het_anchors<NDET, 2, 1>(H, tab, s.e.in, pairs, q0, np, panel, base, s_an, warp, kChainWarps, lane);
    else
      het_anchors<NDET, 2>(H, tab, s.e.in, pairs, q0, np, panel, base, s_an, warp, kChainWarps, lane);
    __syncthreads();
    for (int q = warp; q < np; q += kChainWarps) {
      float4 v[NDET];
      const int qn = min(q + kChainWarps, np - 1);
#pragma unroll
      for (int i = 0; i < NDET; ++i) {
        v[i] = nx[i];
        nx[i] = __ldg(ew + (qn * NDET + i) * 32);
      }
#pragma unroll
      for (int p = 0; p < kCand / 2; ++p)
        if (p < pairs) {
          const HetPrep<NDET>* pp[2] = {&s.e.prep[2 * p], &s.e.prep[2 * p + 1]};
          het_edges<NDET, 2>(H, s_an + ((size_t)p * panel + q) * kHetAncPair, s.e.in[p], pp, q0 + q, lane, v, acc[p]);
        }
    }
  }
#pragma unroll
  for (int i = 0; i < NDET; ++i) {
    float a[32];
#pragma unroll
    for (int p = 0; p < kCand / 2; ++p) {
      PkOps<2>::get(acc[p].zr[i], a + 2 * p);
      PkOps<2>::get(acc[p].zi[i], a + kCand + 2 * p);
      PkOps<2>::get(acc[p].hh[i], a + 2 * kCand + 2 * p);
      a[3 * kCand + 2 * p] = a[3 * kCand + 2 * p + 1] = 0.0f;
    }
    const float v = warp_transpose_sum(a, lane);
    if (lane < 3 * kCand) s.e.part[warp][i][lane] = v;
  }
  __syncthreads();
  if (threadIdx.x < 4 * 3 * kCand * NDET) {  // (whole warps)
    // the warps' sums (double-float, four threads a value), rounded once to FP64
    const int v = threadIdx.x >> 2, i = v / (3 * kCand), j = v - i * (3 * kCand), g0 = threadIdx.x & 3;
    dfl t = {0.0f, 0.0f};
#pragma unroll
    for (int r = 0; r < kChainWarps; r += 4) t = df_add(t, dfl{s.e.part[r + g0][i][j], 0.0f});
#pragma unroll
    for (int o = 1; o < 4; o <<= 1)
      t = df_add(t, dfl{__shfl_xor_sync(0xffffffffu, t.hi, o), __shfl_xor_sync(0xffffffffu, t.lo, o)});
    if (g0 == 0) s.e.tot[i][j] = (double)t.hi + (double)t.lo;
  }
}

// logL and caches of the round's candidates, by warp 0: slot lane / 4, detector
// lane % 4 (het_detector with the reciprocal of the data scale).
template <int NDET>
__device__ __forceinline__ void finish_het(ChainShared<NDET, CHAIN_HET>& s, const HetTables& H, int lane) {
  ChainWork& w = s.w;
  const LikeConst& L = s.L;
  const int a = lane >> 2, i = lane & 3;
  const bool on = a < w.n_act;
  const int k = on ? w.list[a] : 0;
  double Z[2] = {0.0, 0.0}, hh = 0.0, k2[2] = {0.0, 0.0}, vv = 0.0;
  if (on && i < NDET)
    het_detector(L, *H.fid, w.rec[k], i, s.e.tot[i][a], s.e.tot[i][kCand + a], s.e.tot[i][2 * kCand + a], Z, &hh, k2,
                 &vv);
  if (on) {
    w.kap[k][2 * i] = k2[0];
    w.kap[k][2 * i + 1] = k2[1];
    w.vv[k][i] = vv;
  }
  const int l0 = lane & ~3;
  double Zr = 0.0, Zi = 0.0, HH = 0.0;
#pragma unroll
  for (int d = 0; d < NDET; ++d) {
    Zr += __shfl_sync(0xffffffffu, Z[0], l0 + d);
    Zi += __shfl_sync(0xffffffffu, Z[1], l0 + d);
    HH += __shfl_sync(0xffffffffu, hh, l0 + d);
  }
  if (on && i == 0) w.ly[k] = het_epilogue(L, Zr, Zi, HH);
  __syncwarp();
}

// Time-marginalised: a candidate after another, as k_het_tm.
template <int NDET>
__device__ __forceinline__ void eval_het_tm(ChainShared<NDET, CHAIN_HET_TM>& s, const HetTables& H, unsigned char* scratch,
                                            const ChainLayout& lay, int warp, int lane) {
  ChainWork& w = s.w;
  const LikeConst& L = s.L;
  float2* y = reinterpret_cast<float2*>(scratch);
  for (int a = 0; a < w.n_act; ++a) {
    const int k = w.list[a];
    const EvalRecord& r = w.rec[k];
    if (warp == 0) {
      het_prepare_warp<NDET>(L, H, r, s.e.prep, lane);
      het_in_set<NDET, 1>(s.e.in, 0, s.e.prep, lane);
    }
    HetAcc<NDET, 1> acc;
    acc.clear();
    het_products<NDET>(H, s.e.prep, s.e.in, reinterpret_cast<float*>(scratch + lay.anc_off), lay.panel, warp,
                       kChainWarps, lane, acc, y);
#pragma unroll
    for (int i = 0; i < NDET; ++i) {
      float d = acc.hh[i];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
      if (lane == 0) s.e.hh[warp][i] = d;
    }
    __syncthreads();
    float wm, ws;
    if (L.tm_M > 0)
      tm_pass_nufft(L, H, y, tm_nufft_grid(scratch, H.n_bins), tm_nufft_tw(scratch, H.n_bins, L.tm_M), warp,
                    kChainWarps, lane, nullptr, wm, ws);
    else
      tm_pass(L, H, y, warp, kChainWarps, lane, nullptr, wm, ws);
    if (lane == 0) {
      s.e.tm[warp][0] = wm;
      s.e.tm[warp][1] = ws;
    }
    __syncthreads();
    if (warp == 0) {
      const double ll = tm_finish<NDET>(L, r, s.e.hh, s.e.tm, kChainWarps, lane);
      if (lane == 0) w.ly[k] = ll;
    }
    if (threadIdx.x == 0) {
      for (int j = 0; j < 2 * SWIG_MAX_DET; ++j) w.kap[k][j] = 0.0;
      for (int i = 0; i < SWIG_MAX_DET; ++i) w.vv[k][i] = 0.0;
    }
    __syncthreads();
  }
}

template <int NDET, int MODE>
__global__ void __launch_bounds__(kChainBlock, 1)
    k_ns_chain(const ChainEvent* __restrict__ ev, int n_ev, NSGlobal* gb, ChainLayout lay) {
  extern __shared__ __align__(16) unsigned char smem[];
  ChainShared<NDET, MODE>& s = *reinterpret_cast<ChainShared<NDET, MODE>*>(smem);
  unsigned char* scratch = smem + lay.scratch_off;
  ChainWork& w = s.w;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k_chains = ev[0].S.nrep;
  const bool timer = blockIdx.x == 0 && tid == 0;
  unsigned long long t0 = gtimer(), t1;
  if (tid < 8) s.prof[tid] = 0;
  if (tid < 4) s.cta[tid] = 0;
  if (tid == 0) s.event = -1;
  NSGlobal* g0 = ev[0].P.g;
  for (;;) {
    // a CTA without a chain waits here for the longest one: as long as any advances
    if (!grid_sync(gb, lay.n_ctas, lay.spin_limit, &gb->beat)) return;
    if (timer) {
      t1 = gtimer();
      g0->t_wait_sweep += t1 - t0;
      t0 = t1;
      g0->rounds += 1;
    }
    if ((int)blockIdx.x < n_ev) ns_boundary_check(ev[blockIdx.x].L, ev[blockIdx.x].S, ev[blockIdx.x].P, scratch);
    if (!grid_sync(gb, lay.n_ctas, lay.spin_limit)) return;
    bool all_run = true;
    for (int e = 0; e < n_ev; ++e) all_run = all_run && *(volatile int*)&ev[e].P.g->status == ST_RUNNING;
    if (!all_run) return;
    if ((int)blockIdx.x < n_ev) 
      ns_boundary_advance(ev[blockIdx.x].L, ev[blockIdx.x].S, ev[blockIdx.x].P, scratch, lay.scratch_bytes);
    if (timer) *(volatile int*)&gb->task = 0;
    if (!grid_sync(gb, lay.n_ctas, lay.spin_limit)) return;
    if (timer) {
      t1 = gtimer();
      g0->t_bound += t1 - t0;
      t0 = t1;
    }
    for (;;) {
      __syncthreads();
      if (tid == 0) s.task = atomicAdd(&gb->task, 1);
      __syncthreads();
      const int task = s.task;
      if (task >= n_ev * k_chains) break;
      const int e = task / k_chains, c = task - e * k_chains;
      const ChainEvent& E = ev[e];
      if (s.event != e) {  // the event's constants and, resident, its weights and tables
        __syncthreads();
        const unsigned* src = reinterpret_cast<const unsigned*>(&E.L);
        for (int q = tid; q < (int)(sizeof(LikeConst) / 4); q += kChainBlock) reinterpret_cast<unsigned*>(&s.L)[q] = src[q];
        src = reinterpret_cast<const unsigned*>(&E.S);
        for (int q = tid; q < (int)(sizeof(SamplerConst) / 4); q += kChainBlock)
          reinterpret_cast<unsigned*>(&s.S)[q] = src[q];
        if constexpr (MODE == CHAIN_FOLD) {
          for (int q = tid; q < 32 * kFoldKinds; q += kChainBlock) s.e.x[q] = E.F.x[q];
          if (lay.res_off > 0) {
            float4* d = reinterpret_cast<float4*>(smem + lay.res_off);
            const int nw = E.F.nc * NDET * 32, nt = FR_ROWS * E.F.ld / 4;
            const float4* tab4 = reinterpret_cast<const float4*>(E.F.tab);
            for (int q = tid; q < nw; q += kChainBlock) cp_async16(d + q, E.F.w + q);
            for (int q = tid; q < nt; q += kChainBlock) cp_async16(d + nw + q, tab4 + q);
            asm volatile("cp.async.wait_all;" ::: "memory");
          }
        }
        if constexpr (MODE == CHAIN_HET) {
          if (tid < NBASIS) s.e.fc[tid] = E.H.fid->c[tid];
          if (tid < SWIG_MAX_DET) s.e.ft[tid] = E.H.fid->tau[tid];
        }
        if constexpr (MODE == CHAIN_HET)
          if (lay.res_off > 0) {
            float* d = reinterpret_cast<float*>(smem + lay.res_off);
            for (int q = tid; q < HC_ROWS * E.H.n_chunks; q += kChainBlock) cp_async<4>(d + q, E.H.chunk + q);
            cp_async_commit();
            cp_async_wait<0>();
          }
        __syncthreads();
        if (tid == 0) s.event = e;
      }
      if (MODE == CHAIN_HET_TM && E.L.tm_M > 0) tm_load_twiddles(s.L, E.H, scratch, E.H.n_bins);
      const SamplerPtrs& P = E.P;
      float* base = lay.base_off > 0 ? reinterpret_cast<float*>(smem + lay.base_off) : nullptr;
      const float4* W = E.F.w;
      const float* tab = MODE == CHAIN_FOLD ? E.F.tab : E.H.chunk;
      if (MODE == CHAIN_FOLD && lay.res_off > 0) {
        W = reinterpret_cast<const float4*>(smem + lay.res_off);
        tab = reinterpret_cast<const float*>(W + E.F.nc * NDET * 32);
      }
      if (MODE == CHAIN_HET && lay.res_off > 0) tab = reinterpret_cast<const float*>(smem + lay.res_off);
      // written by CTA e at the boundary: read through L2, never a stale L1 line
      const double logl_star = __ldcg(&P.g->logl_star);
      const long long it = __ldcg(&P.g->iter);
      if (warp == 0) {
        warp_copy_cg(&w.ch, &P.chains[c], sizeof(ChainState), lane);
        warp_copy_cg(&w.rx, &P.recx[c], sizeof(EvalRecord), lane);
      }
      unsigned long long* prof = c == 0 && e == 0 ? s.prof : nullptr;
      bool have = false;
      if constexpr (MODE != CHAIN_HET_TM)
        if (tid == 0) s.e.base_ok = 0;
      for (long long guard = 0; guard < (1ll << 24); ++guard) {
        long long tc = 0;
        if (warp == 0) {
          tc = clock64();
          if constexpr (MODE == CHAIN_FOLD)
            if (have) finish_fold<NDET>(s, lane);
          if constexpr (MODE == CHAIN_HET)
            if (have) finish_het<NDET>(s, E.H, lane);
          if (lane == 0 && (guard & 7) == 0) atomicAdd(&gb->beat, 1u);
          chain_control<NDET, MODE != CHAIN_FOLD>(s.L, s.S, P, w, c, it, logl_star, have, lane, prof, &gb->beat);
          if constexpr (MODE != CHAIN_HET_TM)
            if (lane == 0 && w.status == ROUND_EVAL && (w.fl & (BF_INTR | BF_TIDE))) s.e.base_ok = 0;
          if (lane == 0) {
            const long long t2 = clock64();
            s.cta[2] += t2 - tc;
            s.cta[3] += t2 - tc;
            tc = t2;
          }
        }
        __syncthreads();
        if (w.status == ROUND_DONE) break;
        chain_setup<NDET>(s.L, w, warp, lane);
        if (prof && tid == 0) prof[4] += clock64() - tc;
        if constexpr (MODE == CHAIN_FOLD)
          eval_fold<NDET>(s, E.F, W, tab, base, reinterpret_cast<float*>(scratch),
                          lay.scratch_bytes / (int)(kFoldAnchor * sizeof(float)), warp, lane);
        else if constexpr (MODE == CHAIN_HET)
          eval_het<NDET>(s, E.H, tab, base, reinterpret_cast<float*>(scratch), lay.scratch_bytes, warp, lane);
        else
          eval_het_tm<NDET>(s, E.H, scratch, lay, warp, lane);
        __syncthreads();
        if (tid == 0) {
          s.cta[0] += w.n_act;
          s.cta[1] += clock64() - tc;
        }
        have = true;
      }
      if (warp == 0) warp_copy(&P.chains[c], &w.ch, sizeof(ChainState), lane);
    }
    if (tid == 0) {
      if (ev[0].P.cta_prof) {
        unsigned long long* cp = ev[0].P.cta_prof + 4 * (size_t)blockIdx.x;
        for (int j = 0; j < 4; ++j) cp[j] += s.cta[j];
      }
      if (blockIdx.x == 0) {
        g0->f_units += s.cta[0];
        g0->f_unit_cyc += s.cta[1];
        g0->f_idle_cyc += s.cta[2];
      }
      for (int j = 0; j < 4; ++j) s.cta[j] = 0;
      // the CTA that ran the first event's first chain
      if (s.prof[7]) {
        atomicAdd(&g0->c_result, s.prof[0]);
        atomicAdd(&g0->c_step, s.prof[1]);
        atomicAdd(&g0->c_prop, s.prof[2]);
        atomicAdd(&g0->c_free, s.prof[3]);
        atomicAdd(&g0->c_setup, s.prof[4]);
        atomicAdd(&g0->n_free, s.prof[5]);
        atomicAdd(&g0->n_setup, s.prof[6]);
        atomicAdd(&g0->n_step, s.prof[7]);
        for (int j = 0; j < 8; ++j) s.prof[j] = 0;
      }
    }
    if (timer) {
      t1 = gtimer();
      g0->t_ctrl += t1 - t0;
      t0 = t1;
    }
  }
}

namespace {
template <int NDET>
void* chain_kernel_as(int mode) {
  switch (mode) {
    case CHAIN_FOLD: return (void*)k_ns_chain<NDET, CHAIN_FOLD>;
    case CHAIN_HET: return (void*)k_ns_chain<NDET, CHAIN_HET>;
    default: return (void*)k_ns_chain<NDET, CHAIN_HET_TM>;
  }
}
}  // namespace

void* chain_kernel(int n_det, int mode) {
  switch (n_det) {
    case 1: return chain_kernel_as<1>(mode);
    case 2: return chain_kernel_as<2>(mode);
    case 3: return chain_kernel_as<3>(mode);
    default: return chain_kernel_as<4>(mode);
  }
}

}  // namespace swig
