// Heterodyned (relative-binning) likelihood (Sec. 3.4 of the paper) on the device.
//
// With the fiducial waveform h0 the ratio r_i(f) = h_i(f) / h0_i(f) is, for
// this model, (C_i / C0_i) exp(-2 pi i (dP(f) + f dtau_i)) with dP = P - P0 and
// dtau_i = tau_i - tau0_i (the f^-7/6 amplitude cancels).  It is evaluated at
// the N_b + 1 bin edges and taken linear inside each bin:
//   r0_b = (r(e_b) + r(e_b+1)) / 2,  r1_b = (r(e_b+1) - r(e_b)) / (e_b+1 - e_b),
//   Z_i  = sum_b A0_ib r0_b + A1_ib r1_b,
//   HH_i = sum_b B0_ib |r0_b|^2 + 2 B1_ib Re(r0_b conj(r1_b)),
// with the summary data A0, A1, B0, B1 (host FP64, stored FP32).  dP at an
// edge is a double-float sum of (c_j - c0_j) phi_j(f_e) (it can reach hundreds
// of cycles far from the fiducial); the contraction itself is FP32 per bin with
// a pairwise (warp-shuffle) reduction and an FP64 epilogue.
//
// Time marginalisation (t_c marginalised, Sec. 3.1 and App. A).  Z_i is
// linear in the edge values, Z_i = sum_e g_ie r_i(e) with hat-function weights
// g_ie = (A0_ib/2 - A1_ib/w_b) from the bin above the edge plus
// (A0_ib/2 + A1_ib/w_b) from the bin below.  A common geocentric shift dt
// multiplies r_i(e) by exp(-2 pi i f_e dt) in every detector, so the network
// overlap at a grid node is one sum over edges,
//   Z(dt_j) = sum_e y_e exp(-2 pi i f_e dt_j),   y_e = sum_i g_ie r_i(e),
// with the templates built at the fiducial's t_c.  <h|h> is the same at every
// node (a time shift only rotates h) and is taken there once.
#pragma once

#include "device_common.cuh"
#include "packed.cuh"

namespace swig {

struct HetTables {
  int n_bins;                 // N_b
  const float* edge_basis;    // [2 * NBASIS][N_b + 1] phi_j(f_e): row 2j hi parts, row 2j+1 lo parts
  const float* edge_f;        // [2][N_b + 1] f_e: hi parts, lo parts
  const EvalRecord* fid;      // fiducial record
  const float2* tm_w;         // [N_b + 1] exp(-2 pi i f_e dt), one grid step
  // non-uniform FFT form of the time pass (see het_nufft_tables)
  const float* nu_wt;
  const float* nu_corr;
  const float2* nu_tw;
  const int4* nu_piece;  // gather pieces (first entry, entries, first edge)
  const int4* nu_point;  // grid points with entries (point, first piece, pieces)
  // chunk anchors (kernels.h HetChunkRow)
  int n_chunks;
  const float* chunk;  // [HC_ROWS][n_chunks]
  // edge weights of the contraction (het_edge_weights in capi.cu): per chunk,
  // detector and lane (Re g_ie, Im g_ie, B0_ib / 2, f_e - f_a with detector 0)
  const float4* ew;    // [n_chunks][n_det][32]
};

__host__ __device__ inline HetTables het_tables(const DeviceBuffers& B) {
  HetTables H;
  H.n_bins = B.het_nb;
  H.edge_basis = B.het_edge_basis;
  H.edge_f = B.het_edge_f;
  H.fid = B.het_fid;
  H.tm_w = B.het_tm_w;
  H.nu_wt = B.het_nu_wt;
  H.nu_corr = B.het_nu_corr;
  H.nu_tw = B.het_nu_tw;
  H.nu_piece = B.het_nu_piece;
  H.nu_point = B.het_nu_point;
  H.n_chunks = B.het_nc;
  H.chunk = B.het_chunk;
  H.ew = B.het_ew;
  return H;
}

// Per-evaluation constants: coefficient and delay differences from the
// fiducial in double-float, and rho_i = C_i / C0_i.
template <int NDET>
struct HetPrep {
  dfl dc[NBASIS];
  dfl dtau[NDET];
  float rho_re[NDET], rho_im[NDET];
};

// The differences by a warp, one per lane, against the fiducial's c and tau.
template <int NDET>
__device__ __forceinline__ void het_differences(const double* f0c, const double* f0tau, const EvalRecord& r,
                                                HetPrep<NDET>& p, int lane) {
  const bool c = lane < NBASIS, t = lane >= 16 && lane < 16 + NDET;
  const double x = c ? r.c[lane] - f0c[lane] : t ? r.tau[lane - 16] - f0tau[lane - 16] : 0.0;
  const dfl d = df_from_double(x);
  if (c) p.dc[lane] = d;
  if (t) p.dtau[lane - 16] = d;
  __syncwarp();
}

// The constants by a warp, one per lane.
template <int NDET>
__device__ __forceinline__ void het_prepare_warp(const LikeConst& L, const HetTables& H, const EvalRecord& r,
                                                 HetPrep<NDET>& p, int lane) {
  const EvalRecord& f0 = *H.fid;
  if (lane < NDET) {
    const int i = lane;
    const double iden = L.het_fid_iden[i];
    p.rho_re[i] = (float)((r.cre[i] * f0.cre[i] + r.cim[i] * f0.cim[i]) * iden);
    p.rho_im[i] = (float)((r.cim[i] * f0.cre[i] - r.cre[i] * f0.cim[i]) * iden);
  }
  het_differences<NDET>(f0.c, f0.tau, r, p, lane);
}

__device__ __forceinline__ unsigned smem_addr(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_addr(dst)), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// ---------------------------------------------------------------------------
// Contraction by edges.  r_i(e) = rho_i u_i(e) with |u| = 1, so with the hat
// weights g_ie of the header
//   Z_i = rho_i sum_e g_ie u_i(e),
//   <h|h>_i = |rho_i|^2 sum_b B0_ib (1 + Re u_i(e_b) u_i*(e_b+1)) / 2
// (|r| is the same at both ends of a bin, so the B1 term vanishes): one phasor,
// one complex multiply-add and one term of the bin's phase difference per edge
// and detector, on 16 bytes of weights instead of 24 of summary data.  A warp
// takes a chunk of 32 edges for N evaluations at once (N = 2: packed FP32, the
// weights loaded once for all).
// ---------------------------------------------------------------------------
template <int NDET, int N>
struct HetAcc {
  using O = PkOps<N>;
  typename O::T zr[NDET], zi[NDET], hh[NDET];  // sum g u; sum (B0 / 2) (1 - Re u u*')
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < NDET; ++i) zr[i] = zi[i] = hh[i] = O::all(0.0f);
  }
};

// Phase differences of one edge from the double-float sum over the basis
// (chunks whose Taylor form does not serve the evaluation).
template <int NDET>
__device__ __noinline__ void het_exact_phase(const HetTables& H, const HetPrep<NDET>& p, int e, float* out) {
  const size_t ne = (size_t)H.n_bins + 1;
  dfl dp = {0.0f, 0.0f};
  for (int j = 0; j < NBASIS; ++j)
    dp = df_add(dp, df_mul(p.dc[j], dfl{__ldg(H.edge_basis + 2 * j * ne + e),
                                        __ldg(H.edge_basis + (2 * j + 1) * ne + e)}));
  const dfl fe = {__ldg(H.edge_f + e), __ldg(H.edge_f + ne + e)};
#pragma unroll
  for (int i = 0; i < NDET; ++i) out[i] = df_frac(df_add(dp, df_mul(fe, p.dtau[i])));
}

// What the anchors of N evaluations read (interleaved, evaluation k at [..][k]):
// coefficient differences in double-float and their magnitudes, and the delay
// differences.
template <int NDET, int N>
struct __align__(8) HetIn {
  float dc_hi[NBASIS][N], dc_lo[NBASIS][N], dc_abs[NBASIS][N];
  float dt_hi[NDET][N], dt_lo[NDET][N];
};
// Evaluation k's share, one value per lane (after het_prepare_warp).
template <int NDET, int N>
__device__ __forceinline__ void het_in_set(HetIn<NDET, N>& in, int k, const HetPrep<NDET>& p, int lane) {
  if (lane < NBASIS) {
    in.dc_hi[lane][k] = p.dc[lane].hi;
    in.dc_lo[lane][k] = p.dc[lane].lo;
    in.dc_abs[lane][k] = fabsf(p.dc[lane].hi);
  }
  if (lane < NDET) {
    in.dt_hi[lane][k] = p.dtau[lane].hi;
    in.dt_lo[lane][k] = p.dtau[lane].lo;
  }
}

// The basis functions that only the spins move: the other sums (rows of
// kHetBaseRows values per chunk: A, a_1 in double-float, the bound, a_2 ..)
// stand while masses and tides do.
__device__ __forceinline__ constexpr bool het_moved(int j) { return j == B_M23 || j == B_M13; }
enum { HB_A = 0, HB_S = 2, HB_R = 4, HB_POLY = 5 };
static_assert(HB_POLY + kHetPoly == kHetBaseRows, "base rows");

// One quarter (sub 0 .. 3) of the anchors of chunk q for N evaluations, value m
// of evaluation k to out[N m + k]: sub 0 the phases frac(dP(f_a) + f_a dtau_i),
// sub 1 a_1, 1 / S and the exact flag, sub 2 and 3 the Taylor terms.  WITH 1: from the base rows
// (stride nc) and the moved functions; -1: the base rows themselves (N = 1),
// at out[m nc].
template <int NDET, int N, int WITH = 0>
__device__ __forceinline__ void het_anchor_part(const float* __restrict__ chunk, int nc, const HetIn<NDET, N>& in,
                                                int sub, int q, const float* base, float* out) {
  using O = PkOps<N>;
  using T = typename O::T;
  const float* tab = chunk + q;
  auto row = [&](int r) { return O::all(tab[r * nc]); };
  auto from = [&](int m) { return O::all(WITH == 1 ? base[m * nc + q] : 0.0f); };
  auto put = [&](int m, T v) { *reinterpret_cast<T*>(out + N * m) = v; };
  auto dc = [&](int j) { return DflN<N>{O::load(in.dc_hi[j]), O::load(in.dc_lo[j])}; };
  auto takes = [](int j) { return WITH == 0 || het_moved(j) == (WITH == 1); };
  if (sub == 0) {
    DflN<N> A = {from(HB_A), from(HB_A + 1)};
#pragma unroll
    for (int j = 0; j < NBASIS; ++j)
      if (takes(j)) A = dfn_add<N>(A, dfn_mul<N>(dc(j), DflN<N>{row(HC_VAL_HI + j), row(HC_VAL_LO + j)}));
    if constexpr (WITH < 0) {
      out[HB_A * nc] = A.hi;
      out[(HB_A + 1) * nc] = A.lo;
    } else {
      const DflN<N> fa = {row(HC_FA_HI), row(HC_FA_LO)};
#pragma unroll
      for (int i = 0; i < NDET; ++i)
        put(kHetAncPhase + i,
            dfn_frac<N>(dfn_add<N>(A, dfn_mul<N>(fa, DflN<N>{O::load(in.dt_hi[i]), O::load(in.dt_lo[i])}))));
    }
  } else if (sub == 1) {
    DflN<N> S = {from(HB_S), from(HB_S + 1)};
    T R = from(HB_R);
#pragma unroll
    for (int j = 0; j < NBASIS; ++j)
      if (takes(j)) {
        S = dfn_add<N>(S, dfn_mul<N>(dc(j), DflN<N>{row(HC_D1_HI + j), row(HC_D1_LO + j)}));
        R = O::fma(O::load(in.dc_abs[j]), row(HC_BND + j), R);
      }
    if constexpr (WITH < 0) {
      out[HB_S * nc] = S.hi;
      out[(HB_S + 1) * nc] = S.lo;
      out[HB_R * nc] = R;
    } else {
      put(0, O::add(S.hi, S.lo));
      put(kHetAncInvS, row(HC_INV_S));
      float r[N];
      O::get(R, r);
#pragma unroll
      for (int k = 0; k < N; ++k) out[N * kHetAncExact + k] = r[k] > kHetTaylorEps ? 1.0f : 0.0f;
    }
  } else {
    constexpr int kHalf = (kHetPoly + 1) / 2;  // orders 2 .. kHalf + 1, and above
    T a[kHalf];
    const int m0 = sub == 2 ? 0 : kHalf;
#pragma unroll
    for (int m = 0; m < kHalf; ++m) a[m] = m0 + m < kHetPoly ? from(HB_POLY + m0 + m) : O::all(0.0f);
#pragma unroll
    for (int j = 0; j < NBASIS; ++j)
      if (takes(j)) {
        const T c = O::load(in.dc_hi[j]);
#pragma unroll
        for (int m = 0; m < kHalf; ++m)
          if (m0 + m < kHetPoly) a[m] = O::fma(c, row(HC_POLY + (m0 + m) * NBASIS + j), a[m]);
      }
#pragma unroll
    for (int m = 0; m < kHalf; ++m)
      if (m0 + m < kHetPoly) {
        if constexpr (WITH < 0)
          out[(HB_POLY + m0 + m) * nc] = a[m];
        else
          put(1 + m0 + m, a[m]);
      }
  }
}

// Anchors of np chunks from q0 on for `sets` groups of N evaluations by the
// warps first, first + stride, ... of a CTA: quarter by quarter, 32 chunks (of
// all groups, one after the other) per warp and turn.  chunk: H.chunk or its
// copy in shared memory.  Group g's anchors at s_an + (g panel + q) kHetAncPair
// (N = 2) or kHetAncOne.
template <int NDET, int N, int WITH = 0>
__device__ __forceinline__ void het_anchors(const HetTables& H, const float* chunk, const HetIn<NDET, N>* in, int sets,
                                            int q0, int np, int panel, const float* base, float* s_an, int first,
                                            int stride, int lane) {
  const int all = sets * np, per = (all + 31) >> 5;  // warp turns of a quarter
  for (int sub = 0, t = first; sub < 4;) {
    if (t >= per) {
      t -= per;
      ++sub;
      continue;
    }
    const int v = 32 * t + lane;
    if (v < all) {
      const int g = v / np, q = v - g * np;
      het_anchor_part<NDET, N, WITH>(chunk, H.n_chunks, in[g], sub, q0 + q, base,
                                     s_an + (size_t)(g * panel + q) * (N == 2 ? kHetAncPair : kHetAncOne));
    }
    t += stride;
  }
}

// Chunk q of N evaluations.  an: kHetAncStride values per evaluation, value m
// of evaluation k at an[N m + k]; in: their inputs; p[k]: its constants (exact chunks only); w: the chunk's weights
// at this lane.  TM: Z is not formed, y[e] = sum_i rho_i g_ie u_i(e) is stored.
template <int NDET, int N, bool TM = false>
__device__ __forceinline__ void het_edges(const HetTables& H, const float* __restrict__ an,
                                          const HetIn<NDET, N>& in, const HetPrep<NDET>* const* p, int q, int lane,
                                          const float4* w, HetAcc<NDET, N>& acc, float2* y = nullptr) {
  using O = PkOps<N>;
  using T = typename O::T;
  const float d = w[0].w;
  T ph[NDET];
  bool exact = false;
#pragma unroll
  for (int k = 0; k < N; ++k) exact = exact || an[N * kHetAncExact + k] != 0.0f;
  {
    const T d2 = O::all(d), x = O::mul(d2, O::load(an + N * kHetAncInvS));
    T v = O::load(an + N * kHetPoly);
#pragma unroll
    for (int n = kHetPoly - 1; n >= 0; --n) v = O::fma(v, x, O::load(an + N * n));
    v = O::mul(v, x);
#pragma unroll
    for (int i = 0; i < NDET; ++i)
      ph[i] = O::add(O::load(an + N * (kHetAncPhase + i)), O::fma(d2, O::load(in.dt_hi[i]), v));
  }
  if (exact) {  // warp-uniform, rare
    float f[NDET][N];
#pragma unroll
    for (int i = 0; i < NDET; ++i) O::get(ph[i], f[i]);
#pragma unroll
    for (int k = 0; k < N; ++k)
      if (an[N * kHetAncExact + k] != 0.0f) {
        float g[NDET];
        het_exact_phase<NDET>(H, *p[k], min(31 * q + lane, H.n_bins), g);
#pragma unroll
        for (int i = 0; i < NDET; ++i) f[i][k] = g[i];
      }
#pragma unroll
    for (int i = 0; i < NDET; ++i) ph[i] = O::set(f[i]);
  }
  float yr = 0.0f, yi = 0.0f;
#pragma unroll
  for (int i = 0; i < NDET; ++i) {
    const T m = O::all(12582912.0f), nm = O::all(-12582912.0f), mone = O::all(-1.0f);
    const T r = O::mul(O::fma(O::add(O::add(ph[i], m), nm), mone, ph[i]), O::all(6.283185307179586f));
    float a[N], c[N], s[N];
    O::get(r, a);
#pragma unroll
    for (int k = 0; k < N; ++k) __sincosf(a[k], &s[k], &c[k]);  // u = c - i s
    const T co = O::set(c), si = O::set(s);
    float cn[N], sn[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
      cn[k] = __shfl_down_sync(0xffffffffu, c[k], 1);
      sn[k] = __shfl_down_sync(0xffffffffu, s[k], 1);
    }
    const T gr = O::all(w[i].x), gi = O::all(w[i].y);
    if (TM) {
      const float zr = w[i].x * c[0] + w[i].y * s[0], zi = w[i].y * c[0] - w[i].x * s[0];
      yr += p[0]->rho_re[i] * zr - p[0]->rho_im[i] * zi;
      yi += p[0]->rho_re[i] * zi + p[0]->rho_im[i] * zr;
    } else {
      acc.zr[i] = O::fma(gr, co, O::fma(gi, si, acc.zr[i]));
      acc.zi[i] = O::fma(gi, co, O::fma(O::all(-w[i].x), si, acc.zi[i]));
    }
    // 1 - (c c' + s s'), zero-weighted where the lane has no bin
    const T dd = O::fma(O::fma(si, O::set(sn), O::mul(co, O::set(cn))), mone, O::all(1.0f));
    acc.hh[i] = O::fma(O::all(w[i].z), dd, acc.hh[i]);
  }
  if (TM) {
    const int e = 31 * q + lane;
    if (e <= H.n_bins && (lane < 31 || e == H.n_bins)) y[e] = make_float2(yr, yi);
  }
}

// The results of one evaluation from its sums (T_i = sum g u, D_i = sum (B0 /
// 2) (1 - Re u u*'), FP64): Z_i and <h|h>_i of detector i, and the cache of
// projection-only evaluations, kap = (Z_i / C_i) / inv_scale_i and vv = <h|h>_i
// / |C_i|^2 A1^2, in which rho_i drops out.
__device__ __forceinline__ void het_detector(const LikeConst& L, const EvalRecord& fid, const EvalRecord& r, int i,
                                             double tr, double ti, double dsum, double* Z, double* hh, double* kap2,
                                             double* vv) {
  const double c0r = fid.cre[i], c0i = fid.cim[i], iden = L.het_fid_iden[i];
  // (T / C0): kap before the data scale
  const double kr = (tr * c0r + ti * c0i) * iden, ki = (ti * c0r - tr * c0i) * iden;
  const double cr = r.cre[i], ci = r.cim[i];
  Z[0] = cr * kr - ci * ki;
  Z[1] = cr * ki + ci * kr;
  const double b = (L.het_b0[i] - dsum) * iden;
  *hh = (cr * cr + ci * ci) * b;
  kap2[0] = kr * L.rscale[i];
  kap2[1] = ki * L.rscale[i];
  *vv = b * (L.amp1 * L.amp1);
}

// The edge products y_e of one evaluation (time marginalisation) by a whole
// CTA: anchors of a panel of chunks in s_an, then the chunks q = warp, warp +
// n_warps, ... of every panel.  The caller's prep and in are visible after the
// first barrier here; y after the caller's next one.
template <int NDET>
__device__ inline void het_products(const HetTables& H, const HetPrep<NDET>& prep, const HetIn<NDET, 1>& in,
                                    float* s_an, int panel, int warp, int n_warps, int lane, HetAcc<NDET, 1>& acc,
                                    float2* y) {
  const HetPrep<NDET>* pp[1] = {&prep};
  for (int q0 = 0; q0 < H.n_chunks; q0 += panel) {
    const int np = min(panel, H.n_chunks - q0);
    __syncthreads();
    het_anchors<NDET, 1>(H, H.chunk, &in, 1, q0, np, panel, nullptr, s_an, warp, n_warps, lane);
    __syncthreads();
    for (int q = warp; q < np; q += n_warps) {
      float4 w[NDET];
#pragma unroll
      for (int i = 0; i < NDET; ++i) w[i] = __ldg(H.ew + ((size_t)(q0 + q) * NDET + i) * 32 + lane);
      het_edges<NDET, 1, true>(H, s_an + q * kHetAncOne, in, pp, q0 + q, lane, w, acc, y);
    }
  }
}

// Vector k's sums over the warps in warp order (double-float, rounded once to
// FP64): lane 3 i + kind (Re T, Im T, D) of detector i; part[warp][i][K kind +
// vector].
template <int NDET, int K>
__device__ __forceinline__ double het_part_sum(const float (*part)[NDET][3 * K], int n_warps, int k, int lane) {
  double v = 0.0;
  if (lane < 3 * NDET) {
    const int i = lane / 3, kind = lane - 3 * i;
    dfl t = {0.0f, 0.0f};
    for (int w = 0; w < n_warps; ++w) t = df_add(t, dfl{part[w][i][K * kind + k], 0.0f});
    v = (double)t.hi + (double)t.lo;
  }
  __syncwarp();
  return v;
}

// Network Z and <h|h> from those sums, one detector per lane, added in
// detector order (every lane); kap: component j of the cache on lane j, vv:
// detector i's on lane i.
template <int NDET>
__device__ __forceinline__ void het_network(const LikeConst& L, const EvalRecord& fid, const EvalRecord& r, double v,
                                            int lane, double& Zr, double& Zi, double& HH, double& kap, double& vv) {
  const unsigned full = 0xffffffffu;
  const int d = lane < NDET ? lane : 0;
  const double tr = __shfl_sync(full, v, 3 * d), ti = __shfl_sync(full, v, 3 * d + 1);
  const double ds = __shfl_sync(full, v, 3 * d + 2);
  double Z[2], hh, k2[2], vi;
  het_detector(L, fid, r, d, tr, ti, ds, Z, &hh, k2, &vi);
  Zr = Zi = HH = 0.0;
#pragma unroll
  for (int i = 0; i < NDET; ++i) {
    Zr += __shfl_sync(full, Z[0], i);
    Zi += __shfl_sync(full, Z[1], i);
    HH += __shfl_sync(full, hh, i);
  }
  const double k0 = __shfl_sync(full, k2[0], lane < 2 * NDET ? lane >> 1 : 0);
  const double k1 = __shfl_sync(full, k2[1], lane < 2 * NDET ? lane >> 1 : 0);
  kap = lane < 2 * NDET ? ((lane & 1) ? k1 : k0) : 0.0;
  vv = lane < NDET ? vi : 0.0;
}

// FP64 epilogue: plain Re Z or phase-marginalised log I0(|Z|), minus
// <h|h>/2 and <d|d>/2.
__device__ inline double het_epilogue(const LikeConst& L, double Z_re, double Z_im, double HH) {
  const double base_ll = -0.5 * HH - 0.5 * L.DD;
  if (L.phase_marg) {
    const double x = sqrt(Z_re * Z_re + Z_im * Z_im);
    return (L.fast_epilogue ? x + (double)log_i0e_f32((float)x) : log_bessel_i0(x)) + base_ll;
  }
  return Z_re + base_ll;
}

// ---------------------------------------------------------------------------
// Time pass of the time-marginalised likelihood.
// ---------------------------------------------------------------------------
constexpr int kTmNodes = 32;  // grid nodes per warp pass (lane l ends with node j0 + l)

// Log weight of one node: log I0(|Z|) with phi_c marginalised, Re Z otherwise.
__device__ __forceinline__ float tm_node_logw(const LikeConst& L, float zr, float zi) {
  if (L.phase_marg) {
    const float x = sqrtf(zr * zr + zi * zi);
    return x + log_i0e_f32(x);
  }
  return zr;
}

// One level of the halving reduction: lanes with bit O set keep the upper O
// nodes, the others the lower O, each adding its partner's copy of them.
template <int O>
__device__ __forceinline__ void tm_halve(float* ar, float* ai, int lane) {
  const bool up = (lane & O) != 0;
#pragma unroll
  for (int k = 0; k < O; ++k) {
    const float sr = up ? ar[k] : ar[k + O], si = up ? ai[k] : ai[k + O];
    const float kr = up ? ar[k + O] : ar[k], ki = up ? ai[k + O] : ai[k];
    ar[k] = kr + __shfl_xor_sync(0xffffffffu, sr, O);
    ai[k] = ki + __shfl_xor_sync(0xffffffffu, si, O);
  }
}

// One edge's inputs to the time pass: its product y_e, rotation w_e and
// frequency (double-float); an edge past the end reads as y = 0, w = 1.
struct TmEdge {
  float2 y, w;
  dfl f;
};

__device__ __forceinline__ TmEdge tm_load_edge(const HetTables& H, const float2* __restrict__ y, int e, int ne) {
  TmEdge d;
  if (e < ne) {
    d.y = y[e];
    d.w = H.tm_w[e];
    d.f = {H.edge_f[e], H.edge_f[ne + e]};
  } else {
    d.y = make_float2(0.0f, 0.0f);
    d.w = make_float2(1.0f, 0.0f);
    d.f = {0.0f, 0.0f};
  }
  return d;
}

// y_e exp(-2 pi i f_e dt): the term at the chunk's first node.
__device__ __forceinline__ float2 tm_start(const TmEdge& d, dfl dt) {
  const float twopi = 6.283185307179586f;
  float s, co;
  __sincosf(twopi * df_frac(df_mul(d.f, dt)), &s, &co);  // exp(-2 pi i f_e dt) = co - i s
  return make_float2(d.y.x * co + d.y.y * s, d.y.y * co - d.y.x * s);
}

// One warp, nodes [j0, j0 + 32): Z(dt_j) = sum_e y_e exp(-2 pi i f_e dt_j).
// Lane l takes edges l, l + 32, ... two at a time (e and e + 32, added in
// that order, so the sums are those of one edge at a time): one phasor at
// dt_j0 from the double-float phase f_e dt_j0, then a rotation by w_e per
// node (31 steps, FP32 drift ~2e-6 rad).  The next pair's loads are issued
// before the current pair's steps.  The 32 node sums are reduced across the
// warp by halving, after which lane l holds node j0 + l; returns its log
// weight (-inf past the last node).  All 32 lanes call it together.
__device__ inline float tm_nodes_warp(const LikeConst& L, const HetTables& H, const float2* __restrict__ y, int j0,
                                      int lane) {
  float ar[kTmNodes], ai[kTmNodes];
#pragma unroll
  for (int k = 0; k < kTmNodes; ++k) ar[k] = ai[k] = 0.0f;
  const dfl d0 = df_from_double(L.tm_t0 + (double)j0 * L.tm_dt);
  const int ne = H.n_bins + 1;
  TmEdge a = tm_load_edge(H, y, lane, ne), b = tm_load_edge(H, y, lane + 32, ne);
  for (int e = lane; e < ne; e += 64) {
    const TmEdge ca = a, cb = b;
    a = tm_load_edge(H, y, e + 64, ne);
    b = tm_load_edge(H, y, e + 96, ne);
    float2 u = tm_start(ca, d0), v = tm_start(cb, d0);
#pragma unroll
    for (int k = 0; k < kTmNodes; ++k) {
      ar[k] += u.x;
      ai[k] += u.y;
      ar[k] += v.x;
      ai[k] += v.y;
      const float tu = u.x * ca.w.x - u.y * ca.w.y;
      u.y = u.x * ca.w.y + u.y * ca.w.x;
      u.x = tu;
      const float tv = v.x * cb.w.x - v.y * cb.w.y;
      v.y = v.x * cb.w.y + v.y * cb.w.x;
      v.x = tv;
    }
  }
  tm_halve<16>(ar, ai, lane);
  tm_halve<8>(ar, ai, lane);
  tm_halve<4>(ar, ai, lane);
  tm_halve<2>(ar, ai, lane);
  tm_halve<1>(ar, ai, lane);
  return (j0 + lane < L.tm_n) ? tm_node_logw(L, ar[0], ai[0]) : -INFINITY;
}

// The warps of a CTA share the grid's 32-node chunks (chunk q to warp
// q mod n_warps).  Each lane keeps a running max and scaled sum of its
// nodes' exp(log weight); returns the warp's (max, sum), the same on every
// lane.  ell (optional) receives every node's log weight.
__device__ inline void tm_pass(const LikeConst& L, const HetTables& H, const float2* __restrict__ y, int warp,
                               int n_warps, int lane, float* ell, float& wm, float& ws) {
  float m = -INFINITY, s = 0.0f;
  const int nq = (L.tm_n + kTmNodes - 1) / kTmNodes;
  for (int q = warp; q < nq; q += n_warps) {
    const int j = q * kTmNodes + lane;
    const float l = tm_nodes_warp(L, H, y, q * kTmNodes, lane);
    if (j < L.tm_n) {
      if (ell) ell[j] = l;
      if (l > m) {
        s = s * __expf(m - l) + 1.0f;
        m = l;
      } else {
        s += __expf(l - m);
      }
    }
  }
  float M = m;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
  float S = (m > -INFINITY) ? s * __expf(m - M) : 0.0f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) S += __shfl_xor_sync(0xffffffffu, S, o);
  wm = M;
  ws = S;
}

// The gather's per-piece partial sums follow the grid and its twiddles.
__device__ __forceinline__ float2* tm_nufft_parts(const LikeConst& L, float2* g) { return g + 2 * L.tm_M; }

// Gather of the non-uniform FFT's grid values b_l = sum_e w_le c_e (the
// whole block).  A grid point's entries are consecutive edges, cut into
// pieces of at most kNufftPiece entries; lane t sums pieces t, t + nt, ...
// (all of a piece's weight loads issued together) into part[], then thread
// t combines the pieces of grid points t, t + nt, ... in order.  Fixed sum
// orders: deterministic.  Grid points without entries are zeroed.
__device__ inline void nufft_gather(const LikeConst& L, const HetTables& H, const float2* y, float2* g,
                                    float2* part, int lg) {
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int l = tid; l < L.tm_M; l += nt) g[l] = make_float2(0.0f, 0.0f);
  // the descriptors of this thread's first four pieces, loaded together
  constexpr int kPre = 4;
  int4 dp[kPre];
#pragma unroll
  for (int r = 0; r < kPre; ++r)
    dp[r] = tid + r * nt < L.tm_pieces ? __ldg(&H.nu_piece[tid + r * nt]) : make_int4(0, 0, 0, 0);
  for (int p = tid, r = 0; p < L.tm_pieces; p += nt, ++r) {
    int4 d = dp[0];
#pragma unroll
    for (int u = 1; u < kPre; ++u)
      if (r == u) d = dp[u];
    if (r >= kPre) d = __ldg(&H.nu_piece[p]);
    // entry i of 32 pieces in a row
    const float* wt = H.nu_wt + (size_t)(p >> 5) * kNufftPiece * 32 + (p & 31);
    float w[kNufftPiece];
#pragma unroll
    for (int i = 0; i < kNufftPiece; ++i) w[i] = i < d.y ? __ldg(wt + 32 * i) : 0.0f;
    float br = 0.0f, bi = 0.0f;
#pragma unroll
    for (int i = 0; i < kNufftPiece; ++i)
      if (i < d.y) {
        const float2 c = y[d.z + i];
        br = fmaf(w[i], c.x, br);
        bi = fmaf(w[i], c.y, bi);
      }
    part[p] = make_float2(br, bi);
  }
  __syncthreads();
  for (int q = tid; q < L.tm_points; q += nt) {
    const int4 d = __ldg(&H.nu_point[q]);
    float br = 0.0f, bi = 0.0f;
    for (int i = 0; i < d.z; ++i) {
      const float2 v = part[d.y + i];
      br += v.x;
      bi += v.y;
    }
    g[__brev((unsigned)d.x) >> (32 - lg)] = make_float2(br, bi);
  }
}

// The same time pass by non-uniform FFT (tables of het_nufft_tables): the
// edge products become c_e = y_e exp(-2 pi i f_e dt_ref) (double-float phase;
// y is overwritten), every grid point gathers its kernel-weighted c_e in a
// fixed order into bit-reversed position, a radix-2 FFT with exponent
// +2 pi i runs in shared memory, and node j takes Z_j = X[(j - j0) mod M] /
// Phi(j - j0).  Nodes are assigned to warps and lanes as in tm_pass, so the
// (max, sum) pairs and ell have the same layout.  Every thread of the CTA
// calls it (it synchronises the CTA).  Cost per evaluation ~W (N_b + 1)
// multiply-adds for the gather and (M/2) log2 M butterflies, against
// (N_b + 1) N_t terms for the direct sum.
__device__ inline void tm_pass_nufft(const LikeConst& L, const HetTables& H, const float2* y, float2* g,
                                     const float2* tw, int warp, int n_warps, int lane, float* ell, float& wm,
                                     float& ws) {
  const int tid = threadIdx.x, nt = blockDim.x;
  const int M = L.tm_M;
  // y holds c_e (the edge weights carry the reference rotation)
  const int lg = __ffs(M) - 1;
  nufft_gather(L, H, y, g, tm_nufft_parts(L, g), lg);
  __syncthreads();
  // radix-2 stages of spans 1..16 inside 32-point blocks in registers (warp
  // shuffles: no shared-memory bank conflicts, no block barriers), then the
  // wider spans through shared memory
  for (int blk = warp; blk < M / 32; blk += n_warps) {
    const int at = blk * 32 + lane;
    float2 x = g[at];
#pragma unroll
    for (int half = 1; half < 32; half <<= 1) {
      const float2 w = tw[half - 1 + (lane & (half - 1))];
      const float pr = __shfl_xor_sync(0xffffffffu, x.x, half), pi = __shfl_xor_sync(0xffffffffu, x.y, half);
      if ((lane & half) == 0)  // lower point: x + w partner
        x = make_float2(x.x + (w.x * pr - w.y * pi), x.y + (w.x * pi + w.y * pr));
      else  // upper point: partner - w x
        x = make_float2(pr - (w.x * x.x - w.y * x.y), pi - (w.x * x.y + w.y * x.x));
    }
    g[at] = x;
  }
  __syncthreads();
  for (int half = 32; half < M; half <<= 1) {
    for (int b = tid; b < M / 2; b += nt) {
      const int pos = b & (half - 1), i = ((b - pos) << 1) + pos, j = i + half;
      const float2 w = tw[half - 1 + pos];
      const float2 xj = g[j], xi = g[i];
      const float tr = w.x * xj.x - w.y * xj.y, ti = w.x * xj.y + w.y * xj.x;
      g[j] = make_float2(xi.x - tr, xi.y - ti);
      g[i] = make_float2(xi.x + tr, xi.y + ti);
    }
    __syncthreads();
  }
  float m = -INFINITY, s = 0.0f;
  const int nq = (L.tm_n + kTmNodes - 1) / kTmNodes;
  // four nodes per lane at a time, taken up in order
  constexpr int kAhead = 4;
  for (int q0 = warp; q0 < nq; q0 += kAhead * n_warps) {
    float l[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int j = (q0 + u * n_warps) * kTmNodes + lane;
      if (j < L.tm_n) {
        const int mi = j - L.tm_j0;
        const float2 z = g[mi < 0 ? mi + M : mi];
        const float cr = __ldg(H.nu_corr + j);
        l[u] = tm_node_logw(L, z.x * cr, z.y * cr);
      }
    }
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int j = (q0 + u * n_warps) * kTmNodes + lane;
      if (j < L.tm_n) {
        if (ell) ell[j] = l[u];
        if (l[u] > m) {
          s = s * __expf(m - l[u]) + 1.0f;
          m = l[u];
        } else {
          s += __expf(l[u] - m);
        }
      }
    }
  }
  float Mx = m;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) Mx = fmaxf(Mx, __shfl_xor_sync(0xffffffffu, Mx, o));
  float S = (m > -INFINITY) ? s * __expf(m - Mx) : 0.0f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) S += __shfl_xor_sync(0xffffffffu, S, o);
  wm = Mx;
  ws = S;
}

// The NUFFT grid's place in shared memory: after the N_b + 1 edge products;
// its M stage-major twiddles follow the grid (tm_nufft_tw).
__device__ __forceinline__ float2* tm_nufft_grid(unsigned char* smem, int n_bins) {
  return reinterpret_cast<float2*>(smem + ((((size_t)n_bins + 1) * 2 * sizeof(float) + 15) / 16 * 16));
}
__device__ __forceinline__ float2* tm_nufft_tw(unsigned char* smem, int n_bins, int M) {
  return tm_nufft_grid(smem, n_bins) + M;
}
// Copy of the twiddle table into shared memory (whole block).
__device__ __forceinline__ void tm_load_twiddles(const LikeConst& L, const HetTables& H, unsigned char* smem,
                                                 int n_bins) {
  float2* tw = tm_nufft_tw(smem, n_bins, L.tm_M);
  for (int k = threadIdx.x; k < L.tm_M; k += blockDim.x) tw[k] = __ldg(&H.nu_tw[k]);
}

// Time-marginalised logL of record r from the warps' (max, sum) pairs and
// detector sums D, both added in warp order: log((1/N_t) sum_j exp(l_j)) -
// <h|h>/2 - <d|d>/2.  By a warp: a warp's pair, a detector, a logarithm per lane
// (on one thread the FP64 chains took 39,000 cycles of an evaluation's 100,000).
template <int NDET>
__device__ inline double tm_finish(const LikeConst& L, const EvalRecord& r, const float (*hh)[NDET],
                                   const float (*wms)[2], int n_warps, int lane) {
  const unsigned full = 0xffffffffu;
  double d = 0.0, a = 0.0, iden = 0.0;
  if (lane < NDET) {
    for (int w = 0; w < n_warps; ++w) d += (double)hh[w][lane];
    a = (r.cre[lane] * r.cre[lane] + r.cim[lane] * r.cim[lane]) * (L.het_b0[lane] - d);
    iden = L.het_fid_iden[lane];
  }
  double HH = 0.0;
#pragma unroll
  for (int i = 0; i < NDET; ++i) HH += __shfl_sync(full, a, i) * __shfl_sync(full, iden, i);
  float M = -INFINITY;
  for (int w = 0; w < n_warps; ++w) M = fmaxf(M, wms[w][0]);
  const bool on = lane < n_warps && wms[lane][0] > -INFINITY;
  const double e = on ? exp((double)wms[lane][0] - (double)M) : 0.0, ws = on ? (double)wms[lane][1] : 0.0;
  const unsigned some = __ballot_sync(full, on);
  double S = 0.0;
  for (int w = 0; w < n_warps; ++w) {
    const double ew = __shfl_sync(full, e, w), sw = __shfl_sync(full, ws, w);
    if ((some >> w) & 1u) S += sw * ew;
  }
  const double lg = log(lane == 0 ? S : (double)L.tm_n);
  return (double)M + __shfl_sync(full, lg, 0) - __shfl_sync(full, lg, 1) - 0.5 * HH - 0.5 * L.DD;
}

}  // namespace swig
