// Folded full-grid sums (mixed precision), device side.
//
// kappa_i = sum_k D_i(k) exp(-2 pi i (P(f_k) + f_k tau_i)) over a few hundred
// thousand bins samples a smooth function far more finely than it varies: over
// a chunk of bins the phase, less the chunk's reference slope s, turns through
// a few cycles only.  The host cuts the grid into chunks over which every
// template of the prior box keeps below a fixed bandwidth (fold_plan in
// capi.cu).  On such a chunk the template equals its polynomial interpolant
// through 64 Chebyshev nodes to 1e-8, and the sum over the chunk's bins is,
// exactly for that interpolant, a sum over the nodes,
//   sum_k D'_i(k) E'(x_k) = sum_j W_ij E'(x_j),  W_ij = sum_k D'_i(k) l_j(x_k),
// with D'_i(k) = D_i(k) exp(-2 pi i s (f_k - f_c)), l_j the Lagrange basis and
// W formed once per event in FP64.  Where 64 bins hold more phase than that
// (the lowest frequencies) the nodes are the bins themselves.  The 128 s
// three-detector grid's 259,585 bins become about 80 chunks of 64 nodes.
//
// Bound: the FP32 issue slots, with the SFU beside them (two results per node and
// detector, 78 x 64 x 3 nodes instead of 778,755 bins).  Batched, against the direct
// sum over every bin (one GB300): 1000 vectors on the 128 s grid 31 us (668), 4099 on
// the 256 s grid 88 us (4.74 ms), one vector 30 us with the host's part (90); the
// error against FP64 is that of the direct sum (kFoldBlock).
//
// An evaluation checks its own bandwidth and Taylor remainder on every chunk
// against the bound the weights were made for; a parameter vector outside
// (one far from the prior box) is summed bin by bin instead: in a batch by all
// its CTAs (fold.cu fold_strays), in the sampler by the chain's (fold_direct).
#pragma once

#include "packed.cuh"
#include "sweep.cuh"

namespace swig {

constexpr int kFoldWarps = 16;     // warps of an evaluating CTA
constexpr int kFoldAnchor = kFoldAnchorFloats;

// What an evaluation reads of its record: coefficients and time shifts in
// double-float.
struct FoldIn {
  float c_hi[NBASIS], c_lo[NBASIS];
  float tau_hi[SWIG_MAX_DET], tau_lo[SWIG_MAX_DET];
};
static_assert(offsetof(EvalRecord, c_lo) == offsetof(EvalRecord, c_hi) + sizeof(float) * NBASIS &&
                  offsetof(EvalRecord, tau_lo) == offsetof(EvalRecord, tau_hi) + sizeof(float) * SWIG_MAX_DET,
              "FoldIn is two runs of EvalRecord's words");

// Word w (0 .. 29) of FoldIn from a record.
__device__ __forceinline__ float fold_in_word(const EvalRecord& r, int w) {
  return w < 2 * NBASIS ? reinterpret_cast<const float*>(&r.c_hi)[w]
                        : reinterpret_cast<const float*>(&r.tau_hi)[w - 2 * NBASIS];
}

// An anchor's sixteen values lie in four 16-byte blocks whose order turns with
// the chunk, so that the lanes' stores (a chunk each, 64 bytes apart) meet 8
// banks instead of 2.
__device__ __forceinline__ int fold_block(int q, int b) { return 4 * (b ^ ((q >> 1) & 3)); }
__device__ __forceinline__ int fold_at(int q, int m) { return fold_block(q, m >> 2) + (m & 3); }

// One quarter (sub 0 .. 3) of the anchor of chunk q for the evaluation `r` (a
// FoldIn or an EvalRecord), written to out[kFoldAnchor], value m at fold_at(sw, m)
// (sw: the chunk's place in its panel):
//   sub 0: out[i] = frac(P(f_c) + f_c tau_i), double-float sums;
//   sub 1: out[4], out[5] = the scaled slope h (P'(f_c) + tau_0 - s) as a
//          double-float, out[5 + i] = h (tau_i - tau_0), i = 1 .. 3;
//   sub 2: out[9], out[11], out[13], out[15]: even Taylor terms a_2 .. a_8;
//   sub 3: out[10], out[12], out[14]: a_3, a_5, a_7, and the order-9 remainder
//          bound against kFoldTaylorEps.
// Returns false when the remainder is too large.  The serial part of an
// anchor is the eleven-term double-float sums; four lanes of different warps
// share it (a lane per chunk took 2.2x as long alone).
template <int NDET, typename Rec>
__device__ __forceinline__ bool fold_anchor(const float* __restrict__ tab, int ld, const Rec& r, int sub, int q,
                                            int sw, float* out) {
  const float* T = tab + q;
  auto row = [&](int k) { return T[k * ld]; };
  if (sub == 0) {
    dfl A = {0.0f, 0.0f};
#pragma unroll
    for (int j = 0; j < NBASIS; ++j)
      A = df_add(A, df_mul(dfl{r.c_hi[j], r.c_lo[j]}, dfl{row(FR_VAL_HI + j), row(FR_VAL_LO + j)}));
    const dfl fc = {row(FR_FC_HI), row(FR_FC_LO)};
#pragma unroll
    for (int i = 0; i < NDET; ++i) out[fold_at(sw, i)] = df_frac(df_add(A, df_mul(fc, dfl{r.tau_hi[i], r.tau_lo[i]})));
  } else if (sub == 1) {
    const dfl h = {row(FR_H_HI), row(FR_H_LO)};
    dfl S = df_add(df_mul(h, dfl{r.tau_hi[0], r.tau_lo[0]}), dfl{-row(FR_SM_HI), -row(FR_SM_LO)});
#pragma unroll
    for (int j = 0; j < kFoldSlopes; ++j)
      S = df_add(S, df_mul(dfl{r.c_hi[j], r.c_lo[j]}, dfl{row(FR_D1_HI + j), row(FR_D1_LO + j)}));
    out[fold_at(sw, 4)] = S.hi;
    out[fold_at(sw, 5)] = S.lo;
#pragma unroll
    for (int i = 1; i < NDET; ++i)
      out[fold_at(sw, 5 + i)] = h.hi * ((r.tau_hi[i] - r.tau_hi[0]) + (r.tau_lo[i] - r.tau_lo[0]));
  } else {
    const int n0 = sub == 2 ? 2 : 3, nn = sub == 2 ? 4 : 3;
    float a[4] = {0.0f, 0.0f, 0.0f, 0.0f}, R = 0.0f;
#pragma unroll
    for (int j = 0; j < kFoldSlopes; ++j) {
      const float c = r.c_hi[j];
#pragma unroll
      for (int m = 0; m < 4; ++m)
        if (m < nn) a[m] = fmaf(c, row(FR_POLY + (n0 + 2 * m - 2) * kFoldSlopes + j), a[m]);
      if (sub == 3) R = fmaf(fabsf(c), row(FR_BND + j), R);
    }
#pragma unroll
    for (int m = 0; m < 4; ++m)
      if (m < nn) out[fold_at(sw, 7 + n0 + 2 * m)] = a[m];
    return R <= kFoldTaylorEps;  // false for a NaN as well
  }
  return true;
}

// Two evaluations' inputs interleaved: (hi a, hi b, lo a, lo b) per coefficient
// and time shift.
struct FoldPair {
  float4 c[NBASIS], tau[SWIG_MAX_DET];
};
// Word j (0 .. 14) of a pair's inputs from their records (16 threads).
__device__ __forceinline__ void fold_pair_set(FoldPair& in, int j, const EvalRecord& a, const EvalRecord& b) {
  if (j < NBASIS)
    in.c[j] = make_float4(a.c_hi[j], b.c_hi[j], a.c_lo[j], b.c_lo[j]);
  else if (j < NBASIS + SWIG_MAX_DET)
    in.tau[j - NBASIS] = make_float4(a.tau_hi[j - NBASIS], b.tau_hi[j - NBASIS], a.tau_lo[j - NBASIS], b.tau_lo[j - NBASIS]);
}
__device__ __forceinline__ DflN<2> fold_dfl2(const float4& v) { return {f2_make(v.x, v.y), f2_make(v.z, v.w)}; }
// The basis functions of the spin terms come last in every sum, so that the
// sums over the others can be kept while only spins, sky or t_c move.
__device__ constexpr int kFoldRest[NBASIS - 2] = {B_M53, B_M1, B_LOG, B_P13, B_P13LOG, B_P23, B_P53, B_P73, B_ONE};
__device__ constexpr int kFoldSpin[2] = {B_M23, B_M13};

// One quarter of the anchors of chunk q for two evaluations (fold_anchor on
// packed pairs), to oa and ob.  base: the sums over kFoldRest of a point with
// the same masses and tides (rows: value hi, lo, slope hi, lo, a_2 .. a_8), or
// null.  Returns the evaluations (bits) whose Taylor remainder is too large.
template <int NDET>
__device__ __forceinline__ int fold_anchor_pair(const float* __restrict__ tab, int ld, const FoldPair& in,
                                                const float* __restrict__ base, int sub, int q, int sw, float* oa,
                                                float* ob) {
  using O = PkOps<2>;
  const float* T = tab + q;
  auto row = [&](int k) { return O::all(T[k * ld]); };
  auto put = [&](int m, f2 v) { f2_split(v, oa[fold_at(sw, m)], ob[fold_at(sw, m)]); };
  auto pre = [&](int k) { return O::all(base[k * ld + q]); };
  if (sub == 0) {
    DflN<2> A = {O::all(0.0f), O::all(0.0f)};
    auto add = [&](int j) {
      A = dfn_add<2>(A, dfn_mul<2>(fold_dfl2(in.c[j]), DflN<2>{row(FR_VAL_HI + j), row(FR_VAL_LO + j)}));
    };
    if (base) {
      A = {pre(0), pre(1)};
    } else {
#pragma unroll
      for (int r = 0; r < NBASIS - 2; ++r) add(kFoldRest[r]);
    }
    add(kFoldSpin[0]);
    add(kFoldSpin[1]);
    const DflN<2> fc = {row(FR_FC_HI), row(FR_FC_LO)};
#pragma unroll
    for (int i = 0; i < NDET; ++i) put(i, dfn_frac<2>(dfn_add<2>(A, dfn_mul<2>(fc, fold_dfl2(in.tau[i])))));
  } else if (sub == 1) {
    DflN<2> S = {O::all(0.0f), O::all(0.0f)};
    auto add = [&](int j) {
      S = dfn_add<2>(S, dfn_mul<2>(fold_dfl2(in.c[j]), DflN<2>{row(FR_D1_HI + j), row(FR_D1_LO + j)}));
    };
    if (base) {
      S = {pre(2), pre(3)};
    } else {
#pragma unroll
      for (int r = 0; r < NBASIS - 3; ++r) add(kFoldRest[r]);  // (the constant has no slope)
    }
    add(kFoldSpin[0]);
    add(kFoldSpin[1]);
    const DflN<2> h = {row(FR_H_HI), row(FR_H_LO)};
    S = dfn_add<2>(S, dfn_add<2>(dfn_mul<2>(h, fold_dfl2(in.tau[0])), DflN<2>{O::all(-T[FR_SM_HI * ld]), O::all(-T[FR_SM_LO * ld])}));
    put(4, S.hi);
    put(5, S.lo);
    const DflN<2> t0 = fold_dfl2(in.tau[0]);
#pragma unroll
    for (int i = 1; i < NDET; ++i) {
      const DflN<2> ti = fold_dfl2(in.tau[i]);
      put(5 + i, O::mul(h.hi, O::add(pk_sub<2>(ti.hi, t0.hi), pk_sub<2>(ti.lo, t0.lo))));
    }
  } else {
    const int n0 = sub == 2 ? 2 : 3, nn = sub == 2 ? 4 : 3;
    f2 a[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) a[m] = base && m < nn ? pre(2 + n0 + 2 * m) : O::all(0.0f);
    auto add = [&](int j) {
      const f2 c = f2_make(in.c[j].x, in.c[j].y);
#pragma unroll
      for (int m = 0; m < 4; ++m)
        if (m < nn) a[m] = O::fma(c, row(FR_POLY + (n0 + 2 * m - 2) * kFoldSlopes + j), a[m]);
    };
    if (!base) {
#pragma unroll
      for (int r = 0; r < NBASIS - 3; ++r) add(kFoldRest[r]);
    }
    add(kFoldSpin[0]);
    add(kFoldSpin[1]);
#pragma unroll
    for (int m = 0; m < 4; ++m)
      if (m < nn) put(7 + n0 + 2 * m, a[m]);
    if (sub == 3) {
      float ra = 0.0f, rb = 0.0f;
#pragma unroll
      for (int j = 0; j < kFoldSlopes; ++j) {
        const float b = T[(FR_BND + j) * ld];
        ra = fmaf(fabsf(in.c[j].x), b, ra);
        rb = fmaf(fabsf(in.c[j].y), b, rb);
      }
      return (ra <= kFoldTaylorEps ? 0 : 1) | (rb <= kFoldTaylorEps ? 0 : 2);
    }
  }
  return 0;
}

// The same quarter's sums over kFoldRest of one point (both halves of `in`) into
// base (kFoldBaseRows rows of ldb).
__device__ __forceinline__ void fold_base(const float* __restrict__ tab, int ld, const FoldPair& in, int sub, int q,
                                          float* base, int ldb) {
  const float* T = tab + q;
  auto put = [&](int k, float v) { base[k * ldb + q] = v; };
  if (sub < 2) {
    DflN<1> A = {0.0f, 0.0f};
    const int n = sub == 0 ? NBASIS - 2 : NBASIS - 3;
    for (int r = 0; r < n; ++r) {
      const int j = kFoldRest[r];
      const int hi = sub == 0 ? FR_VAL_HI + j : FR_D1_HI + j, lo = sub == 0 ? FR_VAL_LO + j : FR_D1_LO + j;
      A = dfn_add<1>(A, dfn_mul<1>(DflN<1>{in.c[j].x, in.c[j].z}, DflN<1>{T[hi * ld], T[lo * ld]}));
    }
    put(2 * sub, A.hi);
    put(2 * sub + 1, A.lo);
  } else {
    const int n0 = sub == 2 ? 2 : 3, nn = sub == 2 ? 4 : 3;
    float a[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (int r = 0; r < NBASIS - 3; ++r) {
      const int j = kFoldRest[r];
#pragma unroll
      for (int m = 0; m < 4; ++m)
        if (m < nn) a[m] = fmaf(in.c[j].x, T[(FR_POLY + (n0 + 2 * m - 2) * kFoldSlopes + j) * ld], a[m]);
    }
#pragma unroll
    for (int m = 0; m < 4; ++m)
      if (m < nn) put(2 + n0 + 2 * m, a[m]);
  }
}

// Whether the finished anchor of chunk q keeps below the chunk's bandwidth
// (kernels.h FR_LIM): |slope| + sum_n n a^(n-1) |a_n| in cycles, a the half
// axis of the Bernstein ellipse of the interpolation bound.
template <int NDET>
__device__ __forceinline__ bool fold_in_band(const float* __restrict__ tab, int ld, const float* an, int sw, int q) {
  float b = 0.0f;
#pragma unroll
  for (int i = 1; i < NDET; ++i) b = fmaxf(b, fabsf(an[fold_at(sw, 5 + i)]));
  float om = fabsf(an[fold_at(sw, 4)]) + b, g = 1.0f;
#pragma unroll
  for (int n = 2; n <= kFoldDeg; ++n) {
    g *= kFoldEllipse;
    om = fmaf((float)n * g, fabsf(an[fold_at(sw, 7 + n)]), om);
  }
  return om <= tab[FR_LIM * ld + q];  // false for a NaN as well
}

// Accumulators of a lane: per detector the real and imaginary sums, for the
// nodes +x and -x in the two halves of a pair.
template <int NDET>
struct FoldAcc {
  f2 re[NDET], im[NDET];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < NDET; ++i) re[i] = im[i] = 0ull;
  }
  __device__ __forceinline__ void total(int i, float& r, float& m) const {
    float a, b, c, d;
    f2_split(re[i], a, b);
    f2_split(im[i], c, d);
    r = a + b;
    m = c + d;
  }
};

// The rounding of the sums.  A lane adds its nodes in FP32 over a block of chunks;
// across blocks, lanes and warps the sums are double-float.  Error against FP64 of
// 2500 vectors on the 64 s grid, a warp each (root mean square, largest): sums over
// slices of the bins, added in FP64, 2.98e-5, 7.1e-5; one FP32 sum over all chunks
// and lanes 3.26e-5, 10.0e-5; blocks of 32 chunks 2.99e-5, 7.9e-5, of 8 chunks
// 2.95e-5, 7.3e-5 (4099 vectors on the 256 s grid 88.2 -> 90.7 us for it).
constexpr int kFoldBlock = 8;

// A lane's sums over blocks as high words, the FP32 accumulators being their low
// ones: after a block what the accumulators hold moves up and its rounding stays
// behind (Dekker's fast two-sum).
template <int NDET>
struct FoldSum {
  FoldAcc<NDET> hi;
  __device__ __forceinline__ void take(FoldAcc<NDET>& acc) {
    auto up = [](f2& h, f2& a) {
      const f2 s = f2_add(h, a);
      a = pk_sub<2>(a, pk_sub<2>(s, h));
      h = s;
    };
#pragma unroll
    for (int i = 0; i < NDET; ++i) {
      up(hi.re[i], acc.re[i]);
      up(hi.im[i], acc.im[i]);
    }
  }
};

// Warp sums of R evaluations from their lanes' accumulators (acc[e], and where there
// were several blocks the high words hi[e]), value j = 2 (NDET e + i) + part to put(j,
// sum), once each.  The upper lanes of a pair take over half of the values at each
// level (see warp_sums); the sums are double-float from level PLAIN on (the levels
// below it add small parts of a warp's sum).
template <int NDET, int R, int PLAIN, typename Put>
__device__ __forceinline__ void fold_warp_sums(const FoldAcc<NDET>* acc, bool blocks, const FoldAcc<NDET>* hi,
                                               int lane, const Put& put) {
  constexpr int n = 2 * NDET * R, V = n <= 2 ? 2 : n <= 4 ? 4 : n <= 8 ? 8 : 16;
  const auto pair_sum = [](const FoldAcc<NDET>& a, int j) {
    float x, y;
    f2_split(j & 1 ? a.im[j / 2] : a.re[j / 2], x, y);
    return x + y;
  };
  dfl a[V];
#pragma unroll
  for (int j = 0; j < V; ++j) a[j] = {j < n ? pair_sum(acc[j / (2 * NDET)], j % (2 * NDET)) : 0.0f, 0.0f};
  if (blocks)  // warp-uniform
#pragma unroll
    for (int j = 0; j < n; ++j) a[j].hi += pair_sum(hi[j / (2 * NDET)], j % (2 * NDET));
  int which = 0, o = 16;
  const auto across = [&](dfl v, int level) {
    return dfl{__shfl_xor_sync(0xffffffffu, v.hi, o),
               level > PLAIN ? __shfl_xor_sync(0xffffffffu, v.lo, o) : 0.0f};
  };
  const auto sum = [](dfl a, dfl b, int level) {
    return level < PLAIN ? dfl{a.hi + b.hi, 0.0f} : level == PLAIN ? two_sum(a.hi, b.hi) : df_accumulate(a, b);
  };
  int level = 0;
#pragma unroll
  for (int h = V / 2; h >= 1; h >>= 1, o >>= 1, ++level) {
    const bool up = (lane & o) != 0;
    which += up ? h : 0;
#pragma unroll
    for (int k = 0; k < h; ++k) {
      const dfl send = up ? a[k] : a[k + h], keep = up ? a[k + h] : a[k];
      a[k] = sum(keep, across(send, level), level);
    }
  }
#pragma unroll
  for (; o > 0; o >>= 1, ++level) a[0] = sum(a[0], across(a[0], level), level);
  if ((lane & (32 / V - 1)) == 0 && which < n) put(which, a[0]);
}

// The lane's node weights and abscissa of a chunk.
template <int NDET>
struct FoldNode {
  float4 w[NDET];
  float2 x;
};
// w: the chunk's weights at this lane; kind: its node kind, x0 the lane's
// Chebyshev abscissa and x the table of all kinds.
template <int NDET>
__device__ __forceinline__ void fold_load(const float4* __restrict__ w, int kind, float2 x0,
                                          const float2* __restrict__ x, int lane, FoldNode<NDET>& v) {
#pragma unroll
  for (int i = 0; i < NDET; ++i) v.w[i] = w[32 * i];
  v.x = x0;
  if (kind) v.x = x[32 * kind + lane];  // warp-uniform
}

// One chunk of one evaluation by one warp, two nodes (+x, -x) per lane.  The
// phase is E(x) + O(x), even and odd Taylor parts: at the two nodes E + O and
// E - O, so the polynomial is formed once for both; the slope's product with x
// is carried in double-float and reduced to its fractional part.
template <int NDET>
__device__ __forceinline__ void fold_chunk(const float* __restrict__ an, int sw, const FoldNode<NDET>& v,
                                           FoldAcc<NDET>& acc) {
  const float2 xv = v.x;
  const float4 A = *reinterpret_cast<const float4*>(an + fold_block(sw, 0));
  const float4 B = *reinterpret_cast<const float4*>(an + fold_block(sw, 1));
  const float4 C = *reinterpret_cast<const float4*>(an + fold_block(sw, 2));
  const float4 D = *reinterpret_cast<const float4*>(an + fold_block(sw, 3));
  const float x = xv.x, x2 = x * x;
  // C = (b_3, a_2, a_3, a_4), D = (a_5, a_6, a_7, a_8)
  const float ev = x2 * fmaf(x2, fmaf(x2, fmaf(x2, D.w, D.y), C.w), C.y);
  const float oh = x2 * x * fmaf(x2, fmaf(x2, D.z, D.x), C.z);
  const float p = x * B.x;
  float e = fmaf(x, B.x, -p);
  e = fmaf(xv.y, B.x, e);
  e = fmaf(x, B.y, e);
  const float od = (p - round_nearest(p)) + (e + oh);
  const float b[4] = {0.0f, B.z, B.w, C.x}, a0[4] = {A.x, A.y, A.z, A.w};
  const f2 magic = f2_make(12582912.0f, 12582912.0f), nmagic = f2_make(-12582912.0f, -12582912.0f);
  const f2 none = f2_make(-1.0f, -1.0f), twopi = f2_make(6.283185307179586f, 6.283185307179586f);
#pragma unroll
  for (int i = 0; i < NDET; ++i) {
    const float ei = ev + a0[i], oi = i ? fmaf(b[i], x, od) : od;
    f2 ph = f2_make(ei + oi, ei - oi);
    const f2 n = f2_add(f2_add(ph, magic), nmagic);  // nearest integers (see round_nearest)
    ph = f2_mul(f2_fma(n, none, ph), twopi);
    float pa, pb, sa, ca, sb, cb;
    f2_split(ph, pa, pb);
    __sincosf(pa, &sa, &ca);
    __sincosf(pb, &sb, &cb);
    const f2 c2 = f2_make(ca, cb), s2 = f2_make(sa, sb);
    const f2 wr = f2_make(v.w[i].x, v.w[i].y), wi = f2_make(v.w[i].z, v.w[i].w);
    acc.re[i] = f2_fma(wr, c2, f2_fma(wi, s2, acc.re[i]));
    acc.im[i] = f2_fma(wi, c2, f2_fma(f2_mul(wr, none), s2, acc.im[i]));
  }
}

// Bin by bin (rare, the sampler): tiles first, first + stride, ... of the grid by one warp
// from global memory, with the tile anchors of the direct sum (sweep.cuh);
// row: kAnchorStride floats of the warp's own in shared memory.  Lane sums in
// FP64 across tiles; every lane returns the warp's totals.
template <int NDET>
__device__ __noinline__ void fold_direct(const LikeConst& L, const FoldTables& F, const EvalRecord& r, int first,
                                         int stride, int lane, float* row, double* out) {
#pragma unroll
  for (int j = 0; j < 2 * NDET; ++j) out[j] = 0.0;
  for (int t = first; t < L.n_tiles; t += stride) {
    __syncwarp();
    if (lane == 0) compute_anchor(NDET, F.tiles[t], F.basis[t], r, row);
    __syncwarp();
    float v[2 * NDET];
    const int lo = F.tiles[t].k0, hi = lo + F.tiles[t].nbins;
    sweep_warp_mixed<NDET>(L, F.data, L.n_bins, F.bin_tile, 0, lo, hi, F.tiles + t, row, t, r, lane, v);
#pragma unroll
    for (int j = 0; j < 2 * NDET; ++j) out[j] += (double)v[j];
  }
}

// Asynchronous 16-byte copy, global to shared memory.
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// Distance-marginalised logL (distance_marg_logl) by a whole warp: the 64
// nodes on 32 lanes, each exponent formed once.
__device__ inline double distance_marg_logl_warp(const LikeConst& L, double zre, double zim, double H, int lane) {
  const double X = L.phase_marg ? sqrt(zre * zre + zim * zim) : zre;
  double a, b;
  distance_window(L, X, H, &a, &b);
  const double mid = 0.5 * (a + b), half = 0.5 * (b - a);
  static_assert(kGaussLegendre == 64, "two nodes per lane");
  const double e0 = distance_exponent(L, zre, X, H, mid + half * L.gl_x[lane]);
  const double e1 = distance_exponent(L, zre, X, H, mid + half * L.gl_x[lane + 32]);
  double M = fmax(fmax(-INFINITY, e0), e1);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) M = fmax(M, __shfl_xor_sync(0xffffffffu, M, o));
  double sum = L.gl_w[lane] * (double)expf((float)(e0 - M)) + L.gl_w[lane + 32] * (double)expf((float)(e1 - M));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  return M + log(half * sum) - 0.5 * L.DD;
}

// logL of record r by a whole warp from kappa (component j on lane j < 2
// NDET, data-scaled): detector i's terms of Z on lane i, added in detector
// order, then loglike_epilogue's closed forms.  Every lane returns it.
template <int NDET>
__device__ __forceinline__ double loglike_epilogue_warp(const LikeConst& L, const EvalRecord& r, double kapc,
                                                        int lane) {
  const int di = lane < NDET ? lane : 0;
  const double kre = __shfl_sync(0xffffffffu, kapc, 2 * di), kim = __shfl_sync(0xffffffffu, kapc, 2 * di + 1);
  double tr = 0.0, ti = 0.0;
  if (lane < NDET) {
    const double a = kre * L.inv_scale[di], b = kim * L.inv_scale[di];
    tr = r.cre[di] * a - r.cim[di] * b;
    ti = r.cre[di] * b + r.cim[di] * a;
  }
  double zr = __shfl_sync(0xffffffffu, tr, 0), zi = __shfl_sync(0xffffffffu, ti, 0);
#pragma unroll
  for (int i = 1; i < NDET; ++i) {
    zr += __shfl_sync(0xffffffffu, tr, i);
    zi += __shfl_sync(0xffffffffu, ti, i);
  }
  if (!r.valid) return -INFINITY;  // warp-uniform
  if (L.dist_marg) return distance_marg_logl_warp(L, zr, zi, r.hh, lane);
  const double base = -0.5 * r.hh - 0.5 * L.DD;
  if (!L.phase_marg) return zr + base;
  const double x = sqrt(zr * zr + zi * zi);
  return (L.fast_epilogue ? x + (double)log_i0e_f32((float)x) : log_bessel_i0(x)) + base;
}

}  // namespace swig
