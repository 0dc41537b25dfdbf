// Batched matched-filter log-likelihood kernels (Eq. 2 of the paper) on the
// full frequency grid, in two precisions:
//
//  * MIXED: FP32 phases and sums over the folded grid (fold.cuh); here only
//    the set-up of its records.
//  * FP64: every per-bin quantity in FP64 with sincospi, as the reference
//    precision of the small single-detector configuration: one warp per (theta,
//    slice of the grid), one partial sum each, added per theta in a fixed order.
//
// The heterodyned likelihood, post-hoc draws, waveforms and the prior transform
// follow.
#include <cuda_runtime.h>

#include <mutex>
#include <utility>
#include <vector>

#include "kernels.h"
#include "het.cuh"
#include "sweep.cuh"

namespace swig {

// Set-up records (FP64), 32 parameter vectors per block, one per lane, one
// piece of the record per warp: a warp's FP64 instruction takes 64 cycles of
// its scheduler however many lanes it serves, so a record's pieces run side by
// side on schedulers and the vectors ride along in the lanes.  The pieces that
// follow from the masses, spins and tides and those of the projections and
// delays share nothing, so they go to two blocks (blockIdx.y).
// What bounds it are the chains: logarithm, exponential and divisions of the
// mass terms and then a share of the coefficients; or the amplitude and the
// angles' sines, two to a scheduler, and then a detector each.  100
// vectors, evaluated: 19.6 us with all pieces on one SM, 16.4 now.
constexpr int kSetupWarps = 8;

__global__ void __launch_bounds__(32 * kSetupWarps)
    k_setup(LikeConst L, const double* __restrict__ theta, int n, EvalRecord* __restrict__ rec, FoldStrays strays) {
  __shared__ double s_th[SWIG_N_PARAMS][33];
  __shared__ double s_m[8][32];      // MassTerms, in EvalRecord::mterm's order
  __shared__ double s_sc[8][32];     // sines and cosines of RA - GMST, Dec, 2 psi, phi_c
  __shared__ double s_ci[32], s_amp[32], s_hh[SWIG_MAX_DET][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i0 = blockIdx.x * 32, i = i0 + lane;
  // a dependent kernel may start; it waits for this grid's end before it
  // reads a record (griddepcontrol.wait)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (strays.ctl && blockIdx.y == 0 && warp == kSetupWarps - 1) {
    if (i < n) strays.done[i] = 0;
    if (blockIdx.x == 0 && lane < 4) strays.ctl[lane] = 0;
  }
  for (int e = threadIdx.x; e < 32 * SWIG_N_PARAMS; e += blockDim.x) {
    const int v = e / SWIG_N_PARAMS, j = e - v * SWIG_N_PARAMS;
    double x = i0 + v < n ? theta[(size_t)i0 * SWIG_N_PARAMS + e] : 1.0;
    if (j == 6 && L.dist_marg) x = 1.0;      // the marginal is built from the template at 1 Mpc
    if (j == 11 && L.tm_n > 0) x = L.tm_tref;  // templates at the fiducial's t_c, shifted node by node
    s_th[j][v] = x;
  }
  __syncthreads();
  double th[SWIG_N_PARAMS];
#pragma unroll
  for (int j = 0; j < SWIG_N_PARAMS; ++j) th[j] = s_th[j][lane];
  const bool valid = theta_valid_bits(th);
  EvalRecord* r = rec + i;
  if (blockIdx.y == 0) {
    if (valid && warp == 0) {
      MassTerms t;
      taylorf2_scale_terms(th[0], th[1], t);
      s_m[4][lane] = t.A, s_m[5][lane] = t.r, s_m[6][lane] = t.ir, s_m[7][lane] = t.lpm;
    } else if (valid && warp == 1) {
      MassTerms t;
      taylorf2_ratio_terms(th[1], t);
      s_m[0][lane] = t.eta, s_m[1][lane] = t.dm, s_m[2][lane] = t.m1, s_m[3][lane] = t.m2;
    }
    __syncthreads();
    if (warp >= 4 || i >= n) return;
    // a share of the phase coefficients
    double c[NBASIS];
#pragma unroll
    for (int j = 0; j < NBASIS; ++j) c[j] = 0.0;
    MassTerms t;
    t.eta = s_m[0][lane], t.dm = s_m[1][lane], t.m1 = s_m[2][lane], t.m2 = s_m[3][lane];
    t.A = s_m[4][lane], t.r = s_m[5][lane], t.ir = s_m[6][lane], t.lpm = s_m[7][lane];
    auto put = [&](int j) {
      const double v = valid ? c[j] : 0.0;
      const dfl d = df_from_double(v);
      r->c[j] = v;
      r->c_hi[j] = d.hi;
      r->c_lo[j] = d.lo;
    };
    if (warp == 0) {
      taylorf2_low_coeffs(t, c);
      put(B_M53), put(B_M1), put(B_LOG), put(B_ONE);
    } else if (warp == 1) {
      taylorf2_high_coeffs(t, c);
      put(B_P13), put(B_P13LOG), put(B_P23);
    } else if (warp == 2) {
      taylorf2_spin_coeffs(t, th[2], th[3], c);
      put(B_M23), put(B_M13);
    } else {
      taylorf2_tidal_coeffs(t, th[4], th[5], c);
      put(B_P53), put(B_P73);
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (valid) r->mterm[k] = s_m[k][lane];
    }
    return;
  }
  switch (warp) {  // (warps w and w + 4 share a scheduler)
    case 0: s_amp[lane] = valid ? amplitude_per_mpc(th[0]) / th[6] : 0.0; break;
    case 1: sincos(th[9] - L.gmst, &s_sc[0][lane], &s_sc[1][lane]); break;
    case 2: sincos(th[10], &s_sc[2][lane], &s_sc[3][lane]); break;
    case 3: sincos(2.0 * th[8], &s_sc[4][lane], &s_sc[5][lane]); break;
    case 5: s_ci[lane] = cos(th[7]); break;
    case 6:
      if (L.phase_marg)
        s_sc[6][lane] = 0.0, s_sc[7][lane] = 1.0;
      else
        sincos(th[12], &s_sc[6][lane], &s_sc[7][lane]);
      break;
    default: break;
  }
  __syncthreads();
  if (warp < SWIG_MAX_DET) {  // projection and time shift of one detector
    const int d = warp;
    double pre = 0.0, pim = 0.0, term = 0.0, cre = 0.0, cim = 0.0;
    if (d < L.n_det) {
      const double amp = s_amp[lane];
      const double sl = s_sc[0][lane], cl = s_sc[1][lane], sd = s_sc[2][lane], cd = s_sc[3][lane];
      double fp, fx;
      antenna_from_sc(L.dten[d], sl, cl, sd, cd, s_sc[4][lane], s_sc[5][lane], &fp, &fx);
      const double ci = s_ci[lane], sph = s_sc[6][lane], cph = s_sc[7][lane];
      const double re0 = fp * (0.5 * (1.0 + ci * ci)), im0 = -fx * ci;
      pre = re0 * cph - im0 * sph;
      pim = re0 * sph + im0 * cph;
      cre = amp * pre, cim = amp * pim;
      term = (cre * cre + cim * cim) * L.K[d];
    }
    s_hh[d][lane] = term;
    if (i < n) {
      r->pre[d] = pre;
      r->pim[d] = pim;
      r->cre[d] = cre;
      r->cim[d] = cim;
    }
  } else {
    const int d = warp - SWIG_MAX_DET;
    double gd = 0.0, tau = 0.0;
    if (d < L.n_det) {
      const double sl = s_sc[0][lane], cl = s_sc[1][lane], sd = s_sc[2][lane], cd = s_sc[3][lane];
      gd = -(cd * (cl * L.vertex[d][0] + sl * L.vertex[d][1]) + sd * L.vertex[d][2]) * (1.0 / kCSI);
      tau = th[11] + gd;
    }
    if (i < n) {
      const dfl tv = df_from_double(tau);
      r->gdel[d] = gd;
      r->tau[d] = tau;
      r->tau_hi[d] = tv.hi;
      r->tau_lo[d] = tv.lo;
    }
  }
  __syncthreads();
  if (warp == 0 && i < n) {
    double hh = 0.0;
#pragma unroll
    for (int d = 0; d < SWIG_MAX_DET; ++d) hh += s_hh[d][lane];
    r->hh = hh;
    r->amp = s_amp[lane];
    r->valid = valid ? 1 : 0;
  }
}

cudaError_t allow_shared(const void* f) {
  static std::mutex lock;
  static std::vector<std::pair<const void*, int>> limits;  // (one architecture: the same on every device)
  int most = -1;
  {
    const std::lock_guard<std::mutex> hold(lock);
    for (const auto& l : limits)
      if (l.first == f) most = l.second;
  }
  if (most < 0) {
    int device = 0, optin = 0;
    cudaFuncAttributes a;
    cudaError_t e = cudaGetDevice(&device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, f);
    if (e != cudaSuccess) return e;
    most = optin - (int)a.sharedSizeBytes;
    const std::lock_guard<std::mutex> hold(lock);
    limits.emplace_back(f, most);
  }
  return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}

// A kernel whose start overlaps the one before it on st (it waits for that one's
// end before it reads its results).
template <typename... P, typename... A>
cudaError_t launch_after(void (*kern)(P...), dim3 grid, int threads, size_t bytes, cudaStream_t st, A... args) {
  const cudaError_t e = bytes ? allow_shared((const void*)kern) : cudaSuccess;
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = st;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

// k_setup of n vectors.
static void launch_setup(const LikeConst& L, const double* theta, int n, EvalRecord* rec, cudaStream_t st,
                         const FoldStrays& strays = {}) {
  k_setup<<<dim3((n + 31) / 32, 2), 32 * kSetupWarps, 0, st>>>(L, theta, n, rec, strays);
}

template <int NDET>
__global__ void __launch_bounds__(256)
    k_sweep_fp64(LikeConst L, const double2* __restrict__ data, const double* __restrict__ ftab,
                 const int* __restrict__ slice_begin, const EvalRecord* __restrict__ rec, int n,
                 double* __restrict__ partials) {
  const int slice = blockIdx.x;
  const int b0 = slice_begin[slice], b1 = slice_begin[slice + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  for (int th = blockIdx.y * 8 + warp; th < n; th += gridDim.y * 8) {
    sweep_warp_fp64<NDET>(L, data, ftab, b0, b1, rec[th], lane,
                          partials + ((size_t)th * L.n_slices + slice) * kPartialStride);
  }
}

// The basis functions at every bin (rows of n values; f in row B_ONE) from
// f^-1/3, f^1/3 and ln f.
__global__ void k_fp64_basis(const double* __restrict__ base, long long k_min, double df, int n, double* __restrict__ tab) {
  const int bin = blockIdx.x * blockDim.x + threadIdx.x;
  if (bin >= n) return;
  const double um = base[3 * (size_t)bin], up = base[3 * (size_t)bin + 1], lf = base[3 * (size_t)bin + 2];
  const double u2 = um * um, p2 = up * up;
  auto put = [&](int j, double v) { tab[(size_t)j * n + bin] = v; };
  put(B_M53, u2 * u2 * um);
  put(B_M1, u2 * um);
  put(B_M23, u2);
  put(B_M13, um);
  put(B_LOG, lf);
  put(B_P13, up);
  put(B_P13LOG, up * lf);
  put(B_P23, p2);
  put(B_P53, p2 * p2 * up);
  put(B_P73, p2 * p2 * up * p2);
  put(B_ONE, (double)(k_min + bin) * df);
}

cudaError_t launch_fp64_basis(const LikeConst& L, const double* base, double* tab, cudaStream_t st) {
  k_fp64_basis<<<(L.n_bins + 255) / 256, 256, 0, st>>>(base, L.k_min, L.df, L.n_bins, tab);
  return cudaGetLastError();
}

// Per theta: FP64 sum of the slice partials (fixed order), then the epilogue.
__global__ void k_reduce(LikeConst L, const double* __restrict__ partials, int n_units, const EvalRecord* __restrict__ rec,
                         int n, double* __restrict__ out, double* __restrict__ kappa_out) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int th = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (th >= n) return;
  double acc[2 * SWIG_MAX_DET];
#pragma unroll
  for (int j = 0; j < 2 * SWIG_MAX_DET; ++j) acc[j] = 0.0;
  for (int s = lane; s < n_units; s += 32) {
    const double* p = partials + ((size_t)th * n_units + s) * kPartialStride;
#pragma unroll
    for (int j = 0; j < 2 * SWIG_MAX_DET; ++j)
      if (j < 2 * L.n_det) acc[j] += p[j];
  }
#pragma unroll
  for (int j = 0; j < 2 * SWIG_MAX_DET; ++j)
    if (j < 2 * L.n_det)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], o);
  if (lane == 0) {
    double kre[SWIG_MAX_DET], kim[SWIG_MAX_DET];
    for (int i = 0; i < SWIG_MAX_DET; ++i) {
      kre[i] = acc[2 * i];
      kim[i] = acc[2 * i + 1];
    }
    out[th] = loglike_epilogue(L, rec[th], kre, kim);
    if (kappa_out)
      for (int j = 0; j < 2 * SWIG_MAX_DET; ++j) kappa_out[(size_t)th * 2 * SWIG_MAX_DET + j] = acc[j];
  }
}

// ---------------------------------------------------------------------------
// Post-hoc distance of each sample of a distance-marginalised run: the
// q-quantile of p(d_L | theta, data) ~ pi(d) L(d), q from Philox-4x32-10 at
// counter (index lo, index hi, 0x64697374, 5) as a 53-bit uniform.  The
// conditional is tabulated on 1024 trapezoid cells in u = 1/d over the
// marginal's window; the quantile is read off the cumulative from the large-u
// (small-d) end and interpolated linearly inside its cell.
// ---------------------------------------------------------------------------
__global__ void k_distance_draw(LikeConst L, const EvalRecord* __restrict__ rec, const double* __restrict__ kappa,
                                int n, long long first, unsigned k0, unsigned k1, double* __restrict__ theta) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const EvalRecord& r = rec[i];
  double* th = theta + (size_t)SWIG_N_PARAMS * i;
  if (!r.valid) {
    th[6] = NAN;
    return;
  }
  double zr = 0.0, zi = 0.0;
  for (int d = 0; d < L.n_det; ++d) {
    const double a = kappa[(size_t)i * 2 * SWIG_MAX_DET + 2 * d] * L.inv_scale[d];
    const double b = kappa[(size_t)i * 2 * SWIG_MAX_DET + 2 * d + 1] * L.inv_scale[d];
    zr += r.cre[d] * a - r.cim[d] * b;
    zi += r.cre[d] * b + r.cim[d] * a;
  }
  const double H = r.hh;
  const double X = L.phase_marg ? sqrt(zr * zr + zi * zi) : zr;
  double ua, ub;
  distance_window(L, X, H, &ua, &ub);
  constexpr int kCells = 1024;
  const double h = (ub - ua) / kCells;
  double M = -INFINITY;
  for (int j = 0; j <= kCells; ++j) M = fmax(M, distance_exponent(L, zr, X, H, ua + h * j));
  double total = 0.0, fprev = exp(distance_exponent(L, zr, X, H, ua) - M);
  for (int j = 1; j <= kCells; ++j) {
    const double f = exp(distance_exponent(L, zr, X, H, ua + h * j) - M);
    total += 0.5 * (f + fprev);
    fprev = f;
  }
  const long long gi = first + i;
  const uint4 w = philox4x32_10(make_uint4((unsigned)(gi & 0xFFFFFFFFll), (unsigned)(gi >> 32), 0x64697374u, 5u), k0, k1);
  const double q = ((double)(w.x >> 5) * 67108864.0 + (double)(w.y >> 6)) * (1.0 / 9007199254740992.0);
  const double target = q * total;
  double acc = 0.0, uq = ua;
  fprev = exp(distance_exponent(L, zr, X, H, ub) - M);
  for (int j = kCells - 1; j >= 0; --j) {
    const double f = exp(distance_exponent(L, zr, X, H, ua + h * j) - M);
    const double seg = 0.5 * (f + fprev);
    if (acc + seg >= target || j == 0) {
      const double frac = seg > 0.0 ? fmin(1.0, fmax(0.0, (target - acc) / seg)) : 0.5;
      uq = ua + h * (j + 1) - frac * h;
      break;
    }
    acc += seg;
    fprev = f;
  }
  th[6] = 1.0 / uq;
}

// ---------------------------------------------------------------------------
// Post-hoc t_c of time-marginalised samples (App. A): from the node log
// weights of each sample (k_het_tm's ell), the first grid node whose
// cumulative weight reaches q x total, q a 53-bit Philox uniform on the
// sample's global index (stream tag "time").  One warp per sample; the
// cumulative sums run in 32-node chunks (warp inclusive scan) in the same
// order for the total and the search, so the search always ends on a node.
// ---------------------------------------------------------------------------
__device__ inline double warp_inclusive_scan(double v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double u = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += u;
  }
  return v;
}

__global__ void k_time_draw(LikeConst L, const EvalRecord* __restrict__ rec, const float* __restrict__ ell, int n,
                            long long first, unsigned k0, unsigned k1, double* __restrict__ theta) {
  const int i = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= n) return;
  double* th = theta + (size_t)SWIG_N_PARAMS * i;
  if (!rec[i].valid) {
    if (lane == 0) th[11] = NAN;
    return;
  }
  const int N = L.tm_n;
  const float* l = ell + (size_t)i * N;
  float m = -INFINITY;
  for (int j = lane; j < N; j += 32) m = fmaxf(m, l[j]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  double total = 0.0;
  for (int base = 0; base < N; base += 32) {
    const int j = base + lane;
    const double v = warp_inclusive_scan(j < N ? exp((double)l[j] - (double)m) : 0.0, lane);
    total += __shfl_sync(0xffffffffu, v, 31);
  }
  const long long gi = first + i;
  const uint4 w = philox4x32_10(make_uint4((unsigned)(gi & 0xFFFFFFFFll), (unsigned)(gi >> 32), 0x74696d65u, 5u), k0, k1);
  const double q = ((double)(w.x >> 5) * 67108864.0 + (double)(w.y >> 6)) * (1.0 / 9007199254740992.0);
  const double target = q * total;
  double acc = 0.0;
  int pick = N - 1;
  for (int base = 0; base < N; base += 32) {
    const int j = base + lane;
    const double v = warp_inclusive_scan(j < N ? exp((double)l[j] - (double)m) : 0.0, lane);
    const unsigned hit = __ballot_sync(0xffffffffu, j < N && acc + v >= target);
    if (hit) {
      pick = base + __ffs(hit) - 1;
      break;
    }
    acc += __shfl_sync(0xffffffffu, v, 31);
  }
  if (lane == 0) th[11] = L.tm_lo + ((double)pick + 0.5) * L.tm_dt;
}

cudaError_t launch_time_draw(const LikeConst& L, const DeviceBuffers& B, const float* ell, int n, long long first,
                             unsigned k0, unsigned k1, double* theta, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_time_draw<<<(n + 3) / 4, 128, 0, st>>>(L, B.rec, ell, n, first, k0, k1, theta);
  return cudaGetLastError();
}

cudaError_t launch_distance_draw(const LikeConst& L, const DeviceBuffers& B, const double* kappa, int n,
                                 long long first, unsigned k0, unsigned k1, double* theta, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_distance_draw<<<(n + 127) / 128, 128, 0, st>>>(L, B.rec, kappa, n, first, k0, k1, theta);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Heterodyned likelihood: up to eight parameter vectors per CTA, so that a
// chunk's weights are read once for all of them and two share each packed FP32
// instruction.  Anchors of a panel of chunks (a thread per pair, chunk and
// quarter), then a warp per chunk over the vectors' pairs; the warps' sums and the FP64
// epilogue a warp per vector.  (A warp per vector walking all chunks with an
// eleven-term double-float sum per edge took 266 us for 1000 vectors on 5000
// bins, 15 % of the issue slots.)
// ---------------------------------------------------------------------------
constexpr int kHetBatch = 8;
constexpr int kHetWarps = kHetTmThreads / 32;
constexpr int kHetPanel = 256;  // chunks anchored at once

template <int NDET>
__global__ void __launch_bounds__(kHetTmThreads, 1)
    k_het(LikeConst L, HetTables H, const EvalRecord* __restrict__ rec, int n, int per, int tab_off,
          double* __restrict__ out, double* __restrict__ kappa_out, double* __restrict__ vv_out) {
  extern __shared__ __align__(16) float s_an[];  // [pairs][panel][kHetAncPair], the chunk table
  __shared__ HetPrep<NDET> s_prep[kHetBatch];
  __shared__ HetIn<NDET, 2> s_in[kHetBatch / 2];
  __shared__ float s_part[kHetWarps][NDET][3 * kHetBatch];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int panel = min(kHetPanel, H.n_chunks);
  const float* tab = H.chunk;
  if (tab_off > 0) {
    for (int q = threadIdx.x; q < HC_ROWS * H.n_chunks; q += kHetTmThreads) cp_async<4>(s_an + tab_off + q, H.chunk + q);
    cp_async_commit();
    tab = s_an + tab_off;
  }
  // the set-up kernel's records, while this one's start overlapped its end
  asm volatile("griddepcontrol.wait;" ::: "memory");
  cp_async_wait<0>();
  for (int base = blockIdx.x * per; base < n; base += gridDim.x * per) {
    const int m = min(per, n - base), pairs = (m + 1) / 2;
    __syncthreads();
    if (warp < 2 * pairs) {  // (an odd batch's last pair holds its vector twice)
      het_differences<NDET>(H.fid->c, H.fid->tau, rec[base + min(warp, m - 1)], s_prep[warp], lane);
      het_in_set<NDET, 2>(s_in[warp >> 1], warp & 1, s_prep[warp], lane);
    }
    HetAcc<NDET, 2> acc[kHetBatch / 2];
#pragma unroll
    for (int p = 0; p < kHetBatch / 2; ++p) acc[p].clear();
    for (int q0 = 0; q0 < H.n_chunks; q0 += panel) {
      const int np = min(panel, H.n_chunks - q0);
      __syncthreads();
      // the first chunk's weights, then always the next one's: in flight meanwhile
      float4 nx[NDET];
      const float4* ew = H.ew + (size_t)q0 * NDET * 32 + lane;
      if (warp < np)
#pragma unroll
        for (int i = 0; i < NDET; ++i) nx[i] = __ldg(ew + (warp * NDET + i) * 32);
      het_anchors<NDET, 2>(H, tab, s_in, pairs, q0, np, panel, nullptr, s_an, warp, kHetWarps, lane);
      __syncthreads();
      for (int q = warp; q < np; q += kHetWarps) {
        float4 w[NDET];
        const int qn = min(q + kHetWarps, np - 1);
#pragma unroll
        for (int i = 0; i < NDET; ++i) {
          w[i] = nx[i];
          nx[i] = __ldg(ew + (qn * NDET + i) * 32);
        }
#pragma unroll
        for (int p = 0; p < kHetBatch / 2; ++p)
          if (p < pairs) {
            const HetPrep<NDET>* pp[2] = {&s_prep[2 * p], &s_prep[2 * p + 1]};
            het_edges<NDET, 2>(H, s_an + ((size_t)p * panel + q) * kHetAncPair, s_in[p], pp, q0 + q, lane, w,
                               acc[p]);
          }
      }
    }
#pragma unroll
    for (int i = 0; i < NDET; ++i) {
      float a[32];  // value 8 kind + vector
#pragma unroll
      for (int p = 0; p < kHetBatch / 2; ++p) {
        PkOps<2>::get(acc[p].zr[i], a + 2 * p);
        PkOps<2>::get(acc[p].zi[i], a + kHetBatch + 2 * p);
        PkOps<2>::get(acc[p].hh[i], a + 2 * kHetBatch + 2 * p);
        a[3 * kHetBatch + 2 * p] = a[3 * kHetBatch + 2 * p + 1] = 0.0f;
      }
      const float v = warp_transpose_sum(a, lane);
      if (lane < 3 * kHetBatch) s_part[warp][i][lane] = v;
    }
    __syncthreads();
    if (warp < m) {
      const EvalRecord& r = rec[base + warp];
      const double v = het_part_sum<NDET, kHetBatch>(s_part, kHetWarps, warp, lane);
      double Zr, Zi, HH, kap = 0.0, vv = 0.0;
      het_network<NDET>(L, *H.fid, r, v, lane, Zr, Zi, HH, kap, vv);
      const size_t th = base + warp;
      const bool valid = r.valid != 0;
      if (lane == 0) out[th] = valid ? het_epilogue(L, Zr, Zi, HH) : -INFINITY;
      if (kappa_out && lane < 2 * SWIG_MAX_DET) kappa_out[th * 2 * SWIG_MAX_DET + lane] = valid ? kap : 0.0;
      if (vv_out && lane < SWIG_MAX_DET) vv_out[th * SWIG_MAX_DET + lane] = valid ? vv : 0.0;
    }
  }
}

// Time-marginalised heterodyned likelihood, one CTA per theta (the thread
// count and the chunk-to-warp assignment of the persistent sampler, so both
// give the same sums): the warps contract the chunks, storing the edge
// products y_e in shared memory, then share the grid's 32-node chunks.
// ell (optional) receives every node's log weight, [n][tm_n].  The anchors lie
// where the time pass's grid follows (or after it, anc_off).
template <int NDET>
__global__ void __launch_bounds__(kHetTmThreads, 1)
    k_het_tm(LikeConst L, HetTables H, const EvalRecord* __restrict__ rec, int n, int anc_off, int panel,
             double* __restrict__ out, double* __restrict__ kappa_out, double* __restrict__ vv_out,
             float* __restrict__ ell) {
  extern __shared__ __align__(16) unsigned char smem[];
  float2* y = reinterpret_cast<float2*>(smem);
  float* s_an = reinterpret_cast<float*>(smem + anc_off);
  __shared__ HetPrep<NDET> s_prep;
  __shared__ HetIn<NDET, 1> s_in;
  __shared__ float s_hh[kHetWarps][NDET];
  __shared__ float s_tm[kHetWarps][2];
  const int th = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
  if (th >= n) return;
  const EvalRecord& r = rec[th];
  if (L.tm_M > 0) tm_load_twiddles(L, H, smem, H.n_bins);  // read after the barriers below
  // the set-up kernel's records, while this one's start overlapped its end
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (threadIdx.x == 0) {
    // no projection-only reuse under time marginalisation: the caches are zero
    if (kappa_out)
      for (int j = 0; j < 2 * SWIG_MAX_DET; ++j) kappa_out[(size_t)th * 2 * SWIG_MAX_DET + j] = 0.0;
    if (vv_out)
      for (int i = 0; i < SWIG_MAX_DET; ++i) vv_out[(size_t)th * SWIG_MAX_DET + i] = 0.0;
  }
  float* ell_th = ell ? ell + (size_t)th * L.tm_n : nullptr;
  if (!r.valid) {
    if (threadIdx.x == 0) out[th] = -INFINITY;
    if (ell_th)
      for (int j = threadIdx.x; j < L.tm_n; j += blockDim.x) ell_th[j] = -INFINITY;
    return;
  }
  if (warp == 0) {
    het_prepare_warp<NDET>(L, H, r, s_prep, lane);
    het_in_set<NDET, 1>(s_in, 0, s_prep, lane);
  }
  HetAcc<NDET, 1> acc;
  acc.clear();
  het_products<NDET>(H, s_prep, s_in, s_an, panel, warp, n_warps, lane, acc, y);
#pragma unroll
  for (int i = 0; i < NDET; ++i) {
    float d = acc.hh[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
    if (lane == 0) s_hh[warp][i] = d;
  }
  __syncthreads();
  float wm, ws;
  if (L.tm_M > 0)
    tm_pass_nufft(L, H, y, tm_nufft_grid(smem, H.n_bins), tm_nufft_tw(smem, H.n_bins, L.tm_M), warp, n_warps, lane,
                  ell_th, wm, ws);
  else
    tm_pass(L, H, y, warp, n_warps, lane, ell_th, wm, ws);
  if (lane == 0) {
    s_tm[warp][0] = wm;
    s_tm[warp][1] = ws;
  }
  __syncthreads();
  if (warp == 0) {
    const double ll = tm_finish<NDET>(L, r, s_hh, s_tm, n_warps, lane);
    if (lane == 0) out[th] = ll;
  }
}

template <int NDET>
cudaError_t launch_het_tm(const LikeConst& L, const DeviceBuffers& B, int n, double* out, cudaStream_t st,
                          double* kappa_out, double* vv_out, float* ell) {
  const HetTmLayout lay = het_tm_layout(L, B);
  return launch_after(k_het_tm<NDET>, dim3(n), kHetTmThreads, lay.bytes, st, L, het_tables(B), (const EvalRecord*)B.rec, n,
                            lay.anc_off, lay.panel, out, kappa_out, vv_out, ell);
}

template <int NDET>
cudaError_t launch_het_plain(const LikeConst& L, const DeviceBuffers& B, int n, double* out, cudaStream_t st,
                             double* kappa_out, double* vv_out) {
  // as few vectors per CTA as fill the device once
  int per = (n + L.sm_count - 1) / L.sm_count;
  per = per < kHetBatch ? per : kHetBatch;
  const int panel = B.het_nc < kHetPanel ? B.het_nc : kHetPanel, ctas = (n + per - 1) / per;
  size_t bytes = (size_t)((per + 1) / 2) * panel * kHetAncPair * sizeof(float);
  const size_t tab = sizeof(float) * HC_ROWS * (size_t)B.het_nc;
  const int tab_off = bytes + tab <= 200 * 1024 ? (int)(bytes / sizeof(float)) : 0;
  if (tab_off) bytes += tab;
  return launch_after(k_het<NDET>, dim3(ctas < L.sm_count ? ctas : L.sm_count), kHetTmThreads, bytes, st, L, het_tables(B),
                            (const EvalRecord*)B.rec, n, per, tab_off, out, kappa_out, vv_out);
}

cudaError_t launch_loglike_het(const LikeConst& L, const DeviceBuffers& B, const double* theta, int n, double* out,
                               cudaStream_t st, double* kappa_out, double* vv_out, float* ell) {
  if (n <= 0) return cudaSuccess;
  launch_setup(L, theta, n, B.rec, st);
  if (L.tm_n > 0) {
    switch (L.n_det) {
      case 1: return launch_het_tm<1>(L, B, n, out, st, kappa_out, vv_out, ell);
      case 2: return launch_het_tm<2>(L, B, n, out, st, kappa_out, vv_out, ell);
      case 3: return launch_het_tm<3>(L, B, n, out, st, kappa_out, vv_out, ell);
      default: return launch_het_tm<4>(L, B, n, out, st, kappa_out, vv_out, ell);
    }
  }
  switch (L.n_det) {
    case 1: return launch_het_plain<1>(L, B, n, out, st, kappa_out, vv_out);
    case 2: return launch_het_plain<2>(L, B, n, out, st, kappa_out, vv_out);
    case 3: return launch_het_plain<3>(L, B, n, out, st, kappa_out, vv_out);
    default: return launch_het_plain<4>(L, B, n, out, st, kappa_out, vv_out);
  }
}

// ---------------------------------------------------------------------------
// Detector strain on the grid (FP64): h_i(f) = C_i f^-7/6 exp(-2 pi i (P(f) + f tau_i)).
// ---------------------------------------------------------------------------
__global__ void k_waveform(LikeConst L, const EvalRecord* __restrict__ rec, double2* __restrict__ out) {
  const int bin = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = blockIdx.y;
  if (bin >= L.n_bins || i >= L.n_det) return;
  const EvalRecord& r = rec[0];
  const double f = (double)(L.k_min + bin) * L.df;
  const double up = cbrt(f), um = 1.0 / up, lf = log(f);
  const double u2 = um * um, p2 = up * up;
  double P = r.c[B_ONE] + r.c[B_LOG] * lf;
  P += um * (r.c[B_M13] + um * (r.c[B_M23] + um * (r.c[B_M1] + u2 * r.c[B_M53])));
  P += up * (r.c[B_P13] + r.c[B_P13LOG] * lf) + p2 * r.c[B_P23] + p2 * p2 * up * (r.c[B_P53] + p2 * r.c[B_P73]);
  double ph = fma(f, r.tau[i], P);
  ph -= rint(ph);
  double s, co;
  sincospi(2.0 * ph, &s, &co);
  const double a = exp(-7.0 / 6.0 * lf);
  // C_i a (cos - i sin)
  const double re = a * (r.cre[i] * co + r.cim[i] * s), im = a * (r.cim[i] * co - r.cre[i] * s);
  out[(size_t)i * L.n_bins + bin] = make_double2(re, im);
}

cudaError_t launch_waveform(const LikeConst& L, const double* theta_dev, EvalRecord* rec_dev, double2* out,
                            cudaStream_t st) {
  launch_setup(L, theta_dev, 1, rec_dev, st);
  dim3 grid((L.n_bins + 255) / 256, L.n_det);
  k_waveform<<<grid, 256, 0, st>>>(L, rec_dev, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Prior transform (Table I inverse CDFs).
// ---------------------------------------------------------------------------
__global__ void k_prior_transform(const PriorSlot* __restrict__ slots, int n_sampled, const double* __restrict__ u,
                                  int n, double* __restrict__ theta, SkyFrame sky) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  prior_map(slots, u + (size_t)i * n_sampled, theta + (size_t)i * SWIG_N_PARAMS, &sky);
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
cudaError_t launch_loglike_mixed(const LikeConst& L, const DeviceBuffers& B, const double* theta, int n,
                                 double* out, cudaStream_t st, double* kappa_out) {
  if (n <= 0) return cudaSuccess;
  launch_setup(L, theta, n, B.rec, st, fold_strays_at(B.strays, n));
  return launch_fold(L, B, n, out, st, kappa_out);
}

cudaError_t launch_loglike_fp64(const LikeConst& L, const DeviceBuffers& B, const double* theta, int n,
                                double* out, cudaStream_t st, double* kappa_out) {
  if (n <= 0) return cudaSuccess;
  launch_setup(L, theta, n, B.rec, st);
  const int gy = (n + 7) / 8 < 64 ? (n + 7) / 8 : 64;
  dim3 grid(L.n_slices, gy);
  const auto sweep = L.n_det == 1 ? k_sweep_fp64<1> : L.n_det == 2 ? k_sweep_fp64<2> : L.n_det == 3 ? k_sweep_fp64<3>
                                                                                               : k_sweep_fp64<4>;
  cudaError_t e = launch_after(sweep, grid, 256, 0, st, L, (const double2*)B.data64, (const double*)B.ftab,
                               (const int*)B.slice_begin, (const EvalRecord*)B.rec, n, B.partials64);
  if (e == cudaSuccess)
    e = launch_after(k_reduce, dim3((n + 3) / 4), 128, 0, st, L, (const double*)B.partials64, L.n_slices,
                     (const EvalRecord*)B.rec, n, out, kappa_out);
  return e;
}

cudaError_t launch_prior_transform(const PriorSlot* slots, int n_sampled, const double* u, int n, double* theta,
                                   cudaStream_t st, SkyFrame sky) {
  if (n <= 0) return cudaSuccess;
  k_prior_transform<<<(n + 127) / 128, 128, 0, st>>>(slots, n_sampled, u, n, theta, sky);
  return cudaGetLastError();
}

}  // namespace swig
