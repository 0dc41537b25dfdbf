// State and shared device code of the nested samplers: the run's constants and
// state, draws, the bounded grid barrier, the projection-only likelihood and the
// iteration boundary.
#pragma once

#include <cuda_runtime.h>

#include "context.h"
#include "device_common.cuh"

namespace swig {

constexpr int kMaxDim = SWIG_N_PARAMS;
constexpr int kMaxBlocks = 16;
constexpr int kMaxStepOut = 100;
constexpr int kMaxShrink = 100;
constexpr int kMaxSort = 8192;
constexpr int kMaxChains = 2048;

constexpr int kMaxEvents = 4;    // events per multi-event launch
constexpr int kFlowThreads = 512;  // FP64 dataflow sampler: 16 warps
constexpr int kFreeBudget = 8;  // projection-only evaluations per chain per round
#ifndef SWIG_FLOW_PARTS
#define SWIG_FLOW_PARTS 1
#endif
static_assert(SWIG_FLOW_PARTS >= 1 && SWIG_FLOW_PARTS <= 4, "1..4 parts per slice");
// FP64 sampler: PH_LEFT, then PH_RIGHT; chain sampler: PH_OUT, both ends
enum ChainPhase { PH_NEW = 0, PH_LEFT = 1, PH_RIGHT = 2, PH_SHRINK = 3, PH_OUT = 4 };
// What a Gibbs block moves: waveform coefficients, amplitude A(Mc)/d_L,
// projection P_i, time shifts tau_i (BF_SKY: through the geocentric delays;
// BF_TAU alone: t_c).
enum BlockFlag { BF_INTR = 1, BF_AMP = 2, BF_PROJ = 4, BF_TAU = 8, BF_SPIN = 16, BF_TIDE = 32, BF_SKY = 64 };
enum RunStatus { ST_RUNNING = 0, ST_TERMINATED = 1, ST_LIMIT = 2 };

struct SamplerConst {
  int ndim, nlive, nrep, sweeps, steps_per_dim, n_blocks;
  int slot_of_dim[kMaxDim];
  int block_size[kMaxBlocks], block_free[kMaxBlocks], block_flags[kMaxBlocks];
  int block_dims[kMaxBlocks][kMaxDim];
  PriorSlot prior[SWIG_N_PARAMS];
  unsigned key0, key1;
  double dlogz;
  int m_pow2;
  int max_iters;
  long long spin_limit;
  int n_ctas;
  int flow_parts;   // parts per slice (dataflow kernel): fixed summation partition
  SkyFrame sky;     // detector-frame sky parameterisation (slots 9, 10), or off
  int learn_on;     // learned directions available (SWIG_PROPOSAL_LEARNED)
  float learn_mix;  // probability of a learned direction per slice step
  // dimensions of each block as a bit mask and each dimension's rank within
  // its block
  unsigned block_mask[kMaxBlocks];
  int block_rank[kMaxDim];
  int claim_off;  // FP64 sampler: byte offset of the claim words in dynamic shared memory
  // chain sampler (chain.cuh), the launch shape: rungs per bracket end and
  // shrinkage draws evaluated at a time; one end of a bracket after the other
  int spec_out, spec_shr, spec_mix, one_end;
};

struct ChainState {
  double x[kMaxDim], y[kMaxDim], dir[kMaxDim];
  double th[SWIG_N_PARAMS], th_y[SWIG_N_PARAMS];  // theta of x and of the proposal
  double lx, lo, hi, t;
  double kap[2 * SWIG_MAX_DET];
  double vv[SWIG_MAX_DET];  // heterodyned path: <h|h>_i / |C_i|^2 of the current point, times A1^2
  int block, step, sweep, phase, n_out, n_shrink;
  int pending, done, proj_dirty, slot;
  unsigned ctr;
  int n_caps;
  long long n_evals, n_full;
  int side;     // PH_OUT: bit 0 the left end still stepping out, bit 1 the right end
  int n_out_r;  // PH_OUT: expansions of the right end
  int closed;   // ... ends that left the unit cube (bits)
  int score;    // chain sampler: how often its guess held lately (chain.cuh)
};

struct NSGlobal {
  double logx, logz, logl_star;
  long long iter;
  int iters_launch;
  int status;
  int error;
  int chains_done;
  int need_writeback;
  int n_dead;
  unsigned bar_count, bar_gen;
  int task;  // chain sampler: next chain of the iteration
  unsigned beat;  // ... raised as any CTA's chain advances (every eight rounds, or steps)
  // phase timers of CTA 0 [ns, %globaltimer]: boundary, control, wait after
  // control, sweep, wait after sweep; and rounds
  unsigned long long t_bound, t_ctrl, t_wait_ctrl, t_sweep, t_wait_sweep, rounds;
  // chain 0's control breakdown [clock64 cycles]: pending result, new step,
  // proposal + transform, projection-only evaluations, full setup; counts
  unsigned long long c_result, c_step, c_prop, c_free, c_setup, n_free, n_setup, n_step;
  // CTA 0's sweep warps (dataflow kernel): units evaluated, clock64 cycles in
  // units, cycles idle (polling for work)
  unsigned long long f_units, f_unit_cyc, f_idle_cyc;
};

__device__ __forceinline__ unsigned long long gtimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

struct SamplerPtrs {
  double* live_u;      // [m][ndim]
  double* live_logl;   // [m]
  double* live_kap;    // [m][8]
  double* live_vv;     // [m][4] heterodyned path: see ChainState::vv
  ChainState* chains;  // [k]
  EvalRecord* recx;    // [k] setup record of each chain's current point
  int* pending;        // [k]
  float* chol;         // [kMaxBlocks][kMaxDim][kMaxDim]
  NSGlobal* g;
  double* dead_u;      // [max_iters * k][ndim]
  double* dead_logl;
  double* dead_logw;
  const double* harm;  // [k + 1]: sum_{i<j} 1 / (m - i)
  const double* lw;    // [m + 1]: log(1 - exp(-1/n))
  const float* learn_out;  // [m][32] network outputs (u, s) of a frozen live snapshot, or null
  int* req;                // [k] 8 * (sequence number of the chain's latest full-likelihood request) + parts per slice
  int* done_cnt;           // [k] CTAs that finished the chain's latest request
  unsigned long long* cta_prof;  // [n_ctas][4] per CTA: sweep units, cycles in units, cycles polling, control cycles
};

// ---------------------------------------------------------------------------
// Draws built on Philox-4x32-10 (device_common.cuh).
// ---------------------------------------------------------------------------
__device__ __forceinline__ double u01_from(uint4 r) {  // 53-bit uniform in [0, 1)
  const unsigned long long m = ((unsigned long long)(r.x >> 5) << 26) | (r.y >> 6);
  return (double)m * (1.0 / 9007199254740992.0);
}

__device__ __forceinline__ double chain_uniform(const SamplerConst& S, ChainState& ch, int c, long long it) {
  return u01_from(philox4x32_10(make_uint4(ch.ctr++, (unsigned)c, (unsigned)it, 0u), S.key0, S.key1));
}

// Standard normal by Box-Muller from one Philox block.
__device__ __forceinline__ float chain_normal(const SamplerConst& S, ChainState& ch, int c, long long it) {
  const uint4 r = philox4x32_10(make_uint4(ch.ctr++, (unsigned)c, (unsigned)it, 0u), S.key0, S.key1);
  const float u1 = ((float)(r.x >> 8) + 1.0f) * (1.0f / 16777216.0f);  // (0, 1]
  const float u2 = (float)(r.y >> 8) * (1.0f / 16777216.0f);
  return sqrtf(-2.0f * logf(u1)) * cospif(2.0f * u2);
}

// ---------------------------------------------------------------------------
// Bounded grid barrier (all CTAs co-resident by cooperative launch).  beat
// (optional): a count that the other CTAs raise as they work; the limit then
// bounds the polls in which it stands still.
// ---------------------------------------------------------------------------
static __device__ bool grid_sync(NSGlobal* g, int n_ctas, long long limit, const unsigned* beat = nullptr) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* vgen = &g->bar_gen;
    const unsigned gen = *vgen;
    __threadfence();
    const unsigned arrived = atomicAdd(&g->bar_count, 1u) + 1u;
    if (arrived == (unsigned)n_ctas) {
      atomicExch(&g->bar_count, 0u);
      __threadfence();
      atomicAdd(&g->bar_gen, 1u);
    } else {
      long long spins = 0;
      unsigned last = 0;
      while (*vgen == gen) {
        if (beat) {
          const unsigned now = *(const volatile unsigned*)beat;
          if (now != last) {
            last = now;
            spins = 0;
          }
        }
        if (++spins > limit) {
          atomicCAS(&g->error, 0, SWIG_E_TIMEOUT);
          break;
        }
        __nanosleep(100);
      }
    }
    __threadfence();
    s_ok = (*(volatile int*)&g->error) == 0;
  }
  __syncthreads();
  return s_ok != 0;
}

// ---------------------------------------------------------------------------
// Epilogue of blocks that leave kappa unchanged: projection factors in FP32 (an
// error delta of C enters logL as (Z - <h|h>) delta, small near the peak), what they
// multiply, their products and the sums in double-float.  Z and <h|h> / 2 cancel in
// logL and are about SNR^2 and SNR^2 / 2: in FP32, with a loud signal (SNR 170, logL
// -3,975), their rounding alone is 3e-3.  Largest error over 500,000 dead points of
// 32 injections without an SNR cut, in units of 1e-6 |logL| + 1e-6: 1.54 in FP32, 0.59
// (4 iterations of the 128 s run 12.77 -> 12.93 ms).
// ---------------------------------------------------------------------------
__device__ __forceinline__ dfl df_scale(float c, dfl a) {  // c a, not renormalised
  const float p = __fmul_rn(c, a.hi);
  return {p, fmaf(c, a.lo, fmaf(c, a.hi, -p))};
}

// kap: per-detector sums cached at the chain's current point (full grid:
// kappa_i; heterodyned: (Z_i / C_i) / inv_scale_i) times L.amp_s; vv: <h|h>_i /
// |C_i|^2 times A1^2 (full grid: the constant L.amp_k); (hi, lo).
__device__ inline double free_loglike(const LikeConst& L, const float* th, const float2* kap, const float2* vv) {
  const float mc = th[0], dl = th[6], iota = th[7], psi = th[8];
  const float ra = th[9], dec = th[10], phic = th[12];
  if (!(mc > 0.0f && dl > 0.0f)) return -INFINITY;
  const float rel = exp2f(0.8333333333f * log2f(mc)) / dl;  // Mc^(5/6) / d_L
  float sl, cl, sd, cd, sp, cp;
  sincosf(ra - L.gmst_f, &sl, &cl);
  sincosf(dec, &sd, &cd);
  sincosf(psi, &sp, &cp);
  const float east[3] = {-sl, cl, 0.0f};
  const float north[3] = {-sd * cl, -sd * sl, cd};
  float X[3], Y[3];
  for (int k = 0; k < 3; ++k) {
    X[k] = -cp * east[k] + sp * north[k];
    Y[k] = sp * east[k] + cp * north[k];
  }
  const float ci = cosf(iota);
  const float plus = 0.5f * (1.0f + ci * ci), cross = -ci;
  float sph = 0.0f, cph = 1.0f;
  if (!L.phase_marg) sincosf(phic, &sph, &cph);
  dfl zr = {0.0f, 0.0f}, zi = {0.0f, 0.0f}, hh = {0.0f, 0.0f};
  for (int i = 0; i < L.n_det; ++i) {
    float d[6];
    for (int q = 0; q < 6; ++q) d[q] = L.dten_f[i][q];
    auto form = [&d](const float* a, const float* b) {
      return a[0] * (d[0] * b[0] + d[1] * b[1] + d[2] * b[2]) + a[1] * (d[1] * b[0] + d[3] * b[1] + d[4] * b[2]) +
             a[2] * (d[2] * b[0] + d[4] * b[1] + d[5] * b[2]);
    };
    const float fp = form(X, X) - form(Y, Y), fx = 2.0f * form(X, Y);
    const float re0 = rel * fp * plus, im0 = rel * fx * cross;
    const float cre = re0 * cph - im0 * sph, cim = re0 * sph + im0 * cph;
    const dfl a = {kap[2 * i].x, kap[2 * i].y}, b = {kap[2 * i + 1].x, kap[2 * i + 1].y};
    zr = df_accumulate(zr, df_accumulate(df_scale(cre, a), df_scale(-cim, b)));
    zi = df_accumulate(zi, df_accumulate(df_scale(cre, b), df_scale(cim, a)));
    const dfl c2 = df_accumulate(df_scale(cre, dfl{cre, 0.0f}), df_scale(cim, dfl{cim, 0.0f}));
    hh = df_accumulate(hh, df_mul(c2, dfl{vv[i].x, vv[i].y}));
  }
  // with d_L marginalised the template is at 1 Mpc: zr, zi, hh are Z1, H1
  if (L.dist_marg)
    return distance_marg_logl(L, (double)zr.hi + (double)zr.lo, (double)zi.hi + (double)zi.lo,
                              (double)hh.hi + (double)hh.lo);
  dfl core = zr;
  if (L.phase_marg) {
    // |Z|: the root of the high words, and what is left of the squares over 2 |Z|
    const float x = sqrtf(fmaf(zr.hi, zr.hi, zi.hi * zi.hi));
    const dfl s = df_accumulate(df_scale(zr.hi, dfl{zr.hi, 2.0f * zr.lo}), df_scale(zi.hi, dfl{zi.hi, 2.0f * zi.lo}));
    const dfl r = df_accumulate(s, df_scale(-x, dfl{x, 0.0f}));
    core = df_accumulate(dfl{x, x > 0.0f ? 0.5f * (r.hi + r.lo) / x : 0.0f}, dfl{log_i0e_f32(x), 0.0f});
  }
  core = df_accumulate(core, dfl{-0.5f * hh.hi, -0.5f * hh.lo});
  return (double)core.hi + ((double)core.lo - 0.5 * L.DD);
}

// ---------------------------------------------------------------------------
// Chain control.
// ---------------------------------------------------------------------------
// g: count the finished chain there (FP64 sampler).
__device__ inline void finish_step(const SamplerConst& S, ChainState& ch, NSGlobal* g = nullptr) {
  ch.phase = PH_NEW;
  if (++ch.step >= S.steps_per_dim * S.block_size[ch.block]) {
    ch.step = 0;
    if (++ch.block >= S.n_blocks) {
      ch.block = 0;
      if (++ch.sweep >= S.sweeps) {
        ch.done = 1;
        if (g) atomicAdd(&g->chains_done, 1);
      }
    }
  }
}

// Copy n bytes (a multiple of 4) with the whole warp.
__device__ __forceinline__ void warp_copy(void* dst, const void* src, int n, int lane) {
  const unsigned* s4 = static_cast<const unsigned*>(src);
  unsigned* d4 = static_cast<unsigned*>(dst);
  for (int q = lane; q < n / 4; q += 32) d4[q] = s4[q];
  __syncwarp();
}

// The same from global memory written by another SM (through L2).
__device__ __forceinline__ void warp_copy_cg(void* dst, const void* src, int n, int lane) {
  const unsigned* s4 = static_cast<const unsigned*>(src);
  unsigned* d4 = static_cast<unsigned*>(dst);
  for (int q = lane; q < n / 4; q += 32) d4[q] = __ldcg(s4 + q);
  __syncwarp();
}

// ---------------------------------------------------------------------------
// Iteration boundary on CTA 0.
// ---------------------------------------------------------------------------
static __device__ void block_reduce_max_sum(double* vals, int n, double* out_max, double* out_sumexp, double* s_tmp) {
  // two passes over vals[0..n): max, then sum exp(v - max); s_tmp holds at
  // least the block size rounded up to a power of two (tree over it, the
  // padding holding the operation's identity)
  const int nt = blockDim.x, tid = threadIdx.x;
  int np2 = 1;
  while (np2 < nt) np2 <<= 1;
  double m = -INFINITY;
  for (int i = tid; i < n; i += nt) m = fmax(m, vals[i]);
  s_tmp[tid] = m;
  if (tid + nt < np2) s_tmp[tid + nt] = -INFINITY;
  __syncthreads();
  for (int s = np2 / 2; s > 0; s >>= 1) {
    if (tid < s) s_tmp[tid] = fmax(s_tmp[tid], s_tmp[tid + s]);
    __syncthreads();
  }
  m = s_tmp[0];
  __syncthreads();
  double acc = 0.0;
  if (isfinite(m))
    for (int i = tid; i < n; i += nt) acc += exp(vals[i] - m);
  s_tmp[tid] = acc;
  if (tid + nt < np2) s_tmp[tid + nt] = 0.0;
  __syncthreads();
  for (int s = np2 / 2; s > 0; s >>= 1) {
    if (tid < s) s_tmp[tid] += s_tmp[tid + s];
    __syncthreads();
  }
  *out_max = m;
  *out_sumexp = s_tmp[0];
  __syncthreads();
}

// An integer that orders like v (the zeros alike).
__device__ __forceinline__ long long fp64_order(double v) {
  const long long b = __double_as_longlong(v);
  return b >= 0 ? b : (long long)0x8000000000000000ull - b;
}

// First half of the boundary: write the finished chains back into the live
// set and apply the launch's iteration limit and the termination rule.  Fills
// the sort keys in `smem` for the second half.  Returns false (status set)
// when the run stops here.
static __device__ __noinline__ bool ns_boundary_check(const LikeConst& L, const SamplerConst& S, const SamplerPtrs& P,
                                               unsigned char* smem) {
  NSGlobal* g = P.g;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int m = S.nlive, k = S.nrep, d = S.ndim;
  if (g->need_writeback) {
    for (int c = tid; c < k; c += nt) {
      const ChainState& ch = P.chains[c];
      const int slot = __ldcg(&ch.slot);
      for (int j = 0; j < d; ++j) P.live_u[(size_t)slot * d + j] = __ldcg(&ch.x[j]);
      P.live_logl[slot] = __ldcg(&ch.lx);
      for (int j = 0; j < 2 * SWIG_MAX_DET; ++j) P.live_kap[(size_t)slot * 2 * SWIG_MAX_DET + j] = __ldcg(&ch.kap[j]);
      for (int i = 0; i < SWIG_MAX_DET; ++i) P.live_vv[(size_t)slot * SWIG_MAX_DET + i] = __ldcg(&ch.vv[i]);
    }
    __syncthreads();
    if (tid == 0) g->need_writeback = 0;
  }
  __syncthreads();
  if (g->iters_launch >= S.max_iters) {
    if (tid == 0) g->status = ST_LIMIT;
    return false;
  }
  double* key = reinterpret_cast<double*>(smem);
  int* idx = reinterpret_cast<int*>(key + S.m_pow2);
  double* tmp = reinterpret_cast<double*>(idx + S.m_pow2);  // (nt rounded up to a power of two) doubles
  for (int i = tid; i < S.m_pow2; i += nt) {
    key[i] = i < m ? P.live_logl[i] : INFINITY;
    idx[i] = i;
  }
  __syncthreads();
  // termination: log Z_live = log X + log mean L_live
  double mx, se;
  block_reduce_max_sum(key, m, &mx, &se, tmp);
  const double logz_live = g->logx + mx + log(se / (double)m);
  const double logz = g->logz;
  if (isfinite(logz) && logz_live - logz < S.dlogz) {
    if (tid == 0) g->status = ST_TERMINATED;
    return false;
  }
  return true;
}

// Second half: sort, retire the k worst points, update log X / log Z and
// logL*, estimate the block Cholesky factors, start k chains at survivors.
// smem: `bytes` of it (0: as much as the sort takes).
//
// One CTA does this while the others wait, so its latencies count in full: the
// sort compares integers (an FP64 comparison or conversion costs a scheduler
// 64 cycles) and the covariance reads the live points from shared memory,
// converted once, its sums in the order of the points.  nlive 1000, 12
// dimensions, with the first half: 317 -> 147 us per iteration.
static __device__ __noinline__ void ns_boundary_advance(const LikeConst& L, const SamplerConst& S, const SamplerPtrs& P,
                                                 unsigned char* smem, int bytes) {
  NSGlobal* g = P.g;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int m = S.nlive, k = S.nrep, d = S.ndim;
  double* key = reinterpret_cast<double*>(smem);
  int* idx = reinterpret_cast<int*>(key + S.m_pow2);
  double* tmp = reinterpret_cast<double*>(idx + S.m_pow2);
  // bitonic sort (ascending) of (logL, index)
  for (int kk = 2; kk <= S.m_pow2; kk <<= 1) {
    for (int j = kk >> 1; j > 0; j >>= 1) {
      for (int i = tid; i < S.m_pow2; i += nt) {
        const int ixj = i ^ j;
        if (ixj > i) {
          const bool asc = (i & kk) == 0;
          const double a = key[i], b = key[ixj];
          const long long ka = fp64_order(a), kb = fp64_order(b);
          if ((ka > kb) == asc || (ka == kb && ((idx[i] > idx[ixj]) == asc))) {
            key[i] = b;
            key[ixj] = a;
            const int t = idx[i];
            idx[i] = idx[ixj];
            idx[ixj] = t;
          }
        }
      }
      __syncthreads();
    }
  }
  // deaths: w_j = L_j (X_{j-1} - X_j), log X_j = log X_0 - sum_{i<=j} 1/(m - i)
  const int base = g->n_dead;
  int np2 = 1;  // the reduction scratch spans the block size rounded up to a power of two
  while (np2 < nt) np2 <<= 1;
  double* logw = tmp + np2;  // k doubles
  for (int j = tid; j < k; j += nt) {
    const int s = idx[j];
    const double lwj = key[j] + (g->logx - P.harm[j]) + P.lw[m - j];
    logw[j] = lwj;
    P.dead_logl[base + j] = key[j];
    P.dead_logw[base + j] = lwj;
    for (int q = 0; q < d; ++q) P.dead_u[(size_t)(base + j) * d + q] = P.live_u[(size_t)s * d + q];
  }
  __syncthreads();
  double wm, ws;
  block_reduce_max_sum(logw, k, &wm, &ws, tmp);
  if (tid == 0) {
    const double a = g->logz, b = wm + log(ws);
    const double hi = fmax(a, b);
    g->logz = isfinite(hi) ? hi + log(exp(a - hi) + exp(b - hi)) : hi;
    g->logx -= P.harm[k];
    g->logl_star = key[k];
    g->n_dead = base + k;
  }
  // covariance of the live points (FP32; only a proposal scale) and block Cholesky
  float* mean = reinterpret_cast<float*>(logw + k);
  float* cov = mean + kMaxDim;  // kMaxDim x kMaxDim
  // panels of points in FP32: behind the covariance, or over the reductions'
  // scratch where that is longer (an even number of points: 80 at least)
  float* pan = cov + kMaxDim * kMaxDim;
  const int room = max(0, bytes - (int)(reinterpret_cast<unsigned char*>(pan) - smem)) / (int)(d * sizeof(float));
  const int over = (int)((np2 + k) * sizeof(double)) / (int)(d * sizeof(float));
  if (over > room) pan = reinterpret_cast<float*>(tmp);
  const int rows = max(over, room) & ~1;
  float acc0 = 0.0f, acc1 = 0.0f;
  for (int i0 = 0; i0 < m; i0 += rows) {
    const int n = min(rows, m - i0);
    for (int q = tid; q < n * d; q += nt) pan[q] = (float)P.live_u[(size_t)i0 * d + q];
    __syncthreads();
    if (tid < d) {
#pragma unroll 8
      for (int i = 0; i < n; ++i) acc0 += pan[i * d + tid];
    }
    __syncthreads();
  }
  if (tid < d) mean[tid] = acc0 / (float)m;
  __syncthreads();
  const int ca = tid / d, cb = tid % d;
  const bool pair = tid < d * d && cb <= ca;
  acc0 = 0.0f;
  for (int i0 = 0; i0 < m; i0 += rows) {
    const int n = min(rows, m - i0);
    for (int q = tid; q < n * d; q += nt)
      pan[q] = (rows < m ? (float)P.live_u[(size_t)i0 * d + q] : pan[q]) - mean[q % d];
    __syncthreads();
    if (pair) {  // even points and odd ones
#pragma unroll 4
      for (int i = 0; i + 1 < n; i += 2) {
        acc0 = fmaf(pan[i * d + ca], pan[i * d + cb], acc0);
        acc1 = fmaf(pan[(i + 1) * d + ca], pan[(i + 1) * d + cb], acc1);
      }
      if (n & 1) acc0 = fmaf(pan[(n - 1) * d + ca], pan[(n - 1) * d + cb], acc0);
    }
    __syncthreads();
  }
  if (pair) {
    const float v = (acc0 + acc1) / (float)(m - 1);
    cov[ca * kMaxDim + cb] = v;
    cov[cb * kMaxDim + ca] = v;
  }
  __syncthreads();
  if (tid < S.n_blocks) {
    const int b = tid, nb = S.block_size[b];
    float* Lb = P.chol + (size_t)b * kMaxDim * kMaxDim;
    float tr = 0.0f;
    for (int r = 0; r < nb; ++r) tr += cov[S.block_dims[b][r] * kMaxDim + S.block_dims[b][r]];
    const float jitter = fmaxf(1e-6f * tr / (float)nb, 1e-30f);
    for (int r = 0; r < nb; ++r) {
      for (int q = 0; q <= r; ++q) {
        float s = cov[S.block_dims[b][r] * kMaxDim + S.block_dims[b][q]] + (r == q ? jitter : 0.0f);
        for (int p = 0; p < q; ++p) s -= Lb[r * kMaxDim + p] * Lb[q * kMaxDim + p];
        if (r == q)
          Lb[r * kMaxDim + r] = sqrtf(fmaxf(s, jitter));
        else
          Lb[r * kMaxDim + q] = s / Lb[q * kMaxDim + q];
      }
    }
  }
  __syncthreads();
  // chains: replace the c-th worst, start at a uniformly drawn survivor
  const long long it = g->iter;
  for (int c = tid; c < k; c += nt) {
    ChainState& ch = P.chains[c];
    const uint4 r = philox4x32_10(make_uint4(0u, (unsigned)c, (unsigned)it, 1u), S.key0, S.key1);
    int pick = (int)(u01_from(r) * (double)(m - k));
    pick = min(pick, m - k - 1);
    const int s = idx[k + pick];
    ch.slot = idx[c];
    for (int j = 0; j < d; ++j) ch.x[j] = P.live_u[(size_t)s * d + j];
    ch.lx = P.live_logl[s];
    for (int j = 0; j < 2 * SWIG_MAX_DET; ++j) ch.kap[j] = P.live_kap[(size_t)s * 2 * SWIG_MAX_DET + j];
    for (int i = 0; i < SWIG_MAX_DET; ++i) ch.vv[i] = P.live_vv[(size_t)s * SWIG_MAX_DET + i];
    prior_map(S.prior, ch.x, ch.th, &S.sky);
    setup_record(L, ch.th, &P.recx[c]);
    ch.proj_dirty = 0;
    ch.block = ch.step = ch.sweep = 0;
    ch.phase = PH_NEW;
    ch.pending = 0;
    ch.done = 0;
    ch.ctr = 0;
    ch.side = 0;
    ch.n_out_r = 0;
    P.pending[c] = 0;
    P.req[c] = 0;
    P.done_cnt[c] = 0;
  }
  __syncthreads();
  if (tid == 0) {
    g->chains_done = 0;
    g->iter = it + 1;
    g->iters_launch += 1;
    g->need_writeback = 1;
  }
}

static __device__ void ns_boundary(const LikeConst& L, const SamplerConst& S, const SamplerPtrs& P, unsigned char* smem) {
  if (ns_boundary_check(L, S, P, smem)) ns_boundary_advance(L, S, P, smem, 0);
}


}  // namespace swig
