// Persistent Slice-within-Gibbs nested sampler (Sec. 2.2, 2.3, 3.2 of the paper).
//
// One cooperative launch runs up to `max_iters` nested-sampling iterations on
// the device.  The grid meets at a barrier only around the iteration boundary:
//
//   boundary  (CTA 0, once per NS iteration): write the k finished chains back
//             into the live set, sort the live log-likelihoods, test the
//             termination rule log Z_live - log Z_dead < dlogz, retire the k
//             worst points into the dead buffer with weights L_j (X_{j-1} - X_j)
//             (log X shrinks by 1/n per death, n = m, m-1, ..., m-k+1), set
//             logL* to the lowest survivor, estimate the live covariance and
//             its per-block Cholesky factors, and start k chains at survivors.
//
// Within the iteration the mixed-precision and heterodyned runs have a CTA
// advance a chain (chain.cuh).  The FP64 run is a dataflow here (k_ns_flow):
// every CTA owns one slice of the frequency grid (its data staged once in shared
// memory), and
//
//   control   (warp 0 of the chain's home CTA): advance the chain's hit-and-run
//             slice state machine (Neal 2003 stepping-out and shrinkage along a
//             direction drawn from the block covariance, or a learned one)
//             through every proposal that needs no pass over the grid:
//             proposals outside the unit cube, and proposals of blocks that only
//             change the projection factors C_i (d_L, iota, psi, phi_c), which
//             reuse the chain's cached per-detector sums kappa_i.  A proposal
//             that changes the waveform or the time shifts is set up (one lane
//             per piece of the record) and published as a request.
//   sweep     (warps 1.. of every CTA): claim published requests and evaluate
//             the CTA's slice for them, one warp per (chain, slice), partial
//             sums per (chain, slice); the chain's control resumes when every
//             CTA has counted itself done.
//
// Every spin-wait is bounded; on expiry the kernel records SWIG_E_TIMEOUT and
// every CTA returns at its next barrier.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <climits>
#include <cstddef>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "chain.h"
#include "context.h"
#include "mlp.h"
#include "sampler.cuh"
#include "sweep.cuh"

namespace swig {

// ---------------------------------------------------------------------------
// Chain control.
// ---------------------------------------------------------------------------
// Outcome of evaluating the proposal y with log-likelihood ly.  Returns true
// when the shrinkage phase accepts y (the caller moves the chain there and
// then calls finish_step); stepping-out and rejections are handled here.
__device__ inline bool apply_result(const SamplerConst& S, ChainState& ch, double ly, double logl_star,
                                    NSGlobal* g) {
  const bool ok = ly > logl_star;
  switch (ch.phase) {
    case PH_LEFT:
      if (ok) {
        ch.lo -= 1.0;
        if (++ch.n_out >= kMaxStepOut) {
          ch.phase = PH_RIGHT;
          ch.n_out = 0;
        }
      } else {
        ch.phase = PH_RIGHT;
        ch.n_out = 0;
      }
      return false;
    case PH_RIGHT:
      if (ok) {
        ch.hi += 1.0;
        if (++ch.n_out >= kMaxStepOut) {
          ch.phase = PH_SHRINK;
          ch.n_shrink = 0;
        }
      } else {
        ch.phase = PH_SHRINK;
        ch.n_shrink = 0;
      }
      return false;
    default:  // PH_SHRINK
      if (ok) return true;
      if (ch.t < 0.0)
        ch.lo = ch.t;
      else
        ch.hi = ch.t;
      if (++ch.n_shrink >= kMaxShrink) {
        ++ch.n_caps;
        finish_step(S, ch, g);
      }
      return false;
  }
}

__device__ inline void move_to_proposal(const SamplerConst& S, ChainState& ch, double ly) {
  for (int j = 0; j < S.ndim; ++j) ch.x[j] = ch.y[j];
  for (int j = 0; j < SWIG_N_PARAMS; ++j) ch.th[j] = ch.th_y[j];
  ch.lx = ly;
}

// New slice step: direction from the live covariance (n = L_b z, Sec. 2.3),
// or, with probability learn_mix, the learned direction exp(s_b) u_b / |u_b|
// of a live point drawn uniformly from the frozen snapshot; then a bracket
// [-r, 1 - r] of unit width at a uniform offset.
__device__ inline void start_step(const SamplerConst& S, ChainState& ch, const float* chol, const float* learn_out,
                                  int c, long long it) {
  const int b = ch.block, nb = S.block_size[b];
  for (int j = 0; j < S.ndim; ++j) ch.dir[j] = 0.0;
  bool learned = false;
  if (S.learn_on && learn_out && chain_uniform(S, ch, c, it) < (double)S.learn_mix) {
    const int row = min((int)(chain_uniform(S, ch, c, it) * (double)S.nlive), S.nlive - 1);
    const float* o = learn_out + (size_t)row * 32;
    float nrm2 = 0.0f;
    for (int r = 0; r < nb; ++r) {
      const float u = o[S.block_dims[b][r]];
      nrm2 = fmaf(u, u, nrm2);
    }
    const float inv = rsqrtf(nrm2 + 1e-12f);
    for (int r = 0; r < nb; ++r) {
      const int j = S.block_dims[b][r];
      const float s = fminf(fmaxf(o[13 + j], -30.0f), 5.0f);
      ch.dir[j] = (double)(expf(s) * o[j] * inv);
    }
    learned = true;
  }
  if (!learned) {
    float z[kMaxDim];
    for (int j = 0; j < nb; ++j) z[j] = chain_normal(S, ch, c, it);
    const float* Lb = chol + (size_t)b * kMaxDim * kMaxDim;
    for (int r = 0; r < nb; ++r) {
      float v = 0.0f;
      for (int q = 0; q <= r; ++q) v = fmaf(__ldcg(&Lb[r * kMaxDim + q]), z[q], v);
      ch.dir[S.block_dims[b][r]] = (double)v;
    }
  }
  const double r0 = chain_uniform(S, ch, c, it);
  ch.lo = -r0;
  ch.hi = 1.0 - r0;
  ch.phase = PH_LEFT;
  ch.n_out = 0;
  ch.n_shrink = 0;
}

// Advance chain c through the proposals that need no grid pass (outside the
// unit cube, or projection-only blocks, at most kFreeBudget of the latter per
// round) and leave the first full-likelihood proposal pending with its setup
// record in *rec.  Only the Gibbs block's slots are transformed and only the
// pieces of the record that the block moves are recomputed.  Lane 0 only.
__device__ __noinline__ void chain_advance_local(const LikeConst& L, const SamplerConst& S, const SamplerPtrs& P, int c,
                                    const double* kap_in, const double* vv_in, double ly_in, ChainState& ch,
                                    EvalRecord& rx, bool& rx_dirty, EvalRecord& rec, bool& rec_set,
                                    int& setup_fl) {
  NSGlobal* g = P.g;
  // written by CTA 0 at the boundary: read through L2, never a stale L1 line
  const double logl_star = __ldcg(&g->logl_star);
  const long long it = __ldcg(&g->iter);
  if (ch.done) return;
  const bool prof = (c == 0);
  long long tk = clock64();
  unsigned long long acc_res = 0, acc_step = 0, acc_prop = 0, acc_free = 0, acc_setup = 0, cnt_free = 0, cnt_setup = 0,
                     cnt_step = 0;
  struct Flush {
    NSGlobal* g;
    bool on;
    unsigned long long *a0, *a1, *a2, *a3, *a4, *n0, *n1, *n2;
    __device__ ~Flush() {
      if (!on) return;
      g->c_result += *a0;
      g->c_step += *a1;
      g->c_prop += *a2;
      g->c_free += *a3;
      g->c_setup += *a4;
      g->n_free += *n0;
      g->n_setup += *n1;
      g->n_step += *n2;
    }
  } flush{g, prof, &acc_res, &acc_step, &acc_prop, &acc_free, &acc_setup, &cnt_free, &cnt_setup, &cnt_step};
  if (ch.pending) {
    ch.pending = 0;
    ++ch.n_full;
    ++ch.n_evals;
    if (apply_result(S, ch, ly_in, logl_star, g)) {
      move_to_proposal(S, ch, ly_in);
      for (int j = 0; j < 2 * SWIG_MAX_DET; ++j) ch.kap[j] = kap_in[j];
      if (vv_in)
        for (int i = 0; i < SWIG_MAX_DET; ++i) ch.vv[i] = vv_in[i];
      rx = rec;
      rx_dirty = true;
      ch.proj_dirty = 0;
      finish_step(S, ch, g);
    }
  }
  if (prof) {
    const long long t2 = clock64();
    acc_res += t2 - tk;
    tk = t2;
  }
  int free_left = kFreeBudget;
  for (int guard = 0; guard < 1 << 20 && !ch.done; ++guard) {
    const int b = ch.block;
    if (S.block_free[b] && free_left <= 0) return;  // resume next round
    if (ch.phase == PH_NEW) {
      start_step(S, ch, P.chol, P.learn_out, c, it);
      if (prof) {
        const long long t2 = clock64();
        acc_step += t2 - tk;
        cnt_step += 1;
        tk = t2;
      }
    }
    double t;
    if (ch.phase == PH_LEFT)
      t = ch.lo;
    else if (ch.phase == PH_RIGHT)
      t = ch.hi;
    else
      t = ch.lo + (ch.hi - ch.lo) * chain_uniform(S, ch, c, it);
    ch.t = t;
    const int nb = S.block_size[b];
    bool inside = true;
    for (int r = 0; r < nb; ++r) {
      const int j = S.block_dims[b][r];
      const double v = ch.x[j] + t * ch.dir[j];
      ch.y[j] = v;
      inside = inside && (v >= 0.0) && (v <= 1.0);
    }
    if (!inside) {
      apply_result(S, ch, -INFINITY, logl_star, g);
      continue;
    }
    for (int j = 0; j < S.ndim; ++j)
      if (ch.dir[j] == 0.0) ch.y[j] = ch.x[j];
    for (int q = 0; q < SWIG_N_PARAMS; ++q) ch.th_y[q] = ch.th[q];
    bool sky_block = false;
    for (int r = 0; r < nb; ++r) {
      const int j = S.block_dims[b][r], slot = S.slot_of_dim[j];
      ch.th_y[slot] = prior_slot_inverse(S.prior[slot], ch.y[j]);
      sky_block = sky_block || slot == 9 || slot == 10;
    }
    if (S.sky.on && sky_block) sky_frame_to_radec(S.sky, ch.th_y[9], ch.th_y[10], &ch.th_y[9], &ch.th_y[10]);
    if (prof) {
      const long long t2 = clock64();
      acc_prop += t2 - tk;
      tk = t2;
    }
    if (S.block_free[b]) {
      --free_left;
      ++ch.n_evals;
      {
        EvalRecord tmp = rx;
        tmp.valid = theta_valid(ch.th_y) ? 1 : 0;
        setup_amp(ch.th_y, &tmp);
        setup_projection(L, ch.th_y, &tmp);
        setup_combine(L, &tmp);
        double kre[SWIG_MAX_DET], kim[SWIG_MAX_DET];
        for (int i = 0; i < SWIG_MAX_DET; ++i) {
          kre[i] = ch.kap[2 * i];
          kim[i] = ch.kap[2 * i + 1];
        }
        const double ly = loglike_epilogue(L, tmp, kre, kim);
        if (apply_result(S, ch, ly, logl_star, g)) {
          move_to_proposal(S, ch, ly);
          rx = tmp;
          rx_dirty = true;
          finish_step(S, ch, g);
        }
        if (prof) {
          const long long t2 = clock64();
          acc_free += t2 - tk;
          cnt_free += 1;
          tk = t2;
        }
      }
      continue;
    }
    rec = rx;
    setup_fl = S.block_flags[b] | (ch.proj_dirty ? (BF_AMP | BF_PROJ) : 0);
    rec.valid = theta_valid(ch.th_y) ? 1 : 0;
    rec_set = true;
    ch.pending = 1;
    P.pending[c] = 1;
    if (prof) {
      acc_setup += clock64() - tk;
      cnt_setup += 1;
    }
    return;
  }
}

// Chain control on local copies of the chain state and records (local
// memory is cached in L1; the global copies are read and written once).
// Lane 0 only.  Returns the set-up flags of the new pending proposal (its
// record in *rec_out still holds the current point's values for the pieces
// the block moves), or -1 when nothing is pending.
__device__ __noinline__ int chain_advance(const LikeConst& L, const SamplerConst& S, const SamplerPtrs& P, int c,
                                          const double* kap_in, double ly_in, EvalRecord* rec_out,
                                          const double* vv_in = nullptr) {
  if (P.chains[c].done) return -1;
  ChainState ch = P.chains[c];
  EvalRecord rx = P.recx[c];
  EvalRecord rec;
  if (ch.pending) rec = *rec_out;
  bool rx_dirty = false, rec_set = false;
  int fl = -1;
  chain_advance_local(L, S, P, c, kap_in, vv_in, ly_in, ch, rx, rx_dirty, rec, rec_set, fl);
  P.chains[c] = ch;
  if (rx_dirty) P.recx[c] = rx;
  if (rec_set) *rec_out = rec;
  return fl;
}

// The set-up of a pending proposal's record, one piece per lane: lane 0 the
// waveform coefficients (all, or only spin / tidal ones), lane 1 the
// amplitude, lanes 2.. the projection of each detector, lanes 8.. the time
// shift of each detector; then one lane per coefficient splits it into a
// double-float and one lane per detector forms C_i (lane 0 adds <h|h> in
// detector order).  All 32 lanes call it with the same fl (>= 0) and th (the
// proposal's theta).
__device__ __noinline__ void setup_record_warp(const LikeConst& L, const double* th, int fl, bool f32,
                                               EvalRecord* rec, int lane) {
  const bool valid = rec->valid != 0;
  // a sky move: the two FP64 sines/cosines of the delays on lanes 0 and 1 at
  // once (one call's latency), shared with the delay lanes
  double sl = 0.0, cl = 0.0, sd = 0.0, cd = 0.0;
  if (valid && (fl & BF_SKY)) {  // warp-uniform
    double sv, cv;
    sincos((lane & 1) ? th[10] : th[9] - L.gmst, &sv, &cv);
    sl = __shfl_sync(0xffffffffu, sv, 0);
    cl = __shfl_sync(0xffffffffu, cv, 0);
    sd = __shfl_sync(0xffffffffu, sv, 1);
    cd = __shfl_sync(0xffffffffu, cv, 1);
  }
  if (valid) {
    if (lane == 0) {
      if (fl & BF_INTR)
        setup_intrinsic(th, rec, false);
      else if (fl & (BF_SPIN | BF_TIDE))
        setup_intrinsic_partial(th, rec, (fl & BF_SPIN) != 0, (fl & BF_TIDE) != 0, false);
    } else if (lane == 1) {
      if (fl & BF_AMP) {
        if (f32)
          setup_amp_f32(th, rec);
        else
          setup_amp(th, rec);
      }
    } else if (lane >= 2 && lane < 2 + L.n_det) {
      if (fl & BF_PROJ) setup_projection_det(L, th, lane - 2, f32, rec);
    } else if (lane >= 8 && lane < 8 + L.n_det) {
      if (fl & BF_SKY)
        setup_delay_det_sc(L, th, lane - 8, sl, cl, sd, cd, rec);
      else if (fl & BF_TAU)
        setup_tc_det(th, lane - 8, rec);
    }
  } else if (lane == 0) {
    // invalid proposal: the record only has to say so (logL = -inf)
    rec->amp = 0.0;
  }
  __syncwarp();
  if (valid && (fl & (BF_INTR | BF_SPIN | BF_TIDE)) && lane < NBASIS) {
    const dfl v = df_from_double(rec->c[lane]);
    rec->c_hi[lane] = v.hi;
    rec->c_lo[lane] = v.lo;
  }
  double term = 0.0;
  if (lane < SWIG_MAX_DET) {
    const double cre = rec->amp * rec->pre[lane], cim = rec->amp * rec->pim[lane];
    rec->cre[lane] = cre;
    rec->cim[lane] = cim;
    if (lane < L.n_det) term = (cre * cre + cim * cim) * L.K[lane];
  }
  double hh = 0.0;
#pragma unroll
  for (int i = 0; i < SWIG_MAX_DET; ++i) hh += __shfl_sync(0xffffffffu, term, i);
  if (lane == 0) rec->hh = hh;
  __syncwarp();
}

// ---------------------------------------------------------------------------
// The persistent kernel, dataflow form.  Within an NS iteration nothing
// waits on a grid-wide barrier: warp 0 of each CTA runs the control of the
// chains homed there, and publishes each full-likelihood request by bumping
// the chain's sequence number after writing its record; warps 1.. of every
// CTA claim (chain, request) pairs as they appear and evaluate the CTA's
// slice of the grid for them (one warp per pair), then count themselves in
// done_cnt.  A chain's control resumes once all CTAs have counted.  The
// per-slice sums are written in a fixed place and added over slices in a
// fixed order, so results do not depend on timing.  Every wait is bounded.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(int* p, int v) {
  asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Copy the part of a record that a sweep unit reads (the double-float phase
// coefficients and the time shifts: one contiguous run of words), written by
// another SM, into shared memory (through L2).
static_assert(offsetof(EvalRecord, c_lo) > offsetof(EvalRecord, c_hi) &&
                  offsetof(EvalRecord, tau) > offsetof(EvalRecord, c_lo) &&
                  offsetof(EvalRecord, tau_hi) > offsetof(EvalRecord, tau) &&
                  offsetof(EvalRecord, tau_lo) > offsetof(EvalRecord, tau_hi),
              "the sweep's fields of EvalRecord are one run");
// The FP64 sweep also reads the FP64 coefficients c, which precede that run.
__device__ __forceinline__ void load_record_cg(const EvalRecord* src, EvalRecord* dst, int lane) {
  static_assert(offsetof(EvalRecord, c) == 0, "c leads the record");
  constexpr int w1 = (int)((offsetof(EvalRecord, tau_lo) + sizeof(float) * SWIG_MAX_DET) / 4);
  const unsigned* s = reinterpret_cast<const unsigned*>(src);
  unsigned* d = reinterpret_cast<unsigned*>(dst);
  for (int w = lane; w < w1; w += 32) d[w] = __ldcg(s + w);
  __syncwarp();
}

// done_cnt += v with release semantics (orders the unit's partial writes,
// made visible to lane 0 by the preceding __syncwarp, before the count).
__device__ __forceinline__ void red_release_add(int* p, int v) {
  asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// One control step of chain c by a whole warp: add the slice partials of the
// finished request (fixed order), advance the chain's slice state machine and,
// when it needs a full likelihood, set up its record and publish the request.
// Returns true while the chain needs another control step right away
// (projection-only budget used up), false once it waits for a request or is
// done.
template <int NDET>
__device__ bool flow_control(const LikeConst& L, const SamplerConst& S, const DeviceBuffers& B, const SamplerPtrs& P,
                             int c, int lane) {
  NSGlobal* g = P.g;
  double kap_y[2 * SWIG_MAX_DET];
#pragma unroll
  for (int j = 0; j < 2 * SWIG_MAX_DET; ++j) kap_y[j] = 0.0;
  double ly = 0.0;
  const bool pend = P.chains[c].pending != 0;
  if (pend) {
    double acc[2 * SWIG_MAX_DET];
#pragma unroll
    for (int j = 0; j < 2 * SWIG_MAX_DET; ++j) acc[j] = 0.0;
    const int n_units = L.n_slices * S.flow_parts;
    for (int s2 = lane; s2 < n_units; s2 += 32) {
#pragma unroll
      for (int j = 0; j < 2 * NDET; ++j)
        acc[j] += __ldcg(&B.partials64[((size_t)c * n_units + s2) * kPartialStride + j]);
    }
#pragma unroll
    for (int j = 0; j < 2 * NDET; ++j)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], o);
#pragma unroll
    for (int j = 0; j < 2 * SWIG_MAX_DET; ++j) kap_y[j] = acc[j];
    if (lane == 0) {
      double kre[SWIG_MAX_DET], kim[SWIG_MAX_DET];
      for (int i = 0; i < SWIG_MAX_DET; ++i) {
        kre[i] = kap_y[2 * i];
        kim[i] = kap_y[2 * i + 1];
      }
      ly = loglike_epilogue(L, B.rec[c], kre, kim);
    }
  }
  int fl = -1, done = 0;
  if (lane == 0) {
    if (pend) P.pending[c] = 0;
    fl = chain_advance(L, S, P, c, kap_y, ly, &B.rec[c]);
    done = P.chains[c].done;
  }
  fl = __shfl_sync(0xffffffffu, fl, 0);
  done = __shfl_sync(0xffffffffu, done, 0);
  __syncwarp();
  if (fl >= 0) {
    const long long ts = clock64();
    setup_record_warp(L, P.chains[c].th_y, fl, false, &B.rec[c], lane);
    if (lane == 0) {
      if (c == 0) g->c_setup += clock64() - ts;
      P.done_cnt[c] = 0;
      __threadfence();
      // sequence number and unit width in one word (one unit per slice)
      st_release(&P.req[c], (((P.req[c] >> 3) + 1) << 3) | S.flow_parts);
    }
    __syncwarp();
    return false;
  }
  return !done;
}


template <int NDET>
__global__ void __launch_bounds__(kFlowThreads, 1)
    k_ns_flow(LikeConst L, SamplerConst S, DeviceBuffers B, SamplerPtrs P) {
  extern __shared__ __align__(16) unsigned char dyn[];  // per-warp records, or sort buffers (boundary)
  const int slice = blockIdx.x;
  const int b0 = B.slice_begin[slice], b1 = B.slice_begin[slice + 1];
  const int nb = b1 - b0;
  const int tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  NSGlobal* g = P.g;
  EvalRecord* rec = reinterpret_cast<EvalRecord*>(dyn) + warp;
  int* s_claim = reinterpret_cast<int*>(dyn + S.claim_off);  // per request slot: units this CTA has taken
  const int G = S.flow_parts;
  const int target = S.n_ctas * G;  // units per request: G parts of every slice

  const bool timer = blockIdx.x == 0 && tid == 0;
  unsigned long long t0 = gtimer(), t1;
  for (;;) {
    if (!grid_sync(g, S.n_ctas, S.spin_limit)) return;
    if (timer) {
      t1 = gtimer();
      g->t_wait_sweep += t1 - t0;
      t0 = t1;
      g->rounds += 1;
    }
    if (blockIdx.x == 0) ns_boundary(L, S, P, dyn);
    for (int c = tid; c < S.nrep; c += blockDim.x) s_claim[c] = 0;
    if (!grid_sync(g, S.n_ctas, S.spin_limit)) return;
    if (timer) {
      t1 = gtimer();
      g->t_bound += t1 - t0;
      t0 = t1;
    }
    if (*(volatile int*)&g->status != ST_RUNNING) return;

    long long idle = 0;
    unsigned long long my_units = 0, my_unit_cyc = 0, my_idle_cyc = 0, my_ctrl_cyc = 0;
    long long tpoll = clock64();
    if (warp == 0) {
      // ---- control of the chains homed on this CTA (one lane, state in
      // global memory).  A chain is ready when every CTA finished its request
      for (;;) {
        bool all_done = true, progressed = false;
        for (int c = blockIdx.x; c < S.nrep; c += S.n_ctas) {
          int st = 0;  // 0 done, 1 waiting, 2 ready
          if (lane == 0) {
            const ChainState* ch = &P.chains[c];
            if (ch->done)
              st = 0;
            else if (ch->pending)
              st = ld_acquire(&P.done_cnt[c]) >= target ? 2 : 1;
            else
              st = 2;
          }
          st = __shfl_sync(0xffffffffu, st, 0);
          if (st == 0) continue;
          all_done = false;
          if (st == 1) continue;
          progressed = true;
          const long long tc0 = clock64();
          flow_control<NDET>(L, S, B, P, c, lane);
          my_ctrl_cyc += clock64() - tc0;
        }
        if (all_done) break;
        if (*(volatile int*)&g->error) break;
        if (progressed) {
          idle = 0;
        } else {
          if (++idle > S.spin_limit) {
            if (lane == 0) atomicCAS(&g->error, 0, SWIG_E_TIMEOUT);
            break;
          }
          __nanosleep(64);
        }
      }
    } else {
      // ---- sweep: claim (chain, request, part) units, lowest chain first,
      // and evaluate that part of this CTA's slice, one warp per unit (the G
      // parts of a request may run on G warps at once)
      for (;;) {
        if (*(volatile int*)&g->chains_done >= S.nrep) break;
        if (*(volatile int*)&g->error) break;
        // s_claim[c] = units of chain c this CTA has taken: request r owns
        // units (r - 1) G .. r G - 1, one per part
        int cc = -1, part = 0;
        int rq[4];  // request words of four groups of 32 slots, read together
        for (int base = 0; base < S.nrep && cc < 0; base += 32) {
          const int c = base + lane;
          const int gq = (base >> 5) & 3;
          if (gq == 0) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
              rq[q] = base + 32 * q + lane < S.nrep ? *(volatile int*)&P.req[base + 32 * q + lane] : 0;
          }
          int r = 0;
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (q == gq) r = rq[q] >> 3;
          bool cand = false;
          if (c < S.nrep) cand = r * G > *(volatile int*)&s_claim[c];
          unsigned m = __ballot_sync(0xffffffffu, cand);
          while (m) {
            const int leader = __ffs(m) - 1;
            int won = 0, pt = 0;
            if (lane == leader) {
              const int old = *(volatile int*)&s_claim[c];
              if (old < r * G) {
                const int nv = max(old, (r - 1) * G) + 1;
                won = atomicCAS(&s_claim[c], old, nv) == old;
                pt = nv - 1 - (r - 1) * G;
              }
            }
            if (__shfl_sync(0xffffffffu, won, leader)) {
              cc = base + leader;
              part = __shfl_sync(0xffffffffu, pt, leader);
              break;
            }
            m &= ~(1u << leader);
          }
        }
        if (cc < 0) {
          if (++idle > S.spin_limit) {
            if (lane == 0) atomicCAS(&g->error, 0, SWIG_E_TIMEOUT);
            break;
          }
          __nanosleep(100);
          continue;
        }
        idle = 0;
        const long long tu0 = clock64();
        my_idle_cyc += tu0 - tpoll;
        __threadfence();  // acquire: the request word was read relaxed
        load_record_cg(&B.rec[cc], rec, lane);
        {
          const int lo = (int)(((long long)nb * part) / G), hi = (int)(((long long)nb * (part + 1)) / G);
          const size_t pidx = (((size_t)cc * L.n_slices + slice) * G + part) * kPartialStride;
          sweep_warp_fp64<NDET>(L, B.data64, B.ftab, b0 + lo, b0 + hi, *rec, lane, B.partials64 + pidx);
        }
        __syncwarp();
        if (lane == 0) red_release_add(&P.done_cnt[cc], 1);
        tpoll = clock64();
        my_units += 1;
        my_unit_cyc += tpoll - tu0;
      }
    }
    my_idle_cyc += clock64() - tpoll;
    if (blockIdx.x == 0 && lane == 0) {
      atomicAdd(&g->f_units, my_units);
      atomicAdd(&g->f_unit_cyc, my_unit_cyc);
      atomicAdd(&g->f_idle_cyc, my_idle_cyc);
    }
    if (lane == 0 && P.cta_prof) {
      unsigned long long* cp = P.cta_prof + 4 * (size_t)blockIdx.x;
      if (warp == 0) {
        atomicAdd(cp + 3, my_ctrl_cyc);
      } else {
        atomicAdd(cp + 0, my_units);
        atomicAdd(cp + 1, my_unit_cyc);
        atomicAdd(cp + 2, my_idle_cyc);
      }
    }
    __syncthreads();
    if (timer) {
      t1 = gtimer();
      g->t_ctrl += t1 - t0;
      t0 = t1;
    }
  }
}

// Initial live set: m unit-cube draws (Philox, stream tag 2) and their theta.
__global__ void k_init_live(SamplerConst S, double* live_u, double* theta) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= S.nlive) return;
  double u[kMaxDim];
  for (int j = 0; j < S.ndim; ++j) {
    const uint4 r = philox4x32_10(make_uint4((unsigned)j, (unsigned)i, 0xFFFFFFFFu, 2u), S.key0, S.key1);
    u[j] = u01_from(r);
    live_u[(size_t)i * S.ndim + j] = u[j];
  }
  prior_map(S.prior, u, theta + (size_t)i * SWIG_N_PARAMS, &S.sky);
}

__global__ void k_dead_theta(SamplerConst S, const double* u, int n, double* theta) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) prior_map(S.prior, u + (size_t)i * S.ndim, theta + (size_t)i * SWIG_N_PARAMS, &S.sky);
}

// ---------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------
struct SamplerState {
  SamplerPtrs P = {};
  double* harm = nullptr;
  double* lw = nullptr;
  double* init_theta = nullptr;
  ChainEvent* ev = nullptr;  // chain sampler: the run as its kernel reads it
  unsigned long long* cta_prof = nullptr;  // [n_ctas][4]
  int cta_prof_n = 0;
  int cap_iters = 0;
  int nlive = 0, nrep = 0, ndim = 0;
};

namespace {

template <typename T>
void dfree(T*& p) {
  if (p) cudaFree(p);
  p = nullptr;
}

void release(SamplerState* s) {
  if (!s) return;
  dfree(s->P.live_u);
  dfree(s->P.live_logl);
  dfree(s->P.live_kap);
  dfree(s->P.live_vv);
  dfree(s->P.chains);
  dfree(s->P.recx);
  dfree(s->P.pending);
  dfree(s->P.req);
  dfree(s->P.done_cnt);
  dfree(s->P.chol);
  dfree(s->P.g);
  dfree(s->P.dead_u);
  dfree(s->P.dead_logl);
  dfree(s->P.dead_logw);
  dfree(s->harm);
  dfree(s->lw);
  dfree(s->init_theta);
  dfree(s->ev);
  dfree(s->cta_prof);
}

int fail(swig_ctx* c, int code, const std::string& m) {
  c->err = m;
  return code;
}

#define SCUDA(call)                                                                                        \
  do {                                                                                                     \
    cudaError_t e_ = (call);                                                                               \
    if (e_ != cudaSuccess)                                                                                 \
      return fail(c, e_ == cudaErrorMemoryAllocation ? SWIG_E_NOMEM : SWIG_E_CUDA,                         \
                  std::string(#call) + ": " + cudaGetErrorString(e_));                                     \
  } while (0)

void* pick_flow_kernel(int n_det) {
  switch (n_det) {
    case 1: return (void*)k_ns_flow<1>;
    case 2: return (void*)k_ns_flow<2>;
    case 3: return (void*)k_ns_flow<3>;
    default: return (void*)k_ns_flow<4>;
  }
}

}  // namespace
}  // namespace swig

using namespace swig;

void swig_sampler_release(swig_ctx* c) {
  if (c && c->sampler) {
    release(c->sampler);
    delete c->sampler;
    c->sampler = nullptr;
  }
}

extern "C" {

int swig_set_wait_limit(swig_ctx* c, long long spins) {
  if (!c) return SWIG_E_ARG;
  if (spins < 0) return fail(c, SWIG_E_ARG, "wait limit must be >= 0");
  c->wait_limit = spins;
  return SWIG_OK;
}

}  // extern "C"

namespace swig {
namespace {

// Host state of one sampler run between its set-up and its result.
struct RunState {
  SamplerConst S;
  SamplerState* st = nullptr;
  size_t smem = 0;
  int mode = 0;          // ChainMode
  ChainLayout lay = {};  // chain sampler
  void* kern = nullptr;
  int threads = 0;
  bool het = false, mixed = false, learned = false;
  int m = 0, k = 0, nd = 0;
  float learn_lr = 0.0f;
  int learn_steps = 0;
  std::vector<double> du, dl, dw;
  NSGlobal gh, gl;  // after a launch; as uploaded before one (the copies read it)
  long long total_iters = 0;
  double persistent_ms = 0.0, learn_ms = 0.0;
  long long persistent_launches = 0, learn_rounds = 0;
  bool finished = false;
  std::chrono::steady_clock::time_point t_start;
};

}  // namespace
}  // namespace swig

using namespace swig;

namespace {

// Shared memory of the samplers' stated problem size (refused beyond 220 KB):
// full grid in mixed precision, a slice of the weighted data and its tiles'
// anchors for 16 warps; heterodyned, the chunks' anchors and the time pass.
size_t stated_bytes(const swig_ctx* c, bool mixed, bool het, int k, size_t sort_bytes) {
  const LikeConst& L = c->L;
  auto up = [](size_t v) { return (v + 15) & ~(size_t)15; };
  const size_t state = sizeof(ChainState) + sizeof(EvalRecord);
  if (het) {
    const size_t tm = L.tm_n > 0 ? het_tm_smem_bytes(c->B.het_nb, L.tm_M, L.tm_M > 0 ? L.tm_pieces : 0) : 0;
    return up(up(std::max(sort_bytes, tm)) + state) + sizeof(float) * kHetAncStride * (size_t)c->B.het_nc;
  }
  const size_t tail = up(std::max((size_t)(kFlowThreads / 32) * sizeof(EvalRecord), sort_bytes));
  if (!mixed) return tail + sizeof(int) * (size_t)k;
  const int tiles = c->B.max_slice_tiles;
  const size_t data = up((size_t)c->B.max_slice_bins * (L.n_det * sizeof(float2) + sizeof(int)));
  const size_t rows = up(tiles * sizeof(TileInfo)) + up((size_t)16 * tiles * kAnchorStride * sizeof(float));
  const size_t slots = (k + L.n_slices - 1) / L.n_slices;
  return data + rows + up(tail + slots * state) + sizeof(int) * 2 * (size_t)k;
}

// Validation, preparation, sampler constants, buffers, the initial live set
// and the NS state: everything before the first persistent launch.
int run_setup(swig_ctx* c, RunState& R) {
  if (!c->prior_set) return fail(c, SWIG_E_STATE, "prior not set");
  if (!c->cfg_set) return fail(c, SWIG_E_STATE, "sampler not configured");
  if (c->cfg.nlive > kMaxSort) return fail(c, SWIG_E_ARG, "nlive must be <= 8192 for the device sort");
  if (c->cfg.nrep > kMaxChains) return fail(c, SWIG_E_ARG, "nrep must be <= 2048");
  int rc = prepare(c);
  if (rc) return rc;
  R.t_start = std::chrono::steady_clock::now();
  const StreamDrain drain{c->stream};
  const bool het = c->prepared_like == SWIG_LIKE_HET;
  const bool mixed = !het && c->prepared_precision == SWIG_PREC_MIXED;
  R.het = het;
  R.mixed = mixed;
  const int m = c->cfg.nlive, k = c->cfg.nrep;
  R.m = m;
  R.k = k;
  const LikeConst& L = c->L;
  if (!het && k > 32 * L.n_slices) return fail(c, SWIG_E_ARG, "nrep exceeds 32 chains per CTA");
  const int chain_ctas = std::max(1, std::min(c->sm_count, k));

  SamplerConst& S = R.S;
  std::memset(&S, 0, sizeof(S));
  S.nlive = m;
  S.nrep = k;
  S.sweeps = c->cfg.sweeps;
  S.steps_per_dim = c->cfg.steps_per_dim;
  S.dlogz = c->cfg.dlogz;
  S.key0 = (unsigned)(c->cfg.seed & 0xFFFFFFFFu);
  S.key1 = (unsigned)(c->cfg.seed >> 32);
  S.n_ctas = het || mixed ? chain_ctas : L.n_slices;
  S.spin_limit = c->wait_limit;
  if ((rc = make_sky_frame(c, &S.sky))) return rc;
  int nd = 0;
  for (int i = 0; i < SWIG_N_PARAMS; ++i) {
    const swig_param& p = c->params[i];
    S.prior[i] = make_prior_slot(p.kind, p.mode, p.lo, p.hi, p.value);
    if (p.mode == SWIG_MODE_SAMPLE) S.slot_of_dim[nd++] = i;
  }
  S.ndim = nd;
  R.nd = nd;
  // Gibbs blocks in increasing block id
  int ids[kMaxDim], n_ids = 0;
  for (int j = 0; j < nd; ++j) {
    const int b = c->params[S.slot_of_dim[j]].block;
    bool seen = false;
    for (int q = 0; q < n_ids; ++q) seen = seen || ids[q] == b;
    if (!seen) ids[n_ids++] = b;
  }
  std::sort(ids, ids + n_ids);
  S.n_blocks = n_ids;
  for (int b = 0; b < n_ids; ++b) {
    S.block_size[b] = 0;
    bool free_block = true;
    int flags = 0;
    for (int j = 0; j < nd; ++j)
      if (c->params[S.slot_of_dim[j]].block == ids[b]) {
        S.block_dims[b][S.block_size[b]++] = j;
        const int slot = S.slot_of_dim[j];
        free_block = free_block && (slot == 6 || slot == 7 || slot == 8 || slot == 12);
        if (slot <= 1) flags |= BF_INTR;
        if (slot == 2 || slot == 3) flags |= BF_SPIN;
        if (slot == 4 || slot == 5) flags |= BF_TIDE;
        if (slot == 0 || slot == 6) flags |= BF_AMP;
        if (slot == 7 || slot == 8 || slot == 9 || slot == 10 || slot == 12) flags |= BF_PROJ;
        if (slot == 9 || slot == 10 || slot == 11) flags |= BF_TAU;
        if (slot == 9 || slot == 10) flags |= BF_SKY;
      }
    // time marginalisation keeps no per-detector cache at every node, so
    // projection-only blocks take the full evaluation there (and everywhere
    // when the cache is switched off)
    S.block_free[b] = (free_block && L.tm_n == 0 && !c->cfg.cache_off) ? 1 : 0;
    S.block_flags[b] = flags;
    S.block_mask[b] = 0u;
    for (int r = 0; r < S.block_size[b]; ++r) {
      S.block_mask[b] |= 1u << S.block_dims[b][r];
      S.block_rank[S.block_dims[b][r]] = r;
    }
  }
  S.m_pow2 = 1;
  while (S.m_pow2 < m) S.m_pow2 *= 2;
  S.max_iters = (int)std::max(1, std::min(64, c->cfg.max_iter));
  // FP64: the parts of a request's slice, each with its own partial (at most 4:
  // the partial buffers hold 4 per slice and theta)
  S.flow_parts = c->cfg.flow_parts > 0 ? c->cfg.flow_parts : SWIG_FLOW_PARTS;
  // chain sampler: candidates per round (chain.cuh).  Four rungs per end and
  // two draws unless a smaller launch shape is asked for (first iterations of the
  // 128 s run, ms: (rungs, draws) = (4, 2) 12.8, (4, 3) 13.1, (4, 4) 13.3, (4, 8)
  // 13.6, (3, 3) 14.4, (2, 4) 16.5; heterodyned 38.8, 39.1, 38.9, 40.2, 42.2, 47.9);
  // with t_c marginalised
  // an evaluation costs as much as a round's latency: one at a time
  const int shape = c->cfg.flow_parts;
  S.spec_out = L.tm_n > 0 ? 1 : shape >= 3 ? 1 : shape == 2 ? 2 : 4;
  S.spec_shr = L.tm_n > 0 ? 1 : shape >= 4 ? 1 : 2;
  S.spec_mix = L.tm_n > 0 ? 0 : S.spec_shr;
  S.one_end = c->cfg.stepout_one_end ? 1 : 0;
  // learned proposal: retrain every learn_interval iterations (one launch each)
  R.learned = c->cfg.proposal == SWIG_PROPOSAL_LEARNED;
  const double learn_mix = c->cfg.learn_mix > 0.0 ? std::min(1.0, c->cfg.learn_mix) : 0.5;
  R.learn_lr = c->cfg.learn_lr > 0.0 ? (float)c->cfg.learn_lr : 1e-3f;
  R.learn_steps = c->cfg.learn_steps > 0 ? c->cfg.learn_steps : 50;
  const int learn_interval = c->cfg.learn_interval > 0 ? c->cfg.learn_interval : 8;
  if (R.learned) {
    if (2 * nd >= m) return fail(c, SWIG_E_ARG, "the learned proposal needs nlive > 2 x sampled dimensions");
    S.max_iters = std::min(S.max_iters, learn_interval);
    S.learn_on = 1;
    S.learn_mix = (float)learn_mix;
  }

  const size_t sort_bytes = (size_t)S.m_pow2 * (sizeof(double) + sizeof(int)) + kSweepThreads * sizeof(double) +
                            (size_t)k * sizeof(double) + (kMaxDim + kMaxDim * kMaxDim) * sizeof(float) + 64;
  if (const size_t need = stated_bytes(c, mixed, het, k, sort_bytes); need > 220 * 1024)
    return fail(c, SWIG_E_ARG, "problem too large for the persistent kernel's shared memory");
  if (mixed || het) {
    R.mode = mixed ? CHAIN_FOLD : L.tm_n > 0 ? CHAIN_HET_TM : CHAIN_HET;
    ChainLayout& y = R.lay;
    std::memset(&y, 0, sizeof(y));
    y.scratch_off = (int)chain_fixed_bytes(L.n_det, R.mode);
    size_t scratch = sort_bytes;
    if (R.mode == CHAIN_FOLD) {
      // anchors of eight candidates over every chunk, at least of 64 chunks
      scratch = std::max(scratch, sizeof(float) * kFoldAnchorFloats * 8 * (size_t)std::min(c->B.fold_nc, 128));
    } else if (R.mode == CHAIN_HET) {
      scratch = std::max(scratch, sizeof(float) * kHetAncPair * 4 * (size_t)std::max(32, std::min(c->B.het_nc, 256)));
    } else {
      const HetTmLayout lay = het_tm_layout(L, c->B);
      y.anc_off = lay.anc_off;
      y.panel = lay.panel;
      scratch = std::max(scratch, lay.bytes);
    }
    y.scratch_bytes = (int)((scratch + 15) & ~(size_t)15);
    R.smem = (size_t)y.scratch_off + y.scratch_bytes;
    if (R.mode == CHAIN_FOLD) {
      const size_t base = sizeof(float) * kFoldBaseRows * fold_ld(c->B.fold_nc);
      if (R.smem + base <= kChainSmemMax) {
        y.base_off = (int)R.smem;
        R.smem += base;
      }
      const size_t res = fold_resident_bytes(c->B.fold_nc, L.n_det);
      if (R.smem + res <= kChainSmemMax) {
        y.res_off = (int)R.smem;
        R.smem += res;
      }
    }
    if (R.mode == CHAIN_HET) {
      const size_t base = sizeof(float) * kHetBaseRows * ((size_t)c->B.het_nc + 3 & ~(size_t)3);
      if (R.smem + base <= kChainSmemMax) {
        y.base_off = (int)R.smem;
        R.smem += base;
      }
      const size_t res = sizeof(float) * HC_ROWS * (size_t)c->B.het_nc;
      if (R.smem + res <= kChainSmemMax) {
        y.res_off = (int)R.smem;
        R.smem += res;
      }
    }
    if (R.smem > kChainSmemMax)
      return fail(c, SWIG_E_ARG, "problem too large for the persistent kernel's shared memory");
    y.n_ctas = S.n_ctas;
    y.spin_limit = S.spin_limit;
  } else {
    const size_t rec_bytes = (size_t)(kFlowThreads / 32) * sizeof(EvalRecord);
    S.claim_off = (int)((std::max(rec_bytes, sort_bytes) + 15) & ~(size_t)15);
    R.smem = S.claim_off + sizeof(int) * (size_t)k;
  }

  // buffers
  SamplerState* st = c->sampler;
  if (!st || st->nlive != m || st->nrep != k || st->ndim != nd || st->cap_iters < S.max_iters) {
    swig_sampler_release(c);
    st = new SamplerState();
    c->sampler = st;
    st->nlive = m;
    st->nrep = k;
    st->ndim = nd;
    st->cap_iters = S.max_iters;
    SCUDA(cudaMalloc(&st->P.live_u, sizeof(double) * m * nd));
    SCUDA(cudaMalloc(&st->P.live_logl, sizeof(double) * m));
    SCUDA(cudaMalloc(&st->P.live_kap, sizeof(double) * m * 2 * SWIG_MAX_DET));
    SCUDA(cudaMalloc(&st->P.live_vv, sizeof(double) * m * SWIG_MAX_DET));
    SCUDA(cudaMalloc(&st->P.chains, sizeof(ChainState) * k));
    SCUDA(cudaMalloc(&st->P.recx, sizeof(EvalRecord) * k));
    SCUDA(cudaMalloc(&st->P.pending, sizeof(int) * k));
    SCUDA(cudaMalloc(&st->P.req, sizeof(int) * k));
    SCUDA(cudaMalloc(&st->P.done_cnt, sizeof(int) * k));
    SCUDA(cudaMalloc(&st->ev, sizeof(ChainEvent)));
    SCUDA(cudaMalloc(&st->P.chol, sizeof(float) * kMaxBlocks * kMaxDim * kMaxDim));
    SCUDA(cudaMalloc(&st->P.g, sizeof(NSGlobal)));
    SCUDA(cudaMalloc(&st->P.dead_u, sizeof(double) * (size_t)S.max_iters * k * nd));
    SCUDA(cudaMalloc(&st->P.dead_logl, sizeof(double) * (size_t)S.max_iters * k));
    SCUDA(cudaMalloc(&st->P.dead_logw, sizeof(double) * (size_t)S.max_iters * k));
    SCUDA(cudaMalloc(&st->harm, sizeof(double) * (k + 1)));
    SCUDA(cudaMalloc(&st->lw, sizeof(double) * (m + 1)));
    SCUDA(cudaMalloc(&st->init_theta, sizeof(double) * m * SWIG_N_PARAMS));
    std::vector<double> harm(k + 1, 0.0), lw(m + 1, 0.0);
    const StreamDrain drain_weights{c->stream};
    for (int j = 1; j <= k; ++j) harm[j] = harm[j - 1] + 1.0 / (double)(m - (j - 1));
    for (int n = 1; n <= m; ++n) lw[n] = std::log(-std::expm1(-1.0 / (double)n));
    SCUDA(cudaMemcpyAsync(st->harm, harm.data(), sizeof(double) * harm.size(), cudaMemcpyHostToDevice, c->stream));
    SCUDA(cudaMemcpyAsync(st->lw, lw.data(), sizeof(double) * lw.size(), cudaMemcpyHostToDevice, c->stream));
    st->P.harm = st->harm;
    st->P.lw = st->lw;
  }
  R.st = st;
  if (st->cta_prof_n < S.n_ctas) {
    dfree(st->cta_prof);
    SCUDA(cudaMalloc(&st->cta_prof, sizeof(unsigned long long) * 4 * S.n_ctas));
    st->cta_prof_n = S.n_ctas;
  }
  SCUDA(cudaMemsetAsync(st->cta_prof, 0, sizeof(unsigned long long) * 4 * S.n_ctas, c->stream));
  st->P.cta_prof = st->cta_prof;
  st->P.learn_out = nullptr;
  if (R.learned) {
    if (!c->mlp) c->mlp = new Mlp();
    if (c->mlp->cap < m) SCUDA(mlp_alloc(*c->mlp, std::max(m, 1024), c->stream));
  }
  if ((rc = ensure_scratch(c, std::max(m, k)))) return rc;  // FP64: records and partials of k requests

  // initial live set and its likelihoods (with the per-detector sums)
  SCUDA(cudaSetDevice(c->device));
  k_init_live<<<(m + 127) / 128, 128, 0, c->stream>>>(S, st->P.live_u, st->init_theta);
  SCUDA(cudaGetLastError());
  {
    cudaError_t e = cudaMemsetAsync(st->P.live_vv, 0, sizeof(double) * m * SWIG_MAX_DET, c->stream);
    if (e != cudaSuccess) {
    } else if (het) {
      e = launch_loglike_het(L, c->B, st->init_theta, m, st->P.live_logl, c->stream, st->P.live_kap, st->P.live_vv);
    } else {
      e = mixed ? launch_loglike_mixed(L, c->B, st->init_theta, m, st->P.live_logl, c->stream, st->P.live_kap)
                : launch_loglike_fp64(L, c->B, st->init_theta, m, st->P.live_logl, c->stream, st->P.live_kap);
    }
    SCUDA(e);
  }
  NSGlobal& g0 = R.gl;
  std::memset(&g0, 0, sizeof(g0));
  g0.logx = 0.0;
  g0.logz = -INFINITY;
  g0.chains_done = k;
  g0.status = ST_RUNNING;
  SCUDA(cudaMemcpyAsync(st->P.g, &g0, sizeof(g0), cudaMemcpyHostToDevice, c->stream));
  SCUDA(cudaMemsetAsync(st->P.pending, 0, sizeof(int) * k, c->stream));
  SCUDA(cudaMemsetAsync(st->P.req, 0, sizeof(int) * k, c->stream));
  SCUDA(cudaMemsetAsync(st->P.done_cnt, 0, sizeof(int) * k, c->stream));
  SCUDA(cudaMemsetAsync(st->P.chains, 0, sizeof(ChainState) * k, c->stream));
  c->n_launches += het || mixed ? 3 : 4;  // init draw + batched likelihood

  R.kern = het || mixed ? chain_kernel(L.n_det, R.mode) : pick_flow_kernel(L.n_det);
  R.threads = het || mixed ? kChainBlock : kFlowThreads;
  if (R.learned) SCUDA(mlp_init(*c->mlp, c->cfg.seed ^ 0x4D4C5050ull, c->stream, &c->n_launches));
  R.du.clear();
  R.dl.clear();
  R.dw.clear();
  R.total_iters = 0;
  R.finished = false;
  return SWIG_OK;
}

// Reset the per-launch counters of the NS state before a launch.
int run_reset(swig_ctx* c, RunState& R) {
  NSGlobal& gl = R.gl;
  SCUDA(cudaMemcpyAsync(&gl, R.st->P.g, sizeof(gl), cudaMemcpyDeviceToHost, c->stream));
  SCUDA(cudaStreamSynchronize(c->stream));
  gl.iters_launch = 0;
  gl.n_dead = 0;
  gl.status = ST_RUNNING;
  gl.error = 0;
  gl.bar_count = 0;
  SCUDA(cudaMemcpyAsync(R.st->P.g, &gl, sizeof(gl), cudaMemcpyHostToDevice, c->stream));
  return SWIG_OK;
}

// After a launch: the NS state, its dead points, and whether the run is over.
int run_collect(swig_ctx* c, RunState& R) {
  SCUDA(cudaMemcpyAsync(&R.gh, R.st->P.g, sizeof(R.gh), cudaMemcpyDeviceToHost, c->stream));
  SCUDA(cudaStreamSynchronize(c->stream));
  const NSGlobal& gh = R.gh;
  if (gh.error) return fail(c, gh.error, gh.error == SWIG_E_TIMEOUT ? "a bounded device wait expired" : "device error");
  c->d2h_bytes += sizeof(gh);
  const int nd = R.nd;
  if (gh.n_dead > 0) {
    c->d2h_bytes += (size_t)gh.n_dead * (nd + 2) * sizeof(double);
    const size_t n0 = R.dl.size();
    R.du.resize((n0 + gh.n_dead) * nd);
    R.dl.resize(n0 + gh.n_dead);
    R.dw.resize(n0 + gh.n_dead);
    SCUDA(cudaMemcpy(R.du.data() + n0 * nd, R.st->P.dead_u, sizeof(double) * gh.n_dead * nd, cudaMemcpyDeviceToHost));
    SCUDA(cudaMemcpy(R.dl.data() + n0, R.st->P.dead_logl, sizeof(double) * gh.n_dead, cudaMemcpyDeviceToHost));
    SCUDA(cudaMemcpy(R.dw.data() + n0, R.st->P.dead_logw, sizeof(double) * gh.n_dead, cudaMemcpyDeviceToHost));
  }
  R.total_iters = gh.iter;
  R.finished = gh.status == ST_TERMINATED || R.total_iters >= c->cfg.max_iter;
  return SWIG_OK;
}

// Final live points, the samples' parameters (and post-hoc distances), the
// result and the profile counters.
int run_finish(swig_ctx* c, RunState& R, swig_result* out) {
  const int m = R.m, k = R.k, nd = R.nd;
  const bool mixed = R.mixed, het = R.het;
  const LikeConst& L = c->L;
  const SamplerConst& S = R.S;
  SamplerState* st = R.st;
  const NSGlobal& gh = R.gh;
  std::vector<double>& du = R.du;
  std::vector<double>& dl = R.dl;
  std::vector<double>& dw = R.dw;
  // final live points, X/m each
  std::vector<double> lu((size_t)m * nd), ll(m);
  SCUDA(cudaMemcpy(lu.data(), st->P.live_u, sizeof(double) * lu.size(), cudaMemcpyDeviceToHost));
  SCUDA(cudaMemcpy(ll.data(), st->P.live_logl, sizeof(double) * m, cudaMemcpyDeviceToHost));
  std::vector<int> order(m);
  for (int i = 0; i < m; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return ll[a] < ll[b]; });
  double logz = gh.logz;
  for (int i : order) {
    const double w = ll[i] + gh.logx - std::log((double)m);
    du.insert(du.end(), lu.begin() + (size_t)i * nd, lu.begin() + (size_t)(i + 1) * nd);
    dl.push_back(ll[i]);
    dw.push_back(w);
    const double hi = std::max(logz, w);
    logz = std::isfinite(hi) ? hi + std::log(std::exp(logz - hi) + std::exp(w - hi)) : hi;
  }
  const size_t n_dead = dl.size();
  double info = 0.0, sum_p2 = 0.0;
  for (size_t i = 0; i < n_dead; ++i) {
    const double p = std::exp(dw[i] - logz);
    info += p * (dl[i] - logz);
    sum_p2 += p * p;
  }
  // counters
  std::vector<ChainState> ch(k);
  SCUDA(cudaMemcpy(ch.data(), st->P.chains, sizeof(ChainState) * k, cudaMemcpyDeviceToHost));
  // theta of every dead point via the device prior transform
  c->out_theta.assign(n_dead * SWIG_N_PARAMS, 0.0);
  {
    double *du_d = nullptr, *th_d = nullptr;
    SCUDA(cudaMalloc(&du_d, sizeof(double) * std::max<size_t>(1, du.size())));
    SCUDA(cudaMalloc(&th_d, sizeof(double) * std::max<size_t>(1, c->out_theta.size())));
    SCUDA(cudaMemcpyAsync(du_d, du.data(), sizeof(double) * du.size(), cudaMemcpyHostToDevice, c->stream));
    k_dead_theta<<<(unsigned)((n_dead + 127) / 128), 128, 0, c->stream>>>(S, du_d, (int)n_dead, th_d);
    ++c->n_launches;
    if (L.dist_marg) {
      // post-hoc distances: the kappa sums of every sample, then a draw from
      // its conditional distance posterior
      const int chunk = 4096;
      double *kap_d = nullptr, *ll_d = nullptr;
      cudaError_t e = cudaMalloc(&kap_d, sizeof(double) * 2 * SWIG_MAX_DET * chunk);
      if (e == cudaSuccess) e = cudaMalloc(&ll_d, sizeof(double) * chunk);
      for (size_t off = 0; e == cudaSuccess && off < n_dead; off += chunk) {
        const int mm = (int)std::min<size_t>(chunk, n_dead - off);
        if (ensure_scratch(c, mm)) {
          e = cudaErrorMemoryAllocation;
          break;
        }
        e = mixed ? launch_loglike_mixed(L, c->B, th_d + off * SWIG_N_PARAMS, mm, ll_d, c->stream, kap_d)
                  : launch_loglike_fp64(L, c->B, th_d + off * SWIG_N_PARAMS, mm, ll_d, c->stream, kap_d);
        if (e == cudaSuccess)
          e = launch_distance_draw(L, c->B, kap_d, mm, (long long)off, S.key0, S.key1, th_d + off * SWIG_N_PARAMS,
                                   c->stream);
        c->n_launches += mixed ? 3 : 4;
      }
      if (kap_d) cudaFree(kap_d);
      if (ll_d) cudaFree(ll_d);
      if (e != cudaSuccess) {
        cudaFree(du_d);
        cudaFree(th_d);
        SCUDA(e);
      }
    }
    if (L.tm_n > 0) {
      // post-hoc t_c: the node log weights of every sample, then a draw from
      // its conditional on the time grid
      const int chunk = (int)std::max<int64_t>(1, std::min<int64_t>(4096, ((int64_t)1 << 26) / L.tm_n));
      double* ll_d = nullptr;
      float* ell_d = nullptr;
      cudaError_t e = cudaMalloc(&ll_d, sizeof(double) * chunk);
      if (e == cudaSuccess) e = cudaMalloc(&ell_d, sizeof(float) * (size_t)chunk * L.tm_n);
      for (size_t off = 0; e == cudaSuccess && off < n_dead; off += chunk) {
        const int mm = (int)std::min<size_t>(chunk, n_dead - off);
        if (ensure_scratch(c, mm)) {
          e = cudaErrorMemoryAllocation;
          break;
        }
        e = launch_loglike_het(L, c->B, th_d + off * SWIG_N_PARAMS, mm, ll_d, c->stream, nullptr, nullptr, ell_d);
        if (e == cudaSuccess)
          e = launch_time_draw(L, c->B, ell_d, mm, (long long)off, S.key0, S.key1, th_d + off * SWIG_N_PARAMS,
                               c->stream);
        c->n_launches += 3;
      }
      if (ll_d) cudaFree(ll_d);
      if (ell_d) cudaFree(ell_d);
      if (e != cudaSuccess) {
        cudaFree(du_d);
        cudaFree(th_d);
        SCUDA(e);
      }
    }
    c->h2d_bytes += sizeof(double) * du.size();
    c->d2h_bytes += sizeof(double) * c->out_theta.size();
    cudaError_t e = cudaStreamSynchronize(c->stream);
    if (e == cudaSuccess) e = cudaMemcpy(c->out_theta.data(), th_d, sizeof(double) * c->out_theta.size(), cudaMemcpyDeviceToHost);
    cudaFree(du_d);
    cudaFree(th_d);
    SCUDA(e);
  }
  c->out_logl = dl;
  c->out_logw.resize(n_dead);
  for (size_t i = 0; i < n_dead; ++i) c->out_logw[i] = dw[i];
  // normalise so that logsumexp(logw) = log Z (already the case by construction)
  out->logz = logz;
  out->info = info;
  out->logz_err = std::sqrt(std::max(info, 0.0) / m);
  out->ess = sum_p2 > 0 ? 1.0 / sum_p2 : 0.0;
  out->n_dead = (int64_t)n_dead;
  out->n_iter = R.total_iters;
  // evaluations: the initial m plus the chains' counters accumulated on device
  long long ne = m, nf = m;
  for (const ChainState& q : ch) {
    ne += q.n_evals;
    nf += q.n_full;
  }
  out->n_evals = ne;
  out->n_sweep_evals = nf;
  out->status = gh.status == ST_TERMINATED ? 0 : 1;
  out->wall_s = std::chrono::duration<double>(std::chrono::steady_clock::now() - R.t_start).count();
  c->last = *out;
  c->profile[0] = (double)gh.rounds;
  c->profile[1] = gh.t_bound * 1e-9;
  c->profile[2] = gh.t_ctrl * 1e-9;
  c->profile[3] = gh.t_wait_ctrl * 1e-9;
  c->profile[4] = gh.t_sweep * 1e-9;
  c->profile[5] = gh.t_wait_sweep * 1e-9;
  c->profile[6] = R.persistent_ms;
  c->profile[7] = (double)R.persistent_launches;
  c->profile[8] = (double)c->n_launches;
  c->profile[9] = (double)c->h2d_bytes;
  c->profile[10] = (double)c->d2h_bytes;
  // bin-detector evaluations (heterodyned: bins of the coarse grid)
  c->profile[11] = (double)nf * (double)L.n_det * (double)(het ? c->B.het_nb : L.n_bins);
  c->profile[12] = (double)gh.c_result;
  c->profile[13] = (double)gh.c_step;
  c->profile[14] = (double)gh.c_prop;
  c->profile[15] = (double)gh.c_free;
  c->profile[16] = (double)gh.c_setup;
  c->profile[17] = (double)gh.n_free;
  c->profile[18] = (double)gh.n_setup;
  c->profile[19] = (double)gh.n_step;
  c->profile[20] = R.learn_ms;
  c->profile[21] = (double)R.learn_rounds;
  c->profile[22] = (double)gh.f_units;
  c->profile[23] = (double)gh.f_unit_cyc;
  c->profile[24] = (double)gh.f_idle_cyc;
  {
    std::vector<unsigned long long> cp(4 * (size_t)S.n_ctas);
    SCUDA(cudaMemcpy(cp.data(), st->cta_prof, sizeof(unsigned long long) * cp.size(), cudaMemcpyDeviceToHost));
    c->cta_profile.assign(cp.begin(), cp.end());
  }
  return SWIG_OK;
}

// The run as the chain kernel reads it.
ChainEvent chain_event(const swig_ctx* c, const RunState& R) {
  ChainEvent d;
  d.L = c->L;
  d.S = R.S;
  d.F = fold_tables(c->B);
  d.H = het_tables(c->B);
  d.P = R.st->P;
  return d;
}

// The persistent launches of one run until termination or the iteration cap.
int run_loop_single(swig_ctx* c, RunState& R) {
  int rc = SWIG_OK;
  const bool chain = R.mixed || R.het;
  SCUDA(allow_shared(R.kern));
  int per_sm = 0;
  SCUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, R.kern, R.threads, R.smem));
  if (per_sm < 1 || R.S.n_ctas > per_sm * c->sm_count)
    return fail(c, SWIG_E_CUDA, "persistent kernel cannot be co-resident on this device");
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  SCUDA(cudaEventCreate(&ev0));
  SCUDA(cudaEventCreate(&ev1));
  while (!R.finished) {
    if ((rc = run_reset(c, R))) break;
    if (R.learned) {
      // retrain on the current live set, then freeze the output rows of
      // this snapshot for the launch's iterations
      Mlp& N = *c->mlp;
      cudaError_t e = cudaEventRecord(ev0, c->stream);
      if (e == cudaSuccess) e = mlp_targets(N, R.st->P.live_u, R.m, R.nd, 2 * R.nd, c->stream, &c->n_launches);
      if (e == cudaSuccess)
        e = mlp_train(N, R.m, R.nd, R.learn_rounds == 0 ? 4 * R.learn_steps : R.learn_steps, R.learn_lr, c->stream,
                      &c->n_launches);
      if (e == cudaSuccess) e = mlp_forward(N, R.m, c->stream, &c->n_launches);
      if (e == cudaSuccess) e = cudaEventRecord(ev1, c->stream);
      if (e == cudaSuccess) e = cudaEventSynchronize(ev1);
      float ms = 0.0f;
      if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, ev0, ev1);
      if (e != cudaSuccess) {
        rc = fail(c, SWIG_E_CUDA, std::string("learned proposal training: ") + cudaGetErrorString(e));
        break;
      }
      R.learn_ms += ms;
      ++R.learn_rounds;
      R.st->P.learn_out = N.out;
    }
    void* flow_args[] = {(void*)&c->L, (void*)&R.S, (void*)&c->B, (void*)&R.st->P};
    int one = 1;
    void* chain_args[] = {(void*)&R.st->ev, (void*)&one, (void*)&R.st->P.g, (void*)&R.lay};
    void** args = chain ? chain_args : flow_args;
    cudaError_t e = cudaSuccess;
    ChainEvent hev;
    const StreamDrain drain{c->stream};
    if (chain) {
      hev = chain_event(c, R);
      e = cudaMemcpyAsync(R.st->ev, &hev, sizeof(hev), cudaMemcpyHostToDevice, c->stream);
    }
    if (e == cudaSuccess) e = cudaEventRecord(ev0, c->stream);
    if (e == cudaSuccess)
      e = cudaLaunchCooperativeKernel(R.kern, dim3(R.S.n_ctas), dim3(R.threads), args, R.smem, c->stream);
    if (e == cudaSuccess) e = cudaEventRecord(ev1, c->stream);
    if (e == cudaSuccess) e = cudaEventSynchronize(ev1);
    float ms = 0.0f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, ev0, ev1);
    if (e != cudaSuccess) {
      rc = fail(c, SWIG_E_CUDA, std::string("persistent launch: ") + cudaGetErrorString(e));
      break;
    }
    R.persistent_ms += ms;
    ++R.persistent_launches;
    ++c->n_launches;
    if ((rc = run_collect(c, R))) break;
  }
  cudaEventDestroy(ev0);
  cudaEventDestroy(ev1);
  return rc;
}

// Events of one campaign that can share a launch: full grid, mixed precision,
// covariance proposal, the same detector count, chains per event and device.
bool batchable(swig_ctx* const* ctxs, const std::vector<RunState>& R, int i0, int i1) {
  for (int i = i0; i < i1; ++i) {
    if (R[i].het || !R[i].mixed || R[i].learned) return false;
    if (ctxs[i]->L.n_det != ctxs[i0]->L.n_det || R[i].k != R[i0].k || ctxs[i]->device != ctxs[i0]->device) return false;
  }
  return true;
}

// One group of events in shared launches until every one is finished.
int run_loop_multi(swig_ctx* const* ctxs, std::vector<RunState>& R, int i0, int i1) {
  swig_ctx* c0 = ctxs[i0];
  const int n_det = c0->L.n_det, k = R[i0].k;
  // shared memory: the largest scratch; weights and tables resident if every
  // event's fit beside it
  ChainLayout lay = R[i0].lay;
  size_t res = 0, base = 0;
  for (int i = i0; i < i1; ++i) {
    lay.scratch_bytes = std::max(lay.scratch_bytes, R[i].lay.scratch_bytes);
    res = std::max(res, fold_resident_bytes(ctxs[i]->B.fold_nc, n_det));
    base = std::max(base, sizeof(float) * kFoldBaseRows * fold_ld(ctxs[i]->B.fold_nc));
  }
  size_t smem = (size_t)lay.scratch_off + lay.scratch_bytes;
  lay.res_off = lay.base_off = 0;
  if (smem + base <= kChainSmemMax) {
    lay.base_off = (int)smem;
    smem += base;
  }
  if (smem + res <= kChainSmemMax) {
    lay.res_off = (int)smem;
    smem += res;
  }
  const int grid = std::min(c0->sm_count, (i1 - i0) * k);
  lay.n_ctas = std::max(grid, i1 - i0);
  void* kern = chain_kernel(n_det, CHAIN_FOLD);
  cudaError_t e = allow_shared(kern);
  int per_sm = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kChainBlock, smem);
  if (e != cudaSuccess) return fail(c0, SWIG_E_CUDA, std::string("multi-event kernel set-up: ") + cudaGetErrorString(e));
  if (per_sm < 1 || lay.n_ctas > per_sm * c0->sm_count)
    return fail(c0, SWIG_E_CUDA, "multi-event persistent kernel cannot be co-resident on this device");
  NSGlobal* gb = nullptr;
  ChainEvent* evd = nullptr;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  int rc = SWIG_OK;
  e = cudaMalloc(&gb, sizeof(NSGlobal));
  if (e == cudaSuccess) e = cudaMalloc(&evd, sizeof(ChainEvent) * (i1 - i0));
  if (e == cudaSuccess) e = cudaEventCreate(&ev0);
  if (e == cudaSuccess) e = cudaEventCreate(&ev1);
  std::vector<ChainEvent> hd;
  std::vector<int> idx;
  NSGlobal g0;
  std::memset(&g0, 0, sizeof(g0));
  const StreamDrain drain{c0->stream};
  while (e == cudaSuccess && rc == SWIG_OK) {
    hd.clear();
    idx.clear();
    for (int i = i0; i < i1; ++i) {
      if (R[i].finished) continue;
      if ((rc = run_reset(ctxs[i], R[i]))) break;
      hd.push_back(chain_event(ctxs[i], R[i]));
      hd.back().P.cta_prof = nullptr;  // (rows of one event's CTAs; this launch has more)
      idx.push_back(i);
    }
    if (rc || hd.empty()) break;
    for (int i : idx) {
      e = cudaStreamSynchronize(ctxs[i]->stream);
      if (e != cudaSuccess) break;
    }
    // on the launch's stream, which does not wait for the default stream's copies
    if (e == cudaSuccess) e = cudaMemcpyAsync(gb, &g0, sizeof(g0), cudaMemcpyHostToDevice, c0->stream);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(evd, hd.data(), sizeof(ChainEvent) * hd.size(), cudaMemcpyHostToDevice, c0->stream);
    int n_ev = (int)hd.size();
    void* args[] = {(void*)&evd, (void*)&n_ev, (void*)&gb, (void*)&lay};
    if (e == cudaSuccess) e = cudaEventRecord(ev0, c0->stream);
    if (e == cudaSuccess) e = cudaLaunchCooperativeKernel(kern, dim3(lay.n_ctas), dim3(kChainBlock), args, smem, c0->stream);
    if (e == cudaSuccess) e = cudaEventRecord(ev1, c0->stream);
    if (e == cudaSuccess) e = cudaEventSynchronize(ev1);
    float ms = 0.0f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, ev0, ev1);
    NSGlobal gh;
    if (e == cudaSuccess) e = cudaMemcpy(&gh, gb, sizeof(gh), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) break;
    if (gh.error) {
      rc = fail(c0, gh.error, gh.error == SWIG_E_TIMEOUT ? "a bounded device wait expired" : "device error");
      break;
    }
    for (int i : idx) {
      R[i].persistent_ms += ms;  // the launch's wall time, shared by its events
      ++R[i].persistent_launches;
      if ((rc = run_collect(ctxs[i], R[i]))) break;
    }
    ++c0->n_launches;
  }
  if (e != cudaSuccess && rc == SWIG_OK)
    rc = fail(c0, SWIG_E_CUDA, std::string("multi-event launch: ") + cudaGetErrorString(e));
  if (gb) cudaFree(gb);
  if (evd) cudaFree(evd);
  if (ev0) cudaEventDestroy(ev0);
  if (ev1) cudaEventDestroy(ev1);
  return rc;
}

}  // namespace

extern "C" {

int swig_autotune(swig_ctx* c, int iters, double* out, int n) {
  if (!c) return SWIG_E_ARG;
  if (iters < 1) return fail(c, SWIG_E_ARG, "autotune needs at least one iteration");
  if (out && n > 0) out[0] = 0.0;
  const swig_sampler_cfg saved = c->cfg;
  if (!c->cfg_set) return fail(c, SWIG_E_STATE, "sampler settings not set");
  if (saved.likelihood != SWIG_LIKE_FULL || saved.precision != SWIG_PREC_MIXED ||
      saved.proposal != SWIG_PROPOSAL_COV)
    return SWIG_OK;
  const int cand[4][2] = {{1, 0}, {1, 1}, {2, 0}, {3, 0}};
  double rate[4] = {0.0, 0.0, 0.0, 0.0};
  int best = 0;
  for (int i = 0; i < 4; ++i) {
    c->cfg = saved;
    c->cfg.flow_parts = cand[i][0];
    c->cfg.stepout_one_end = cand[i][1];
    c->cfg.max_iter = iters;
    swig_result r;
    const int rc = swig_run(c, &r);
    if (rc != SWIG_OK) {
      c->cfg = saved;
      return rc;
    }
    rate[i] = c->profile[6] > 0.0 ? (double)r.n_sweep_evals / (c->profile[6] * 1e-3) : 0.0;
    if (rate[i] > rate[best]) best = i;
  }
  c->cfg = saved;
  c->cfg.flow_parts = cand[best][0];
  c->cfg.stepout_one_end = cand[best][1];
  if (out && n > 0) {
    out[0] = 4.0;
    for (int i = 0; i < 4; ++i)
      for (int j = 0; j < 3; ++j)
        if (1 + 3 * i + j < n) out[1 + 3 * i + j] = j == 0 ? cand[i][0] : j == 1 ? cand[i][1] : rate[i];
  }
  return SWIG_OK;
}

int swig_run(swig_ctx* c, swig_result* out) {
  if (!c) return SWIG_E_ARG;
  if (!out) return fail(c, SWIG_E_ARG, "null result pointer");
  std::memset(out, 0, sizeof(*out));
  RunState R;
  int rc = run_setup(c, R);
  if (!rc) rc = run_loop_single(c, R);
  if (rc) return rc;
  return run_finish(c, R, out);
}

int swig_run_batch(swig_ctx** ctxs, int n_ctx, swig_result* outs) {
  if (!ctxs || !outs || n_ctx < 1) return SWIG_E_ARG;
  for (int i = 0; i < n_ctx; ++i) {
    if (!ctxs[i]) return SWIG_E_ARG;
    for (int j = 0; j < i; ++j)
      if (ctxs[j] == ctxs[i]) return fail(ctxs[i], SWIG_E_ARG, "a context appears twice in the batch");
    std::memset(&outs[i], 0, sizeof(outs[i]));
  }
  std::vector<RunState> R(n_ctx);
  for (int i = 0; i < n_ctx; ++i) {
    const int rc = run_setup(ctxs[i], R[i]);
    if (rc) return rc;
  }
  // Events share a launch in groups of similar grid size: the events of a
  // launch advance their NS iterations in step, so a short event grouped with
  // a long one would wait for it.  Greedy groups over the events sorted by
  // grid size: at most kMaxEvents, within 1.5x of the group's smallest grid,
  // their chains within kMaxChains, their slices within one CTA's shared
  // memory.
  std::vector<int> order(n_ctx);
  for (int i = 0; i < n_ctx; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return ctxs[a]->L.n_bins < ctxs[b]->L.n_bins; });
  std::vector<swig_ctx*> oc(n_ctx);
  std::vector<RunState> orr(n_ctx);
  for (int i = 0; i < n_ctx; ++i) {
    oc[i] = ctxs[order[i]];
    orr[i] = R[order[i]];
  }
  int i0 = 0;
  while (i0 < n_ctx) {
    int i1 = i0 + 1;
    if (batchable(oc.data(), orr, i0, i0 + 1)) {
      while (i1 < n_ctx && i1 - i0 < kMaxEvents && batchable(oc.data(), orr, i0, i1 + 1) &&
             (i1 + 1 - i0) * orr[i0].k <= kMaxChains && oc[i1]->L.n_bins <= 1.5 * oc[i0]->L.n_bins)
        ++i1;
    }
    int rc = i1 - i0 == 1 ? run_loop_single(oc[i0], orr[i0]) : run_loop_multi(oc.data(), orr, i0, i1);
    if (rc) return rc;
    for (int i = i0; i < i1; ++i)
      if ((rc = run_finish(oc[i], orr[i], &outs[order[i]]))) return rc;
    i0 = i1;
  }
  return SWIG_OK;
}

int swig_get_profile(swig_ctx* c, double* out, int n) {
  if (!c) return SWIG_E_ARG;
  if (!out || n < 0) return fail(c, SWIG_E_ARG, "null output");
  for (int i = 0; i < n && i < 25; ++i) out[i] = c->profile[i];
  for (int i = 25; i < n && i - 25 < (int)c->cta_profile.size(); ++i) out[i] = c->cta_profile[i - 25];
  return SWIG_OK;
}

int swig_get_samples(swig_ctx* c, double* theta, double* logl, double* logw, int64_t cap, int64_t* n_out) {
  if (!c) return SWIG_E_ARG;
  if (!n_out) return fail(c, SWIG_E_ARG, "null n_out");
  const int64_t n = (int64_t)c->out_logl.size();
  *n_out = n;
  if (cap == 0) return SWIG_OK;
  if (cap < n || !theta || !logl || !logw) return fail(c, SWIG_E_ARG, "capacity below the number of samples or null buffer");
  std::memcpy(theta, c->out_theta.data(), sizeof(double) * n * SWIG_N_PARAMS);
  std::memcpy(logl, c->out_logl.data(), sizeof(double) * n);
  std::memcpy(logw, c->out_logw.data(), sizeof(double) * n);
  return SWIG_OK;
}

}  // extern "C"
