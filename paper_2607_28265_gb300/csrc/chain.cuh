// Chain control of the mixed-precision samplers: one CTA advances one chain.
//
// A slice step (Neal 2003) looks at its points in a fixed order: the left end
// and its expansions, the right end and its, then the shrinkage draws.  Which
// of them the step needs is known only as they are evaluated, but where they
// lie is known ahead: the rungs lo, lo - 1, ... and hi, hi + 1, ... are fixed,
// and a shrinkage draw follows from the ones before it being rejected (the
// uniforms are counter-based).  So a round takes several candidates at once, the
// control then reads their results in the step's own order and stops where the
// step would have stopped; what lies beyond is dropped and not counted.  The
// decisions, draws and counts are those of one candidate after another.
//
// Measured (one GB300, first iterations of the 128 s three-detector run, nlive
// 1000, nrep 100): 4 iterations 145 ms with one candidate at a time across all
// SMs (a request to every SM's slice of the grid, control on one warp), 18.7 ms
// here; heterodyned, 8 iterations 133 -> 47.9 ms.  1.3 candidates are evaluated
// per candidate used; with fewer per round the latencies dominate.
//
// A round costs its latency once: the set-up's FP64 chains (64 cycles an
// instruction whatever the lanes do) serve all candidates, one per lane, and the
// 16 warps share the candidates' sums.
#pragma once

#include "chain.h"
#include "fold.cuh"
#include "het.cuh"
#include "sampler.cuh"

namespace swig {

constexpr int kCand = 8;          // candidates per round at most
constexpr int kChainWarps = kChainBlock / 32;
constexpr int kFoldGroups = 4;    // groups of chunks (partial sums) of a full round's pairs
static_assert(kChainBlock == kHetTmThreads, "the sampler and the batched time-marginalised kernel share sum orders");

// What the control keeps of a chain between its rounds, and a round's
// candidates, in shared memory.
struct ChainWork {
  ChainState ch;
  EvalRecord rx;             // record of the chain's current point
  EvalRecord rec[kCand];     // ... of the candidates
  double th[kCand][SWIG_N_PARAMS];
  double y[kCand][kMaxDim];  // the block's coordinates
  double t[kCand];
  double ly[kCand];
  double kap[kCand][2 * SWIG_MAX_DET];
  double vv[kCand][SWIG_MAX_DET];
  double sc[4][kCand];       // sines and cosines of RA - GMST and Dec
  unsigned inside, act;      // candidate bits: in the unit cube; to be evaluated
  int list[kCand], n_act;    // the latter's numbers
  int n_cand, n_left;        // candidates; stepping out: of them on the left
  int fl;                    // record pieces that the block moves
  int status;
  int bad[kCand];            // folded sums: outside the band, summed bin by bin
};

enum { ROUND_EVAL = 0, ROUND_DONE = 1 };

// Sign and unit-interval tests on the bits: an FP64 comparison costs the
// scheduler 64 cycles.
__device__ __forceinline__ bool fp64_negative(double v) {  // v < 0 (not -0); v is no NaN
  return __double_as_longlong(v) < 0 && (__double_as_longlong(v) << 1) != 0;
}
__device__ __forceinline__ bool fp64_in_unit(double v) {  // 0 <= v <= 1, false for a NaN
  const long long b = __double_as_longlong(v);
  return (b >= 0 && b <= 0x3FF0000000000000ll) || (b << 1) == 0;
}

// Apply the results of the pending candidates in the step's order.  ok: the
// candidates whose logL exceeds logL* (bits).  Returns the accepted candidate
// or -1.  Lane-uniform.
__device__ __forceinline__ int chain_consume(const SamplerConst& S, ChainState& ch, const ChainWork& w, unsigned ok,
                                             bool full) {
  const int n = w.n_cand, nl = w.n_left;
  const unsigned inside = w.inside;
  int evals = 0, hit = -1;
  if (ch.phase == PH_OUT) {
    for (int k = 0; k < nl && (ch.side & 1); ++k) {
      if ((inside >> k) & 1u) {
        ++evals;
        if ((ok >> k) & 1u) {
          ch.lo -= 1.0;
          if (++ch.n_out >= kMaxStepOut) ch.side &= ~1;
          continue;
        }
      }
      ch.side &= ~1;
    }
    for (int k = nl; k < n && (ch.side & 2); ++k) {
      if ((inside >> k) & 1u) {
        ++evals;
        if ((ok >> k) & 1u) {
          ch.hi += 1.0;
          if (++ch.n_out_r >= kMaxStepOut) ch.side &= ~2;
          continue;
        }
      }
      ch.side &= ~2;
    }
    if (ch.side == 0) {
      ch.phase = PH_SHRINK;
      ch.n_shrink = 0;
    }
  } else {
    for (int k = 0; k < n; ++k) {
      ++ch.ctr;  // its uniform
      if ((inside >> k) & 1u) {
        ++evals;
        if ((ok >> k) & 1u) {
          hit = k;
          break;
        }
      }
      const double t = w.t[k];
      if (fp64_negative(t))
        ch.lo = t;
      else
        ch.hi = t;
      if (++ch.n_shrink >= kMaxShrink) {
        ++ch.n_caps;
        finish_step(S, ch);
        break;
      }
    }
  }
  ch.n_evals += evals;
  if (full) ch.n_full += evals;
  return hit;
}

// The direction and bracket of a new slice step (start_step across the warp:
// row r of the Cholesky product on lane r).
__device__ __forceinline__ void chain_start_step(const SamplerConst& S, ChainState& ch, const float* chol,
                                                 const float* learn_out, int c, long long it, int lane) {
  const int b = ch.block, nb = S.block_size[b];
  const bool inb = lane < S.ndim && ((S.block_mask[b] >> lane) & 1u);
  unsigned ctr = ch.ctr;
  auto uniform = [&] {
    return u01_from(philox4x32_10(make_uint4(ctr++, (unsigned)c, (unsigned)it, 0u), S.key0, S.key1));
  };
  double dir = 0.0;
  bool learned = false;
  if (S.learn_on && learn_out && uniform() < (double)S.learn_mix) {
    const int row = min((int)(uniform() * (double)S.nlive), S.nlive - 1);
    const float* o = learn_out + (size_t)row * 32;
    float nrm2 = 0.0f;
    for (int r = 0; r < nb; ++r) {
      const float u = o[S.block_dims[b][r]];
      nrm2 = fmaf(u, u, nrm2);
    }
    const float inv = rsqrtf(nrm2 + 1e-12f);
    if (inb) {
      const float sv = fminf(fmaxf(o[13 + lane], -30.0f), 5.0f);
      dir = (double)(expf(sv) * o[lane] * inv);
    }
    learned = true;
  }
  if (!learned) {
    // z_r, r < nb, one Philox block each at consecutive counters
    float z = 0.0f;
    if (lane < nb) {
      const uint4 r = philox4x32_10(make_uint4(ctr + (unsigned)lane, (unsigned)c, (unsigned)it, 0u), S.key0, S.key1);
      const float u1 = ((float)(r.x >> 8) + 1.0f) * (1.0f / 16777216.0f);
      const float u2 = (float)(r.y >> 8) * (1.0f / 16777216.0f);
      z = sqrtf(-2.0f * logf(u1)) * cospif(2.0f * u2);
    }
    ctr += (unsigned)nb;
    const float* Lb = chol + (size_t)b * kMaxDim * kMaxDim;
    float v = 0.0f;
    for (int q = 0; q < nb; ++q) {
      const float zq = __shfl_sync(0xffffffffu, z, q);
      if (lane < nb && q <= lane) v = fmaf(__ldcg(&Lb[lane * kMaxDim + q]), zq, v);  // CTA 0 writes L_b
    }
    const float vd = __shfl_sync(0xffffffffu, v, lane < S.ndim ? S.block_rank[lane] : 0);
    if (inb) dir = (double)vd;
  }
  const double r0 = uniform();
  __syncwarp();
  if (lane < S.ndim) ch.dir[lane] = dir;
  if (lane == 0) {
    ch.ctr = ctr;
    ch.lo = -r0;
    ch.hi = 1.0 - r0;
    ch.phase = PH_OUT;
    ch.side = 3;
    ch.n_out = ch.n_out_r = ch.n_shrink = 0;
  }
  __syncwarp();
}

// The round's candidates: bracket coordinates, points and theta, one candidate
// per lane, written to w.  All lanes.
__device__ __forceinline__ void chain_candidates(const SamplerConst& S, ChainWork& w, int c, long long it, int lane) {
  ChainState& ch = w.ch;
  const int b = ch.block, nb = S.block_size[b];
  int n, nl = 0;
  double t = 0.0;
  if (ch.phase == PH_OUT) {
    const bool l = ch.side & 1, r = (ch.side & 2) && !(S.one_end && l);
    // an end alone may use both ends' rungs
    const int d = l && r ? S.spec_out : min(2 * S.spec_out, kCand);
    nl = l ? min(d, kMaxStepOut - ch.n_out) : 0;
    n = nl + (r ? min(d, kMaxStepOut - ch.n_out_r) : 0);
    // rung by rung, as the step moves its end (each addition rounds)
    const int m = lane < nl ? lane : lane - nl;
    t = lane < nl ? ch.lo : ch.hi;
    for (int i = 1; i < max(nl, n - nl); ++i)
      if (i <= m) t += lane < nl ? -1.0 : 1.0;
  } else {
    n = min(S.spec_shr, kMaxShrink - ch.n_shrink);
    const double u = u01_from(philox4x32_10(make_uint4(ch.ctr + (unsigned)lane, (unsigned)c, (unsigned)it, 0u), S.key0,
                                            S.key1));
    double lo = ch.lo, hi = ch.hi;
    for (int k = 0; k < n; ++k) {
      const double tk = lo + (hi - lo) * __shfl_sync(0xffffffffu, u, k);
      if (lane == k) t = tk;
      if (fp64_negative(tk))
        lo = tk;
      else
        hi = tk;
    }
  }
  const bool on = lane < n;
  bool inside = on;
  if (on) {
#pragma unroll
    for (int s = 0; s < SWIG_N_PARAMS; ++s) w.th[lane][s] = ch.th[s];
    w.t[lane] = t;
  }
  bool sky = false;
  for (int r = 0; r < nb; ++r) {
    const int j = S.block_dims[b][r], slot = S.slot_of_dim[j];
    if (on) {
      const double v = ch.x[j] + t * ch.dir[j];
      w.y[lane][j] = v;
      if (!fp64_in_unit(v)) inside = false;
      // the sky angles go through FP64: the delays need them to ~1e-10
      if (inside)
        w.th[lane][slot] = (S.sky.on && (slot == 9 || slot == 10)) ? prior_slot_inverse(S.prior[slot], v)
                                                                   : prior_slot_inverse_f32(S.prior[slot], v);
    }
    sky = sky || slot == 9 || slot == 10;
  }
  if (S.sky.on && sky && inside) sky_frame_to_radec(S.sky, w.th[lane][9], w.th[lane][10], &w.th[lane][9], &w.th[lane][10]);
  const unsigned m = __ballot_sync(0xffffffffu, inside);
  if (lane == 0) {
    w.n_cand = n;
    w.n_left = nl;
    w.inside = m;
  }
  __syncwarp();
}

// Accept candidate k: point, theta, logL and, from a full evaluation, the
// per-detector sums and the record.  All lanes.
__device__ __forceinline__ void chain_accept(const SamplerConst& S, ChainWork& w, int k, bool full, int lane) {
  ChainState& ch = w.ch;
  const int b = ch.block;
  if (lane < S.ndim && ((S.block_mask[b] >> lane) & 1u)) ch.x[lane] = w.y[k][lane];
  if (lane < SWIG_N_PARAMS) ch.th[lane] = w.th[k][lane];
  if (full) {
    if (lane < 2 * SWIG_MAX_DET) ch.kap[lane] = w.kap[k][lane];
    if (lane < SWIG_MAX_DET) ch.vv[lane] = w.vv[k][lane];
    warp_copy(&w.rx, &w.rec[k], sizeof(EvalRecord), lane);
  }
  __syncwarp();
  if (lane == 0) {
    ch.lx = w.ly[k];
    ch.proj_dirty = full ? 0 : 1;
    finish_step(S, ch);
  }
  __syncwarp();
}

// Warp 0 between two evaluations: apply the results (have: a round is pending,
// its logL in w.ly), then advance to the next round that needs the CTA.
// Projection-only blocks are evaluated here, a candidate per lane.
template <int NDET, bool HET>
__device__ __forceinline__ void chain_control(const LikeConst& L, const SamplerConst& S, const SamplerPtrs& P,
                                              ChainWork& w, int c, long long it, double logl_star, bool have,
                                              int lane, unsigned long long* prof) {
  ChainState& ch = w.ch;
  long long tk = clock64();
  auto lap = [&](int slot) {
    if (prof && lane == 0) {
      const long long t2 = clock64();
      prof[slot] += t2 - tk;
      tk = t2;
    }
  };
  auto apply = [&](bool full) {
    const bool in = lane < w.n_cand && ((w.inside >> lane) & 1u);
    const unsigned ok = __ballot_sync(0xffffffffu, in && w.ly[lane < kCand ? lane : 0] > logl_star);
    int hit = -1;
    if (lane == 0) hit = chain_consume(S, ch, w, ok, full);
    hit = __shfl_sync(0xffffffffu, hit, 0);
    __syncwarp();
    if (hit >= 0) chain_accept(S, w, hit, full, lane);
  };
  if (have) apply(true);
  lap(0);
  for (int guard = 0; guard < 1 << 20; ++guard) {
    if (ch.done) break;
    if (ch.phase == PH_NEW) {
      chain_start_step(S, ch, P.chol, P.learn_out, c, it, lane);
      if (prof && lane == 0) prof[7] += 1;
      lap(1);
    }
    chain_candidates(S, w, c, it, lane);
    lap(2);
    const unsigned inside = w.inside;
    if (inside == 0u) {
      apply(!S.block_free[ch.block]);
      continue;
    }
    if (S.block_free[ch.block]) {
      if ((inside >> lane) & 1u) w.ly[lane] = free_loglike_mixed(L, w.th[lane], ch.kap, HET ? ch.vv : nullptr);
      __syncwarp();
      if (prof && lane == 0) prof[5] += __popc(inside);
      apply(false);
      lap(3);
      continue;
    }
    bool valid = false;
    if ((inside >> lane) & 1u) {
      valid = theta_valid(w.th[lane]);
      if (!valid) w.ly[lane] = -INFINITY;
    }
    const unsigned act = __ballot_sync(0xffffffffu, valid);
    if (act == 0u) {
      apply(true);
      continue;
    }
    if (valid) {
      w.list[__popc(act & ((1u << lane) - 1u))] = lane;
      w.bad[lane] = 0;
    }
    if (lane == 0) {
      w.act = act;
      w.n_act = __popc(act);
      w.fl = S.block_flags[ch.block] | (ch.proj_dirty ? (BF_AMP | BF_PROJ) : 0);
      w.status = ROUND_EVAL;
      if (prof) prof[6] += __popc(inside);
    }
    __syncwarp();
    return;
  }
  if (lane == 0) w.status = ROUND_DONE;
  __syncwarp();
}

// Records of the round's candidates by the whole CTA: the current point's with
// the block's pieces formed anew, one piece per warp and one candidate per lane
// (see k_setup).  Ends with a barrier.
template <int NDET>
__device__ __forceinline__ void chain_setup(const LikeConst& L, ChainWork& w, int warp, int lane) {
  const int fl = w.fl;
  const unsigned act = w.act;
  constexpr int kWords = sizeof(EvalRecord) / 4;
  for (int k = warp; k < w.n_cand; k += kChainWarps)
    if ((act >> k) & 1u) {
      const unsigned* s = reinterpret_cast<const unsigned*>(&w.rx);
      unsigned* d = reinterpret_cast<unsigned*>(&w.rec[k]);
      for (int q = lane; q < kWords; q += 32) d[q] = s[q];
    }
  __syncthreads();
  const int k = lane < kCand ? lane : 0;
  const bool on = (act >> lane) & 1u;
  EvalRecord& r = w.rec[k];
  const double* th = w.th[k];
  if (fl & (BF_INTR | BF_SKY | BF_AMP | BF_PROJ)) {  // uniform
    if (warp == 0) {
      if ((fl & BF_INTR) && on) {
        const MassTerms t = taylorf2_mass_terms(th[0], th[1]);
        r.mterm[0] = t.eta, r.mterm[1] = t.dm, r.mterm[2] = t.m1, r.mterm[3] = t.m2;
        r.mterm[4] = t.A, r.mterm[5] = t.r, r.mterm[6] = t.ir, r.mterm[7] = t.lpm;
      }
    } else if (warp == 1) {
      if ((fl & BF_AMP) && on) setup_amp_f32(th, &r);
    } else if (warp == 2) {
      if ((fl & BF_SKY) && on) sincos(th[9] - L.gmst, &w.sc[0][k], &w.sc[1][k]);
    } else if (warp == 3) {
      if ((fl & BF_SKY) && on) sincos(th[10], &w.sc[2][k], &w.sc[3][k]);
    } else if (warp >= 4 && warp < 4 + NDET) {
      if ((fl & BF_PROJ) && on) setup_projection_det(L, th, warp - 4, true, &r);
    }
    __syncthreads();
  }
  if (warp < 4) {
    const bool need = (fl & BF_INTR) || (warp == 2 && (fl & BF_SPIN)) || (warp == 3 && (fl & BF_TIDE));
    if (need && on) {
      MassTerms t;
      t.eta = r.mterm[0], t.dm = r.mterm[1], t.m1 = r.mterm[2], t.m2 = r.mterm[3];
      t.A = r.mterm[4], t.r = r.mterm[5], t.ir = r.mterm[6], t.lpm = r.mterm[7];
      double cc[NBASIS];
#pragma unroll
      for (int j = 0; j < NBASIS; ++j) cc[j] = 0.0;
      auto put = [&](int j) {
        const dfl d = df_from_double(cc[j]);
        r.c[j] = cc[j];
        r.c_hi[j] = d.hi;
        r.c_lo[j] = d.lo;
      };
      if (warp == 0) {
        taylorf2_low_coeffs(t, cc);
        put(B_M53), put(B_M1), put(B_LOG), put(B_ONE);
      } else if (warp == 1) {
        taylorf2_high_coeffs(t, cc);
        put(B_P13), put(B_P13LOG), put(B_P23);
      } else if (warp == 2) {
        taylorf2_spin_coeffs(t, th[2], th[3], cc);
        put(B_M23), put(B_M13);
      } else {
        taylorf2_tidal_coeffs(t, th[4], th[5], cc);
        put(B_P53), put(B_P73);
      }
    }
  } else if (warp < 4 + NDET) {
    if (on) {
      if (fl & BF_SKY)
        setup_delay_det_sc(L, th, warp - 4, w.sc[0][k], w.sc[1][k], w.sc[2][k], w.sc[3][k], &r);
      else if (fl & BF_TAU)
        setup_tc_det(th, warp - 4, &r);
    }
  } else if (warp == 8) {
    // C_i and <h|h>: candidate lane / 4, detector lane % 4
    const int kk = lane >> 2, i = lane & 3;
    double term = 0.0;
    if ((act >> kk) & 1u) {
      EvalRecord& q = w.rec[kk];
      const double cre = q.amp * q.pre[i], cim = q.amp * q.pim[i];
      q.cre[i] = cre;
      q.cim[i] = cim;
      if (i < L.n_det) term = (cre * cre + cim * cim) * L.K[i];
    }
    double hh = 0.0;
#pragma unroll
    for (int d = 0; d < SWIG_MAX_DET; ++d) hh += __shfl_sync(0xffffffffu, term, (lane & ~3) + d);
    if (i == 0 && ((act >> kk) & 1u)) w.rec[kk].hh = hh;
  }
  __syncthreads();
}

}  // namespace swig
