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
// SMs (a request to every SM's slice of the grid, control on one warp), 12.9 ms
// here; heterodyned, 8 iterations 133 -> 38.9 ms.  1.3 candidates are evaluated
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
constexpr int kFreeRungs = 8;     // rungs per end of a projection-only step, and its draws at a time
constexpr int kChainWarps = kChainBlock / 32;
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
  int n_cand, n_left;        // candidates; stepping out: of them on the left,
  int n_rung;                // ... on both ends (the others are draws ahead)
  double lo, hi;             // the bracket that those draws assume
  int fl;                    // record pieces that the block moves
  int status;
  int bad[kCand];            // folded sums: outside the band, summed bin by bin
  // projection-only steps: a lane's theta, the current point's sums
  float fth[2 * kFreeRungs][SWIG_N_PARAMS];
  float2 fkap[2 * SWIG_MAX_DET], fvv[SWIG_MAX_DET];  // free_loglike's, (hi, lo)
};

enum { ROUND_EVAL = 0, ROUND_DONE = 1 };
constexpr int kGuess0 = 96;  // of 128: the share of right guesses that a chain starts from

// Sign and unit-interval tests on the bits: an FP64 comparison costs the
// scheduler 64 cycles.
__device__ __forceinline__ bool fp64_negative(double v) {  // v < 0 (not -0); v is no NaN
  return __double_as_longlong(v) < 0 && (__double_as_longlong(v) << 1) != 0;
}
__device__ __forceinline__ bool fp64_in_unit(double v) {  // 0 <= v <= 1, false for a NaN
  const long long b = __double_as_longlong(v);
  return (b >= 0 && b <= 0x3FF0000000000000ll) || (b << 1) == 0;
}

// What the rungs of one end say: n of them (candidates first ..), `room` more
// expansions allowed.  moved: expansions; evals: points that the step looked at;
// shut: the end stays; left: it left the unit cube.
struct EndResult {
  int moved, evals;
  bool shut, left;
};
__device__ __forceinline__ EndResult end_result(unsigned inside, unsigned ok, int first, int n, int room) {
  const unsigned in = inside >> first, go = in & (ok >> first);
  EndResult e;
  e.moved = min(__ffs(~go) - 1, n);
  const bool more = e.moved < n;  // a rung that was not taken: the end
  e.left = more && !((in >> e.moved) & 1u);
  e.evals = e.moved + (more && !e.left);
  e.shut = more || e.moved >= room;
  return e;
}

// Apply the results of the pending candidates in the step's order.  ok: the
// candidates whose logL exceeds logL* (bits).  Returns the accepted candidate
// or -1.  All lanes compute; lane 0 writes the state.
__device__ __forceinline__ int chain_consume(const SamplerConst& S, ChainWork& w, unsigned ok, int lane) {
  ChainState& ch = w.ch;
  const int n = w.n_cand, nl = w.n_left, nr = w.n_rung;
  const unsigned inside = w.inside;
  double lo = ch.lo, hi = ch.hi;
  int evals = 0, hit = -1, k = 0, phase = ch.phase, n_shrink = ch.n_shrink;
  if (phase == PH_OUT) {
    int side = ch.side, closed = ch.closed, out = ch.n_out, outr = ch.n_out_r, score = ch.score;
    if (nl > 0) {
      const EndResult e = end_result(inside, ok, 0, nl, kMaxStepOut - out);
      evals += e.evals;
      out += e.moved;
      if (e.moved > 0) lo = e.moved < nl ? w.t[e.moved] : w.t[nl - 1] - 1.0;
      if (e.shut) side &= ~1;
      if (e.left) closed |= 1;
    }
    if (nr > nl) {
      const EndResult e = end_result(inside, ok, nl, nr - nl, kMaxStepOut - outr);
      evals += e.evals;
      outr += e.moved;
      if (e.moved > 0) hi = e.moved < nr - nl ? w.t[nl + e.moved] : w.t[nr - 1] + 1.0;
      if (e.shut) side &= ~2;
      if (e.left) closed |= 2;
    }
    k = n;
    if (side == 0) {
      phase = PH_SHRINK;
      n_shrink = 0;
      score += 16 * (closed == 3) - ((kGuess0 + score) >> 3);
      closed = 0;
      // the draws ahead stand if the bracket became the one they assume
      if (__double_as_longlong(lo) == __double_as_longlong(w.lo) &&
          __double_as_longlong(hi) == __double_as_longlong(w.hi))
        k = nr;
    }
    __syncwarp();
    if (lane == 0) ch.side = side, ch.closed = closed, ch.n_out = out, ch.n_out_r = outr, ch.score = score;
  }
  bool capped = false;
  unsigned ctr = ch.ctr;
  for (; k < n; ++k) {
    ++ctr;  // its uniform
    if ((inside >> k) & 1u) {
      ++evals;
      if ((ok >> k) & 1u) {
        hit = k;
        break;
      }
    }
    const double t = w.t[k];
    if (fp64_negative(t))
      lo = t;
    else
      hi = t;
    if (++n_shrink >= kMaxShrink) {
      capped = true;
      break;
    }
  }
  __syncwarp();
  if (lane == 0) {
    ch.lo = lo, ch.hi = hi, ch.phase = phase, ch.n_shrink = n_shrink, ch.ctr = ctr;
    ch.n_evals += evals;
    ch.n_full += evals;
    if (capped) {
      ++ch.n_caps;
      finish_step(S, ch);
    }
  }
  __syncwarp();
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
    const float* Lb = chol + (size_t)b * kMaxDim * kMaxDim;
    float row[kMaxDim];  // (CTA 0 writes L_b: through L2)
#pragma unroll
    for (int q = 0; q < kMaxDim; ++q) row[q] = q < nb && q <= lane && lane < nb ? __ldcg(&Lb[lane * kMaxDim + q]) : 0.0f;
    // z_r, r < nb, one Philox block each at consecutive counters
    float z = 0.0f;
    if (lane < nb) {
      const uint4 r = philox4x32_10(make_uint4(ctr + (unsigned)lane, (unsigned)c, (unsigned)it, 0u), S.key0, S.key1);
      const float u1 = ((float)(r.x >> 8) + 1.0f) * (1.0f / 16777216.0f);
      const float u2 = (float)(r.y >> 8) * (1.0f / 16777216.0f);
      z = sqrtf(-2.0f * logf(u1)) * cospif(2.0f * u2);
    }
    ctr += (unsigned)nb;
    float v = 0.0f;
#pragma unroll
    for (int q = 0; q < kMaxDim; ++q)
      if (q < nb) {
        const float zq = __shfl_sync(0xffffffffu, z, q);
        if (lane < nb && q <= lane) v = fmaf(row[q], zq, v);
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
//
// While most steps come to the cube's boundary on both ends (75 % in a run's
// first iterations, 22 % late), a round that steps out also takes the first
// draws of the shrinkage, from the bracket that this would leave: both ends at
// the last rung inside.  A right guess saves the step a round; a wrong one costs
// two candidates.  Taken where the guess held for half of the chain's last eight
// steps or so (late, with either this guess or that neither end moves, the
// candidates cost more than the rounds: 250 iterations 1.28 -> 1.43 s).
__device__ __forceinline__ void chain_candidates(const SamplerConst& S, ChainWork& w, int c, long long it, int lane) {
  ChainState& ch = w.ch;
  const int b = ch.block, nb = S.block_size[b];
  const auto at = [&](int j, double t) { return ch.x[j] + t * ch.dir[j]; };
  // draws first .. first + n - 1 (lanes) of a bracket, each after the ones
  // before it were rejected
  const auto draws = [&](double lo, double hi, int first, int n) {
    const double u = u01_from(philox4x32_10(make_uint4(ch.ctr + (unsigned)(lane - first), (unsigned)c, (unsigned)it, 0u),
                                            S.key0, S.key1));
    double t = 0.0;
    for (int k = first; k < first + n; ++k) {
      const double tk = lo + (hi - lo) * __shfl_sync(0xffffffffu, u, k);
      if (lane == k) t = tk;
      if (fp64_negative(tk))
        lo = tk;
      else
        hi = tk;
    }
    return t;
  };
  int n, nl = 0, nr = 0;
  double t = 0.0;
  if (ch.phase == PH_OUT) {
    const bool l = ch.side & 1, r = (ch.side & 2) && !(S.one_end && l);
    // an end alone may use both ends' rungs; rungs 0 .. 7 on lanes 0 .. 7
    // (left) and 8 .. 15 (right)
    const int d = l && r ? S.spec_out : min(2 * S.spec_out, kCand);
    const int dl = l ? min(d, kMaxStepOut - ch.n_out) : 0, dr = r ? min(d, kMaxStepOut - ch.n_out_r) : 0;
    const bool right = lane & 8;
    const int m = lane & 7;
    // rung by rung, as the step moves its end (each addition rounds)
    t = right ? ch.hi : ch.lo;
    for (int i = 1; i < max(dl, dr); ++i)
      if (i <= m) t += right ? 1.0 : -1.0;
    bool in = lane < 16 && m < (right ? dr : dl);
    if (in)
      for (int q = 0; q < nb; ++q)
        if (!fp64_in_unit(at(S.block_dims[b][q], t))) in = false;
    const unsigned ins = __ballot_sync(0xffffffffu, in);
    // rungs inside the cube in a row; the next one closes the end unseen
    const int cl = __ffs(~(ins & 0xffu)) - 1, cr = __ffs(~((ins >> 8) & 0xffu)) - 1;
    nl = min(cl + 1, dl);
    nr = nl + min(cr + 1, dr);
    const double lo = l ? __shfl_sync(0xffffffffu, t, min(cl, 7)) : ch.lo;
    const double hi = r ? __shfl_sync(0xffffffffu, t, 8 + min(cr, 7)) : ch.hi;
    // (a guess needs the rungs that leave the cube, on every open end)
    const bool ahead = S.spec_mix > 0 && kGuess0 + ch.score >= 64 && r == ((ch.side & 2) != 0) &&
                       (!l || cl < dl) && (!r || cr < dr);
    int nd = 0;
    if (ahead) {
      nd = S.spec_mix;
      if (nd > 1) nd += (min(cl, dl) + min(cr, dr) + nd) & 1;  // candidates go in pairs
      nd = min(nd, kCand - nr);
    }
    n = nr + nd;
    t = __shfl_sync(0xffffffffu, t, lane < nl ? lane : lane < nr ? 8 + lane - nl : 0);
    const double td = draws(lo, hi, nr, nd);
    if (lane >= nr) t = td;
    if (lane == 0) {
      w.lo = lo;
      w.hi = hi;
    }
  } else {
    n = min(S.spec_shr, kMaxShrink - ch.n_shrink);
    t = draws(ch.lo, ch.hi, 0, n);
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
      const double v = at(j, t);
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
    w.n_rung = nr;
    w.inside = m;
  }
  __syncwarp();
}

// Accept candidate k: point, theta, logL, per-detector sums and the record.
// All lanes.
__device__ __forceinline__ void chain_accept(const SamplerConst& S, ChainWork& w, int k, int lane) {
  ChainState& ch = w.ch;
  const int b = ch.block;
  if (lane < S.ndim && ((S.block_mask[b] >> lane) & 1u)) ch.x[lane] = w.y[k][lane];
  if (lane < SWIG_N_PARAMS) ch.th[lane] = w.th[k][lane];
  if (lane < 2 * SWIG_MAX_DET) ch.kap[lane] = w.kap[k][lane];
  if (lane < SWIG_MAX_DET) ch.vv[lane] = w.vv[k][lane];
  warp_copy(&w.rx, &w.rec[k], sizeof(EvalRecord), lane);
  __syncwarp();
  if (lane == 0) {
    ch.lx = w.ly[k];
    ch.proj_dirty = 0;
    finish_step(S, ch);
  }
  __syncwarp();
}

// A whole slice step of a projection-only block, whose logL follows from the
// current point's sums: a candidate per lane, up to kFreeRungs rungs of each end
// (left on lanes 0 .. 7, right on 8 .. 15) or as many draws at a time, the
// decisions by ballots.  Points, draws and counts are those of one candidate
// after another.  Returns the points evaluated.
template <bool HET>
__device__ __forceinline__ int chain_free_step(const LikeConst& L, const SamplerConst& S, ChainWork& w, int c,
                                               long long it, double logl_star, int lane) {
  ChainState& ch = w.ch;
  const int b = ch.block, nb = S.block_size[b];
  const int row = lane & (2 * kFreeRungs - 1);
  float* th = w.fth[row];
  {
    // rounded once, a value per lane
    const int j = lane - SWIG_N_PARAMS, i = j - 2 * SWIG_MAX_DET;
    double x = 0.0;
    if (j < 0)
      x = ch.th[lane];
    else if (i < 0)
      x = ch.kap[j] * L.amp_s[j >> 1];
    else if (i < SWIG_MAX_DET)
      x = HET ? ch.vv[i] : L.amp_k[i];
    const dfl v = df_from_double(x);
    const float f = v.hi;
    if (j >= 0 && i < 0) w.fkap[j] = make_float2(v.hi, v.lo);
    if (i >= 0 && i < SWIG_MAX_DET) w.fvv[i] = make_float2(v.hi, v.lo);
#pragma unroll
    for (int s = 0; s < SWIG_N_PARAMS; ++s) {
      const float v = __shfl_sync(0xffffffffu, f, s);
      if (lane < 2 * kFreeRungs) th[s] = v;
    }
    __syncwarp();
  }
  // logL at bracket coordinate t of the lanes that are on (bits: inside, above logL*)
  double ly = 0.0;
  const auto look = [&](double t, bool on, unsigned& inside, unsigned& ok) {
    bool in = on;
    if (on)
      for (int r = 0; r < nb; ++r) {
        const int j = S.block_dims[b][r], slot = S.slot_of_dim[j];
        const double v = ch.x[j] + t * ch.dir[j];
        if (!fp64_in_unit(v)) in = false;
        if (in) th[slot] = (float)prior_slot_inverse_f32(S.prior[slot], v);
      }
    inside = __ballot_sync(0xffffffffu, in);
    if (in) ly = free_loglike(L, th, w.fkap, w.fvv);
    ok = __ballot_sync(0xffffffffu, in && ly > logl_star);
    __syncwarp();
  };
  double lo = ch.lo, hi = ch.hi;
  int evals = 0, seen = 0, side = 3, out = 0, outr = 0;
  unsigned inside, ok;
  while (side) {
    const int dl = side & 1 ? min(kFreeRungs, kMaxStepOut - out) : 0;
    const int dr = side & 2 ? min(kFreeRungs, kMaxStepOut - outr) : 0;
    const bool right = lane >= kFreeRungs;
    const int m = lane & (kFreeRungs - 1);
    double t = right ? hi : lo;  // rung by rung (each addition rounds)
    for (int i = 1; i < kFreeRungs; ++i)
      if (i <= m) t += right ? 1.0 : -1.0;
    look(t, lane < 2 * kFreeRungs && m < (right ? dr : dl), inside, ok);
    seen += __popc(inside);
    if (dl > 0) {
      const EndResult e = end_result(inside & ((1u << kFreeRungs) - 1u), ok, 0, dl, kMaxStepOut - out);
      evals += e.evals;
      out += e.moved;
      const double tn = __shfl_sync(0xffffffffu, t, min(e.moved, kFreeRungs - 1));
      lo = e.moved < kFreeRungs ? tn : tn - 1.0;
      if (e.shut) side &= ~1;
    }
    if (dr > 0) {
      const EndResult e = end_result(inside, ok, kFreeRungs, dr, kMaxStepOut - outr);
      evals += e.evals;
      outr += e.moved;
      const double tn = __shfl_sync(0xffffffffu, t, kFreeRungs + min(e.moved, kFreeRungs - 1));
      hi = e.moved < kFreeRungs ? tn : tn + 1.0;
      if (e.shut) side &= ~2;
    }
  }
  unsigned ctr = ch.ctr;
  int n_shrink = 0, hit = -1;
  double t = 0.0;
  while (hit < 0 && n_shrink < kMaxShrink) {
    const int n = min(kFreeRungs, kMaxShrink - n_shrink);
    const double u = u01_from(philox4x32_10(make_uint4(ctr + (unsigned)lane, (unsigned)c, (unsigned)it, 0u), S.key0,
                                            S.key1));
    for (int k = 0; k < n; ++k) {  // each draw after the ones before it were rejected
      const double tk = lo + (hi - lo) * __shfl_sync(0xffffffffu, u, k);
      if (lane == k) t = tk;
      if (fp64_negative(tk))
        lo = tk;
      else
        hi = tk;
    }
    look(t, lane < n, inside, ok);
    seen += __popc(inside);
    hit = __ffs(ok) - 1;
    const int used = hit >= 0 ? hit + 1 : n;
    evals += __popc(inside & ((1u << used) - 1u));
    ctr += (unsigned)used;
    n_shrink += used;
  }
  __syncwarp();
  if (hit >= 0) {
    if (lane == hit) {
      for (int r = 0; r < nb; ++r) {
        const int j = S.block_dims[b][r], slot = S.slot_of_dim[j];
        const double v = ch.x[j] + t * ch.dir[j];
        ch.x[j] = v;
        ch.th[slot] = prior_slot_inverse_f32(S.prior[slot], v);
      }
      ch.lx = ly;
      ch.proj_dirty = 1;
    }
  }
  __syncwarp();
  if (lane == 0) {
    ch.ctr = ctr;
    ch.n_evals += evals;
    if (hit < 0) ++ch.n_caps;
    finish_step(S, ch);
  }
  __syncwarp();
  return seen;
}

// Warp 0 between two evaluations: apply the results (have: a round is pending,
// its logL in w.ly), then advance to the next round that needs the CTA.
// Projection-only blocks are evaluated here, a candidate per lane.  beat: raised
// after eight of their steps (grid_sync).
template <int NDET, bool HET>
__device__ __forceinline__ void chain_control(const LikeConst& L, const SamplerConst& S, const SamplerPtrs& P,
                                              ChainWork& w, int c, long long it, double logl_star, bool have,
                                              int lane, unsigned long long* prof, unsigned* beat) {
  ChainState& ch = w.ch;
  long long tk = clock64();
  auto lap = [&](int slot) {
    if (prof && lane == 0) {
      const long long t2 = clock64();
      prof[slot] += t2 - tk;
      tk = t2;
    }
  };
  auto apply = [&] {
    const bool in = lane < w.n_cand && ((w.inside >> lane) & 1u);
    const unsigned ok = __ballot_sync(0xffffffffu, in && w.ly[lane < kCand ? lane : 0] > logl_star);
    const int hit = chain_consume(S, w, ok, lane);
    if (hit >= 0) chain_accept(S, w, hit, lane);
  };
  if (have) apply();
  lap(0);
  for (int guard = 0; guard < 1 << 20; ++guard) {
    if (ch.done) break;
    if (ch.phase == PH_NEW) {
      chain_start_step(S, ch, P.chol, P.learn_out, c, it, lane);
      if (prof && lane == 0) prof[7] += 1;
      lap(1);
    }
    if (S.block_free[ch.block]) {
      const int seen = chain_free_step<HET>(L, S, w, c, it, logl_star, lane);
      if (prof && lane == 0) prof[5] += seen;
      if (lane == 0 && (guard & 7) == 7) atomicAdd(beat, 1u);
      lap(3);
      continue;
    }
    chain_candidates(S, w, c, it, lane);
    const unsigned inside = w.inside;
    if (inside == 0u) {
      lap(2);
      apply();
      continue;
    }
    bool valid = false;
    if ((inside >> lane) & 1u) {
      valid = theta_valid_bits(w.th[lane]);
      if (!valid) w.ly[lane] = -INFINITY;
    }
    const unsigned act = __ballot_sync(0xffffffffu, valid);
    if (act == 0u) {
      lap(2);
      apply();
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
    lap(2);
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
