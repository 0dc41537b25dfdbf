// Learned slice proposal on the device: initialisation, training targets,
// BF16 tensor-core matrix products (FP32 accumulation), loss and Adam, two
// kernels a training step.  See mlp.h for the model.
//
// Every kernel is deterministic (fixed summation orders, split-K partials
// summed in split order); the same inputs give bit-identical parameters.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>

#include "device_common.cuh"
#include "kernels.h"
#include "mlp.h"

namespace swig {

namespace {

constexpr int kTargetWarps = 4;
constexpr int kMaxNbr = 2 * kMlpIn;
constexpr int kMaxCand = 128;
constexpr int kPowerIters = 600;
constexpr int kRowThreads = 512;
constexpr int kBiasBlocks = 2 * (kMlpH / 4) + (kMlpOut + 3) / 4;
constexpr int kColChunk = 64;  // rows of a stage of the gradients' ring
constexpr int kLdC = 48 + 8;   // their length in shared memory: 16-byte units, an odd number

// rows with the padding that the products read
__host__ __device__ constexpr int mlp_rows(int n) { return (n + 15) / 16 * 16; }

__device__ __forceinline__ float silu_f(float z) { return z / (1.0f + expf(-z)); }
__device__ __forceinline__ float dsilu_f(float z) {
  const float s = 1.0f / (1.0f + expf(-z));
  return s * (1.0f + z * (1.0f - s));
}

// ---------------------------------------------------------------------------
// Initial weights: W[i][j] = Box-Muller(Philox(j, i, layer, 9)) / sqrt(fan_in)
// ---------------------------------------------------------------------------
__global__ void k_mlp_init(float* params, unsigned k0, unsigned k1) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= kMlpParams) return;
  int layer, fan_in, cols, base;
  if (p < kMlpOffB1) {
    layer = 0, fan_in = kMlpIn, cols = kMlpH, base = kMlpOffW1;
  } else if (p < kMlpOffW2) {
    params[p] = 0.0f;
    return;
  } else if (p < kMlpOffB2) {
    layer = 2, fan_in = kMlpH, cols = kMlpH, base = kMlpOffW2;
  } else if (p < kMlpOffW3) {
    params[p] = 0.0f;
    return;
  } else if (p < kMlpOffB3) {
    layer = 4, fan_in = kMlpH, cols = kMlpOut, base = kMlpOffW3;
  } else {
    params[p] = 0.0f;
    return;
  }
  const int q = p - base, i = q / cols, j = q % cols;
  const uint4 r = philox4x32_10(make_uint4((unsigned)j, (unsigned)i, (unsigned)layer, 9u), k0, k1);
  const double u1 = ((double)(r.x >> 8) + 1.0) * (1.0 / 16777216.0);
  const double u2 = (double)(r.y >> 8) * (1.0 / 16777216.0);
  params[p] = (float)(sqrt(-2.0 * log(u1)) * cos(6.283185307179586 * u2) / sqrt((double)fan_in));
}

// BF16 copies of the weights in the padded layouts of the matrix products.
__device__ __forceinline__ void write_bf16_weight(int p, float w, __nv_bfloat16* w1b, __nv_bfloat16* w2b,
                                                  __nv_bfloat16* w3b) {
  if (p < kMlpOffB1) {
    w1b[p - kMlpOffW1] = __float2bfloat16_rn(w);  // [13][256] inside [16][256]
  } else if (p >= kMlpOffW2 && p < kMlpOffB2) {
    w2b[p - kMlpOffW2] = __float2bfloat16_rn(w);
  } else if (p >= kMlpOffW3 && p < kMlpOffB3) {
    const int q = p - kMlpOffW3;
    w3b[(q / kMlpOut) * kMlpOutPad + q % kMlpOut] = __float2bfloat16_rn(w);
  }
}

__global__ void k_mlp_bf16_weights(const float* params, __nv_bfloat16* w1b, __nv_bfloat16* w2b, __nv_bfloat16* w3b) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < kMlpParams) write_bf16_weight(p, params[p], w1b, w2b, w3b);
}

// ---------------------------------------------------------------------------
// Live-set statistics, network inputs and local-PCA targets
// ---------------------------------------------------------------------------
// mean and population standard deviation (floored at 1e-12) per dimension;
// one warp and block per dimension, fixed-order lane sums and shuffle tree
__global__ void k_live_stats(const double* u, int n, int d, double* stats) {
  const int w = blockIdx.x, lane = threadIdx.x;
  double s = 0.0;
#pragma unroll 8
  for (int i = lane; i < n; i += 32) s += u[(size_t)i * d + w];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  const double mu = s / (double)n;
  double v = 0.0;
#pragma unroll 8
  for (int i = lane; i < n; i += 32) {
    const double t = u[(size_t)i * d + w] - mu;
    v += t * t;
  }
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) {
    stats[w] = mu;
    stats[kMlpIn + w] = fmax(sqrt(v / (double)n), 1e-12);
  }
}

// standardised coordinates (FP64, n x d; FP32 by dimension, rows ld apart) and
// the BF16 network inputs (n x 16, zero rows up to the next multiple of 16)
__global__ void k_standardise(const double* u, int n, int d, const double* stats, double* xs, float* xf, int ld,
                              __nv_bfloat16* xb) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= mlp_rows(n) * kMlpInPad) return;
  const int i = e / kMlpInPad, j = e % kMlpInPad;
  if (i < n && j < d) {
    const double x = (u[(size_t)i * d + j] - stats[j]) / stats[kMlpIn + j];
    xs[(size_t)i * d + j] = x;
    xf[(size_t)j * ld + i] = (float)x;
    xb[e] = __float2bfloat16_rn((float)x);
  } else {
    xb[e] = __float2bfloat16_rn(0.0f);
  }
}

__global__ void k_inputs_f32(const float* x, int n, __nv_bfloat16* xb) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= mlp_rows(n) * kMlpInPad) return;
  const int i = e / kMlpInPad, j = e % kMlpInPad;
  xb[e] = __float2bfloat16_rn(i < n && j < kMlpIn ? x[(size_t)i * kMlpIn + j] : 0.0f);
}

struct PcaWarp {
  double dist[kMaxCand];          // exact squared distances of the candidates
  int cand[kMaxCand];             // candidates, by index
  int nb[kMaxNbr];                // neighbours, nearest first
  double x[kMaxNbr * kMlpIn];     // neighbours' coordinates about their mean
  double mean[kMlpIn], sig[kMlpIn], v[kMlpIn];
  double m[2][kMlpIn * kMlpIn];   // correlation matrix and its powers
};

// y = M v, then v = y / |y| (v stays where y vanishes)
__device__ __forceinline__ void power_step(const double* m, double* v, int d, int lane) {
  double y = 0.0;
  if (lane < d)
    for (int b = 0; b < d; ++b) y += m[lane * d + b] * v[b];
  double nn = lane < d ? y * y : 0.0;
  for (int o = 8; o > 0; o >>= 1) nn += __shfl_xor_sync(0xffffffffu, nn, o);
  __syncwarp();
  if (lane < d && nn > 0.0) v[lane] = y / sqrt(nn);
  __syncwarp();
}

// One warp per live point: the k nearest other points in standardised
// coordinates (ties by index), their covariance in unit-cube coordinates, log
// standard deviations, and the leading eigenvector of the correlation matrix R
// by kPowerIters power iterations from (1, .., 1) (sign: largest-magnitude
// entry positive).
//
// FP64 instructions bound this kernel: each occupies a scheduler for 64
// cycles, whatever the lanes in use.  So the distances are first taken in FP32
// with a bound on their error, and in FP64 only for the points that may be
// among the k nearest: with T the k-th smallest of the lanes' minima (k <= 26
// lanes have a point at most that far away), those whose FP32 distance less
// its bound is at most T plus its bound, about 1.4 x 32 points however large n
// is.  FP64 distances decide, as they would over all points.  More than
// kMaxCand candidates (many equal points) take FP64 distances over all.
// The power iterations are R^600 = R^8 R^16 R^64 R^512, each power by
// squaring (scaled by powers of two) and one product with the vector: 9
// symmetric squarings and 4 products for 600 dependent ones.
// 1000 points x 12 dimensions: 2.9 ms with FP64 distances per neighbour and
// 600 products, 0.10 ms now.
__global__ void __launch_bounds__(32 * kTargetWarps) k_local_pca(const double* u, const double* xs, const float* xf,
                                                               int ld, int n, int d, int k, float* tdir, float* tls,
                                                               int* nbr) {
  __shared__ PcaWarp s_w[kTargetWarps];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * kTargetWarps + w;
  if (i >= n) return;
  PcaWarp& s = s_w[w];
  float xi[kMlpIn];
#pragma unroll
  for (int q = 0; q < kMlpIn; ++q) xi[q] = q < d ? xf[(size_t)q * ld + i] : 0.0f;
  const auto dist32 = [&](int j) {
    float f = 0.0f;
#pragma unroll
    for (int q = 0; q < kMlpIn; ++q)
      if (q < d) {
        const float t = xf[(size_t)q * ld + j] - xi[q];
        f += t * t;
      }
    return f;
  };
  const auto dist64 = [&](int j) {
    double dd = 0.0;
    for (int q = 0; q < d; ++q) {
      const double t = xs[(size_t)j * d + q] - xs[(size_t)i * d + q];
      dd += t * t;
    }
    return dd;
  };
  float lo = INFINITY;
  for (int j = lane; j < n; j += 32) {
    const float f = dist32(j);
    if (j != i && f < lo) lo = f;
  }
  int below = 0;
  for (int o = 0; o < 32; ++o) {
    const float t = __shfl_sync(0xffffffffu, lo, o);
    below += t < lo || (t == lo && o < lane);
  }
  const unsigned kth = __ballot_sync(0xffffffffu, below == k - 1);
  // |x| <= sqrt(n) (standardised over n points), so a difference is off by at
  // most a = 4 x 2^-24 sqrt(n), and the sum f of d squares by
  // E(f) = 2 a sqrt(d f) + d a^2 + 2^-20 f; thr solves f - E(f) = T + E(T)
  float thr = INFINITY;
  if (kth) {
    const float T = __shfl_sync(0xffffffffu, lo, __ffs(kth) - 1);
    const float eps = 9.5367432e-7f, a = 2.4e-7f * sqrtf((float)n);
    const float b = 1.01f * a * sqrtf((float)d), c = 1.01f * (float)d * a * a;
    const float rhs = T + 2.0f * b * sqrtf(T) + c + eps * T + c;
    const float r = (b + sqrtf(b * b + rhs)) / (1.0f - eps);
    thr = r * r * (1.0f + 1e-5f);
  }
  int nc = 0;
  for (int j0 = 0; j0 < n; j0 += 32) {
    const int j = j0 + lane;
    const bool in = j < n && j != i && dist32(min(j, n - 1)) <= thr;
    const unsigned m = __ballot_sync(0xffffffffu, in);
    const int at = nc + __popc(m & ((1u << lane) - 1u));
    if (in && at < kMaxCand) s.cand[at] = j;
    nc += __popc(m);
  }
  __syncwarp();
  if (nc >= k && nc <= kMaxCand) {
    for (int c = lane; c < nc; c += 32) s.dist[c] = dist64(s.cand[c]);
    __syncwarp();
    for (int c = lane; c < nc; c += 32) {
      // non-negative doubles compare like their bits
      const long long mine = __double_as_longlong(s.dist[c]);
      int rank = 0;
      for (int o = 0; o < nc; ++o) {
        const long long other = __double_as_longlong(s.dist[o]);
        rank += other < mine || (other == mine && o < c);
      }
      if (rank < k) s.nb[rank] = s.cand[c];
    }
  } else {
    double last_d = -1.0;
    int last_j = -1;
    for (int r = 0; r < k; ++r) {
      double bd = INFINITY;
      int bj = INT_MAX;
      for (int j = lane; j < n; j += 32) {
        if (j == i) continue;
        const double dd = dist64(j);
        const bool after = dd > last_d || (dd == last_d && j > last_j);
        const bool better = dd < bd || (dd == bd && j < bj);
        if (after && better) {
          bd = dd;
          bj = j;
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const double od = __shfl_xor_sync(0xffffffffu, bd, o);
        const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
        if (od < bd || (od == bd && oj < bj)) {
          bd = od;
          bj = oj;
        }
      }
      last_d = bd;
      last_j = bj;
      if (lane == 0) s.nb[r] = bj < n ? bj : i;  // no comparable distance: coordinates that are not numbers
    }
  }
  __syncwarp();
  // covariance of the neighbours (1/k normalisation)
  if (lane < d) {
    double t = 0.0;
    for (int r = 0; r < k; ++r) t += u[(size_t)s.nb[r] * d + lane];
    s.mean[lane] = t / (double)k;
  }
  __syncwarp();
  for (int e = lane; e < k * d; e += 32) s.x[e] = u[(size_t)s.nb[e / d] * d + e % d] - s.mean[e % d];
  __syncwarp();
  const int pairs = d * (d + 1) / 2;
  const auto pair_of = [&](int e, int& a, int& b) {  // a <= b
    a = 0;
    while (e >= d - a) e -= d - a, ++a;
    b = a + e;
  };
  int pa[3], pb[3];  // this lane's entries of a symmetric matrix (91 at most)
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    pa[q] = pb[q] = 0;
    if (lane + 32 * q < pairs) pair_of(lane + 32 * q, pa[q], pb[q]);
  }
#pragma unroll
  for (int q = 0; q < 3; ++q)
    if (lane + 32 * q < pairs) {
      double t = 0.0;
      for (int r = 0; r < k; ++r) t += s.x[r * d + pa[q]] * s.x[r * d + pb[q]];
      s.m[1][pa[q] * d + pb[q]] = t / (double)k;
    }
  __syncwarp();
  double sig = 1.0;
  if (lane < d) {
    sig = fmax(sqrt(s.m[1][lane * d + lane]), 1e-12);
    s.sig[lane] = sig;
    s.v[lane] = 1.0 / sqrt((double)d);
  }
  __syncwarp();
  // R_ab = C_ab / (sig_a sig_b)
#pragma unroll
  for (int q = 0; q < 3; ++q)
    if (lane + 32 * q < pairs) {
      const int a = pa[q], b = pb[q];
      s.m[0][a * d + b] = s.m[0][b * d + a] = s.m[1][a * d + b] / (s.sig[a] * s.sig[b]);
    }
  __syncwarp();
  if (d == 2) {
    // (1, 1) is an eigenvector of every 2 x 2 correlation matrix and only
    // rounding moves the iteration off it: the products one by one, as the
    // definition has them
    for (int it = 0; it < kPowerIters; ++it) power_step(s.m[0], s.v, d, lane);
  } else {
    int cur = 0;
    for (int p = 1; p <= kPowerIters; p *= 2) {
      const double* m = s.m[cur];
      if (kPowerIters & p) power_step(m, s.v, d, lane);
      if (2 * p > kPowerIters) break;
      double* m2 = s.m[cur ^ 1];
      // the largest entry, on the diagonal, grows from 1 by 13 at most and
      // then as its square: a power of two brings it back when it is large
      long long top = 0;  // (non-negative doubles compare like their bits)
      for (int a = 0; a < d; ++a) top = max(top, __double_as_longlong(m[a * d + a]));
      const int ex = (int)(top >> 52) - 1023;
      const bool large = ex >= 128 && ex < 1024;
      const double sc = __hiloint2double((1023 - (large ? 2 * min(ex, 500) : 0)) << 20, 0);
#pragma unroll
      for (int q = 0; q < 3; ++q)
        if (lane + 32 * q < pairs) {
          const int a = pa[q], b = pb[q];
          double t = 0.0;
          for (int c = 0; c < d; ++c) t += m[a * d + c] * m[c * d + b];
          if (large) t *= sc;
          m2[a * d + b] = m2[b * d + a] = t;
        }
      __syncwarp();
      cur ^= 1;
    }
  }
  // sign: the largest-magnitude entry (first on ties) positive
  double best = -1.0;
  int arg = 0;
  for (int b = 0; b < d; ++b) {
    const double a = fabs(s.v[b]);
    if (a > best) {
      best = a;
      arg = b;
    }
  }
  const double sgn = s.v[arg] < 0.0 ? -1.0 : 1.0;
  if (lane < kMlpIn) {
    tdir[(size_t)i * kMlpIn + lane] = lane < d ? (float)(sgn * s.v[lane]) : 0.0f;
    tls[(size_t)i * kMlpIn + lane] = lane < d ? (float)log(sig) : 0.0f;
  }
  if (lane < k && nbr) nbr[(size_t)i * kMaxNbr + lane] = s.nb[lane];
}

// ---------------------------------------------------------------------------
// Matrix products: BF16 operands, FP32 accumulation with mma.sync m16n8k16,
// from zero in the order of k.  The operands of one step are small (W2 is 128
// KB) and the step is a chain of five dependent products, so launches, not
// tensor throughput, bound it: a row kernel takes 16 rows through the forward
// pass, the loss and the backward pass with the activations in registers and
// shared memory, and a column kernel forms the weight gradients and applies
// Adam to them.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void mma_bf16_16816(float* d, const unsigned* a, const unsigned* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

template <bool TRANS>
__device__ __forceinline__ void ldsm4(unsigned* r, const __nv_bfloat16* p) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  if constexpr (TRANS)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}
__device__ __forceinline__ void ldsm2_trans(unsigned* r, const __nv_bfloat16* p) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(a) : "memory");
}
__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// The next kernel of the step may be set up while this one runs; it waits for
// this grid's end before it touches memory.
__device__ __forceinline__ void chain_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

struct RowArgs {
  const float* params;
  const __nv_bfloat16 *w1b, *w2b, *w3b, *xb;
  const float *tdir, *tls;
  int n, d;
  float* out;  // [n][32], or null
  float *dout, *dz2, *dz1;
  __nv_bfloat16 *h1b, *h2b, *doutb, *dz2b, *dz1b;
  double* row_loss;  // or null
};

// Row lengths in shared memory: 16 bytes more than a multiple of 128, so that
// the eight rows of a matrix load meet all banks.
constexpr int kLdH = kMlpH + 8, kLdO = kMlpOutPad + 8, kLdX = kMlpInPad + 8;
struct RowShared {
  __nv_bfloat16 w2[kMlpH * kLdH];
  __nv_bfloat16 w1[kMlpInPad * kLdH];
  __nv_bfloat16 w3[kMlpH * kLdO];
  __nv_bfloat16 ha[16 * kLdH];  // h1, then dz2
  __nv_bfloat16 hb[16 * kLdH];  // h2, then dz1
  __nv_bfloat16 dO[16 * kLdO];
  __nv_bfloat16 x[16 * kLdX];
  float out[16 * kMlpOutPad];
  float bias[2 * kMlpH + kMlpOutPad];
};

// One block per 16 rows (blocks stride over tiles beyond one per SM, keeping
// the weights in shared memory), a warp per 16 of the 256 hidden units: z1 and
// z2 stay in the registers that the backward pass wants them in.
// TRAIN false: outputs only.  1000 rows: about 9 us, of which 2.6 us until the
// weights are there (taken in the order of their use, W2 in four groups: a step
// 20.5 -> 19.9 us) and 1.1 us for each 256 x 256 product (the shared memory they
// are read from); 16 rows are the least that the product takes, so 63 SMs work.
template <bool TRAIN>
__global__ void __launch_bounds__(kRowThreads) k_mlp_rows(RowArgs g) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  RowShared& s = *reinterpret_cast<RowShared*>(s_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3;
  const int c0 = 16 * warp;  // this warp's hidden units
  chain_launch();
  chain_wait();
  for (int e = tid; e < kMlpInPad * (kMlpH / 8); e += kRowThreads)
    copy16(s.w1 + (e / (kMlpH / 8)) * kLdH + e % (kMlpH / 8) * 8, g.w1b + e * 8);
  if (tid < kMlpH / 4) copy16(s.bias + 4 * tid, g.params + kMlpOffB1 + 4 * tid);
  const int tiles = mlp_rows(g.n) / 16;
  // lane addresses of the fragments: A [row][k]; B from [k][col] (transposed
  // on the way) and from [col][k]
  const int la = (lane & 7) + ((lane >> 3) & 1) * 8, lk = (lane >> 4) * 8;
  const int lb = (lane & 7) + (lane >> 4) * 8, lc = ((lane >> 3) & 1) * 8;
  bool first = true;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int r0 = 16 * tile;
    if (tid < 32) copy16(s.x + (tid >> 1) * kLdX + (tid & 1) * 8, g.xb + (size_t)r0 * kMlpInPad + tid * 8);
    copy_commit();
    // the first tile's weights follow in the order of their use, a group each
    if (first) {
#pragma unroll
      for (int part = 0; part < 4; ++part) {
        for (int e = part * (kMlpH / 4) * (kMlpH / 8) + tid; e < (part + 1) * (kMlpH / 4) * (kMlpH / 8); e += kRowThreads)
          copy16(s.w2 + (e / (kMlpH / 8)) * kLdH + e % (kMlpH / 8) * 8, g.w2b + e * 8);
        if (part == 0 && tid < kMlpH / 4) copy16(s.bias + kMlpH + 4 * tid, g.params + kMlpOffB2 + 4 * tid);
        copy_commit();
      }
      for (int e = tid; e < kMlpH * (kMlpOutPad / 8); e += kRowThreads)
        copy16(s.w3 + (e / (kMlpOutPad / 8)) * kLdO + e % (kMlpOutPad / 8) * 8, g.w3b + e * 8);
      if (tid < kMlpOutPad / 4) copy16(s.bias + 2 * kMlpH + 4 * tid, g.params + kMlpOffB3 + 4 * tid);
      copy_commit();
    }
    float tgt = 0.0f;  // this lane's target of the warp's row: direction, then log-widths
    if (TRAIN && r0 + warp < g.n) {
      if (lane < kMlpIn) tgt = g.tdir[(size_t)(r0 + warp) * kMlpIn + lane];
      else if (lane < 2 * kMlpIn) tgt = g.tls[(size_t)(r0 + warp) * kMlpIn + lane - kMlpIn];
    }
    if (first)
      copy_wait<5>();
    else
      copy_wait<0>();
    __syncthreads();
    // Z1 = X W1 + b1
    float z1[2][4], z2[2][4];
    const auto zero = [](float (&a)[2][4]) {
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int q = 0; q < 4; ++q) a[t][q] = 0.0f;
    };
    // pre-activation and BF16 activation of an accumulated tile
    const auto hidden = [&](float (&z)[2][4], const float* bias, __nv_bfloat16* h) {
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int col = c0 + 8 * t + 2 * tig;
          float v0 = 0.0f + z[t][2 * r], v1 = 0.0f + z[t][2 * r + 1];
          v0 += bias[col];
          v1 += bias[col + 1];
          z[t][2 * r] = v0;
          z[t][2 * r + 1] = v1;
          __nv_bfloat162 p;
          p.x = __float2bfloat16_rn(silu_f(v0));
          p.y = __float2bfloat16_rn(silu_f(v1));
          *reinterpret_cast<__nv_bfloat162*>(h + (gid + 8 * r) * kLdH + col) = p;
        }
    };
    // rows of a shared tile to global memory; zero beyond the last row, which
    // the gradients' products read to a multiple of 16
    const auto put_rows = [&](const __nv_bfloat16* h, __nv_bfloat16* dst) {
      const int row = tid >> 5, col = (tid & 31) * 8;
      const uint4 v = r0 + row < g.n ? *reinterpret_cast<const uint4*>(h + row * kLdH + col) : make_uint4(0, 0, 0, 0);
      *reinterpret_cast<uint4*>(dst + (size_t)(r0 + row) * kMlpH + col) = v;
    };
    unsigned a[4], b[4];
    zero(z1);
    ldsm4<false>(a, s.x + la * kLdX + lk);
    ldsm4<true>(b, s.w1 + la * kLdH + c0 + lk);
    mma_bf16_16816(z1[0], a, b);
    mma_bf16_16816(z1[1], a, b + 2);
    hidden(z1, s.bias, s.ha);
    if (first) copy_wait<4>();
    __syncthreads();
    // Z2 = H1 W2 + b2
    if (TRAIN) put_rows(s.ha, g.h1b);
    zero(z2);
#pragma unroll
    for (int part = 0; part < 4; ++part) {
      if (first && part > 0) {
        if (part == 1) copy_wait<3>();
        if (part == 2) copy_wait<2>();
        if (part == 3) copy_wait<1>();
        __syncthreads();
      }
#pragma unroll
      for (int k0 = part * (kMlpH / 4); k0 < (part + 1) * (kMlpH / 4); k0 += 16) {
        ldsm4<false>(a, s.ha + la * kLdH + k0 + lk);
        ldsm4<true>(b, s.w2 + (k0 + la) * kLdH + c0 + lk);
        mma_bf16_16816(z2[0], a, b);
        mma_bf16_16816(z2[1], a, b + 2);
      }
    }
    hidden(z2, s.bias + kMlpH, s.hb);
    if (first) copy_wait<0>();
    __syncthreads();
    // O = H2 W3 + b3
    if (TRAIN) put_rows(s.hb, g.h2b);
    if (warp < kMlpOutPad / 8) {
      float o[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 4
      for (int k0 = 0; k0 < kMlpH; k0 += 16) {
        ldsm4<false>(a, s.hb + la * kLdH + k0 + lk);
        ldsm2_trans(b, s.w3 + (k0 + (lane & 15)) * kLdO + 8 * warp);
        mma_bf16_16816(o, a, b);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int row = gid + 8 * (q >> 1), col = 8 * warp + 2 * tig + (q & 1);
        float v = 0.0f + o[q];
        v += s.bias[2 * kMlpH + col];
        s.out[row * kMlpOutPad + col] = col < kMlpOut ? v : 0.0f;
      }
    }
    __syncthreads();
    if (g.out && r0 + warp < g.n) g.out[(size_t)(r0 + warp) * kMlpOutPad + lane] = s.out[warp * kMlpOutPad + lane];
    if (TRAIN) {
      // loss and its gradient: a warp per row, a lane per output
      const float* o = s.out + warp * kMlpOutPad;
      const float mine = o[lane];
      float nrm2 = 0.0f;
      for (int j = 0; j < g.d; ++j) nrm2 += o[j] * o[j];
      const float nrm = sqrtf(nrm2 + 1e-12f);
      const float unit = mine / nrm;
      float c = 0.0f;
      for (int j = 0; j < g.d; ++j)
        c += __shfl_sync(0xffffffffu, unit, j) * __shfl_sync(0xffffffffu, tgt, j);
      const float inv_n = 1.0f / (float)g.n;
      float v = 0.0f, df = 0.0f;
      if (lane < g.d) {
        v = -2.0f * c * (tgt - c * unit) / nrm * inv_n;
      } else if (lane >= kMlpIn && lane < kMlpIn + g.d) {
        df = mine - tgt;
        v = 2.0f * df * inv_n;
      }
      const bool in = r0 + warp < g.n;
      if (!in) v = 0.0f;
      s.dO[warp * kLdO + lane] = __float2bfloat16_rn(v);
      const size_t at = (size_t)(r0 + warp) * kMlpOutPad + lane;
      if (in) g.dout[at] = v;
      g.doutb[at] = __float2bfloat16_rn(v);
      if (g.row_loss) {
        double l = 1.0 - (double)c * (double)c;
        for (int j = kMlpIn; j < kMlpIn + g.d; ++j) {
          const float t = __shfl_sync(0xffffffffu, df, j);
          l += (double)t * (double)t;
        }
        if (in && lane == 0) g.row_loss[r0 + warp] = l;
      }
      __syncthreads();
      // gradient of a pre-activation: FP32 for the bias, BF16 for the products
      const auto back = [&](float (&acc)[2][4], const float (&z)[2][4], __nv_bfloat16* h, float* dst) {
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            const int row = gid + 8 * r, col = c0 + 8 * t + 2 * tig;
            float v0 = 0.0f + acc[t][2 * r], v1 = 0.0f + acc[t][2 * r + 1];
            v0 *= dsilu_f(z[t][2 * r]);
            v1 *= dsilu_f(z[t][2 * r + 1]);
            if (r0 + row < g.n)
              *reinterpret_cast<float2*>(dst + (size_t)(r0 + row) * kMlpH + col) = make_float2(v0, v1);
            __nv_bfloat162 p;
            p.x = __float2bfloat16_rn(v0);
            p.y = __float2bfloat16_rn(v1);
            *reinterpret_cast<__nv_bfloat162*>(h + row * kLdH + col) = p;
          }
      };
      // dZ2 = (dO W3^T) silu'(Z2)
      float acc[2][4];
      zero(acc);
#pragma unroll
      for (int k0 = 0; k0 < kMlpOutPad; k0 += 16) {
        ldsm4<false>(a, s.dO + la * kLdO + k0 + lk);
        ldsm4<false>(b, s.w3 + (c0 + lb) * kLdO + k0 + lc);
        mma_bf16_16816(acc[0], a, b);
        mma_bf16_16816(acc[1], a, b + 2);
      }
      back(acc, z2, s.ha, g.dz2);
      __syncthreads();
      // dZ1 = (dZ2 W2^T) silu'(Z1)
      put_rows(s.ha, g.dz2b);
      zero(acc);
#pragma unroll 4
      for (int k0 = 0; k0 < kMlpH; k0 += 16) {
        ldsm4<false>(a, s.ha + la * kLdH + k0 + lk);
        ldsm4<false>(b, s.w2 + (c0 + lb) * kLdH + k0 + lc);
        mma_bf16_16816(acc[0], a, b);
        mma_bf16_16816(acc[1], a, b + 2);
      }
      back(acc, z1, s.hb, g.dz1);
      __syncthreads();
      put_rows(s.hb, g.dz1b);
    }
    first = false;
    __syncthreads();
  }
}

struct ColArgs {
  const __nv_bfloat16 *xb, *h1b, *h2b, *dz1b, *dz2b, *doutb;
  const float *dz1, *dz2, *dout;
  int n, splits, k_split;
  float* grad;  // gradients out; null: Adam instead
  float *params, *m, *v;
  __nv_bfloat16 *w1b, *w2b, *w3b;
  int t;  // Adam's step number
  float lr;
};

// (1 - b1^t, 1 - b2^t) of Adam's bias correction
__device__ __forceinline__ float2 adam_corrections(int t) {
  return make_float2(1.0f - powf(0.9f, (float)t), 1.0f - powf(0.999f, (float)t));
}

// (double)x without the FP64 pipe (subnormal, infinite and NaN x aside)
__device__ __forceinline__ double widen(float x) {
  const unsigned b = __float_as_uint(x), e = b & 0x7f800000u;
  if ((b << 1) == 0) return __hiloint2double((int)b, 0);
  if (e == 0 || e == 0x7f800000u) return (double)x;
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), (int)(b << 29));
}

__device__ __forceinline__ void take_gradient(const ColArgs& g, int p, float gr, float2 corr) {
  if (g.grad) {
    g.grad[p] = gr;
    return;
  }
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float mm = b1 * g.m[p] + (1.0f - b1) * gr;
  const float vv = b2 * g.v[p] + (1.0f - b2) * gr * gr;
  g.m[p] = mm;
  g.v[p] = vv;
  const float mh = mm / corr.x;
  const float vh = vv / corr.y;
  const float w = g.params[p] - g.lr * mh / (sqrtf(vh) + eps);
  g.params[p] = w;
  write_bf16_weight(p, w, g.w1b, g.w2b, g.w3b);
}

// Weight gradients A^T B over the rows, and bias gradients (column sums in
// FP64), each applied by Adam where it is formed.
// A block per tile of 48 operand columns: 32 x 16 outputs of W2 and W3, 16 x
// 32 of W1 (8 inputs more than the 13 there are).  The rows are cut into
// `splits` parts, summed in the order of the parts; a part's four warps (one
// 16 x 8 product each) read it through a ring of 64-row stages.  The bias
// blocks, 4 columns each, come first: an FP64 add (or conversion) occupies a
// scheduler for 64 cycles, so the 538 columns are spread over 135 SMs and
// widened by integer instructions.  1000 rows: about 8 us.  A step of the two
// kernels takes 19.9 us; products, epilogues, loss, column sums (one thread a
// column) and Adam as 16 kernels of a graph took 560 us.
template <int STAGES>
__global__ void __launch_bounds__(128 * kMlpMaxSplit) k_mlp_cols(ColArgs g) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  __shared__ float2 s_corr;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) s_corr = adam_corrections(g.t);
  chain_launch();
  chain_wait();
  int blk = blockIdx.x;
  if (blk < kBiasBlocks) {
    const float* src = blk < 64 ? g.dz1 : blk < 128 ? g.dz2 : g.dout;
    const int ld = blk < 128 ? kMlpH : kMlpOutPad, col0 = 4 * (blk < 128 ? blk & 63 : blk - 128);
    const int off = blk < 64 ? kMlpOffB1 : blk < 128 ? kMlpOffB2 : kMlpOffB3;
    const int nw = blockDim.x >> 5, col = col0 + (lane & 3);
    double* s_sum = reinterpret_cast<double*>(s_raw);
    double sum = 0.0;
#pragma unroll 8
    for (int i = 8 * warp + (lane >> 2); i < g.n; i += 8 * nw) sum += widen(src[(size_t)i * ld + col]);
    for (int o = 4; o < 32; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane < 4) s_sum[warp * 4 + lane] = sum;
    __syncthreads();
    if (warp == 0) {
      double t = 0.0;
      for (int w = lane >> 2; w < nw; w += 8) t += s_sum[w * 4 + (lane & 3)];
      for (int o = 4; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane < 4 && (blk < 128 || col < kMlpOut)) take_gradient(g, off + col, (float)t, s_corr);
    }
    return;
  }
  blk -= kBiasBlocks;
  const __nv_bfloat16 *A, *B;
  int lda, ldb, ca, cb, wa = 32, off, cols, rows;
  if (blk < 128) {
    A = g.h1b, B = g.dz2b, lda = ldb = kMlpH, ca = 32 * (blk >> 4), cb = 16 * (blk & 15);
    off = kMlpOffW2, rows = cols = kMlpH;
  } else if (blk < 144) {
    blk -= 128;
    A = g.h2b, B = g.doutb, lda = kMlpH, ldb = kMlpOutPad, ca = 32 * (blk >> 1), cb = 16 * (blk & 1);
    off = kMlpOffW3, rows = kMlpH, cols = kMlpOut;
  } else {
    blk -= 144;
    A = g.xb, B = g.dz1b, lda = kMlpInPad, ldb = kMlpH, ca = 0, cb = 32 * blk, wa = 16;
    off = kMlpOffW1, rows = kMlpIn, cols = kMlpH;
  }
  const int wb = 48 - wa, part = warp >> 2, tid4 = tid & 127;
  const int mt = wa == 32 ? (warp >> 1) & 1 : 0, nt = wa == 32 ? warp & 1 : warp & 3;
  __nv_bfloat16* ring = reinterpret_cast<__nv_bfloat16*>(s_raw) + (size_t)part * STAGES * kColChunk * kLdC;
  const int kbeg = part * g.k_split, kend = min(mlp_rows(g.n), kbeg + g.k_split);
  const int chunks = (kend - kbeg + kColChunk - 1) / kColChunk;
  const auto load = [&](int c) {
    if (c < chunks) {
      __nv_bfloat16* dst = ring + (c % STAGES) * kColChunk * kLdC;
      const int k0 = kbeg + c * kColChunk, nr = min(kColChunk, kend - k0);
      for (int e = tid4; e < nr * 6; e += 128) {
        const int r = e / 6, q = (e - 6 * r) * 8;
        const __nv_bfloat16* src =
            q < wa ? A + (size_t)(k0 + r) * lda + ca + q : B + (size_t)(k0 + r) * ldb + cb + (q - wa);
        copy16(dst + r * kLdC + q, src);
      }
    }
    copy_commit();
  };
#pragma unroll
  for (int c = 0; c < STAGES - 1; ++c) load(c);
  float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  const int ar = (lane & 7) + (lane >> 4) * 8, ac = 16 * mt + ((lane >> 3) & 1) * 8, bc = wa + 8 * nt;
  for (int c = 0; c < chunks; ++c) {
    copy_wait<STAGES - 2>();
    asm volatile("bar.sync %0, 128;" ::"r"(1 + part) : "memory");
    load(c + STAGES - 1);
    const __nv_bfloat16* st = ring + (c % STAGES) * kColChunk * kLdC;
    const int nr = min(kColChunk, kend - kbeg - c * kColChunk);
    for (int k0 = 0; k0 < nr; k0 += 16) {
      unsigned a[4], b[2];
      ldsm4<true>(a, st + (k0 + ar) * kLdC + ac);
      ldsm2_trans(b, st + (k0 + (lane & 15)) * kLdC + bc);
      mma_bf16_16816(acc, a, b);
    }
  }
  // the parts' sums, in order
  copy_wait<0>();
  __syncthreads();
  float* s_part = reinterpret_cast<float*>(s_raw);  // [splits][wa][wb]
#pragma unroll
  for (int q = 0; q < 4; ++q)
    s_part[part * 512 + (16 * mt + (lane >> 2) + 8 * (q >> 1)) * wb + 8 * nt + 2 * (lane & 3) + (q & 1)] = acc[q];
  __syncthreads();
  for (int e = tid; e < 512; e += blockDim.x) {
    const int r = e / wb, c = e - r * wb;
    if (ca + r >= rows || cb + c >= cols) continue;
    float v = 0.0f;
    for (int z = 0; z < g.splits; ++z) v += s_part[z * 512 + e];
    take_gradient(g, off + (ca + r) * cols + cb + c, v, s_corr);
  }
}

// deterministic mean of row_loss (one block, fixed tree)
__global__ void k_mean(const double* v, int n, double* out) {
  __shared__ double s[256];
  double a = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) a += v[i];
  s[threadIdx.x] = a;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = s[0] / (double)n;
}

// ---------------------------------------------------------------------------
// Host helpers
// ---------------------------------------------------------------------------
template <typename T>
cudaError_t dalloc(T*& p, size_t n) {
  return cudaMalloc(&p, sizeof(T) * (n ? n : 1));
}

// A launch whose set-up overlaps the kernel before it.
template <typename Args>
cudaError_t launch_chained(void (*kern)(Args), int grid, int threads, size_t smem, const Args& a, cudaStream_t st) {
  cudaError_t e = allow_shared((const void*)kern);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

cudaError_t launch_rows(Mlp& M, int n, int d, bool train, float* out, double* row_loss, cudaStream_t st, long long* L) {
  RowArgs g{M.params, M.w1b, M.w2b, M.w3b, M.xb,    M.tdir, M.tls,  n,      d,
            out,      M.dout, M.dz2, M.dz1, M.h1b, M.h2b, M.doutb, M.dz2b, M.dz1b, row_loss};
  if (L) *L += 1;
  const int grid = std::min(mlp_rows(n) / 16, M.sms);
  return launch_chained(train ? k_mlp_rows<true> : k_mlp_rows<false>, grid, kRowThreads, sizeof(RowShared), g, st);
}

// t 0: gradients into M.grad; otherwise Adam's step t
cudaError_t launch_cols(Mlp& M, int n, int t, float lr, cudaStream_t st, long long* L) {
  // the parts of the rows: from 512 rows on, 256 or more each
  int splits = n >= 512 ? std::min(kMlpMaxSplit, n / 256) : 1;
  const int ks = ((n + splits - 1) / splits + 15) / 16 * 16;
  splits = (n + ks - 1) / ks;
  ColArgs g{M.xb,   M.h1b,  M.h2b,  M.dz1b, M.dz2b, M.doutb, M.dz1, M.dz2, M.dout, n, splits, ks, t ? nullptr : M.grad,
            M.params, M.adam_m, M.adam_v, M.w1b, M.w2b, M.w3b, t, lr};
  const int stages = splits <= 7 ? 4 : 3;  // 200 KB at most
  if (L) *L += 1;
  return launch_chained(stages == 4 ? k_mlp_cols<4> : k_mlp_cols<3>, kBiasBlocks + 128 + 16 + 8, 128 * splits,
                        sizeof(__nv_bfloat16) * splits * stages * kColChunk * kLdC, g, st);
}

}  // namespace

cudaError_t mlp_alloc(Mlp& M, int cap, cudaStream_t st) {
  mlp_free(M);
  cudaError_t e = cudaSuccess;
  auto A = [&](cudaError_t r) {
    if (e == cudaSuccess) e = r;
  };
  const size_t rows = mlp_rows(cap);
  int dev = 0;
  A(cudaGetDevice(&dev));
  A(cudaDeviceGetAttribute(&M.sms, cudaDevAttrMultiProcessorCount, dev));
  A(dalloc(M.params, kMlpParams + 6));  // (the output biases are read as 32)
  A(dalloc(M.adam_m, kMlpParams));
  A(dalloc(M.adam_v, kMlpParams));
  A(dalloc(M.grad, kMlpParams));
  A(dalloc(M.w1b, kMlpInPad * kMlpH));
  A(dalloc(M.w2b, kMlpH * kMlpH));
  A(dalloc(M.w3b, kMlpH * kMlpOutPad));
  A(dalloc(M.xb, rows * kMlpInPad));
  A(dalloc(M.h1b, rows * kMlpH));
  A(dalloc(M.h2b, rows * kMlpH));
  A(dalloc(M.out, rows * kMlpOutPad));
  A(dalloc(M.dout, rows * kMlpOutPad));
  A(dalloc(M.doutb, rows * kMlpOutPad));
  A(dalloc(M.dz2, rows * kMlpH));
  A(dalloc(M.dz2b, rows * kMlpH));
  A(dalloc(M.dz1, rows * kMlpH));
  A(dalloc(M.dz1b, rows * kMlpH));
  A(dalloc(M.tdir, rows * kMlpIn));
  A(dalloc(M.tls, rows * kMlpIn));
  A(dalloc(M.nbr, rows * kMaxNbr));
  A(dalloc(M.stats, 2 * kMlpIn));
  A(dalloc(M.live, rows * kMlpIn));
  A(dalloc(M.xs, rows * kMlpIn));
  A(dalloc(M.xf, rows * kMlpIn));
  A(dalloc(M.row_loss, rows));
  A(dalloc(M.loss, 1));
  if (e == cudaSuccess) {
    // padded rows/columns of the weight copies stay zero (on the stream of the
    // kernels that write the others)
    A(cudaMemsetAsync(M.w1b, 0, sizeof(__nv_bfloat16) * kMlpInPad * kMlpH, st));
    A(cudaMemsetAsync(M.w3b, 0, sizeof(__nv_bfloat16) * kMlpH * kMlpOutPad, st));
  }
  if (e != cudaSuccess) {
    mlp_free(M);
    return e;
  }
  M.cap = cap;
  return cudaSuccess;
}

void mlp_free(Mlp& M) {
  auto F = [](auto*& p) {
    if (p) cudaFree(p);
    p = nullptr;
  };
  F(M.params), F(M.adam_m), F(M.adam_v), F(M.grad), F(M.w1b), F(M.w2b), F(M.w3b), F(M.xb);
  F(M.h1b), F(M.h2b), F(M.out), F(M.dout), F(M.doutb), F(M.dz2), F(M.dz2b), F(M.dz1), F(M.dz1b);
  F(M.tdir), F(M.tls), F(M.nbr), F(M.stats), F(M.live), F(M.xs), F(M.xf), F(M.row_loss), F(M.loss);
  M.step = 0;
  M.cap = 0;
}

static cudaError_t reset_adam(Mlp& M, cudaStream_t st, long long* L) {
  cudaError_t e = cudaMemsetAsync(M.adam_m, 0, sizeof(float) * kMlpParams, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(M.adam_v, 0, sizeof(float) * kMlpParams, st);
  if (e != cudaSuccess) return e;
  M.step = 0;
  k_mlp_bf16_weights<<<(kMlpParams + 255) / 256, 256, 0, st>>>(M.params, M.w1b, M.w2b, M.w3b);
  if (L) *L += 1;
  return cudaGetLastError();
}

cudaError_t mlp_init(Mlp& M, uint64_t seed, cudaStream_t st, long long* L) {
  k_mlp_init<<<(kMlpParams + 255) / 256, 256, 0, st>>>(M.params, (unsigned)(seed & 0xFFFFFFFFu),
                                                       (unsigned)(seed >> 32));
  if (L) *L += 1;
  const cudaError_t e = cudaGetLastError();
  return e != cudaSuccess ? e : reset_adam(M, st, L);
}

cudaError_t mlp_load(Mlp& M, const float* params, cudaStream_t st, long long* L) {
  const cudaError_t e = cudaMemcpyAsync(M.params, params, sizeof(float) * kMlpParams, cudaMemcpyHostToDevice, st);
  return e != cudaSuccess ? e : reset_adam(M, st, L);
}

cudaError_t mlp_targets(Mlp& M, const double* live_u, int n, int d, int k, cudaStream_t st, long long* L) {
  if (n > M.cap || d < 1 || d > kMlpIn || k < 1 || k > kMaxNbr || k >= n) return cudaErrorInvalidValue;
  const int ld = mlp_rows(M.cap);
  k_live_stats<<<d, 32, 0, st>>>(live_u, n, d, M.stats);
  k_standardise<<<(mlp_rows(n) * kMlpInPad + 255) / 256, 256, 0, st>>>(live_u, n, d, M.stats, M.xs, M.xf, ld, M.xb);
  k_local_pca<<<(n + kTargetWarps - 1) / kTargetWarps, 32 * kTargetWarps, 0, st>>>(live_u, M.xs, M.xf, ld, n, d, k,
                                                                                  M.tdir, M.tls, M.nbr);
  if (L) *L += 3;
  return cudaGetLastError();
}

cudaError_t mlp_inputs(Mlp& M, const float* x_std, int n, cudaStream_t st, long long* L) {
  if (n > M.cap) return cudaErrorInvalidValue;
  k_inputs_f32<<<(mlp_rows(n) * kMlpInPad + 255) / 256, 256, 0, st>>>(x_std, n, M.xb);
  if (L) *L += 1;
  return cudaGetLastError();
}

cudaError_t mlp_forward(Mlp& M, int n, cudaStream_t st, long long* L) {
  if (n > M.cap) return cudaErrorInvalidValue;
  return launch_rows(M, n, 0, false, M.out, nullptr, st, L);
}

cudaError_t mlp_loss_grad(Mlp& M, int n, int d, cudaStream_t st, long long* L) {
  if (n > M.cap) return cudaErrorInvalidValue;
  cudaError_t e = launch_rows(M, n, d, true, M.out, M.row_loss, st, L);
  if (e == cudaSuccess) e = launch_cols(M, n, 0, 0.0f, st, L);
  if (e != cudaSuccess) return e;
  k_mean<<<1, 256, 0, st>>>(M.row_loss, n, M.loss);
  if (L) *L += 1;
  return cudaGetLastError();
}

cudaError_t mlp_train(Mlp& M, int n, int d, int steps, float lr, cudaStream_t st, long long* L) {
  if (n > M.cap) return cudaErrorInvalidValue;
  for (int s = 0; s < steps; ++s) {
    cudaError_t e = launch_rows(M, n, d, true, nullptr, nullptr, st, L);
    if (e == cudaSuccess) e = launch_cols(M, n, ++M.step, lr, st, L);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace swig

// ---------------------------------------------------------------------------
// C-ABI: the network's pieces on host buffers (verification and tooling)
// ---------------------------------------------------------------------------
#include <string>
#include <vector>

#include "context.h"
#include "swig.h"

using namespace swig;

namespace {

int mfail(swig_ctx* c, int code, const std::string& m) {
  c->err = m;
  return code;
}

#define MCUDA(call)                                                                                         \
  do {                                                                                                      \
    cudaError_t e_ = (call);                                                                                \
    if (e_ != cudaSuccess)                                                                                  \
      return mfail(c, e_ == cudaErrorMemoryAllocation ? SWIG_E_NOMEM : SWIG_E_CUDA,                         \
                   std::string(#call) + ": " + cudaGetErrorString(e_));                                     \
  } while (0)

// The context's network, with buffers for at least n rows.
int ensure_mlp(swig_ctx* c, int n) {
  if (n < 1 || n > 8192) return mfail(c, SWIG_E_ARG, "need 1 <= n <= 8192");
  MCUDA(cudaSetDevice(c->device));
  if (!c->mlp) c->mlp = new Mlp();
  if (c->mlp->cap < n) MCUDA(mlp_alloc(*c->mlp, std::max(n, 1024), c->stream));
  return SWIG_OK;
}

// Host parameters -> master weights (fresh Adam state and BF16 copies).
int upload_params(swig_ctx* c, const float* params) {
  MCUDA(mlp_load(*c->mlp, params, c->stream, &c->n_launches));
  c->h2d_bytes += sizeof(float) * kMlpParams;
  return SWIG_OK;
}

// Live points -> the network's buffer.
int upload_live(swig_ctx* c, const double* live_u, int64_t n, int d) {
  MCUDA(cudaMemcpyAsync(c->mlp->live, live_u, sizeof(double) * n * d, cudaMemcpyHostToDevice, c->stream));
  c->h2d_bytes += sizeof(double) * n * d;
  return SWIG_OK;
}

template <typename T>
int upload(swig_ctx* c, T* dst, const T* src, size_t n) {
  MCUDA(cudaMemcpyAsync(dst, src, sizeof(T) * n, cudaMemcpyHostToDevice, c->stream));
  c->h2d_bytes += sizeof(T) * n;
  return SWIG_OK;
}

// rows of a [n][ld] device array -> [n][w] host array
template <typename T>
int download_rows(swig_ctx* c, T* dst, const T* src, int n, int ld, int w) {
  std::vector<T> tmp((size_t)n * ld);
  MCUDA(cudaMemcpy(tmp.data(), src, sizeof(T) * tmp.size(), cudaMemcpyDeviceToHost));
  c->d2h_bytes += sizeof(T) * tmp.size();
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < w; ++j) dst[(size_t)i * w + j] = tmp[(size_t)i * ld + j];
  return SWIG_OK;
}

}  // namespace

void swig_mlp_release(swig_ctx* c) {
  if (c && c->mlp) {
    mlp_free(*c->mlp);
    delete c->mlp;
    c->mlp = nullptr;
  }
}

extern "C" {

int swig_mlp_init(swig_ctx* c, uint64_t seed, float* params_out) {
  if (!c) return SWIG_E_ARG;
  if (!params_out) return mfail(c, SWIG_E_ARG, "null output");
  int rc = ensure_mlp(c, 1);
  if (rc) return rc;
  MCUDA(mlp_init(*c->mlp, seed, c->stream, &c->n_launches));
  MCUDA(cudaStreamSynchronize(c->stream));
  MCUDA(cudaMemcpy(params_out, c->mlp->params, sizeof(float) * kMlpParams, cudaMemcpyDeviceToHost));
  c->d2h_bytes += sizeof(float) * kMlpParams;
  return SWIG_OK;
}

int swig_mlp_forward(swig_ctx* c, const float* params, const float* x_std, int64_t n, float* out) {
  if (!c) return SWIG_E_ARG;
  if (!params || !x_std || !out) return mfail(c, SWIG_E_ARG, "null buffer");
  int rc = ensure_mlp(c, (int)std::min<int64_t>(n, 1 << 30));
  if (rc) return rc;
  if ((rc = upload_params(c, params))) return rc;
  float* xd = nullptr;
  MCUDA(cudaMalloc(&xd, sizeof(float) * n * kMlpIn));
  cudaError_t e = cudaMemcpyAsync(xd, x_std, sizeof(float) * n * kMlpIn, cudaMemcpyHostToDevice, c->stream);
  if (e == cudaSuccess) e = mlp_inputs(*c->mlp, xd, (int)n, c->stream, &c->n_launches);
  if (e == cudaSuccess) e = mlp_forward(*c->mlp, (int)n, c->stream, &c->n_launches);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  cudaFree(xd);
  MCUDA(e);
  c->h2d_bytes += sizeof(float) * n * kMlpIn;
  return download_rows(c, out, c->mlp->out, (int)n, kMlpOutPad, kMlpOut);
}

int swig_mlp_loss_grad(swig_ctx* c, const float* params, const float* x_std, const float* tdir, const float* tls,
                       int64_t n, int d, double* loss_out, float* grad_out) {
  if (!c) return SWIG_E_ARG;
  if (!params || !x_std || !tdir || !tls || !loss_out || !grad_out) return mfail(c, SWIG_E_ARG, "null buffer");
  if (d < 1 || d > kMlpIn) return mfail(c, SWIG_E_ARG, "need 1 <= d <= 13");
  int rc = ensure_mlp(c, (int)std::min<int64_t>(n, 1 << 30));
  if (rc) return rc;
  if ((rc = upload_params(c, params))) return rc;
  Mlp& M = *c->mlp;
  if ((rc = upload(c, M.tdir, tdir, (size_t)n * kMlpIn))) return rc;
  if ((rc = upload(c, M.tls, tls, (size_t)n * kMlpIn))) return rc;
  float* xd = nullptr;
  MCUDA(cudaMalloc(&xd, sizeof(float) * n * kMlpIn));
  cudaError_t e = cudaMemcpyAsync(xd, x_std, sizeof(float) * n * kMlpIn, cudaMemcpyHostToDevice, c->stream);
  if (e == cudaSuccess) e = mlp_inputs(M, xd, (int)n, c->stream, &c->n_launches);
  if (e == cudaSuccess) e = mlp_loss_grad(M, (int)n, d, c->stream, &c->n_launches);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  cudaFree(xd);
  MCUDA(e);
  c->h2d_bytes += sizeof(float) * n * kMlpIn;
  MCUDA(cudaMemcpy(loss_out, M.loss, sizeof(double), cudaMemcpyDeviceToHost));
  MCUDA(cudaMemcpy(grad_out, M.grad, sizeof(float) * kMlpParams, cudaMemcpyDeviceToHost));
  c->d2h_bytes += sizeof(double) + sizeof(float) * kMlpParams;
  return SWIG_OK;
}

int swig_mlp_targets(swig_ctx* c, const double* live_u, int64_t n, int d, float* tdir, float* tls, int* nbr) {
  if (!c) return SWIG_E_ARG;
  if (!live_u || !tdir || !tls) return mfail(c, SWIG_E_ARG, "null buffer");
  if (d < 1 || d > kMlpIn || 2 * d >= n) return mfail(c, SWIG_E_ARG, "need 1 <= d <= 13 and 2d < n");
  int rc = ensure_mlp(c, (int)std::min<int64_t>(n, 1 << 30));
  if (rc) return rc;
  Mlp& M = *c->mlp;
  if ((rc = upload_live(c, live_u, n, d))) return rc;
  MCUDA(mlp_targets(M, M.live, (int)n, d, 2 * d, c->stream, &c->n_launches));
  MCUDA(cudaStreamSynchronize(c->stream));
  if ((rc = download_rows(c, tdir, M.tdir, (int)n, kMlpIn, kMlpIn))) return rc;
  if ((rc = download_rows(c, tls, M.tls, (int)n, kMlpIn, kMlpIn))) return rc;
  if (nbr && (rc = download_rows(c, nbr, M.nbr, (int)n, 2 * kMlpIn, 2 * kMlpIn))) return rc;
  return SWIG_OK;
}

int swig_mlp_train(swig_ctx* c, const double* live_u, int64_t n, int d, int steps, double lr, float* params_inout,
                   float* out_rows) {
  if (!c) return SWIG_E_ARG;
  if (!live_u || !params_inout) return mfail(c, SWIG_E_ARG, "null buffer");
  if (d < 1 || d > kMlpIn || 2 * d >= n) return mfail(c, SWIG_E_ARG, "need 1 <= d <= 13 and 2d < n");
  if (steps < 0 || !(lr > 0.0)) return mfail(c, SWIG_E_ARG, "need steps >= 0 and lr > 0");
  int rc = ensure_mlp(c, (int)std::min<int64_t>(n, 1 << 30));
  if (rc) return rc;
  if ((rc = upload_params(c, params_inout))) return rc;
  Mlp& M = *c->mlp;
  if ((rc = upload_live(c, live_u, n, d))) return rc;
  cudaError_t e = mlp_targets(M, M.live, (int)n, d, 2 * d, c->stream, &c->n_launches);
  if (e == cudaSuccess) e = mlp_train(M, (int)n, d, steps, (float)lr, c->stream, &c->n_launches);
  if (e == cudaSuccess && out_rows) e = mlp_forward(M, (int)n, c->stream, &c->n_launches);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  MCUDA(e);
  MCUDA(cudaMemcpy(params_inout, M.params, sizeof(float) * kMlpParams, cudaMemcpyDeviceToHost));
  c->d2h_bytes += sizeof(float) * kMlpParams;
  if (out_rows && (rc = download_rows(c, out_rows, M.out, (int)n, kMlpOutPad, kMlpOut))) return rc;
  return SWIG_OK;
}

}  // extern "C"
