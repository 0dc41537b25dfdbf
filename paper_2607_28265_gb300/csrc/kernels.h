// Launch interface between the C-ABI host code and the CUDA kernels.
#pragma once

#include <cuda_runtime.h>

#include "swig_internal.h"

namespace swig {

struct PriorSlot {
  int kind;
  int mode;
  double lo, hi, value;
  double c1, c2;  // SINE: cos lo, cos hi; COSINE: sin lo, sin hi; POWER2: lo^3, hi^3
};

inline PriorSlot make_prior_slot(int kind, int mode, double lo, double hi, double value);

// Detector-frame sky parameterisation: slots 9 and 10 hold the azimuth and
// zenith of the source about the baseline between two detectors (ez, from
// detector b to detector a; ex towards the Earth's north pole), mapped to
// (RA, Dec) at the reference sidereal time before any use.
struct SkyFrame {
  int on;
  double ex[3], ey[3], ez[3];
  double gmst;
};

// Time-marginalised heterodyned likelihood: threads per CTA (one theta or
// one chain per CTA), the largest bin count (the edge products y_e live in
// shared memory) and the shared-memory bytes of those products.
constexpr int kHetTmThreads = 512;
constexpr int kMaxTmBins = 16384;
// Non-uniform FFT time pass: node counts it serves (the direct sum below and
// above), the kernel width in grid points; its grid of M complex values
// follows the edge products in shared memory.
constexpr int kNufftMinNodes = 64;
constexpr int kNufftMaxNodes = 4096;
constexpr int kNufftWidth = 8;
// entries per gather piece (one lane sums a piece)
// (odd, so that the pieces of one grid point start in different banks)
constexpr int kNufftPiece = 31;
// (edge products, then the non-uniform FFT's grid of M and stage-major
// twiddle table of M complex values, then the gather's per-piece partial sums)
inline size_t het_tm_smem_bytes(int n_bins, int nufft_m = 0, int pieces = 0) {
  return (((size_t)n_bins + 1) * 2 * sizeof(float) + 15) / 16 * 16 + (size_t)nufft_m * 4 * sizeof(float) +
         (size_t)pieces * 2 * sizeof(float);
}

// Heterodyned contraction by chunk anchors.  A warp step covers one chunk of
// 32 edges (31 bins).  Per chunk the host tabulates, at its first edge f_a,
// the basis values and first derivative (double-float) and the scaled
// derivatives of orders 2..kHetTaylorDeg (float), as rows of a [HC_ROWS][chunks]
// table; per evaluation the phase difference from the fiducial is anchored
// there in double-float and carried across the chunk by an FP32 Taylor form
// in x = (f_e - f_a) / S (S the chunk's span).  Rows HC_BND + j hold the
// remainder bound of basis j, max |phi_j^(11)| S^11 / 11! over the chunk: an
// evaluation whose sum_j |c_j - c0_j| HC_BND_j exceeds kHetTaylorEps cycles
// takes the chunk edge by edge in double-float instead.
constexpr int kHetChunkEdges = 32;
constexpr float kHetTaylorEps = 1e-6f;
// degree of the chunk Taylor form (wider than the full grid's tiles: a chunk
// of 31 heterodyned bins spans up to ~10 % of its frequency mid-band)
constexpr int kHetTaylorDeg = 10;
constexpr int kHetPoly = kHetTaylorDeg - 1;  // orders 2..kHetTaylorDeg
enum HetChunkRow {
  HC_VAL_HI = 0,
  HC_VAL_LO = NBASIS,
  HC_D1_HI = 2 * NBASIS,
  HC_D1_LO = 3 * NBASIS,
  HC_POLY = 4 * NBASIS,  // HC_POLY + (n - 2) * NBASIS + j: phi_j^(n)(f_a) S^n / n!
  HC_FA_HI = 4 * NBASIS + kHetPoly * NBASIS,
  HC_FA_LO,
  HC_INV_S,
  HC_BND,
  HC_ROWS = HC_BND + NBASIS
};
// Per-evaluation chunk anchor in shared memory: a_1 .. a_kHetTaylorDeg, then
// frac(dP(f_a) + f_a dtau_i) per detector, 1 / S and the exact flag of this
// evaluation.
constexpr int kHetAncStride = 16;
constexpr int kHetAncPhase = kHetPoly + 1;
constexpr int kHetAncInvS = kHetAncPhase + SWIG_MAX_DET;
constexpr int kHetAncExact = kHetAncInvS + 1;
static_assert(kHetAncExact < kHetAncStride, "chunk anchor layout");
// Floats from one chunk's anchor to the next: two evaluations interleaved, and
// one, padded so that the lanes' stores (a chunk each) meet all banks.
constexpr int kHetAncPair = 2 * kHetAncStride + 2;
constexpr int kHetAncOne = kHetAncStride + 1;
// Partial sums of a chain's current point per chunk (het.cuh).
constexpr int kHetBaseRows = 5 + kHetPoly;

// Folded full-grid sums (fold.cuh): the grid in chunks of kFoldNodes nodes.
// Rows of the [FR_ROWS][ld] table (a column per chunk): at the chunk's centre f_c, with h the
// half width [Hz] that scales the node abscissae to |x| <= 1, the basis values
// and first derivatives times h (double-float; the constant basis function,
// last, has no derivatives), derivatives of orders 2..kFoldDeg times h^n / n!
// (float), the order-9 remainder bound max |phi_j^(9)| h^9 / 9!, f_c, h and the
// reference slope times h (double-float), the bandwidth the weights serve
// [cycles] and the node kind (an int's bits).
constexpr int kFoldNodes = 64;
constexpr int kFoldAnchorFloats = 16;  // per (evaluation, chunk)
constexpr int kFoldBaseRows = 11;      // rows [ld] of a point's partial sums (fold.cuh fold_base)
constexpr int kFoldDeg = 8;
constexpr int kFoldSlopes = NBASIS - 1;
enum FoldRow {
  FR_VAL_HI = 0,
  FR_VAL_LO = NBASIS,
  FR_D1_HI = 2 * NBASIS,
  FR_D1_LO = FR_D1_HI + kFoldSlopes,
  FR_POLY = FR_D1_LO + kFoldSlopes,  // FR_POLY + (n - 2) * kFoldSlopes + j
  FR_BND = FR_POLY + (kFoldDeg - 1) * kFoldSlopes,
  FR_FC_HI = FR_BND + kFoldSlopes,
  FR_FC_LO,
  FR_H_HI,
  FR_H_LO,
  FR_SM_HI,
  FR_SM_LO,
  FR_LIM,
  FR_KIND,
  FR_ROWS
};
// Node kinds: 0 the 64 Chebyshev nodes; s = 1 .. kFoldKinds - 1 the bins of a
// block of w = 128 >> s themselves, x = +-(2 l + 1) / w.
constexpr int kFoldKinds = 7;
// Interpolation of exp(2 pi i delta(x)) through n Chebyshev nodes errs by at
// most 4 M rho^(1 - n) / (rho - 1), M its bound on the Bernstein ellipse of
// parameter rho: M <= exp(2 pi b omega) with omega = |delta_1| + sum_n n
// a^(n-1) |delta_n|, a and b the ellipse's half axes.  rho = 3 gave the fewest
// chunks on the 128 s grid (78; 2: 130, 4: 82, 5: 87).
constexpr float kFoldRho = 3.0f;
constexpr float kFoldEllipse = 0.5f * (kFoldRho + 1.0f / kFoldRho);
// Taylor remainder [cycles] and interpolation error an evaluation may have
// (the host plans for a fifth and a tenth of them over the prior box).
constexpr float kFoldTaylorEps = 1e-7f;
constexpr double kFoldEps = 1e-7;

struct FoldChunk {
  int k0, nbins;   // bins [k0, k0 + nbins)
  int kind;        // node kind
  int pad;
  double slope_h;  // reference slope times h [cycles]
};

struct FoldTables {
  int nc;             // chunks
  int ld;             // row length of tab: nc rounded up to 4
  const float* tab;   // [FR_ROWS][ld]
  const float4* w;    // [nc][n_det][32] node weights (+x re, -x re, +x im, -x im)
  const float2* x;    // [kFoldKinds][32] the lanes' node abscissae (hi, lo)
  // bin by bin (fold_direct, fold_strays)
  const float2* data;
  const TileInfo* tiles;
  const TileBasis* basis;
  const int* bin_tile;
  const int* slice_begin;
};

// Vectors of a batch that the node weights do not serve (fold.cu fold_strays), in
// the scratch of the batch; the set-up kernel clears ctl and done.
struct FoldStrays {
  int* ctl;     // [4] vectors decided, strays among them (one 64-bit count), units taken, list entries
  int* list;    // [n] the strays
  int* done;    // [n] slices summed of stray i
  float* part;  // [n][n_slices][kPartialStride] their sums
};
inline size_t fold_strays_bytes(int n, int n_slices) {
  return sizeof(int) * (4 + 2 * (size_t)n) + sizeof(float) * kPartialStride * (size_t)n_slices * n + 16;
}
inline FoldStrays fold_strays_at(void* p, int n) {
  FoldStrays s;
  s.ctl = static_cast<int*>(p);
  s.list = s.ctl + 4;
  s.done = s.list + n;
  const size_t off = (sizeof(int) * (4 + 2 * (size_t)n) + 15) / 16 * 16;
  s.part = reinterpret_cast<float*>(static_cast<char*>(p) + off);
  return s;
}

// Device buffers owned by a context (all allocated with cudaMalloc).
struct DeviceBuffers {
  // problem data
  float2* data32 = nullptr;      // [n_det][n_bins] scaled D_i (MIXED)
  double2* data64 = nullptr;     // [n_det][n_bins] D_i (FP64)
  double* ftab = nullptr;        // [NBASIS][n_bins] basis functions, f in row B_ONE (FP64)
  TileInfo* tiles = nullptr;     // [n_tiles]
  TileBasis* basis = nullptr;    // [n_tiles]
  int* slice_begin = nullptr;    // [n_slices + 1] first bin of each slice
  int* bin_tile = nullptr;       // [n_bins] tile of each bin
  PriorSlot* prior = nullptr;    // [13]
  int fold_nc = 0;               // folded full-grid sums (FoldTables)
  float* fold_tab = nullptr;
  float4* fold_w = nullptr;
  float2* fold_x = nullptr;
  int max_slice_bins = 0;        // largest slice: bins, and (mixed) tiles that overlap it
  int max_slice_tiles = 1;
  // heterodyned likelihood tables (SWIG_LIKE_HET)
  int het_nb = 0;
  float* het_edge_basis = nullptr;  // [2 * NBASIS][N_b + 1] (row per basis function, hi / lo)
  float* het_edge_f = nullptr;      // [2][N_b + 1] (hi row, lo row)
  int het_nc = 0;                   // chunks of kHetChunkEdges edges
  float* het_chunk = nullptr;       // [HC_ROWS][het_nc] chunk anchor tables
  EvalRecord* het_fid = nullptr;    // fiducial record
  float4* het_ew = nullptr;         // [het_nc][n_det][32] edge weights (HetTables::ew)
  // time marginalisation on the heterodyned bins (t_c marginalised)
  float2* het_tm_w = nullptr;       // [N_b + 1] exp(-2 pi i f_e dt), the step between grid nodes
  // ... by non-uniform FFT (L.tm_M > 0): kernel weight of every (grid point,
  // edge) entry in grid-point order, deconvolution 1 / Phi per node, twiddles
  float* het_nu_wt = nullptr;       // [pieces / 32][kNufftPiece][32]
  float* het_nu_corr = nullptr;     // [N_t]
  float2* het_nu_tw = nullptr;      // [M] stage-major twiddles: span h at h - 1 + p, exp(2 pi i p / (2 h))
  int4* het_nu_piece = nullptr;     // [pieces] (first entry, entries, first edge, 0)
  int4* het_nu_point = nullptr;     // [points] (grid point, first piece, pieces, 0)
  // scratch for batched evaluation, sized for `cap` thetas
  int cap = 0;
  EvalRecord* rec = nullptr;     // [cap]
  double* partials64 = nullptr;  // [cap][n_slices][kPartialStride]
  void* strays = nullptr;        // FoldStrays of cap vectors (mixed, full grid)
  double* theta = nullptr;       // [cap][13] staging for host calls
  double* out = nullptr;         // [cap]
  double* u = nullptr;           // [cap][13]
};

// Shared memory of a time-marginalised evaluation: het_tm_smem_bytes with the
// anchors of a panel of chunks over the time pass's grid, or appended where the
// grid is smaller.
struct HetTmLayout {
  size_t bytes;
  int anc_off, panel;
};
inline HetTmLayout het_tm_layout(const LikeConst& L, const DeviceBuffers& B) {
  HetTmLayout lay;
  lay.panel = B.het_nc < 128 ? B.het_nc : 128;
  const size_t anc = (size_t)lay.panel * kHetAncOne * sizeof(float);
  const size_t ys = (((size_t)B.het_nb + 1) * 2 * sizeof(float) + 15) / 16 * 16;
  lay.bytes = (het_tm_smem_bytes(B.het_nb, L.tm_M, L.tm_M > 0 ? L.tm_pieces : 0) + 15) / 16 * 16;
  if ((size_t)L.tm_M * 2 * sizeof(float) >= anc) {
    lay.anc_off = (int)ys;
  } else {
    lay.anc_off = (int)lay.bytes;
    lay.bytes += anc;
  }
  return lay;
}

inline __host__ __device__ int fold_ld(int nc) { return (nc + 3) & ~3; }
inline __host__ __device__ FoldTables fold_tables(const DeviceBuffers& B) {
  return {B.fold_nc, fold_ld(B.fold_nc), B.fold_tab, B.fold_w, B.fold_x, B.data32, B.tiles, B.basis, B.bin_tile,
          B.slice_begin};
}

// Bytes of the weights and table (weights first) in shared memory.
inline __host__ __device__ size_t fold_resident_bytes(int nc, int n_det) {
  return (size_t)nc * n_det * 32 * sizeof(float4) + sizeof(float) * FR_ROWS * fold_ld(nc);
}

// Lets kernel f take all the dynamic shared memory that a block of its device may
// have.  The limit belongs to the function, not to a context or a launch, and
// contexts may be used by several threads at once: every launch asks for the same
// value, so that none lowers it between another's call and its launch.
cudaError_t allow_shared(const void* f);

// FP64 path: the basis functions at every bin, tab [NBASIS][n_bins] (f in row
// B_ONE), from base [n_bins][3] (f^-1/3, f^1/3, ln f).
cudaError_t launch_fp64_basis(const LikeConst& L, const double* base, double* tab, cudaStream_t st);
// Node weights of the event (B.fold_w) from its weighted data (B.data32) and
// the chunks (device pointer); synchronises the stream.
cudaError_t launch_fold_weights(const LikeConst& L, const DeviceBuffers& B, const FoldChunk* chunks, cudaStream_t st);
// The folded evaluation of n records in B.rec (launch_loglike_mixed after its
// set-up).
cudaError_t launch_fold(const LikeConst& L, const DeviceBuffers& B, int n, double* out, cudaStream_t st,
                        double* kappa_out);

// logL of n thetas (device pointers) into out; kappa_out (optional, n x 8
// doubles) receives the unscaled per-detector sums (re, im) for each theta.
cudaError_t launch_loglike_mixed(const LikeConst& L, const DeviceBuffers& B, const double* theta, int n,
                                 double* out, cudaStream_t st, double* kappa_out = nullptr);
cudaError_t launch_loglike_fp64(const LikeConst& L, const DeviceBuffers& B, const double* theta, int n,
                                double* out, cudaStream_t st, double* kappa_out = nullptr);
// Setup record and detector strain of one theta (FP64) into out [n_det][n_bins].
cudaError_t launch_waveform(const LikeConst& L, const double* theta_dev, EvalRecord* rec_dev, double2* out,
                            cudaStream_t st);
// Post-hoc d_L of n samples of a distance-marginalised run (records in B.rec
// and their kappa sums from the preceding likelihood launch); writes theta[6].
cudaError_t launch_distance_draw(const LikeConst& L, const DeviceBuffers& B, const double* kappa, int n,
                                 long long first, unsigned k0, unsigned k1, double* theta, cudaStream_t st);
// Heterodyned logL of n thetas (device pointers), up to eight per CTA.
// kappa_out (n x 8) / vv_out (n x 4), optional: the per-detector cache of
// projection-only evaluations (het.cuh het_detector).
// With t_c marginalised (L.tm_n > 0) one CTA of kHetTmThreads per theta
// instead, and ell (optional, n x tm_n) receives each node's log weight.
cudaError_t launch_loglike_het(const LikeConst& L, const DeviceBuffers& B, const double* theta, int n, double* out,
                               cudaStream_t st, double* kappa_out = nullptr, double* vv_out = nullptr,
                               float* ell = nullptr);
// Post-hoc t_c of n time-marginalised samples from their node log weights
// (records of the same samples in B.rec); sample i uses the Philox counter of
// global index first + i under key (k0, k1).  Writes theta[i][11].
cudaError_t launch_time_draw(const LikeConst& L, const DeviceBuffers& B, const float* ell, int n, long long first,
                             unsigned k0, unsigned k1, double* theta, cudaStream_t st);
cudaError_t launch_prior_transform(const PriorSlot* slots, int n_sampled, const double* u, int n, double* theta,
                                   cudaStream_t st, SkyFrame sky);

// Shared memory that a slice of the bins is planned for (plan_slices): data (float2
// per detector and bin) plus the tile index of each bin.
inline size_t sweep_smem_bytes(int n_det, int slice_bins) {
  return (size_t)slice_bins * (n_det * sizeof(float2) + sizeof(int));
}

}  // namespace swig
