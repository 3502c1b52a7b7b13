// Randomized QR factorisations of a tall and skinny block K = Q R (Sec. 2 of
// the paper: the randomized orthogonalisation processes an rKS basis can be
// built with), on the double-float kernels of the solver:
//
//  * RKS_QR_RGS: randomized Gram-Schmidt, the process of Algorithm 2 without
//    the product with A.  The sketches z_j = Omega k_j of all columns first
//    (one launch, which also converts the block); r = S_j^T z_j with a second
//    pass in the sketch (host, FP64: S_j is d x j), q~ = k_j - Q_j r by panels
//    of 8 columns against all earlier ones, then column by column inside the
//    panel fused with the partial sketches of q~ (the solver's update kernel),
//    beta = ||Omega q~||.  Columns stay unscaled on the
//    device (their scale 1/beta goes into the next coefficients and the
//    final conversion), as in the solver.
//  * RKS_QR_WHITEN: sketch and whiten (the whitening of Sec. 3.3 on a whole
//    block): Omega K = Q_s R by Householder QR on the host, Q = K R^{-1} by
//    one double-float product.
//  * RKS_QR_RCHOLQR: randomized Cholesky QR: Q_1 = K R_1^{-1} as above, the
//    Gram matrix Q_1^T Q_1 (double-float dot kernel), its Cholesky factor R_2,
//    Q = Q_1 R_2^{-1}, R = R_2 R_1: a Euclidean-orthonormal Q.
//  * RKS_QR_RHQR: randomized Householder QR: Householder QR of the sketched
//    block Theta K, Theta = [[I_s, 0], [0, Omega']] (rows 0..s-1 kept,
//    Omega' the embedding of dimension n - s on the others), on the host,
//    with every reflector applied to the double-float columns on the device
//    and Q accumulated from the reflectors: Theta Q orthonormal.
//
// Omega is the solver's sparse-sign embedding (SplitMix64 hash, zeta rows per
// column, values +-1/sqrt(zeta)), applied through the deterministic per-tile
// bin lists, so the results do not depend on scheduling.

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "../../include/rks.h"
#include "convert.cuh"
#include "dense.h"
#include "pdl.cuh"
#include "rks_impl.h"

namespace {

// Q[i, j] = (x.hi + x.lo)[i, j] * scale[j] in FP64, four rows a thread with
// their loads in flight together
__global__ void __launch_bounds__(256) k_df2d_scaled(int64_t n, const float2* __restrict__ x, int64_t ldx,
                                                     const double* __restrict__ scale, double* __restrict__ y,
                                                     int64_t ldy) {
  const int j = blockIdx.y;
  const double sc = scale[j];
  x += (int64_t)j * ldx;
  y += (int64_t)j * ldy;
  for (int64_t i0 = blockIdx.x * (int64_t)1024 + threadIdx.x; i0 < n; i0 += (int64_t)gridDim.x * 1024) {
    float2 v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (i0 + 256 * q < n) v[q] = x[i0 + 256 * q];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (i0 + 256 * q < n) y[i0 + 256 * q] = rks::df_to_double(v[q]) * sc;
  }
}

constexpr int kRgsThreads = 256;
constexpr int kMaxD = 8192;      // largest sketch size

// Device state of the randomized Gram-Schmidt (column-major arrays).
struct RgsState {
  int s, d;
  double zscale;
  const double* Z;     // d x s: sums of Omega k_j, unscaled
  double* sum;         // d: sums of the sketch of the column just updated, unscaled
  double* P;           // d x kPanelCols: the panel's sketches after the earlier panels' projection
  double* S;           // d x s: the sketches of the orthonormal columns
  double* R;           // s x s
  double* cs;          // s: 1 / beta_j, the scale of a stored column
  float2* nrs;         // coefficients of the next update
  int* flag;           // 1: a column vanished or is not finite
};

// a[c] = S[:, c0 + c]^T z for c < nc, then z -= S[:, c0 ..] a, a warp per
// column and a thread per row; z and a in shared memory.
__device__ void rgs_project(const RgsState& g, int c0, int nc, double* z, double* a) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int c = warp; c < nc; c += kRgsThreads / 32) {
    const double* sc = g.S + (size_t)(c0 + c) * g.d;
    double v = 0.0;
    for (int i = lane; i < g.d; i += 32) v += sc[i] * z[i];
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) a[c] = v;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < g.d; i += kRgsThreads) {
    double v = z[i];
#pragma unroll 4
    for (int c = 0; c < nc; ++c) v -= g.S[i + (size_t)(c0 + c) * g.d] * a[c];
    z[i] = v;
  }
  __syncthreads();
}

// Column k of a panel against the p0 earlier columns, twice: its coefficients
// for the panel update (zero for k >= nb), its part of R and its sketch after
// it.  One CTA per column; bound by FP64 at two lanes a clock: 31 us on average
// over the ten panels of 80 columns, d = 320.
__global__ void __launch_bounds__(kRgsThreads) k_rgs_panel(RgsState g, int p0, int nb) {
  extern __shared__ double rgs_sm[];
  double* z = rgs_sm;
  double* a = rgs_sm + g.d;
  constexpr int B = rks::kPanelCols;
  const int k = blockIdx.x;
  if (k >= nb) {
    for (int c = threadIdx.x; c < p0; c += kRgsThreads) g.nrs[(size_t)c * B + k] = make_float2(0.f, 0.f);
    return;
  }
  for (int i = threadIdx.x; i < g.d; i += kRgsThreads) z[i] = g.Z[i + (size_t)(p0 + k) * g.d] * g.zscale;
  __syncthreads();
  for (int pass = 0; pass < 2 && p0 > 0; ++pass) {
    rgs_project(g, 0, p0, z, a);
    for (int c = threadIdx.x; c < p0; c += kRgsThreads) {
      double* r = g.R + c + (size_t)(p0 + k) * g.s;
      const double v = pass ? *r + a[c] : a[c];
      *r = v;
      if (pass) g.nrs[(size_t)c * B + k] = rks::df_from_double(-v * g.cs[c]);
    }
    __syncthreads();
  }
  for (int i = threadIdx.x; i < g.d; i += kRgsThreads) g.P[i + (size_t)k * g.d] = z[i];
}

// Column p0 + done of a panel has been updated: beta, its sketch, its scale.
// Then (next >= 0) column p0 + next against the panel's columns before it,
// twice: the coefficients of its update.  One CTA, 11 us at d = 320, in place
// of a copy to the host, its loops and a copy back; with the panels' share the
// 80-column RGS at n = 1e6 went from 8.8 to 8.0 ms, and from 7.4 to 7.0 ms with
// the division per row gone and the launch overlapped with the fold.
__global__ void __launch_bounds__(kRgsThreads) k_rgs_col(RgsState g, int p0, int done, int next) {
  extern __shared__ double rgs_sm[];
  double* z = rgs_sm;
  double* a = rgs_sm + g.d;
  __shared__ double red[kRgsThreads / 32 + 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int j = p0 + done;
  rks::pdl_next();
  if (next >= 0)                       // written before the update in front of the fold
    for (int i = threadIdx.x; i < g.d; i += kRgsThreads) z[i] = g.P[i + (size_t)next * g.d];
  rks::pdl_wait();
  double bb = 0.0;
  for (int i = threadIdx.x; i < g.d; i += kRgsThreads) {
    const double v = g.sum[i] * g.zscale;
    bb += v * v;
  }
  for (int o = 16; o; o >>= 1) bb += __shfl_xor_sync(0xffffffffu, bb, o);
  if (lane == 0) red[warp] = bb;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int q = 0; q < kRgsThreads / 32; ++q) t += red[q];
    const double beta = sqrt(t);
    if (!(beta > 0.0) || !isfinite(beta)) *g.flag = 1;
    g.R[j + (size_t)j * g.s] = beta;
    g.cs[j] = red[kRgsThreads / 32] = 1.0 / beta;
  }
  __syncthreads();
  const double inv = red[kRgsThreads / 32];
  for (int i = threadIdx.x; i < g.d; i += kRgsThreads) {
    g.S[i + (size_t)j * g.d] = g.sum[i] * g.zscale * inv;   // a division per row is nine FP64 operations
  }
  if (next < 0) return;
  __syncthreads();
  for (int pass = 0; pass < 2; ++pass) {
    rgs_project(g, p0, next, z, a);
    if ((int)threadIdx.x < next) {
      const int c = threadIdx.x;
      double* r = g.R + p0 + c + (size_t)(p0 + next) * g.s;
      const double v = pass ? *r + a[c] : a[c];
      *r = v;
      if (pass) g.nrs[c] = rks::df_from_double(-v * g.cs[p0 + c]);
    }
    __syncthreads();
  }
}

float2 to_df(double v) {
  const float h = (float)v;
  return make_float2(h, (float)(v - (double)h));
}

// Device state of one call, freed on every exit path.
struct QrWork {
  int64_t n = 0, ldu = 0;
  int s = 0, d = 0, zeta = 0, chunk = 1;
  double zscale = 0.0;
  cudaStream_t st = nullptr;
  float2* U = nullptr;        // ldu x 2s double-float columns: [0, s) and [s, 2s)
  uint16_t* otab = nullptr;
  rks::SketchTiles tiles;
  bool have_tiles = false;
  double* part = nullptr;     // per-CTA partial sums (G x d per column; the Gram matrix's)
  double* sums = nullptr;     // folded sums (d per column; the Gram matrix's pairs)
  float2* Q2 = nullptr;       // s x s double-float factor
  float2* nrs = nullptr;      // update coefficients (s x 8 of a panel, or 2 s)
  float2* sj = nullptr;       // scale of the updated column
  double* scale = nullptr;    // s column scales for the output
  double* dense = nullptr;    // small matrices of the randomized Gram-Schmidt
  char* small = nullptr;      // the block that holds sums, Q2, nrs, sj, scale, dense and flag
  int* flag = nullptr;
  std::vector<double> host;   // sums read back
  ~QrWork() {
    cudaFree(U); cudaFree(otab); cudaFree(part); cudaFree(small);
    if (have_tiles) rks::free_sketch_tiles(&tiles);
  }
};

#define QK(x)                                   \
  do {                                          \
    if ((x) != cudaSuccess) return RKS_ECUDA;   \
  } while (0)

// nsk: rows the sketch covers (n, or n - s for RHQR's Omega' on rows s..n-1);
// ncol: double-float columns (s, or 2 s for the methods that form Q beside K)
int setup(QrWork& w, int64_t n, int s, int d, int zeta, uint64_t seed, cudaStream_t st, int64_t nsk, int ncol) {
  w.n = n; w.s = s; w.d = d; w.zeta = zeta; w.st = st;
  w.zscale = 1.0 / std::sqrt((double)zeta);
  w.ldu = (n + 31) / 32 * 32;
  const size_t nsum = std::max((size_t)d * s, (size_t)rks::gram_pairs(s));
  // one block for the small arrays (and two for the tiles): seven allocations
  // fewer took randomized Cholesky QR of 50 021 x 24 from 832 to 740 us
  const size_t small[7] = {nsum * sizeof(double), (size_t)s * s * sizeof(float2),
                           (size_t)rks::kPanelCols * s * sizeof(float2), sizeof(float2), (size_t)s * sizeof(double),
                           ((size_t)d * (1 + rks::kPanelCols + s) + (size_t)s * s) * sizeof(double), sizeof(int)};
  size_t at[7], total = 0;
  for (int q = 0; q < 7; ++q) {
    at[q] = total;
    total += (small[q] + 255) & ~(size_t)255;
  }
  if (cudaMalloc(&w.U, (size_t)w.ldu * ncol * sizeof(float2)) != cudaSuccess ||
      cudaMalloc(&w.otab, (size_t)nsk * rks::omega_slots(zeta) * sizeof(uint16_t)) != cudaSuccess ||
      cudaMalloc(&w.small, total) != cudaSuccess)
    return RKS_ENOMEM;
  w.sums = reinterpret_cast<double*>(w.small + at[0]);
  w.Q2 = reinterpret_cast<float2*>(w.small + at[1]);
  w.nrs = reinterpret_cast<float2*>(w.small + at[2]);
  w.sj = reinterpret_cast<float2*>(w.small + at[3]);
  w.scale = reinterpret_cast<double*>(w.small + at[4]);
  w.dense = reinterpret_cast<double*>(w.small + at[5]);
  w.flag = reinterpret_cast<int*>(w.small + at[6]);
  w.host.assign(nsum, 0.0);
  QK(cudaMemsetAsync(w.flag, 0, sizeof(int), st));
  rks::launch_omega_table(nsk, d, zeta, seed, w.otab, w.flag, st);
  int bad = 0;
  QK(cudaMemcpyAsync(&bad, w.flag, sizeof(int), cudaMemcpyDeviceToHost, st));
  QK(cudaStreamSynchronize(st));
  if (bad) return RKS_EINVAL;
  if (rks::configure_df_kernels() != cudaSuccess) return RKS_ECUDA;
  if (rks::build_sketch_tiles(nsk, d, zeta, w.otab, &w.tiles, st) != 0) return RKS_ECUDA;
  w.have_tiles = true;
  cudaFree(w.otab);
  w.otab = nullptr;
  if (rks::sketch_tile_smem(w.tiles, s) > 200 * 1024) return RKS_EINVAL;
  // partial sketches of as many columns at a time as 256 MB hold
  w.chunk = (int)std::max<size_t>(1, std::min<size_t>(s, ((size_t)256 << 20) / ((size_t)w.tiles.G * d * sizeof(double))));
  const size_t npart = std::max((size_t)w.tiles.G * d * w.chunk, (size_t)rks::gram_ctas(n) * rks::gram_pairs(s));
  if (cudaMalloc(&w.part, npart * sizeof(double)) != cudaSuccess) return RKS_ENOMEM;
  return RKS_OK;
}

// The largest shared memory of the small steps, once per device: a limit set
// call by call could be lowered by another thread's smaller problem between
// this one's setting and its launch.
cudaError_t configure_qr_kernels_once() {
  const int sm = (int)((kMaxD + RKS_SKETCH_QR_MAX_S) * sizeof(double));
  cudaError_t e = cudaFuncSetAttribute(k_rgs_panel, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_rgs_col, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
  return e;
}

float2* col(QrWork& w, int j) { return w.U + (size_t)j * w.ldu; }

// U[:, c0 + o] = sum_l U[:, a0 + l] F[l, o] for o < s (F s x s, host FP64),
// out of place, in blocks of at most 64 outputs
int product(QrWork& w, int a0, const std::vector<double>& F, int c0) {
  const int s = w.s;
  std::vector<float2> F2((size_t)s * s);
  for (size_t t = 0; t < F2.size(); ++t) F2[t] = to_df(F[t]);
  QK(cudaMemcpyAsync(w.Q2, F2.data(), F2.size() * sizeof(float2), cudaMemcpyHostToDevice, w.st));
  for (int o0 = 0; o0 < s; o0 += 64) {
    const int nb = std::min(64, s - o0);
    rks::launch_df_rows_gemm(w.n, w.U, w.ldu, a0, s, w.Q2 + (size_t)o0 * s, nb, c0 + o0, -1, false, w.st);
  }
  QK(cudaGetLastError());
  QK(cudaStreamSynchronize(w.st));   // F2 is a host temporary
  return RKS_OK;
}

// inverse of an upper-triangular s x s R (back substitution)
std::vector<double> upper_inverse(int s, const std::vector<double>& R) {
  std::vector<double> X((size_t)s * s, 0.0);
  for (int j = 0; j < s; ++j) {
    X[j + (size_t)j * s] = 1.0 / R[j + (size_t)j * s];
    for (int i = j - 1; i >= 0; --i) {
      double acc = 0.0;
      for (int l = i + 1; l <= j; ++l) acc += R[i + (size_t)l * s] * X[l + (size_t)j * s];
      X[i + (size_t)j * s] = -acc / R[i + (size_t)i * s];
    }
  }
  return X;
}

// Sk (d x s) = the sketches of s columns; launch(j, m) leaves the partials of
// columns j .. j + m - 1 in w.part
template <class F>
int sketches(QrWork& w, std::vector<double>& Sk, F launch) {
  const int s = w.s, d = w.d;
  for (int j = 0; j < s; j += w.chunk) {
    const int m = std::min(w.chunk, s - j);
    launch(j, m);
    rks::launch_df_fold(w.part, d, w.tiles.G, w.sums + (size_t)j * d, w.st, m);
  }
  QK(cudaGetLastError());
  QK(cudaMemcpyAsync(w.host.data(), w.sums, (size_t)d * s * sizeof(double), cudaMemcpyDeviceToHost, w.st));
  QK(cudaStreamSynchronize(w.st));
  Sk.assign((size_t)d * s, 0.0);
  for (size_t t = 0; t < Sk.size(); ++t) Sk[t] = w.host[t] * w.zscale;
  return RKS_OK;
}

// Sk = Omega U[row0:, c0 .. c0+s)
int sketch_block(QrWork& w, int c0, std::vector<double>& Sk, int row0 = 0) {
  return sketches(w, Sk, [&](int j, int m) {
    rks::launch_df_sketch_cols(col(w, c0 + j) + row0, w.ldu, m, w.tiles, w.part, w.st);
  });
}

// U[:, 0 .. s) = K in double-float and Sk = Omega K
int sketch_input(QrWork& w, const double* K, int64_t ldk, std::vector<double>& Sk) {
  return sketches(w, Sk, [&](int j, int m) {
    rks::launch_sketch_cols_f64(K + (size_t)j * ldk, ldk, m, col(w, j), w.ldu, w.tiles, w.part, w.st);
  });
}

// Omega K = Q_s R1 (host); U[:, s..2s) = K R1^{-1}.  Sk receives Q_s.
int whiten(QrWork& w, const double* K, int64_t ldk, std::vector<double>& R1, std::vector<double>& Sk) {
  const int s = w.s, d = w.d;
  int rc = sketch_input(w, K, ldk, Sk);
  if (rc) return rc;
  R1.assign((size_t)s * s, 0.0);
  rks_dense::house_qr(d, s, Sk.data(), R1.data());
  for (int j = 0; j < s; ++j)
    if (!(R1[j + (size_t)j * s] > 0.0) || !std::isfinite(R1[j + (size_t)j * s])) return RKS_EBREAKDOWN;
  return product(w, 0, upper_inverse(s, R1), s);
}

// Randomized Gram-Schmidt by panels of kPanelCols columns: the coefficients of
// a column against all earlier panels are its projection in the sketch, which
// does not depend on the panel's own columns, so one pass over the earlier
// columns updates the whole panel (they were read once per column, 26 GB at
// n = 1e6, s = 80); inside the panel a column at a time, its sketch measured
// after its update.  Every projection is made twice (r = S^T z,
// r += S^T (z - S r): S is sketch-orthonormal).  The small steps are kernels
// (k_rgs_panel, k_rgs_col), so that the host waits once, at the end.
int rgs(QrWork& w, const double* K, int64_t ldk, std::vector<double>& R, std::vector<double>& S) {
  constexpr int B = rks::kPanelCols;
  const int s = w.s, d = w.d;
  RgsState g;
  g.s = s; g.d = d; g.zscale = w.zscale;
  g.Z = w.sums; g.cs = w.scale; g.nrs = w.nrs; g.flag = w.flag;
  g.sum = w.dense; g.P = g.sum + d; g.S = g.P + (size_t)d * B; g.R = g.S + (size_t)d * s;
  if (rks::once_per_device(rks::kCfgQr, configure_qr_kernels_once) != cudaSuccess) return RKS_ECUDA;
  const size_t sm = (size_t)(d + s) * sizeof(double);
  const float2 one = make_float2(1.f, 0.f);
  QK(cudaMemcpyAsync(w.sj, &one, sizeof(float2), cudaMemcpyHostToDevice, w.st));
  QK(cudaMemsetAsync(g.R, 0, (size_t)s * s * sizeof(double), w.st));
  // z_j = Omega k_j does not depend on the process: all of them at once
  for (int j = 0; j < s; j += w.chunk) {
    const int m = std::min(w.chunk, s - j);
    rks::launch_sketch_cols_f64(K + (size_t)j * ldk, ldk, m, col(w, j), w.ldu, w.tiles, w.part, w.st);
    rks::launch_df_fold(w.part, d, w.tiles.G, w.sums + (size_t)j * d, w.st, m);
  }
  for (int p0 = 0; p0 < s; p0 += B) {
    const int nb = std::min(B, s - p0);
    k_rgs_panel<<<B, kRgsThreads, sm, w.st>>>(g, p0, nb);
    if (p0 > 0) rks::launch_df_panel(w.n, w.U, w.ldu, p0, p0, nb, w.nrs, w.st);
    for (int jj = 0; jj < nb; ++jj) {
      // q~ = k_j - sum_c (q~_c / beta_c) r_c, fused with its partial sketches
      if (jj > 0) rks::launch_pdl(k_rgs_col, 1, kRgsThreads, sm, w.st, g, p0, jj - 1, jj);
      rks::launch_df_update_sketch(col(w, p0), w.ldu, jj, w.nrs, w.sj, w.tiles, w.part, false, w.st);
      rks::launch_df_fold(w.part, d, w.tiles.G, g.sum, w.st);
    }
    rks::launch_pdl(k_rgs_col, 1, kRgsThreads, sm, w.st, g, p0, nb - 1, -1);
  }
  QK(cudaGetLastError());
  int bad = 0;
  R.resize((size_t)s * s);
  S.resize((size_t)d * s);
  QK(cudaMemcpyAsync(&bad, w.flag, sizeof(int), cudaMemcpyDeviceToHost, w.st));
  QK(cudaMemcpyAsync(R.data(), g.R, R.size() * sizeof(double), cudaMemcpyDeviceToHost, w.st));
  QK(cudaMemcpyAsync(S.data(), g.S, S.size() * sizeof(double), cudaMemcpyDeviceToHost, w.st));
  QK(cudaStreamSynchronize(w.st));
  return bad ? RKS_EBREAKDOWN : RKS_OK;
}

// Randomized Householder QR: Householder QR of Theta K ((s + d) x s, Theta =
// [[I_s, 0], [0, Omega']], Omega' on rows s..n-1) on the host in FP64, its
// reflectors H_j = I - beta_j u_j (Theta u_j)^T Theta applied to the
// double-float columns on the device (u_j is column j after the earlier
// reflectors with its entries above j dropped and rho_j taken off entry j,
// so Theta u_j = v_j), then Q = H_0 ... H_{s-1} [I_s; 0] accumulated
// backwards into columns s..2s-1.  The coefficient of every column update is
// a sketched inner product: the sketches of the later columns are updated on
// the host (Theta H_j = (I - beta v v^T) Theta), each pivot column is
// re-read and re-sketched from the device before its reflector is formed.
int rhqr(QrWork& w, std::vector<double>& R, std::vector<double>& scale) {
  const int s = w.s, d = w.d, ns = s + d;
  const int64_t nb = w.n - s;
  std::vector<double> Y((size_t)ns * s, 0.0), V((size_t)ns * s, 0.0), beta(s, 0.0);
  std::vector<float2> top((size_t)s * s), cf(s), colv(s);
  // top blocks (rows 0..s-1) and sketches of the bottom rows of every column
  QK(cudaMemcpy2DAsync(top.data(), s * sizeof(float2), w.U, w.ldu * sizeof(float2), s * sizeof(float2), s,
                       cudaMemcpyDeviceToHost, w.st));
  std::vector<double> Z0;
  int rc = sketch_block(w, 0, Z0, s);
  if (rc) return rc;
  for (int l = 0; l < s; ++l) {
    for (int i = 0; i < s; ++i) {
      const float2 t = top[i + (size_t)l * s];
      Y[i + (size_t)l * ns] = (double)t.x + (double)t.y;
    }
    for (int i = 0; i < d; ++i) Y[s + i + (size_t)l * ns] = Z0[i + (size_t)l * d];
  }
  R.assign((size_t)s * s, 0.0);
  for (int j = 0; j < s; ++j) {
    double* y = &Y[(size_t)j * ns];
    double* v = &V[(size_t)j * ns];
    if (j > 0) {
      // the pivot column as the device holds it (its top rows and the sketch
      // of the others), so that the reflector is consistent with the vector
      // it is built from: Theta u_j = v_j to rounding
      QK(cudaMemcpyAsync(colv.data(), col(w, j), (size_t)s * sizeof(float2), cudaMemcpyDeviceToHost, w.st));
      rks::launch_df_sketch_vec(col(w, j) + s, w.tiles, w.part, false, w.st);
      rks::launch_df_fold(w.part, d, w.tiles.G, w.sums, w.st);
      QK(cudaGetLastError());
      QK(cudaMemcpyAsync(w.host.data(), w.sums, (size_t)d * sizeof(double), cudaMemcpyDeviceToHost, w.st));
      QK(cudaStreamSynchronize(w.st));
      for (int i = 0; i < s; ++i) y[i] = (double)colv[i].x + (double)colv[i].y;
      for (int i = 0; i < d; ++i) y[s + i] = w.host[i] * w.zscale;
    }
    double nn = 0.0;
    for (int i = j; i < ns; ++i) nn += y[i] * y[i];
    const double nrm = std::sqrt(nn);
    if (!(nrm > 0.0) || !std::isfinite(nrm)) return RKS_EBREAKDOWN;
    const double rho = y[j] >= 0.0 ? -nrm : nrm;     // -sign(y_j) ||y(j:)||
    for (int i = 0; i < j; ++i) R[i + (size_t)j * s] = y[i];
    R[j + (size_t)j * s] = rho;
    for (int i = j; i < ns; ++i) v[i] = y[i];
    v[j] -= rho;
    double vv = 0.0;
    for (int i = j; i < ns; ++i) vv += v[i] * v[i];
    beta[j] = 2.0 / vv;
    // column j becomes u_j: its top rows are v's (zeros above j)
    for (int i = 0; i < s; ++i) colv[i] = to_df(v[i]);
    QK(cudaMemcpyAsync(col(w, j), colv.data(), (size_t)s * sizeof(float2), cudaMemcpyHostToDevice, w.st));
    // H_j on the later columns: y_l -= c_l u_j, c_l = beta v^T Theta y_l
    const int nl = s - 1 - j;
    for (int l = j + 1; l < s; ++l) {
      double* yl = &Y[(size_t)l * ns];
      double a = 0.0;
      for (int i = j; i < ns; ++i) a += v[i] * yl[i];
      const double c = beta[j] * a;
      for (int i = j; i < ns; ++i) yl[i] -= c * v[i];
      cf[l - j - 1] = to_df(c);
    }
    if (nl > 0) {
      QK(cudaMemcpyAsync(w.nrs, cf.data(), (size_t)nl * sizeof(float2), cudaMemcpyHostToDevice, w.st));
      rks::launch_df_axpy_cols(w.n, w.U, w.ldu, j, j + 1, nl, w.nrs, w.st);
    }
  }
  // Q = H_0 ... H_{s-1} [I_s; 0] in columns s..2s-1, Theta Q tracked on the host
  QK(cudaMemsetAsync(col(w, s), 0, (size_t)w.ldu * s * sizeof(float2), w.st));
  std::vector<float2> eye((size_t)s * s, make_float2(0.f, 0.f));
  for (int l = 0; l < s; ++l) eye[l + (size_t)l * s] = make_float2(1.f, 0.f);
  QK(cudaMemcpy2DAsync(col(w, s), w.ldu * sizeof(float2), eye.data(), s * sizeof(float2), s * sizeof(float2), s,
                       cudaMemcpyHostToDevice, w.st));
  std::vector<double> Z((size_t)ns * s, 0.0);
  for (int l = 0; l < s; ++l) Z[l + (size_t)l * ns] = 1.0;
  for (int j = s - 1; j >= 0; --j) {
    const double* v = &V[(size_t)j * ns];
    for (int l = j; l < s; ++l) {
      double* zl = &Z[(size_t)l * ns];
      double a = 0.0;
      for (int i = j; i < ns; ++i) a += v[i] * zl[i];
      const double c = beta[j] * a;
      for (int i = j; i < ns; ++i) zl[i] -= c * v[i];
      cf[l - j] = to_df(c);
    }
    QK(cudaMemcpyAsync(w.nrs + s, cf.data(), (size_t)(s - j) * sizeof(float2), cudaMemcpyHostToDevice, w.st));
    rks::launch_df_axpy_cols(w.n, w.U, w.ldu, j, s + j, s - j, w.nrs + s, w.st);
  }
  QK(cudaGetLastError());
  // positive diagonal: flip Q's column j and R's row j where rho_j < 0
  scale.assign(s, 1.0);
  for (int j = 0; j < s; ++j)
    if (R[j + (size_t)j * s] < 0.0) {
      scale[j] = -1.0;
      for (int c = j; c < s; ++c) R[j + (size_t)c * s] = -R[j + (size_t)c * s];
    }
  (void)nb;
  QK(cudaStreamSynchronize(w.st));
  return RKS_OK;
}

}  // namespace

extern "C" int rks_sketch_qr(int64_t n, int s, const double* K, int64_t ldk, int d, int zeta, uint64_t seed,
                             int method, double* Q, int64_t ldq, double* R, double* S, void* stream) {
  if (n < 2 || s < 1 || s > RKS_SKETCH_QR_MAX_S || zeta < 1 || zeta > 16 || d < 2 * zeta || d > kMaxD || s > d ||
      s > n || !K || !Q || !R || ldk < n || ldq < n)
    return RKS_EINVAL;
  if (method != RKS_QR_RGS && method != RKS_QR_WHITEN && method != RKS_QR_RCHOLQR && method != RKS_QR_RHQR)
    return RKS_EINVAL;
  if (method == RKS_QR_RHQR && n - s < 2) return RKS_EINVAL;
  if (Q == K && ldq != ldk) return RKS_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  QrWork w;
  int rc = setup(w, n, s, d, zeta, seed, st, method == RKS_QR_RHQR ? n - s : n, method == RKS_QR_RGS ? s : 2 * s);
  if (rc) return rc;
  std::vector<double> Rh, Sh;
  int out0 = 0;                 // first column of the result in U
  std::vector<double> ones(s, 1.0);
  if (method == RKS_QR_RGS) {
    rc = rgs(w, K, ldk, Rh, Sh);
    if (rc) return rc;
  } else if (method == RKS_QR_RHQR) {
    std::vector<double> sc;
    rks::launch_d2df_cols(n, K, ldk, w.U, w.ldu, s, st);
    rc = rhqr(w, Rh, sc);
    if (rc) return rc;
    out0 = s;
    QK(cudaMemcpyAsync(w.scale, sc.data(), (size_t)s * sizeof(double), cudaMemcpyHostToDevice, st));
    if (S) {                    // Omega' Q[s:, :], measured: the sketched rows of Theta Q
      rc = sketch_block(w, s, Sh, s);
      if (rc) return rc;
      for (int j = 0; j < s; ++j)
        for (int i = 0; i < d; ++i) Sh[i + (size_t)j * d] *= sc[j];
    }
  } else {
    std::vector<double> R1;
    rc = whiten(w, K, ldk, R1, Sh);
    if (rc) return rc;
    out0 = s;
    Rh = R1;
    if (method == RKS_QR_RCHOLQR) {
      // G = Q1^T Q1 (columns s .. 2s-1)
      std::vector<double> G((size_t)s * s, 0.0);
      const int np = rks::gram_pairs(s);
      rks::launch_df_gram(n, col(w, s), w.ldu, s, w.part, st);
      rks::launch_df_fold(w.part, np, rks::gram_ctas(n), w.sums, st);
      QK(cudaGetLastError());
      QK(cudaMemcpyAsync(w.host.data(), w.sums, (size_t)np * sizeof(double), cudaMemcpyDeviceToHost, st));
      QK(cudaStreamSynchronize(st));
      for (int q = 0, bj = 0, bi = 0; q < np / 16; ++q) {
        for (int u = 0; u < 4; ++u)
          for (int v = 0; v < 4; ++v) {
            const int l = 4 * bi + u, cv = 4 * bj + v;
            if (l <= cv && cv < s) G[l + (size_t)cv * s] = G[cv + (size_t)l * s] = w.host[(size_t)q * 16 + 4 * u + v];
          }
        if (bi++ == bj) { bi = 0; ++bj; }
      }
      // Cholesky G = R2^T R2 (R2 upper)
      std::vector<double> R2((size_t)s * s, 0.0);
      for (int j = 0; j < s; ++j) {
        double dd = G[j + (size_t)j * s];
        for (int l = 0; l < j; ++l) dd -= R2[l + (size_t)j * s] * R2[l + (size_t)j * s];
        if (!(dd > 0.0) || !std::isfinite(dd)) return RKS_EDENSE;
        const double rjj = std::sqrt(dd);
        R2[j + (size_t)j * s] = rjj;
        for (int c = j + 1; c < s; ++c) {
          double a = G[j + (size_t)c * s];
          for (int l = 0; l < j; ++l) a -= R2[l + (size_t)j * s] * R2[l + (size_t)c * s];
          R2[j + (size_t)c * s] = a / rjj;
        }
      }
      rc = product(w, s, upper_inverse(s, R2), 0);   // Q = Q1 R2^{-1} into columns 0 .. s-1
      if (rc) return rc;
      out0 = 0;
      for (int j = 0; j < s; ++j)                   // R = R2 R1
        for (int i = 0; i <= j; ++i) {
          double a = 0.0;
          for (int l = i; l <= j; ++l) a += R2[i + (size_t)l * s] * R1[l + (size_t)j * s];
          Rh[i + (size_t)j * s] = a;
        }
    }
    QK(cudaMemcpyAsync(w.scale, ones.data(), (size_t)s * sizeof(double), cudaMemcpyHostToDevice, st));
    if (S) {                    // the sketch of the computed Q, measured
      rc = sketch_block(w, out0, Sh);
      if (rc) return rc;
    }
  }
  dim3 grid((unsigned)std::min<int64_t>((n + 1023) / 1024, 1024), (unsigned)s);
  k_df2d_scaled<<<grid, 256, 0, st>>>(n, col(w, out0), w.ldu, w.scale, Q, ldq);
  QK(cudaGetLastError());
  QK(cudaStreamSynchronize(st));
  std::copy(Rh.begin(), Rh.end(), R);
  if (S) std::copy(Sh.begin(), Sh.end(), S);
  return RKS_OK;
}
