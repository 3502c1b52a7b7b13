// CUDA kernels of the rKS hot path (sm_103a), FP64 basis.
//
// One Arnoldi step of Algorithm 2 (Sec. 3.1) for the new column c = j + 1:
//   k_spmv_sketch   w = A u_j (u_j = U[:, j] * colscale[j]) -> U[:, c];
//                   z_raw += sum_i sign * w_i  (z = Omega w, Sec. 5 sketch)
//   k_ls_dot        r1 = S^T z                    (S = Omega U[:, 0..j])
//   k_ls_resid      z1 = z - S r1
//   k_ls_dot2       r = r1 + S^T z1, rs = r .* colscale   (CGS2 in the sketch
//                   for b_{j+1} = S^+ z; locked columns included: Thm 4.3)
//   k_update_sketch U[:, c] <- U[:, c] - U[:, 0..j] rs   (u~ = w - U b);
//                   s_raw += sum_i sign * u~_i            (s~ = Omega u~)
//   k_finish        beta = ||s~||, S[:, c] = s~/beta, colscale[c] = 1/beta,
//                   coefficient column, zero the accumulators.
// The basis is stored unnormalised: column c holds u~_c and colscale[c] =
// 1/beta_c (u_c = u~_c / beta_c), so no pass over n is spent on scaling.
//
// Restart (Algorithm 1, truncation; Eqs. 3.5-3.6): k_restart_gemm computes
// U[:, q..q+ka-1] = U[:, q..m-1] Q' in place, row by row, and moves the last
// vector u to column q + ka.
//
// Sketch: column i of Omega has zeta distinct rows from the SplitMix64 hash
// of (seed, i) (see rks.h); entries are sign/sqrt(zeta).  The kernels
// accumulate sign * v in FP64 shared-memory bins per CTA and fold the bins
// into a global d-vector with one atomic add per bin; the 1/sqrt(zeta) scale
// is applied by the consumers of the sums.

#include <mutex>

#include "rks_impl.h"

namespace rks {

__device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ull;

// Rows and signs (+1/-1) of column i of Omega.  Returns false if the draw cap
// was reached (cannot happen for d >= 2*zeta in practice).
template <int MAXZ>
__device__ __forceinline__ bool omega_column(uint64_t seed, uint64_t i, int d, int zeta,
                                             int (&rows)[MAXZ], double (&sgn)[MAXZ]) {
  const uint64_t base = mix64(seed * kGamma + i);
  int cnt = 0;
  const int cap = 32 * zeta;
#pragma unroll
  for (int t = 0; t < MAXZ; ++t) { rows[t] = -1; sgn[t] = 0.0; }
  for (int r = 0; r < cap && cnt < zeta; ++r) {
    uint64_t h = mix64(base + (uint64_t)(r + 1) * kGamma);
    int row = (int)(((h >> 32) * (uint64_t)d) >> 32);
    bool dup = false;
#pragma unroll
    for (int t = 0; t < MAXZ; ++t) dup |= (rows[t] == row);
    if (dup) continue;
    double s = (h & 1ull) ? -1.0 : 1.0;
#pragma unroll
    for (int t = 0; t < MAXZ; ++t) {
      if (t == cnt) { rows[t] = row; sgn[t] = s; }
    }
    ++cnt;
  }
  return cnt == zeta;
}

template <int MAXZ>
__device__ __forceinline__ void sketch_add(double* bins, uint64_t seed, uint64_t i, int d, int zeta,
                                           double v, int* flag) {
  int rows[MAXZ];
  double sgn[MAXZ];
  if (!omega_column<MAXZ>(seed, i, d, zeta, rows, sgn)) atomicOr(flag, RKS_FLAG_HASH);
#pragma unroll
  for (int t = 0; t < MAXZ; ++t)
    if (t < zeta && rows[t] >= 0) atomicAdd(&bins[rows[t]], sgn[t] * v);
}

__device__ __forceinline__ void bins_zero(double* bins, int d) {
  for (int r = threadIdx.x; r < d; r += blockDim.x) bins[r] = 0.0;
  __syncthreads();
}

__device__ __forceinline__ void bins_flush(const double* bins, double* out, int d) {
  __syncthreads();
  for (int r = threadIdx.x; r < d; r += blockDim.x) {
    double v = bins[r];
    if (v != 0.0) atomicAdd(&out[r], v);
  }
}

// ---------------------------------------------------------------------------

template <int MAXZ>
__global__ void k_sketch_pairs(int64_t n, int d, int zeta, uint64_t seed, int32_t* rows_out,
                               int8_t* signs_out, int* flag) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    int rows[MAXZ];
    double sgn[MAXZ];
    if (!omega_column<MAXZ>(seed, (uint64_t)i, d, zeta, rows, sgn)) atomicOr(flag, RKS_FLAG_HASH);
#pragma unroll
    for (int t = 0; t < MAXZ; ++t)
      if (t < zeta) {
        rows_out[i * zeta + t] = rows[t];
        signs_out[i * zeta + t] = (int8_t)(sgn[t] > 0 ? 1 : -1);
      }
  }
}

// out += scale * sum_i sign * x_i, FP64 bins (sketches too large for the
// integer bins of k_sketch_vec_fix).
template <int MAXZ>
__global__ void k_sketch_vec(int64_t n, const double* __restrict__ x, double scale, int d, int zeta,
                             uint64_t seed, double* out, int* flag) {
  extern __shared__ double bins[];
  bins_zero(bins, d);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    sketch_add<MAXZ>(bins, seed, (uint64_t)i, d, zeta, x[i] * scale, flag);
  bins_flush(bins, out, d);
}

// The same sums in fixed point.  What bounds the FP64 form is the shared-
// memory FP64 atomic (a compare-and-swap loop) and the sequential hash; here
// a tile's values become integers in units of 2^-78 of a shared power of two,
// cut into 20-bit limbs that are added with native 32-bit integer atomics (a
// tile has at most 2048 rows and a row meets a bin at most once, so a limb sum
// stays below 2^31), and all zeta draws of a row are hashed at once, repeats
// redrawn afterwards.  The limbs go to 80-bit sums per tile; FP64 appears only
// when a CTA hands its bins over (at its end, or when a tile's largest value
// leaves the power of two).
//
// No addend loses a bit: a value takes the limbs its 53 bits reach, three
// within 2^-4 of the tile's largest, four within 2^-24, and one that is
// smaller still, or is no number, goes to FP64 bins beside the integers.  (With
// three limbs for everything a bin without large entries lost the low bits
// of its small ones.)
// Measured, n = 4 096 000, d = 600, zeta = 8, the whole rks_sketch_apply call
// (the shared atomics are the bound; HBM would take 5 us): 453 us with FP64
// bins, allocations and a copy of the sums to the host and back; 204 us here
// (186 us with three limbs and rounded values); 207 -> 27 us at n = 20 000.
// With exponents at random over the whole range, where the FP64 bins take all:
// 423 -> 383 us.
constexpr int kFixSpan = 8;       // binades a tile's largest value may lie below the power of two
constexpr int kFixThreads = 512;
constexpr int kFixTile = 2048;
constexpr int kFixMaxD = 3072;    // 40 bytes a bin

// One distinct-row draw set: rows[t] and signs (bit t of the result) of
// column i; false if the draw cap was reached.
template <int MAXZ>
__device__ __forceinline__ bool omega_rows(uint64_t seed, uint64_t i, int d, int zeta, int (&rows)[MAXZ],
                                           unsigned& neg) {
  const uint64_t base = mix64(seed * kGamma + i);
  neg = 0u;
#pragma unroll
  for (int t = 0; t < MAXZ; ++t) {
    const uint64_t h = mix64(base + (uint64_t)(t + 1) * kGamma);
    rows[t] = t < zeta ? (int)__umulhi((unsigned)(h >> 32), (unsigned)d) : -2 - t;
    neg |= (unsigned)(h & 1ull) << t;
  }
  unsigned dup = 0u;
#pragma unroll
  for (int t = 1; t < MAXZ; ++t) {
    bool e = false;
#pragma unroll
    for (int u = 0; u < MAXZ; ++u) e |= u < t && rows[u] == rows[t];
    dup |= (unsigned)e << t;
  }
  if (dup == 0u) return true;
  // the draws after the first zeta fill the repeated slots in turn
#pragma unroll
  for (int t = 1; t < MAXZ; ++t)
    if ((dup >> t) & 1u) rows[t] = -1;
  int r = zeta;
  const int cap = 32 * zeta;
#pragma unroll
  for (int t = 1; t < MAXZ; ++t) {
    while (rows[t] == -1) {
      if (r >= cap) return false;
      const uint64_t h = mix64(base + (uint64_t)(++r) * kGamma);
      const int row = (int)__umulhi((unsigned)(h >> 32), (unsigned)d);
      bool e = false;
#pragma unroll
      for (int u = 0; u < MAXZ; ++u) e |= rows[u] == row;
      if (e) continue;
      rows[t] = row;
      neg = (neg & ~(1u << t)) | ((unsigned)(h & 1ull) << t);
    }
  }
  return true;
}

template <int MAXZ>
__global__ void __launch_bounds__(kFixThreads) k_sketch_vec_fix(int64_t n, int tile, const double* __restrict__ x,
                                                                double scale, int d, int zeta, uint64_t seed,
                                                                double* __restrict__ out, int* flag) {
  constexpr int RPT = kFixTile / kFixThreads;
  extern __shared__ __align__(8) unsigned char fixmem[];
  long long* hi = reinterpret_cast<long long*>(fixmem);   // d: sums in units of 2^60
  long long* lo = hi + d;                                  // d: remainders in -2^59 .. 2^59
  double* fb = reinterpret_cast<double*>(lo + d);          // d: FP64 sums of what the limbs do not take
  int* limb = reinterpret_cast<int*>(fb + d);              // 4 x d, lowest first
  __shared__ int wmax[kFixThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int b = tid; b < d; b += kFixThreads) {
    hi[b] = 0;
    lo[b] = 0;
    fb[b] = 0.0;
#pragma unroll
    for (int q = 0; q < 4; ++q) limb[b + q * d] = 0;
  }
  // a bin's integer sum in FP64; its owner thread alone reads and writes it
  auto sum_of = [&](int b, int es) {
    return scalbn((double)hi[b] * 1152921504606846976.0 + (double)lo[b], es - 1101);
  };
  const int64_t ntile = (n + tile - 1) / tile;
  const int64_t t0 = blockIdx.x * ntile / gridDim.x, t1 = (blockIdx.x + 1) * ntile / gridDim.x;
  int es = -1;                     // |x| < 2^(es - 1022) for the integers; -1: none yet
  for (int64_t t = t0; t < t1; ++t) {
    const int64_t r0 = t * tile;
    const int rows = (int)(n - r0 < tile ? n - r0 : tile);
    unsigned long long xb[RPT];
    int em = 0;                    // largest exponent of the tile's numbers, 0: all are zero
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
      const int l = tid + k * kFixThreads;
      xb[k] = l < rows ? (unsigned long long)__double_as_longlong(x[r0 + l]) : 0ull;
      const int E = (int)((xb[k] >> 52) & 0x7FF);
      if ((xb[k] << 1) != 0 && E != 0x7FF) em = max(em, max(E, 1));
    }
    em = __reduce_max_sync(0xffffffffu, em);
    if (lane == 0) wmax[warp] = em;
    __syncthreads();
    em = __reduce_max_sync(0xffffffffu, wmax[lane & (kFixThreads / 32 - 1)]);
    if (em > es || (em > 0 && em < es - kFixSpan)) {
      for (int b = tid; b < d; b += kFixThreads) {
        const double v = es >= 0 ? sum_of(b, es) : 0.0;
        if (v != 0.0) atomicAdd(&out[b], v * scale);
        hi[b] = 0;
        lo[b] = 0;
      }
      es = em + 2;
    }
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
      const int l = tid + k * kFixThreads;
      if (l >= rows) break;
      int rw[MAXZ];
      unsigned neg;
      if (!omega_rows<MAXZ>(seed, (uint64_t)(r0 + l), d, zeta, rw, neg)) { atomicOr(flag, RKS_FLAG_HASH); continue; }
      int E = (int)((xb[k] >> 52) & 0x7FF);
      unsigned long long m = xb[k] & 0xFFFFFFFFFFFFFull;
      if (E) m |= 1ull << 52; else E = 1;
      const int sh = E - es + 6;   // at most 6
      if (E == 0x7FF || sh < -20) {
        const double v = __longlong_as_double((long long)xb[k]);
        if (v != 0.0)
#pragma unroll
          for (int u = 0; u < MAXZ; ++u)
            if (u < zeta) atomicAdd(&fb[rw[u]], (neg >> u) & 1u ? -v : v);
        continue;
      }
      int lf = 0;
      if (sh >= 0) {
        m <<= sh;
      } else {
        lf = (int)((m & ((1ull << -sh) - 1)) << (20 + sh));
        m >>= -sh;
      }
      const int l0 = (int)(m & 0xFFFFF), l1 = (int)((m >> 20) & 0xFFFFF), l2 = (int)(m >> 40);
      neg ^= (xb[k] >> 63) ? ~0u : 0u;
#pragma unroll
      for (int u = 0; u < MAXZ; ++u)
        if (u < zeta) {
          const int sg = -(int)((neg >> u) & 1u);
          int* q = limb + rw[u];
          if (lf) atomicAdd(q, (lf ^ sg) - sg);
          atomicAdd(q + d, (l0 ^ sg) - sg);
          atomicAdd(q + 2 * d, (l1 ^ sg) - sg);
          atomicAdd(q + 3 * d, (l2 ^ sg) - sg);
        }
    }
    __syncthreads();
    for (int b = tid; b < d; b += kFixThreads) {
      const int mid = limb[b + 2 * d];
      const long long s = lo[b] + limb[b] + ((long long)limb[b + d] << 20) + ((long long)(mid & 0xFFFFF) << 40);
      const long long c = (s + (1ll << 59)) >> 60;
      hi[b] += limb[b + 3 * d] + (mid >> 20) + c;
      lo[b] = s - (c << 60);
#pragma unroll
      for (int q = 0; q < 4; ++q) limb[b + q * d] = 0;
    }
    __syncthreads();
  }
  for (int b = tid; b < d; b += kFixThreads) {
    const double v = (es >= 0 ? sum_of(b, es) : 0.0) + fb[b];
    if (v != 0.0) atomicAdd(&out[b], v * scale);
  }
}

// w = A (x * xscale[0]); out_raw += Omega-sums of w.
template <int MAXZ>
__global__ void k_spmv_sketch(int64_t n, const int32_t* __restrict__ rowptr,
                              const int32_t* __restrict__ colind, const double* __restrict__ vals,
                              const double* __restrict__ x, const double* __restrict__ xscale,
                              double* __restrict__ w, int d, int zeta, uint64_t seed,
                              double* out_raw, int* flag) {
  extern __shared__ double bins[];
  bins_zero(bins, d);
  const double sc = xscale[0];
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (int p = rowptr[i]; p < rowptr[i + 1]; ++p) acc = fma(vals[p], x[colind[p]], acc);
    acc *= sc;
    w[i] = acc;
    sketch_add<MAXZ>(bins, seed, (uint64_t)i, d, zeta, acc, flag);
  }
  bins_flush(bins, out_raw, d);
}

// r[col] = sum_row S[row, col] * z_raw[row] * zscale, one warp per column.
__global__ void k_ls_dot(int c, int d, const double* __restrict__ S, const double* __restrict__ z,
                         double zscale, double* __restrict__ r) {
  int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int lane = threadIdx.x & 31;
  if (warp >= c) return;
  const double* s = S + (size_t)warp * d;
  double acc = 0.0;
  for (int row = lane; row < d; row += 32) acc = fma(s[row], z[row], acc);
  for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) r[warp] = acc * zscale;
}

// z1[row] = z_raw[row] * zscale - sum_col S[row, col] r1[col], one warp per row.
__global__ void k_ls_resid(int c, int d, const double* __restrict__ S, const double* __restrict__ z,
                           double zscale, const double* __restrict__ r1, double* __restrict__ z1) {
  int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int lane = threadIdx.x & 31;
  if (row >= d) return;
  double acc = 0.0;
  for (int col = lane; col < c; col += 32) acc = fma(S[row + (size_t)col * d], r1[col], acc);
  for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) z1[row] = z[row] * zscale - acc;
}

// r = r1 + S^T z1 ; rs = r .* colscale
__global__ void k_ls_dot2(int c, int d, const double* __restrict__ S, const double* __restrict__ z1,
                          const double* __restrict__ r1, const double* __restrict__ colscale,
                          double* __restrict__ r, double* __restrict__ rs) {
  int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int lane = threadIdx.x & 31;
  if (warp >= c) return;
  const double* s = S + (size_t)warp * d;
  double acc = 0.0;
  for (int row = lane; row < d; row += 32) acc = fma(s[row], z1[row], acc);
  for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) {
    double v = r1[warp] + acc;
    r[warp] = v;
    rs[warp] = v * colscale[warp];
  }
}

// U[:, c] <- U[:, c] - U[:, 0..c-1] rs ; out_raw += Omega-sums of the result.
template <int MAXZ>
__global__ void k_update_sketch(int64_t n, double* __restrict__ U, int64_t ldu, int c,
                                const double* __restrict__ rs, int d, int zeta, uint64_t seed,
                                double* out_raw, int* flag) {
  extern __shared__ double sh[];
  double* bins = sh;
  double* rsh = sh + d;
  for (int col = threadIdx.x; col < c; col += blockDim.x) rsh[col] = rs[col];
  bins_zero(bins, d);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double acc = U[i + (int64_t)c * ldu];
    const double* up = U + i;
    int col = 0;
    for (; col + 4 <= c; col += 4) {
      double a0 = up[(int64_t)(col + 0) * ldu], a1 = up[(int64_t)(col + 1) * ldu];
      double a2 = up[(int64_t)(col + 2) * ldu], a3 = up[(int64_t)(col + 3) * ldu];
      acc = fma(-a0, rsh[col + 0], acc);
      acc = fma(-a1, rsh[col + 1], acc);
      acc = fma(-a2, rsh[col + 2], acc);
      acc = fma(-a3, rsh[col + 3], acc);
    }
    for (; col < c; ++col) acc = fma(-up[(int64_t)col * ldu], rsh[col], acc);
    U[i + (int64_t)c * ldu] = acc;
    sketch_add<MAXZ>(bins, seed, (uint64_t)i, d, zeta, acc, flag);
  }
  bins_flush(bins, out_raw, d);
}

// One CTA: finish step c (see file header).  coef column c-1 gets (r, beta).
__global__ void k_finish(int c, int d, double zscale, double* __restrict__ s_raw,
                         double* __restrict__ z_raw, double* __restrict__ S,
                         double* __restrict__ colscale, const double* __restrict__ r,
                         double* __restrict__ coef, int ldcoef, int* flag) {
  __shared__ double red[2][32];
  double ss = 0.0, zz = 0.0;
  for (int row = threadIdx.x; row < d; row += blockDim.x) {
    double v = s_raw[row] * zscale;
    double w = z_raw[row] * zscale;
    ss = fma(v, v, ss);
    zz = fma(w, w, zz);
  }
  for (int o = 16; o; o >>= 1) {
    ss += __shfl_xor_sync(0xffffffffu, ss, o);
    zz += __shfl_xor_sync(0xffffffffu, zz, o);
  }
  int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { red[0][warp] = ss; red[1][warp] = zz; }
  __syncthreads();
  if (warp == 0) {
    int nw = blockDim.x >> 5;
    ss = lane < nw ? red[0][lane] : 0.0;
    zz = lane < nw ? red[1][lane] : 0.0;
    for (int o = 16; o; o >>= 1) {
      ss += __shfl_xor_sync(0xffffffffu, ss, o);
      zz += __shfl_xor_sync(0xffffffffu, zz, o);
    }
    if (lane == 0) { red[0][0] = ss; red[1][0] = zz; }
  }
  __syncthreads();
  const double beta = sqrt(red[0][0]);
  const double znorm = sqrt(red[1][0]);
  const bool finite = isfinite(beta) && isfinite(znorm);
  const bool brk = finite && !(beta > 1e-14 * znorm);
  const double inv = (finite && !brk) ? 1.0 / beta : 0.0;
  for (int row = threadIdx.x; row < d; row += blockDim.x) {
    S[row + (size_t)c * d] = s_raw[row] * zscale * inv;
    s_raw[row] = 0.0;
    z_raw[row] = 0.0;
  }
  double* cc = coef + (size_t)(c - 1) * ldcoef;
  for (int i = threadIdx.x; i < c; i += blockDim.x) cc[i] = r[i];
  if (threadIdx.x == 0) {
    cc[c] = beta;
    colscale[c] = inv;
    if (!finite) atomicOr(flag, RKS_FLAG_NAN);
    else if (brk) atomicOr(flag, RKS_FLAG_BREAKDOWN);
  }
}

// Initial vector: S[:, 0] = s/beta, colscale[0] = 1/beta from s_raw.
__global__ void k_start_finish(int d, double zscale, double* __restrict__ s_raw, double* __restrict__ S,
                               double* __restrict__ colscale, int* flag) {
  __shared__ double red[32];
  double ss = 0.0;
  for (int row = threadIdx.x; row < d; row += blockDim.x) {
    double v = s_raw[row] * zscale;
    ss = fma(v, v, ss);
  }
  for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) red[warp] = ss;
  __syncthreads();
  if (warp == 0) {
    int nw = blockDim.x >> 5;
    ss = lane < nw ? red[lane] : 0.0;
    for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if (lane == 0) red[0] = ss;
  }
  __syncthreads();
  double beta = sqrt(red[0]);
  bool ok = isfinite(beta) && beta > 0.0;
  double inv = ok ? 1.0 / beta : 0.0;
  for (int row = threadIdx.x; row < d; row += blockDim.x) {
    S[row] = s_raw[row] * zscale * inv;
    s_raw[row] = 0.0;
  }
  if (threadIdx.x == 0) {
    colscale[0] = inv;
    if (!ok) atomicOr(flag, isfinite(beta) ? RKS_FLAG_BREAKDOWN : RKS_FLAG_NAN);
  }
}

// Default start vector: N(0,1) entries, SplitMix64 stream of `seed`
// (draw r = mix(seed + (r+1) gamma)), Box-Muller on draws (2i, 2i+1).
__global__ void k_start_vector(int64_t n, uint64_t seed, double* __restrict__ x) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    uint64_t h1 = mix64(seed + (uint64_t)(2 * i + 1) * kGamma);
    uint64_t h2 = mix64(seed + (uint64_t)(2 * i + 2) * kGamma);
    double u1 = (double)(h1 >> 11) * (1.0 / 9007199254740992.0);
    double u2 = (double)(h2 >> 11) * (1.0 / 9007199254740992.0);
    x[i] = sqrt(-2.0 * log1p(-u1)) * cospi(2.0 * u2);
  }
}

// Row-blocked small GEMM: C[i, 0..nout-1] = sum_l A[i, l] * B[l, o] for the
// rows of this CTA, A = columns a0..a0+nin-1 of (lda), C = columns c0.. of
// (ldc).  All reads of a row happen before its writes, so C may alias A.
// If move_src >= 0, column move_src of A is copied to column c0 + nout after.
// Dynamic shared memory: B (nin * nout) then tmp (blockDim * nout).
__global__ void k_rows_gemm(int64_t n, const double* A, int64_t lda, int a0, int nin,
                            const double* __restrict__ B, int nout, double* C, int64_t ldc, int c0,
                            int move_src) {
  extern __shared__ double sh[];
  double* Bs = sh;
  double* tmp = sh + (size_t)nin * nout;
  for (int t = threadIdx.x; t < nin * nout; t += blockDim.x) Bs[t] = B[t];
  __syncthreads();
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double* ap = A + i + (int64_t)a0 * lda;
  for (int o0 = 0; o0 < nout; o0 += 8) {
    double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    int no = min(8, nout - o0);
    for (int l = 0; l < nin; ++l) {
      double a = ap[(int64_t)l * lda];
      const double* b = Bs + l + (size_t)o0 * nin;
#pragma unroll
      for (int o = 0; o < 8; ++o)
        if (o < no) acc[o] = fma(a, b[(size_t)o * nin], acc[o]);
    }
#pragma unroll
    for (int o = 0; o < 8; ++o)
      if (o < no) tmp[(size_t)(o0 + o) * blockDim.x + threadIdx.x] = acc[o];
  }
  double mv = move_src >= 0 ? A[i + (int64_t)move_src * lda] : 0.0;
  for (int o = 0; o < nout; ++o) C[i + (int64_t)(c0 + o) * ldc] = tmp[(size_t)o * blockDim.x + threadIdx.x];
  if (move_src >= 0) C[i + (int64_t)(c0 + nout) * ldc] = mv;
}

// y = A x for several columns: Y[:, j] = A X[:, j], j < ncols.
// Residual sums of Ritz vectors, the product with A formed on the way (A X is
// never stored): for slot t = slots[blockIdx.y * C ..], columns col[t] (re) and
// colim[t] (im, CPLX only), lambda = (a, b):
//   {||r||^2, ||x||^2, Re x^H A x, Im x^H A x}, r = A x - lambda x,
// per CTA to out[(t * 4 + q) * gridDim.x + cta], added on the host in CTA order.
// FP64 throughput bounds it: a real column costs its row's products and four
// FMAs (the two-pass form spent 16 on the sums alone and stored A X); C = 4
// real columns share the reads of A.  Rows of more than kLongRow entries are
// taken by the whole warp (one thread on a row of 10^4 entries held the pass
// up for 1.6 ms), unless so many of the warp's 32 rows are long that a thread
// each takes fewer FP64 operations: a row by the warp is its entries / 32
// products and 5 additions, a thread each as many products as the longest row
// has entries.  Measured, n = 1e6, 20 columns, 5 entries per row: 0.79 -> 0.35
// ms; 100 003 rows with one of 10^4 entries, 8 columns: 1.65 -> 0.24 ms; all
// rows of 101, n = 1e5, 8 columns: 0.55 ms in two passes, 0.72 with every row
// by the warp, 0.24.
constexpr int kLongRow = 64;
template <bool CPLX, int C>
__global__ void __launch_bounds__(256) k_resid(int64_t n, const int32_t* __restrict__ rowptr,
                                               const int32_t* __restrict__ colind, const double* __restrict__ vals,
                                               const double* __restrict__ X, int64_t ld, const int* __restrict__ slots,
                                               int nslot, const int* __restrict__ col, const int* __restrict__ colim,
                                               const double* __restrict__ lre, const double* __restrict__ lim,
                                               double* __restrict__ out) {
  constexpr int V = CPLX ? 2 : C;              // vectors read per row
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int slot[C];
  const double* xv[V];
  double la[C];
#pragma unroll
  for (int q = 0; q < C; ++q) {
    slot[q] = slots[min((int)blockIdx.y * C + q, nslot - 1)];
    la[q] = lre[slot[q]];
    xv[q] = X + (int64_t)col[slot[q]] * ld;
  }
  if (CPLX) xv[1] = X + (int64_t)colim[slot[0]] * ld;
  const double lb = CPLX ? lim[slot[0]] : 0.0;
  double s[C][4];
#pragma unroll
  for (int q = 0; q < C; ++q)
#pragma unroll
    for (int k = 0; k < 4; ++k) s[q][k] = 0.0;
  for (int64_t i0 = ((int64_t)blockIdx.x * 8 + warp) * 32; i0 < n; i0 += (int64_t)gridDim.x * 256) {
    const int64_t i = i0 + lane;
    const int p0 = i < n ? rowptr[i] : 0, p1 = i < n ? rowptr[i + 1] : 0;
    bool big = p1 - p0 > kLongRow;
    unsigned m = __ballot_sync(0xffffffffu, big);
    if (m) {
      const int longest = __reduce_max_sync(0xffffffffu, p1 - p0);
      if (__popc(m) * (longest / 32 + 6) >= longest) { m = 0u; big = false; }
    }
    double ax[V];
#pragma unroll
    for (int v = 0; v < V; ++v) ax[v] = 0.0;
    if (!big) {
#pragma unroll 4
      for (int p = p0; p < p1; ++p) {
        const double a = vals[p];
        const int j = colind[p];
#pragma unroll
        for (int v = 0; v < V; ++v) ax[v] = fma(a, xv[v][j], ax[v]);
      }
    }
    for (; m; m &= m - 1) {
      const int src = __ffs(m) - 1;
      const int b0 = __shfl_sync(0xffffffffu, p0, src), b1 = __shfl_sync(0xffffffffu, p1, src);
      double part[V];
#pragma unroll
      for (int v = 0; v < V; ++v) part[v] = 0.0;
#pragma unroll 4
      for (int p = b0 + lane; p < b1; p += 32) {
        const double a = vals[p];
        const int j = colind[p];
#pragma unroll
        for (int v = 0; v < V; ++v) part[v] = fma(a, xv[v][j], part[v]);
      }
#pragma unroll
      for (int v = 0; v < V; ++v) {
        for (int o = 16; o; o >>= 1) part[v] += __shfl_xor_sync(0xffffffffu, part[v], o);
        if (lane == src) ax[v] = part[v];
      }
    }
    if (i < n) {
      if (CPLX) {
        const double xr = xv[0][i], xi = xv[1][i];
        const double rre = ax[0] - la[0] * xr + lb * xi, rim = ax[1] - la[0] * xi - lb * xr;
        s[0][0] += rre * rre + rim * rim;
        s[0][1] += xr * xr + xi * xi;
        s[0][2] += xr * ax[0] + xi * ax[1];
        s[0][3] += xr * ax[1] - xi * ax[0];
      } else {
#pragma unroll
        for (int q = 0; q < C; ++q) {
          const double x = xv[q][i], r = fma(-la[q], x, ax[q]);
          s[q][0] = fma(r, r, s[q][0]);
          s[q][1] = fma(x, x, s[q][1]);
          s[q][2] = fma(x, ax[q], s[q][2]);
        }
      }
    }
  }
  __shared__ double red[C][4][8];
#pragma unroll
  for (int q = 0; q < C; ++q)
#pragma unroll
    for (int k = 0; k < (CPLX ? 4 : 3); ++k) {
      double v = s[q][k];
      for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) red[q][k][warp] = v;
    }
  __syncthreads();
  if (threadIdx.x < C * 4) {
    const int q = threadIdx.x >> 2, k = threadIdx.x & 3;
    if ((int)blockIdx.y * C + q < nslot) {
      double v = 0.0;
      if (CPLX || k < 3)
        for (int w = 0; w < 8; ++w) v += red[q][k][w];
      out[((size_t)slots[blockIdx.y * C + q] * 4 + k) * gridDim.x + blockIdx.x] = v;
    }
  }
}

__global__ void k_f32_to_f64(int64_t n, const float* __restrict__ a, double* __restrict__ b) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    b[i] = (double)a[i];
}

__global__ void k_check_csr(int64_t n, int64_t nnz, const int32_t* __restrict__ rowptr,
                            const int32_t* __restrict__ colind, int* bad) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    int a = rowptr[i], b = rowptr[i + 1];
    if (a > b || a < 0 || b > nnz) { atomicOr(bad, 1); continue; }
    for (int p = a; p < b; ++p)
      if (colind[p] < 0 || colind[p] >= n) { atomicOr(bad, 2); break; }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0 && (rowptr[0] != 0 || rowptr[n] != nnz)) atomicOr(bad, 4);
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------

static int grid_for(int64_t n, int threads, int max_ctas) {
  int64_t g = (n + threads - 1) / threads;
  if (g > max_ctas) g = max_ctas;
  if (g < 1) g = 1;
  return (int)g;
}


void launch_sketch_pairs(int64_t n, int d, int zeta, uint64_t seed, int32_t* rows, int8_t* signs,
                         int* flag, cudaStream_t st) {
  int g = grid_for(n, 256, 152 * 8);
  if (zeta <= 4) k_sketch_pairs<4><<<g, 256, 0, st>>>(n, d, zeta, seed, rows, signs, flag);
  else if (zeta <= 8) k_sketch_pairs<8><<<g, 256, 0, st>>>(n, d, zeta, seed, rows, signs, flag);
  else k_sketch_pairs<16><<<g, 256, 0, st>>>(n, d, zeta, seed, rows, signs, flag);
}

void launch_sketch_vec(int64_t n, const double* x, double scale, int d, int zeta, uint64_t seed, double* out,
                       int* flag, cudaStream_t st) {
  if (d <= kFixMaxD) {
    // tiles of 2048 rows (a flush of d bins each) once every SM has one,
    // smaller ones before, so that short vectors still use many SMs
    const int tile = n >= (int64_t)152 * kFixTile ? kFixTile : (n >= (int64_t)76 * kFixTile ? kFixTile / 2 : kFixThreads);
    // two CTAs per SM: a third adds contention for the bins (226 us instead of
    // 204 at n = 4 096 000, d = 600; 471 instead of 383 where FP64 bins take all)
    const int g = (int)((n + tile - 1) / tile < 152 * 2 ? (n + tile - 1) / tile : 152 * 2);
    const size_t sm = (size_t)d * 40;
    if (zeta <= 4) k_sketch_vec_fix<4><<<g, kFixThreads, sm, st>>>(n, tile, x, scale, d, zeta, seed, out, flag);
    else if (zeta <= 8) k_sketch_vec_fix<8><<<g, kFixThreads, sm, st>>>(n, tile, x, scale, d, zeta, seed, out, flag);
    else k_sketch_vec_fix<16><<<g, kFixThreads, sm, st>>>(n, tile, x, scale, d, zeta, seed, out, flag);
    return;
  }
  int g = grid_for(n, 256, kSketchCtas);
  size_t sm = (size_t)d * sizeof(double);
  if (zeta <= 4) k_sketch_vec<4><<<g, 256, sm, st>>>(n, x, scale, d, zeta, seed, out, flag);
  else if (zeta <= 8) k_sketch_vec<8><<<g, 256, sm, st>>>(n, x, scale, d, zeta, seed, out, flag);
  else k_sketch_vec<16><<<g, 256, sm, st>>>(n, x, scale, d, zeta, seed, out, flag);
}

void launch_spmv_sketch(const Csr& A, const double* x, const double* xscale, double* w, int d, int zeta,
                        uint64_t seed, double* out_raw, int* flag, cudaStream_t st) {
  int g = grid_for(A.n, 256, kSketchCtas);
  size_t sm = (size_t)d * sizeof(double);
  if (zeta <= 4)
    k_spmv_sketch<4><<<g, 256, sm, st>>>(A.n, A.rowptr, A.colind, A.vals, x, xscale, w, d, zeta, seed, out_raw, flag);
  else if (zeta <= 8)
    k_spmv_sketch<8><<<g, 256, sm, st>>>(A.n, A.rowptr, A.colind, A.vals, x, xscale, w, d, zeta, seed, out_raw, flag);
  else
    k_spmv_sketch<16><<<g, 256, sm, st>>>(A.n, A.rowptr, A.colind, A.vals, x, xscale, w, d, zeta, seed, out_raw, flag);
}

void launch_ls(int c, int d, const double* S, const double* z_raw, double zscale, const double* colscale,
               double* r1, double* z1, double* r, double* rs, cudaStream_t st) {
  int warps_per_cta = 4;
  int g1 = (c + warps_per_cta - 1) / warps_per_cta;
  k_ls_dot<<<g1, 32 * warps_per_cta, 0, st>>>(c, d, S, z_raw, zscale, r1);
  int g2 = (d + warps_per_cta - 1) / warps_per_cta;
  k_ls_resid<<<g2, 32 * warps_per_cta, 0, st>>>(c, d, S, z_raw, zscale, r1, z1);
  k_ls_dot2<<<g1, 32 * warps_per_cta, 0, st>>>(c, d, S, z1, r1, colscale, r, rs);
}

void launch_update_sketch(int64_t n, double* U, int64_t ldu, int c, const double* rs, int d, int zeta,
                          uint64_t seed, double* out_raw, int* flag, cudaStream_t st) {
  int g = grid_for(n, 256, kSketchCtas);
  size_t sm = (size_t)(d + c) * sizeof(double);
  if (zeta <= 4) k_update_sketch<4><<<g, 256, sm, st>>>(n, U, ldu, c, rs, d, zeta, seed, out_raw, flag);
  else if (zeta <= 8) k_update_sketch<8><<<g, 256, sm, st>>>(n, U, ldu, c, rs, d, zeta, seed, out_raw, flag);
  else k_update_sketch<16><<<g, 256, sm, st>>>(n, U, ldu, c, rs, d, zeta, seed, out_raw, flag);
}

void launch_finish(int c, int d, double zscale, double* s_raw, double* z_raw, double* S, double* colscale,
                   const double* r, double* coef, int ldcoef, int* flag, cudaStream_t st) {
  k_finish<<<1, 512, 0, st>>>(c, d, zscale, s_raw, z_raw, S, colscale, r, coef, ldcoef, flag);
}

void launch_start_finish(int d, double zscale, double* s_raw, double* S, double* colscale, int* flag,
                         cudaStream_t st) {
  k_start_finish<<<1, 512, 0, st>>>(d, zscale, s_raw, S, colscale, flag);
}

void launch_start_vector(int64_t n, uint64_t seed, double* x, cudaStream_t st) {
  k_start_vector<<<grid_for(n, 256, 152 * 8), 256, 0, st>>>(n, seed, x);
}

// Opt every kernel with dynamic shared memory into the large carve-out
// (sketch bins of up to d = 8192 doubles, restart product tiles).
cudaError_t once_per_device(int slot, cudaError_t (*f)()) {
  constexpr int kMaxDev = 64;
  static std::mutex mu;
  static bool done[kCfgSlots][kMaxDev] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (slot < 0 || slot >= kCfgSlots || dev < 0 || dev >= kMaxDev) return cudaErrorInvalidValue;
  std::lock_guard<std::mutex> lock(mu);
  if (done[slot][dev]) return cudaSuccess;
  e = f();
  if (e == cudaSuccess) done[slot][dev] = true;
  return e;
}

static cudaError_t configure_kernels_once() {
  const int big = 200 * 1024;
  cudaError_t e = cudaSuccess;
#define RKS_SMEM(f) if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, big)
  RKS_SMEM(k_sketch_vec<4>); RKS_SMEM(k_sketch_vec<8>); RKS_SMEM(k_sketch_vec<16>);
  RKS_SMEM(k_sketch_vec_fix<4>); RKS_SMEM(k_sketch_vec_fix<8>); RKS_SMEM(k_sketch_vec_fix<16>);
  RKS_SMEM(k_spmv_sketch<4>); RKS_SMEM(k_spmv_sketch<8>); RKS_SMEM(k_spmv_sketch<16>);
  RKS_SMEM(k_update_sketch<4>); RKS_SMEM(k_update_sketch<8>); RKS_SMEM(k_update_sketch<16>);
  RKS_SMEM(k_rows_gemm);
#undef RKS_SMEM
  return e;
}

cudaError_t configure_kernels() { return once_per_device(kCfgBase, configure_kernels_once); }

int rows_gemm_smem(int nin, int nout, int threads) {
  return (int)(((size_t)nin * nout + (size_t)threads * nout) * sizeof(double));
}

void launch_rows_gemm(int64_t n, const double* A, int64_t lda, int a0, int nin, const double* B, int nout,
                      double* C, int64_t ldc, int c0, int move_src, cudaStream_t st) {
  const int threads = 128;
  size_t sm = (size_t)rows_gemm_smem(nin, nout, threads);
  int g = (int)((n + threads - 1) / threads);
  k_rows_gemm<<<g, threads, sm, st>>>(n, A, lda, a0, nin, B, nout, C, ldc, c0, move_src);
}

int launch_resid(const Csr& A, const double* X, int64_t ld, int nreal, int npair, const int* slots, const int* col,
                 const int* colim, const double* lre, const double* lim, double* out, cudaStream_t st) {
  const int g = grid_for(A.n, 256, kResidCtas);
  // real columns four at a time, the last one to three by a kernel of that many
  // (rows of 27, n = 5e5, one column: 257 us with the group of four, 190 us)
  const int full = nreal & ~3;
  if (full > 0) {
    dim3 grid((unsigned)g, (unsigned)(full / 4));
    k_resid<false, 4><<<grid, 256, 0, st>>>(A.n, A.rowptr, A.colind, A.vals, X, ld, slots, full, col, colim, lre, lim,
                                            out);
  }
  if (nreal > full) {
    auto k = nreal - full == 1 ? k_resid<false, 1> : nreal - full == 2 ? k_resid<false, 2> : k_resid<false, 3>;
    k<<<g, 256, 0, st>>>(A.n, A.rowptr, A.colind, A.vals, X, ld, slots + full, nreal - full, col, colim, lre, lim, out);
  }
  if (npair > 0) {
    dim3 grid((unsigned)g, (unsigned)npair);
    k_resid<true, 1><<<grid, 256, 0, st>>>(A.n, A.rowptr, A.colind, A.vals, X, ld, slots + nreal, npair, col, colim,
                                           lre, lim, out);
  }
  return g;
}

void launch_f32_to_f64(int64_t n, const float* a, double* b, cudaStream_t st) {
  k_f32_to_f64<<<grid_for(n, 256, 152 * 8), 256, 0, st>>>(n, a, b);
}

void launch_check_csr(int64_t n, int64_t nnz, const int32_t* rowptr, const int32_t* colind, int* bad,
                      cudaStream_t st) {
  k_check_csr<<<grid_for(n, 256, 152 * 8), 256, 0, st>>>(n, nnz, rowptr, colind, bad);
}

}  // namespace rks
