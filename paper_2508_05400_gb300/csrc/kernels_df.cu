// Double-float (DF) kernels of the rKS hot path: FP64-class accuracy on the
// FP32 pipes of sm_103a.
//
// GB300 executes FP64 at about 2 FMA/clock/SM (measured: 0.6 T FMA/s for the
// whole GPU), 60x below FP32, so FP64 arithmetic, not HBM, bounds an FP64
// Arnoldi step.  Here every n-dimensional quantity keeps 8 bytes per value but
// as an unevaluated sum of two floats (hi + lo, |lo| <= ulp(hi)/2, a 48-bit
// significand), and products/sums use error-free transformations (TwoSum,
// TwoProd via fmaf) on the FP32 pipes.  The d-dimensional sketch data and the
// host-side dense work stay FP64; final residuals are computed in FP64.
//
// One Arnoldi step of Algorithm 2 (Sec. 3.1), new column c = j + 1, is three
// kernels:
//   k_df_spmv_ell / k_df_spmv_sketch
//                     w' = A u~_j (unscaled, u_j = u~_j / beta_j), z' = Omega w'
//                     (A as interleaved ELLPACK when that is compact, else CSR)
//   k_df_ls_coop      fold of the sketch partials, finish column j (beta_j =
//                     ||s~_j||, S, scale, coefficient column), then b = S^+ z by
//                     CGS2 in the sketch against the locked and active columns
//                     (Thm 4.3), z = z' / beta_j (k_df_fold + k_df_ls1 +
//                     k_df_ls_gram when a cooperative launch is unavailable)
//   k_df_update_sketch u~_{j+1} = w'/beta_j - U b, s~_{j+1} = Omega u~_{j+1}
//
// Sketch accumulation is deterministic: no atomics.  Each CTA owns a fixed,
// contiguous range of rows, cut into tiles of at most kTileRows rows.  For
// every tile a transposed copy of Omega restricted to the tile (the "bin
// lists", built once by k_tiles_build) gives, per sketch row, the tile rows
// that contribute to it and their signs, in a fixed order.  A tile's values
// are staged in shared memory; then the threads that own the tile's sketch
// rows sum their lists (DF, TwoSum) into per-CTA DF accumulators.  Each CTA
// writes its d partial sums; the consumer adds the CTA partials in a fixed
// order (fold_row).  The result is the same bits on every run.

#include <algorithm>
#include <type_traits>
#include <vector>

#include "convert.cuh"
#include "pdl.cuh"
#include "rks_impl.h"

namespace rks {

// ---------------------------------------------------------------------------
// double-float helpers
// ---------------------------------------------------------------------------

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  e = b - (s - a);
}

// (s, t) += (ah + al) * (bh + bl), (s, t) an unnormalised accumulator
__device__ __forceinline__ void df_mac(float ah, float al, float bh, float bl, float& s, float& t) {
  float p = ah * bh;
  float e = fmaf(ah, bh, -p);
  e = fmaf(ah, bl, e);
  e = fmaf(al, bh, e);
  float s2, e2;
  two_sum(s, p, s2, e2);
  s = s2;
  t += e2 + e;
}

// (s, t) += (bh + bl)
__device__ __forceinline__ void df_add(float bh, float bl, float& s, float& t) {
  float s2, e2;
  two_sum(s, bh, s2, e2);
  s = s2;
  t += e2 + bl;
}

// (s, t) += a * b for values stored as TA and TB: an FP32 value has no low
// word, so its terms are left out (df_mac's operations otherwise, in its
// order; the sums differ from df_mac's at most in the sign of a zero)
template <class TA, class TB>
__device__ __forceinline__ void mac_st(float2 a, float2 b, float& s, float& t) {
  constexpr bool A1 = sizeof(TA) == 4, B1 = sizeof(TB) == 4;
  if constexpr (!A1 && !B1) {
    df_mac(a.x, a.y, b.x, b.y, s, t);
  } else {
    const float p = a.x * b.x;
    float e = fmaf(a.x, b.x, -p);
    if constexpr (!B1) e = fmaf(a.x, b.y, e);
    if constexpr (!A1) e = fmaf(a.y, b.x, e);
    float s2, e2;
    two_sum(s, p, s2, e2);
    s = s2;
    t += e2 + e;
  }
}

__device__ __forceinline__ float2 df_norm(float s, float t) {
  float h, l;
  fast_two_sum(s, t, h, l);
  return make_float2(h, l);
}

// DF warp reduction of (s, t) pairs
__device__ __forceinline__ void df_warp_sum(float& s, float& t) {
  for (int o = 16; o; o >>= 1) {
    float s2 = __shfl_xor_sync(0xffffffffu, s, o);
    float t2 = __shfl_xor_sync(0xffffffffu, t, o);
    float ss, e;
    two_sum(s, s2, ss, e);
    s = ss;
    t = t + t2 + e;
  }
}

// Basis / matrix storage: float2 = double-float pair, float = FP32 (the
// mixed-precision basis of the paper's future-work direction, Sec. 6).  Loads
// widen to a pair; stores round the pair to the stored type, and the sketch
// is always taken of the value as stored.
__device__ __forceinline__ float2 ldv(const float2* p) { return *p; }
__device__ __forceinline__ float2 ldv(const float* p) { return make_float2(*p, 0.f); }
__device__ __forceinline__ float2 stv(float2* p, float2 v) { *p = v; return v; }
__device__ __forceinline__ float2 stv(float* p, float2 v) {
  float r = v.x + v.y;
  *p = r;
  return make_float2(r, 0.f);
}

// ---------------------------------------------------------------------------
// sketch (same hash as kernels.cu; see rks.h)
// ---------------------------------------------------------------------------

__device__ __forceinline__ uint64_t mix64_df(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Packed Omega table: for column i, MAXZ uint16 entries (row in bits 0..14,
// bit 15 set for a negative sign), written once by k_omega_table from the same
// hash; unused slots (t >= zeta) are 0xFFFF.  The tile bin lists are built
// from it.

// ---------------------------------------------------------------------------
// kernels
// ---------------------------------------------------------------------------

// The packed Omega table from the hash of rks.h.
template <int MAXZ>
__global__ void k_omega_table(int64_t n, int d, int zeta, uint64_t seed, uint16_t* __restrict__ tab, int* flag) {
  const uint64_t gamma = 0x9E3779B97F4A7C15ull;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t base = mix64_df(seed * gamma + (uint64_t)i);
    int rows[MAXZ];
    uint16_t ent[MAXZ];
#pragma unroll
    for (int t = 0; t < MAXZ; ++t) { rows[t] = -1; ent[t] = 0xFFFF; }
    int cnt = 0;
    const int cap = 32 * zeta;
    for (int r = 0; r < cap && cnt < zeta; ++r) {
      uint64_t h = mix64_df(base + (uint64_t)(r + 1) * gamma);
      int row = (int)(((h >> 32) * (uint64_t)d) >> 32);
      bool dup = false;
#pragma unroll
      for (int t = 0; t < MAXZ; ++t) dup |= (rows[t] == row);
      if (dup) continue;
#pragma unroll
      for (int t = 0; t < MAXZ; ++t)
        if (t == cnt) { rows[t] = row; ent[t] = (uint16_t)(row | ((h & 1ull) ? 0x8000 : 0)); }
      ++cnt;
    }
    if (cnt < zeta) atomicOr(flag, RKS_FLAG_HASH);
#pragma unroll
    for (int t = 0; t < MAXZ; ++t) tab[i * MAXZ + t] = ent[t];
  }
}

// ---------------------------------------------------------------------------
// tile bin lists (built once per context from the packed table)
// ---------------------------------------------------------------------------

// Largest number of entries of one sketch row within one tile (atomicMax into
// *lmax; the per-bin counts are integers, so their order does not matter).
template <int MAXZ>
__global__ void __launch_bounds__(256) k_tiles_count(const int64_t* __restrict__ trow, int d,
                                                     const uint16_t* __restrict__ otab, int* lmax) {
  extern __shared__ int cnt[];   // d
  const int64_t t = blockIdx.x;
  for (int b = threadIdx.x; b < d; b += blockDim.x) cnt[b] = 0;
  __syncthreads();
  const int64_t q1 = trow[t + 1] * MAXZ;
  for (int64_t q = trow[t] * MAXZ + threadIdx.x; q < q1; q += blockDim.x) {
    const uint32_t e = otab[q];
    if (e != 0xFFFFu) atomicAdd(&cnt[e & 0x7FFF], 1);
  }
  __syncthreads();
  int m = 0;
  for (int b = threadIdx.x; b < d; b += blockDim.x) m = max(m, cnt[b]);
  for (int o = 16; o; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(lmax, m);
}

// Bin lists of one tile (one CTA per tile), jagged-diagonal layout:
//   positions p = 0..d-1 rank the sketch rows by entry count (descending,
//   ties by row index); meta[t*d + p] = row | count << 16;
//   slot s holds entry s of every position whose count exceeds s, the
//   positions in order, from off[t*(L+1) + s] = sum_p min(count_p, s);
//   an entry is (tile row) | 0x8000 for a negative sign.
// The entries of a sketch row are listed in (32-row chunk, slot, lane) order,
// fixed by the table alone.
template <int MAXZ>
__global__ void __launch_bounds__(256) k_tiles_build(const int64_t* __restrict__ trow, int d, int zeta, int L,
                                                     const uint16_t* __restrict__ otab, uint32_t* __restrict__ meta,
                                                     int* __restrict__ off, uint16_t* __restrict__ ent) {
  extern __shared__ int sm[];
  int* cnt = sm;          // d: entries per sketch row
  int* rank = cnt + d;    // d: position of each sketch row
  int* scnt = rank + d;   // d: counts by position
  int* cur = scnt + d;    // d: fill cursor per sketch row
  int* offs = cur + d;    // L + 1
  const int64_t t = blockIdx.x;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int64_t r0 = trow[t], r1 = trow[t + 1];
  for (int b = tid; b < d; b += nt) { cnt[b] = 0; cur[b] = 0; }
  __syncthreads();
  for (int64_t q = r0 * MAXZ + tid; q < r1 * MAXZ; q += nt) {
    const uint32_t e = otab[q];
    if (e != 0xFFFFu) atomicAdd(&cnt[e & 0x7FFF], 1);
  }
  __syncthreads();
  for (int b = tid; b < d; b += nt) {
    const int cb = cnt[b];
    int r = 0;
    for (int b2 = 0; b2 < d; ++b2) {
      const int c2 = cnt[b2];
      r += (c2 > cb) || (c2 == cb && b2 < b);
    }
    rank[b] = r;
  }
  __syncthreads();
  for (int b = tid; b < d; b += nt) {
    scnt[rank[b]] = cnt[b];
    meta[t * d + rank[b]] = (uint32_t)b | ((uint32_t)cnt[b] << 16);
  }
  __syncthreads();
  for (int s = tid; s <= L; s += nt) {
    int o = 0;
    for (int p = 0; p < d; ++p) o += min(scnt[p], s);
    offs[s] = o;
    off[t * (L + 1) + s] = o;
  }
  __syncthreads();
  if (tid < 32) {
    const int lane = tid;
    uint16_t* et = ent + r0 * zeta;
    const int rows = (int)(r1 - r0);
    for (int c0 = 0; c0 < rows; c0 += 32) {
      const int l = c0 + lane;
      for (int s = 0; s < MAXZ; ++s) {
        const uint32_t e = l < rows ? (uint32_t)otab[(r0 + l) * MAXZ + s] : 0xFFFFu;
        const bool v = e != 0xFFFFu;
        const uint32_t key = v ? (e & 0x7FFFu) : (0x10000u + lane);   // no two invalid lanes match
        const unsigned grp = __match_any_sync(0xffffffffu, key);
        if (v) {
          const int b = (int)(e & 0x7FFFu);
          const int kk = cur[b] + __popc(grp & ((1u << lane) - 1u));
          et[offs[kk] + rank[b]] = (uint16_t)(l | (e & 0x8000u));
        }
        __syncwarp();
        if (v && lane == __ffs(grp) - 1) cur[e & 0x7FFFu] += __popc(grp);
        __syncwarp();
      }
    }
  }
}

// (s, e) += sign * vals[row] for one bin-list entry: the loads (32-bit shared
// addresses) and the addition
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
template <int OFF>
__device__ __forceinline__ uint32_t lds32(uint32_t a) {
  uint32_t x;
  asm volatile("ld.shared.b32 %0, [%1+%2];" : "=r"(x) : "r"(a), "n"(OFF));
  return x;
}
__device__ __forceinline__ uint32_t lds16(uint32_t a) {   // sign-extended: bit 15 in bit 31
  uint32_t x;
  asm volatile("ld.shared.s16 %0, [%1];" : "=r"(x) : "r"(a));
  return x;
}
__device__ __forceinline__ void lds_val(uint32_t a, uint32_t row, float2& v) {
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a + row * 8u));
}
__device__ __forceinline__ void lds_val(uint32_t a, uint32_t row, float& v) {
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a + row * 4u));
}
__device__ __forceinline__ float flip(float v, uint32_t x) {   // -v for a negative entry
  return __uint_as_float(__float_as_uint(v) ^ (x & 0x80000000u));
}

// (s, e) += sign * v for a bin-list entry x; FP32 values have no low word, so
// its terms are left out
__device__ __forceinline__ void tile_add(uint32_t x, float2 v, float& s, float& e) {
  df_add(flip(v.x, x), flip(v.y, x), s, e);
}
__device__ __forceinline__ void tile_add(uint32_t x, float v, float& s, float& e) {
  float s2, e2;
  two_sum(s, flip(v, x), s2, e2);
  s = s2;
  e += e2;
}
__device__ __forceinline__ void zero_val(float2& v) { v = make_float2(0.f, 0.f); }
__device__ __forceinline__ void zero_val(float& v) { v = 0.f; }

// a stored value (stv) into the tile's value buffer
__device__ __forceinline__ void tile_put(float2* p, float2 v) { *p = v; }
__device__ __forceinline__ void tile_put(float* p, float2 v) { *p = v.x; }

// Sketch of one staged tile: acc[row] += sum over the row's bin list of
// sign * vals[tile row], entries in their stored order.  The tile's slot
// offsets (offs), positions (ms) and entries (es) are in shared memory.
// H adjacent lanes share a position (each takes every H-th entry) when d is
// small; their sums are combined by a fixed xor tree.  A sketch row has one
// position per tile, so acc[row] has one writer per tile.
//
// Bound by instruction issue (a 7-point FP32 SpMV with zeta = 8 issues in 70%
// of the cycles, more than half of them here): hence H as a constant (the slot offsets at constant
// distances), 32-bit shared addresses, a sign by one exclusive or, and the
// last one to three entries of a list as one masked round (adding an exact
// zero changes no bit) instead of one by one.  FP32 values are kept as 4 bytes:
// at random banks a warp's read takes 3 to 4 passes instead of 6.  With the
// lists fetched by the CTA's last warps only, at n = 4.1e6, d = 96: the update
// of 2 to 27 columns 119 -> 93 us on average, the SpMV 73 -> 64 us; pairs,
// n = 1e6, d = 320, 1 to 80 columns: update 70 -> 62 us.
template <int H, class TV>
__device__ __forceinline__ void tile_gather_h(int d, const TV* vals, const int* offs, const uint32_t* ms,
                                              const uint16_t* es, float2* acc) {
  const int total = d * H;
  const int lane = threadIdx.x & 31;
  const uint32_t va = smem_addr(vals);
  for (int base = threadIdx.x & ~31; base < total; base += blockDim.x) {
    const int pp = base + lane;
    const int p = pp / H, h = pp % H;
    float s = 0.f, e = 0.f;
    int b = -1, cnt = 0;
    if (pp < total) {
      const uint32_t mt = ms[p];
      b = (int)(mt & 0xFFFFu);
      cnt = (int)(mt >> 16);
      const uint32_t ea = smem_addr(es) + 2u * p;
      uint32_t oa = smem_addr(offs) + 4u * h;
      int k = (cnt - h + H - 1) / H;          // entries of this lane
      for (; k >= 4; k -= 4, oa += 16u * H) {
        uint32_t x[4];
        TV v[4];
        x[0] = lds32<0>(oa);
        x[1] = lds32<4 * H>(oa);
        x[2] = lds32<8 * H>(oa);
        x[3] = lds32<12 * H>(oa);
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = lds16(ea + 2u * x[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) lds_val(va, x[u] & 0x7FFFu, v[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) tile_add(x[u], v[u], s, e);
      }
      if (k > 0) {
        uint32_t x[3];
        TV v[3];
#pragma unroll
        for (int u = 0; u < 3; ++u) x[u] = lds32<0>(u < k ? oa + 4u * H * u : oa);
#pragma unroll
        for (int u = 0; u < 3; ++u) x[u] = lds16(ea + 2u * x[u]);
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          lds_val(va, x[u] & 0x7FFFu, v[u]);
          if (u >= k) zero_val(v[u]);
        }
#pragma unroll
        for (int u = 0; u < 3; ++u) tile_add(x[u], v[u], s, e);
      }
    }
#pragma unroll
    for (int o = 1; o < H; o <<= 1) {
      const float s2 = __shfl_xor_sync(0xffffffffu, s, o);
      const float e2 = __shfl_xor_sync(0xffffffffu, e, o);
      float ss, er;
      two_sum(s, s2, ss, er);
      s = ss;
      e = e + e2 + er;
    }
    if (h == 0 && cnt > 0) {
      const float2 a = acc[b];
      float as = a.x, ae = a.y;
      df_add(s, e, as, ae);
      acc[b] = df_norm(as, ae);
    }
  }
}
template <class TV>
__device__ __forceinline__ void tile_gather(int d, int H, const TV* vals, const int* offs, const uint32_t* ms,
                                            const uint16_t* es, float2* acc) {
  switch (H) {
    case 1: tile_gather_h<1>(d, vals, offs, ms, es, acc); return;
    case 2: tile_gather_h<2>(d, vals, offs, ms, es, acc); return;
    case 4: tile_gather_h<4>(d, vals, offs, ms, es, acc); return;
    default: tile_gather_h<8>(d, vals, offs, ms, es, acc); return;
  }
}

// Shared memory of a tile kernel: DF accumulators (d), two value buffers,
// the update's coefficients (c), then two buffers each of the tile's entries,
// positions and slot offsets.
struct TileSmem {
  size_t acc, vb, rsh, es, ms, offs, total;
};

__host__ __device__ inline TileSmem tile_smem_layout(int d, int L, int c, int zeta) {
  TileSmem s;
  size_t o = 0;
  s.acc = o; o += (size_t)d * sizeof(float2);
  s.vb = o; o += (size_t)2 * kTileRows * sizeof(float2);
  s.rsh = o; o += (size_t)c * sizeof(float2);
  o = (o + 15) & ~(size_t)15;
  s.es = o; o += (size_t)2 * kTileRows * zeta * sizeof(uint16_t);
  s.ms = o; o += (size_t)2 * d * sizeof(uint32_t);
  s.offs = o; o += (size_t)2 * (L + 1) * sizeof(int);
  s.total = o;
  return s;
}

__host__ __device__ inline size_t tile_smem_bytes(int d, int L, int c, int zeta) {
  return tile_smem_layout(d, L, c, zeta).total;
}

// Stage tile t's slot offsets, positions and entries (coalesced copies; the
// entries with 16-byte loads when aligned).
__device__ __forceinline__ void tile_stage(const SketchTiles& tv, int64_t t, int64_t r0, int rows, int* of,
                                           uint32_t* ms, uint16_t* es) {
  const int L1 = tv.L + 1, d = tv.d;
  for (int q = threadIdx.x; q < L1; q += blockDim.x) of[q] = tv.off[t * L1 + q];
  const uint32_t* mg = tv.meta + t * d;
  for (int q = threadIdx.x; q < d; q += blockDim.x) ms[q] = __ldg(mg + q);
  const uint16_t* src = tv.ent + r0 * tv.zeta;
  const int cnt = rows * tv.zeta;
  int q0 = 0;
  if (((r0 * tv.zeta) & 7) == 0) {
    const int nv = cnt >> 3;
    for (int q = threadIdx.x; q < nv; q += blockDim.x)
      reinterpret_cast<uint4*>(es)[q] = __ldg(reinterpret_cast<const uint4*>(src) + q);
    q0 = nv << 3;
  }
  for (int q = q0 + threadIdx.x; q < cnt; q += blockDim.x) es[q] = src[q];
}

// The CTA's tiles: their rows are consecutive and all but the last tile have
// kTileRows of them, so no tile has to read its bounds first.  rev: taken last
// to first.
struct TileRange {
  int t0, nt;
  bool rev;
  int64_t ra;
  int len;                                        // rows of the CTA
  __device__ __forceinline__ TileRange(const SketchTiles& tv, bool rev_) : rev(rev_) {
    t0 = tv.ctile[blockIdx.x];
    const int t1 = tv.ctile[blockIdx.x + 1];
    nt = t1 - t0;
    ra = tv.row[t0];
    len = (int)(tv.row[t1] - ra);
  }
  __device__ __forceinline__ int at(int k) const { return rev ? nt - 1 - k : k; }   // tile of step k, from t0
  __device__ __forceinline__ int64_t row(int k) const { return ra + at(k) * kTileRows; }
  __device__ __forceinline__ int rows(int k) const { return min(kTileRows, len - at(k) * kTileRows); }
};

// The shared buffers of step k (two sets, taken in turn).
template <class TV>
struct TileBuf {
  TV* v;
  int* of;
  uint32_t* ms;
  uint16_t* es;
  __device__ __forceinline__ TileBuf(uint8_t* sm, const TileSmem& lay, const SketchTiles& tv, int k) {
    const int buf = k & 1;
    v = reinterpret_cast<TV*>(reinterpret_cast<float2*>(sm + lay.vb) + buf * kTileRows);
    of = reinterpret_cast<int*>(sm + lay.offs) + buf * (tv.L + 1);
    ms = reinterpret_cast<uint32_t*>(sm + lay.ms) + buf * tv.d;
    es = reinterpret_cast<uint16_t*>(sm + lay.es) + (size_t)buf * kTileRows * tv.zeta;
  }
};

__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src));
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src));
}

constexpr int kFetchThreads = 128;
// Starts the copy of the bin lists of step k's tile into its buffers, by the
// CTA's last warps (for most d they have no sketch row of their own in the
// gather), and ends with tile_wait; the bytes are those of tile_stage.  Issued a tile
// ahead: staged at the tile's start instead, the bounds' load, then those of
// the lists, were waited for one after the other (FP32 update, n = 4.1e6,
// d = 96, one basis column: 84 -> 64 us; 26 columns: 150 -> 134 us; pairs,
// n = 1e6, d = 320, one column: 30 -> 23 us).
template <class TV>
__device__ __forceinline__ void tile_fetch(uint8_t* sm, const TileSmem& lay, const SketchTiles& tv,
                                           const TileRange& tr, int k) {
  const int f = (int)threadIdx.x - ((int)blockDim.x - kFetchThreads);
  if (f < 0) return;
  const TileBuf<TV> b(sm, lay, tv, k);
  const int L1 = tv.L + 1, d = tv.d;
  const int64_t t = tr.t0 + tr.at(k), e0 = tr.row(k) * tv.zeta;
  const int cnt = tr.rows(k) * tv.zeta;
  const int* og = tv.off + t * L1;
  const uint32_t* mg = tv.meta + t * d;
  const uint16_t* eg = tv.ent + e0;
  int q0;
  if ((e0 & 7) == 0) {
#pragma unroll 4
    for (int q = f; q < cnt >> 3; q += kFetchThreads) cp_async16(b.es + 8 * q, eg + 8 * q);
    q0 = cnt & ~7;
  } else {                       // tiles start at even rows: 4-byte aligned
    for (int q = f; q < cnt >> 1; q += kFetchThreads) cp_async4(b.es + 2 * q, eg + 2 * q);
    q0 = cnt & ~1;
  }
  if ((d & 3) == 0) {
    for (int q = f; q < d >> 2; q += kFetchThreads) cp_async16(b.ms + 4 * q, mg + 4 * q);
  } else {
    for (int q = f; q < d; q += kFetchThreads) cp_async4(b.ms + q, mg + q);
  }
  for (int q = f; q < L1; q += kFetchThreads) cp_async4(b.of + q, og + q);
  for (int q = q0 + f; q < cnt; q += kFetchThreads) b.es[q] = eg[q];
}
__device__ __forceinline__ void tile_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The end of step k: every value of the tile is in its buffer.  Starts the
// next tile's lists (their buffers were last read before this barrier) and
// adds this tile's sums.
template <class TV>
__device__ __forceinline__ void tile_finish(uint8_t* sm, const TileSmem& lay, const SketchTiles& tv,
                                            const TileRange& tr, int k, float2* acc) {
  tile_wait();
  __syncthreads();
  if (k + 1 < tr.nt) tile_fetch<TV>(sm, lay, tv, tr, k + 1);
  const TileBuf<TV> b(sm, lay, tv, k);
  tile_gather(tv.d, tv.H, b.v, b.of, b.ms, b.es, acc);
}

// Asks for p[0 .. cnt) to be brought into L2 (16-byte units; p[cnt] up to the
// next unit is inside the padded column).
template <class TU>
__device__ __forceinline__ void prefetch_rows(const TU* p, int cnt) {
  const uint64_t a = reinterpret_cast<uint64_t>(p) & ~(uint64_t)15;
  const uint64_t e = (reinterpret_cast<uint64_t>(p + cnt) + 15) & ~(uint64_t)15;
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"((uint32_t)(e - a)));
}

__device__ __forceinline__ void tile_write_part(const float2* acc, int d, double* part) {
  __syncthreads();
  for (int r = threadIdx.x; r < d; r += blockDim.x) part[(size_t)blockIdx.x * d + r] = df_to_double(acc[r]);
}

// w'[i] = sum_p A_p x[col_p] (DF) over the CTA's tiles; part[cta] = the
// CTA's Omega-sums of w' as stored.  512 threads; thread l takes the tile
// rows l and l + 512 together, four entries of each per round, so that the
// loads of both rows are in flight at once (the products of a row are still
// accumulated in entry order).
// SK = false: the plain SpMV (Krylov-Schur with Euclidean CGS2), no sketch.
// Two CTAs per SM as in k_df_spmv_ell (99 registers otherwise; rows of 1 to 13
// entries, n = 7e5, d = 320, pairs: 43.2 us a launch, 35.4 us with two).
template <class TA, class TU, bool SK>
__global__ void __launch_bounds__(512, 2) k_df_spmv_sketch(
    const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colind, const TA* __restrict__ vals,
    const TU* __restrict__ x, TU* __restrict__ w, const SketchTiles tv, double* __restrict__ part) {
  static_assert(kTileRows == 1024, "two rows per thread of a 512-thread CTA");
  extern __shared__ __align__(16) uint8_t smraw[];
  const int d = tv.d;
  const TileSmem lay = tile_smem_layout(d, tv.L, 0, tv.zeta);
  float2* acc = reinterpret_cast<float2*>(smraw + lay.acc);
  if (SK)
    for (int r = threadIdx.x; r < d; r += blockDim.x) acc[r] = make_float2(0.f, 0.f);
  const TileRange tr(tv, false);
  if (SK && tr.nt > 0) tile_fetch<TU>(smraw, lay, tv, tr, 0);
  pdl_next();
  pdl_wait();
  x = pdl_fresh(x);
  for (int k = 0; k < tr.nt; ++k) {
    TU* v = TileBuf<TU>(smraw, lay, tv, k).v;
    const int64_t r0 = tr.row(k);
    const int rows = tr.rows(k);
    const int la = threadIdx.x, lb = threadIdx.x + 512;
    int pa = 0, ea = 0, pb = 0, eb = 0;
    if (la < rows) { pa = rowptr[r0 + la]; ea = rowptr[r0 + la + 1]; }
    if (lb < rows) { pb = rowptr[r0 + lb]; eb = rowptr[r0 + lb + 1]; }
    float sa = 0.f, ta = 0.f, sb = 0.f, tb = 0.f;
    const int len = max(ea - pa, eb - pb);
    for (int q = 0; q < len; q += 4) {
      int ca[4], cb[4];
      float2 va[4], vbv[4], xa[4], xb[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int p = pa + q + u, p2 = pb + q + u;
        ca[u] = p < ea ? colind[p] : -1;
        cb[u] = p2 < eb ? colind[p2] : -1;
        va[u] = p < ea ? ldv(vals + p) : make_float2(0.f, 0.f);
        vbv[u] = p2 < eb ? ldv(vals + p2) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        xa[u] = ca[u] >= 0 ? ldv(x + ca[u]) : make_float2(0.f, 0.f);
        xb[u] = cb[u] >= 0 ? ldv(x + cb[u]) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (ca[u] >= 0) mac_st<TA, TU>(va[u], xa[u], sa, ta);
        if (cb[u] >= 0) mac_st<TA, TU>(vbv[u], xb[u], sb, tb);
      }
    }
    if (la < rows) tile_put(v + la, stv(w + r0 + la, df_norm(sa, ta)));
    if (lb < rows) tile_put(v + lb, stv(w + r0 + lb, df_norm(sb, tb)));
    if (SK) tile_finish<TU>(smraw, lay, tv, tr, k, acc);
  }
  if (SK) tile_write_part(acc, d, part);
}

// The SpMV+sketch of k_df_spmv_sketch on the ELLPACK copy of A (CsrDF): a
// thread's entries sit at fixed offsets from its row index, so the loads of a
// round need no row pointer first and each is one contiguous segment per warp.
// Entries are taken in CSR order and padding (column -1) is skipped, so the
// products and sums are those of the CSR kernel, bit for bit.
// WC > 0: rows of at most WC entries, all of a row's loads in one round
// (5-point stencils: W = 5 fits WC = 6 without spilling at two CTAs per SM).
// Two CTAs per SM (the grid is two per SM) must be asked for: with the gather's
// four forms inlined the kernel takes 102 registers otherwise, one CTA per SM
// (W = 12, n = 5e5, d = 320, pairs: 44.1 us a launch, 36.8 us with two).
template <class TA, class TU, bool SK, int WC>
__global__ void __launch_bounds__(512, 2) k_df_spmv_ell(
    const int32_t* __restrict__ ecol, const TA* __restrict__ evals, int W,
    const TU* __restrict__ x, TU* __restrict__ w, const SketchTiles tv, double* __restrict__ part) {
  static_assert(kTileRows == 1024, "two rows per thread of a 512-thread CTA");
  extern __shared__ __align__(16) uint8_t smraw[];
  const int d = tv.d;
  const TileSmem lay = tile_smem_layout(d, tv.L, 0, tv.zeta);
  float2* acc = reinterpret_cast<float2*>(smraw + lay.acc);
  if (SK)
    for (int r = threadIdx.x; r < d; r += blockDim.x) acc[r] = make_float2(0.f, 0.f);
  const TileRange tr(tv, false);
  if (SK && tr.nt > 0) tile_fetch<TU>(smraw, lay, tv, tr, 0);
  pdl_next();
  pdl_wait();
  x = pdl_fresh(x);
  for (int k = 0; k < tr.nt; ++k) {
    TU* v = TileBuf<TU>(smraw, lay, tv, k).v;
    const int64_t r0 = tr.row(k);
    const int rows = tr.rows(k);
    const int la = threadIdx.x, lb = threadIdx.x + 512;
    const bool oka = la < rows, okb = lb < rows;
    const int64_t ia = r0 + la, ib = r0 + lb;
    const int64_t ba = (((ia >> 5) * W) << 5) + (ia & 31), bb = (((ib >> 5) * W) << 5) + (ib & 31);
    float sa = 0.f, ta = 0.f, sb = 0.f, tb = 0.f;
    if (WC > 0) {                                 // one round: every column and value, then x
      constexpr int R1 = WC > 0 ? WC : 1;
      int ca[R1], cb[R1];
      float2 va[R1], vbv[R1];
#pragma unroll
      for (int e = 0; e < R1; ++e) {
        const int64_t oa = ba + ((int64_t)e << 5), ob = bb + ((int64_t)e << 5);
        ca[e] = (oka && e < W) ? ecol[oa] : -1;
        cb[e] = (okb && e < W) ? ecol[ob] : -1;
        va[e] = (oka && e < W) ? ldv(evals + oa) : make_float2(0.f, 0.f);
        vbv[e] = (okb && e < W) ? ldv(evals + ob) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int e = 0; e < R1; ++e) {
        const float2 xa = ca[e] >= 0 ? ldv(x + ca[e]) : make_float2(0.f, 0.f);
        const float2 xb = cb[e] >= 0 ? ldv(x + cb[e]) : make_float2(0.f, 0.f);
        if (ca[e] >= 0) mac_st<TA, TU>(va[e], xa, sa, ta);
        if (cb[e] >= 0) mac_st<TA, TU>(vbv[e], xb, sb, tb);
      }
    }
    constexpr int RU = 4;                         // rounds of four entries
    for (int q = 0; WC == 0 && q < W; q += RU) {
      int ca[RU], cb[RU];
      float2 va[RU], vbv[RU], xa[RU], xb[RU];
#pragma unroll
      for (int u = 0; u < RU; ++u) {
        const int e = q + u;
        const int64_t oa = ba + ((int64_t)e << 5), ob = bb + ((int64_t)e << 5);
        ca[u] = (oka && e < W) ? ecol[oa] : -1;
        cb[u] = (okb && e < W) ? ecol[ob] : -1;
        va[u] = (oka && e < W) ? ldv(evals + oa) : make_float2(0.f, 0.f);
        vbv[u] = (okb && e < W) ? ldv(evals + ob) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < RU; ++u) {
        xa[u] = ca[u] >= 0 ? ldv(x + ca[u]) : make_float2(0.f, 0.f);
        xb[u] = cb[u] >= 0 ? ldv(x + cb[u]) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < RU; ++u) {
        if (ca[u] >= 0) mac_st<TA, TU>(va[u], xa[u], sa, ta);
        if (cb[u] >= 0) mac_st<TA, TU>(vbv[u], xb[u], sb, tb);
      }
    }
    if (oka) tile_put(v + la, stv(w + ia, df_norm(sa, ta)));
    if (okb) tile_put(v + lb, stv(w + ib, df_norm(sb, tb)));
    if (SK) tile_finish<TU>(smraw, lay, tv, tr, k, acc);
  }
  if (SK) tile_write_part(acc, d, part);
}

// w = A x (+ partial sketches) with one warp per row inside each sketch tile
// (rows of many entries): lanes take the row's entries with a stride of 32,
// then a fixed xor tree adds the lanes' double-float sums.  The bound of two
// CTAs per SM leaves registers for the row loop's loads (40 otherwise, a third
// CTA's room): rows of 27, n = 1e6: 156 us a launch, 123 us with the bound;
// rows of 41 at random columns, n = 5e5, 80 columns: the first restart
// 21.2 -> 16.5 ms.
template <class TA, class TU, bool SK, int LPR>
__global__ void __launch_bounds__(512, 2) k_df_spmv_warp(const int32_t* __restrict__ rowptr,
                                                         const int32_t* __restrict__ colind,
                                                         const TA* __restrict__ vals, const TU* __restrict__ x,
                                                         TU* __restrict__ w, const SketchTiles tv,
                                                         double* __restrict__ part) {
  extern __shared__ __align__(16) uint8_t smraw[];
  const int d = tv.d;
  const TileSmem lay = tile_smem_layout(d, tv.L, 0, tv.zeta);
  float2* acc = reinterpret_cast<float2*>(smraw + lay.acc);
  if (SK)
    for (int r = threadIdx.x; r < d; r += blockDim.x) acc[r] = make_float2(0.f, 0.f);
  // groups of LPR lanes per row (LPR = 32: a warp per row)
  const int grp = threadIdx.x / LPR, lane = threadIdx.x % LPR, ngrp = blockDim.x / LPR;
  const TileRange tr(tv, false);
  if (SK && tr.nt > 0) tile_fetch<TU>(smraw, lay, tv, tr, 0);
  pdl_next();
  pdl_wait();
  x = pdl_fresh(x);
  for (int k = 0; k < tr.nt; ++k) {
    TU* v = TileBuf<TU>(smraw, lay, tv, k).v;
    const int64_t r0 = tr.row(k);
    const int rows = tr.rows(k);
    const int nit = (rows + ngrp - 1) / ngrp;        // the same trip count for every lane
    for (int it = 0; it < nit; ++it) {
      const int l = it * ngrp + grp;
      float sh = 0.f, sl = 0.f;
      if (l < rows) {
        const int p0 = rowptr[r0 + l], p1 = rowptr[r0 + l + 1];
        for (int p = p0 + lane; p < p1; p += LPR) {
          const float2 a = ldv(vals + p), xv = ldv(x + colind[p]);
          mac_st<TA, TU>(a, xv, sh, sl);
        }
      }
#pragma unroll
      for (int o = LPR / 2; o; o >>= 1) {              // fixed xor tree inside the group
        const float s2 = __shfl_xor_sync(0xffffffffu, sh, o);
        const float t2 = __shfl_xor_sync(0xffffffffu, sl, o);
        float ss, e;
        two_sum(sh, s2, ss, e);
        sh = ss;
        sl = sl + t2 + e;
      }
      if (l < rows && lane == 0) tile_put(v + l, stv(w + r0 + l, df_norm(sh, sl)));
    }
    if (SK) tile_finish<TU>(smraw, lay, tv, tr, k, acc);
  }
  if (SK) tile_write_part(acc, d, part);
}

// Merge-path split: the number of rows i whose end marker lies before merge
// position dd (marker of row i at rowptr[i + 1] + i); dd - i entries precede.
__device__ __forceinline__ int64_t merge_split(int64_t dd, int64_t n, int64_t nnz, const int32_t* __restrict__ rowptr) {
  int64_t lo = dd > nnz ? dd - nnz : 0, hi = dd < n ? dd : n;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if ((int64_t)rowptr[mid + 1] + mid < dd) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

constexpr int kMergeBlk = kMergeCta * kMergeItems;   // merge items per CTA

// part_row[b] = rows whose end precedes merge position b * kMergeBlk, b <= nb
__global__ void k_merge_partition(int64_t n, int64_t nnz, const int32_t* __restrict__ rowptr, int64_t nb,
                                  int64_t* __restrict__ part_row) {
  const int64_t total = n + nnz;
  for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b <= nb; b += (int64_t)gridDim.x * blockDim.x) {
    const int64_t dd = b * kMergeBlk < total ? b * kMergeBlk : total;
    part_row[b] = merge_split(dd, n, nnz, rowptr);
  }
}

// w' = A x by merge path.  CTA b owns merge positions [b B, (b + 1) B)
// (B = kMergeBlk rows + entries): first its entries' double-float products
// a_p x[col_p] (coalesced, many loads in flight) and its rows' end offsets go
// to shared memory, then thread t walks positions [t K, (t + 1) K) of them
// (K = kMergeItems): a row ending in its range is written to wd (partial when
// it began before), the row still open at its end goes to (mp_row, mp_val).
// The products and their order within a row are those of the CSR kernel.
template <class TA>
__global__ void __launch_bounds__(kMergeCta) k_df_spmv_merge(
    int64_t n, int64_t nnz, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colind,
    const TA* __restrict__ vals, const float2* __restrict__ x2, const float* __restrict__ x1,
    const int64_t* __restrict__ part_row, float2* __restrict__ wd, int* __restrict__ mp_row,
    float2* __restrict__ mp_val, int64_t nthreads) {
  __shared__ float2 prod[kMergeBlk];
  __shared__ int32_t rend[kMergeBlk + 1];
  __shared__ int crow[kMergeCta];       // row open at the end of each thread's range (-1: none)
  __shared__ float2 cval[kMergeCta];    // its partial sum
  __shared__ float2 fval[kMergeCta];    // partial sum of the first row the thread completes
  __shared__ int fhas[kMergeCta];       // whether the thread completes a row
  const int64_t total = n + nnz;
  const int64_t b = blockIdx.x;
  const int64_t rlo = part_row[b], rhi = part_row[b + 1];
  const int64_t dlo = b * kMergeBlk, dhi = dlo + kMergeBlk < total ? dlo + kMergeBlk : total;
  const int64_t jlo = dlo - rlo, jhi = dhi - rhi;     // entries of the CTA's range
  const int ne = (int)(jhi - jlo), nr = (int)(rhi - rlo);
  // products a_p x[col_p], eight entries per thread in flight at a time
  for (int e0 = threadIdx.x; e0 < ne; e0 += 8 * kMergeCta) {
    int c[8];
    float2 a[8], xv[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int e = e0 + u * kMergeCta;
      c[u] = e < ne ? colind[jlo + e] : 0;
      a[u] = e < ne ? ldv(vals + jlo + e) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) xv[u] = x2 ? x2[c[u]] : make_float2(x1[c[u]], 0.f);   // c = 0 past the end
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int e = e0 + u * kMergeCta;
      if (e < ne) {
        const float pr = a[u].x * xv[u].x;
        float er = fmaf(a[u].x, xv[u].x, -pr);
        er = fmaf(a[u].x, xv[u].y, er);
        er = fmaf(a[u].y, xv[u].x, er);
        prod[e] = make_float2(pr, er);
      }
    }
  }
  for (int r = threadIdx.x; r <= nr; r += kMergeCta) rend[r] = rowptr[rlo + r + 1 <= n ? rlo + r + 1 : n];
  crow[threadIdx.x] = -1;
  cval[threadIdx.x] = make_float2(0.f, 0.f);
  fval[threadIdx.x] = make_float2(0.f, 0.f);
  fhas[threadIdx.x] = 0;
  __syncthreads();
  const int64_t t = b * kMergeCta + threadIdx.x;
  const int64_t d0 = t * kMergeItems;
  const int64_t d1 = d0 + kMergeItems < total ? d0 + kMergeItems : total;
  if (t < nthreads && d0 < total) {
    // split inside the CTA's rows: marker of row rlo + q at rend[q] + rlo + q
    auto split = [&](int64_t dd) {
      int lo = 0, hi = nr;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if ((int64_t)rend[mid] + rlo + mid < dd) lo = mid + 1;
        else hi = mid;
      }
      return lo;
    };
    int q = split(d0);
    const int qe = split(d1);
    int64_t j = d0 - (rlo + q);
    const int64_t je = d1 - (rlo + qe);
    float sh = 0.f, sl = 0.f;
    bool first = true;
    for (; q < qe; ++q) {
      const int64_t pe = rend[q];
      for (; j < pe; ++j) {
        const float2 v = prod[j - jlo];
        df_add(v.x, v.y, sh, sl);
      }
      // the first row this thread completes is the one it started in, which
      // may have begun in earlier ranges: its sum is finished by the fold
      if (first) {
        fval[threadIdx.x] = df_norm(sh, sl);
        fhas[threadIdx.x] = 1;
        first = false;
      } else {
        wd[rlo + q] = df_norm(sh, sl);
      }
      sh = 0.f;
      sl = 0.f;
    }
    for (; j < je; ++j) {
      const float2 v = prod[j - jlo];
      df_add(v.x, v.y, sh, sl);
    }
    crow[threadIdx.x] = rlo + qe < n ? (int)(rlo + qe) : -1;
    cval[threadIdx.x] = df_norm(sh, sl);
  }
  __syncthreads();
  // Fold in thread order, by warp 0: lane L folds the records of threads
  // 8L .. 8L+7 (the partial sums of the row it enters with, up to and with
  // its first completion, and the rows it completes after that, written
  // here), then lane 0 chains the 32 lanes: the running row collects each
  // lane's leading partial and is written at the lane's first completion.
  // The row open at the CTA's end becomes the CTA's carry (mp_row[b],
  // mp_val[b]; -1: none), added by k_df_merge_fix.  A fixed order: the sums
  // are the same bits on every run.
  if (threadIdx.x < 32) {
    constexpr int kSeg = kMergeCta / 32;
    const int lane = threadIdx.x;
    float ph = 0.f, pl = 0.f;          // contribution to the row the lane enters with
    float oh = 0.f, ol = 0.f;          // partial of the row open at the lane's end (after a completion)
    int has = 0, orow = -1;
    for (int q = 0; q < kSeg; ++q) {
      const int u = lane * kSeg + q;
      if (fhas[u]) {
        const float2 f = fval[u];
        if (!has) {
          df_add(f.x, f.y, ph, pl);
          has = 1;
        } else {
          df_add(f.x, f.y, oh, ol);
          if (orow >= 0) wd[orow] = df_norm(oh, ol);
        }
        orow = crow[u];
        const float2 v = cval[u];
        oh = 0.f;
        ol = 0.f;
        df_add(v.x, v.y, oh, ol);
      } else if (crow[u] >= 0) {
        const float2 v = cval[u];
        if (has) df_add(v.x, v.y, oh, ol);
        else df_add(v.x, v.y, ph, pl);
      }
    }
    const float2 pre = df_norm(ph, pl), post = df_norm(oh, ol);
    __shared__ float2 s_pre[32], s_post[32];
    __shared__ int s_has[32], s_orow[32];
    s_pre[lane] = pre;
    s_post[lane] = post;
    s_has[lane] = has;
    s_orow[lane] = orow;
    __syncwarp();
    if (lane == 0) {
      int rc = (int)rlo;
      float ch = 0.f, cl = 0.f;
      for (int L = 0; L < 32; ++L) {
        const float2 v = s_pre[L];
        df_add(v.x, v.y, ch, cl);
        if (s_has[L]) {
          if (rc >= 0) wd[rc] = df_norm(ch, cl);
          rc = s_orow[L];
          const float2 w2 = s_post[L];
          ch = 0.f;
          cl = 0.f;
          df_add(w2.x, w2.y, ch, cl);
        }
      }
      mp_row[b] = rc >= 0 && rc < n ? rc : -1;
      mp_val[b] = df_norm(ch, cl);
    }
  }
}

// Fold of the merge-path carries of the CTAs: the first CTA of each run of
// equal carry rows adds the run's partial sums, in CTA order, to that row.
__global__ void k_df_merge_fix(const int* __restrict__ mp_row, const float2* __restrict__ mp_val, int64_t nthreads,
                               float2* __restrict__ wd) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nthreads;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int r = mp_row[t];
    if (r < 0 || (t > 0 && mp_row[t - 1] == r)) continue;
    float sh = 0.f, sl = 0.f;
    for (int64_t u = t; u < nthreads && mp_row[u] == r; ++u) df_add(mp_val[u].x, mp_val[u].y, sh, sl);
    const float2 cur = wd[r];
    df_add(cur.x, cur.y, sh, sl);
    wd[r] = df_norm(sh, sl);
  }
}

// FP32 copy of a double-float vector (the stored basis vector of the FP32 phase)
__global__ void k_df_round_f32(int64_t n, const float2* __restrict__ a, float* __restrict__ b) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    b[i] = a[i].x + a[i].y;
}

// Offsets of the diagonal copy, passed by value.
struct DiaOffs {
  int o[16];
  int lo = 0, hi = 0;   // smallest and largest offset (the SpMV's interior-tile test)
};

// w = A x (+ the per-CTA partial sketches of w when SK) on the diagonal copy
// of A: every load independent of the others and coalesced (value of
// diagonal e at row i, x at i + off_e), the products in increasing column
// order (the CSR kernel's order, the same bits); two rows per thread, the
// tiles and the sketch gather of k_df_spmv_ell.
// ND > 0: exactly ND diagonals, so that an interior tile's loads need neither
// a test nor a zero (rows past a ragged tile's end are read, not stored): pairs,
// 5 diagonals, n = 1e6, d = 320: 29.4 -> 24.2 us; FP32, 7 diagonals,
// n = 4.1e6, d = 96: 73 -> 71 us (64 us with the gather's last form).
template <class TU, class TA, bool SK, int DMAX, int ND = 0>
__global__ void __launch_bounds__(512, 2) k_df_spmv_dia(const DiaOffs offs, int D, const TA* __restrict__ dv,
                                                     int64_t ldd, int64_t n, const TU* __restrict__ x,
                                                     TU* __restrict__ w, const SketchTiles tv,
                                                     double* __restrict__ part) {
  static_assert(kTileRows == 1024, "two rows per thread of a 512-thread CTA");
  extern __shared__ __align__(16) uint8_t smraw[];
  const int d = tv.d;
  const TileSmem lay = tile_smem_layout(d, tv.L, 0, tv.zeta);
  float2* acc = reinterpret_cast<float2*>(smraw + lay.acc);
  if (SK)
    for (int r = threadIdx.x; r < d; r += blockDim.x) acc[r] = make_float2(0.f, 0.f);
  const TileRange tr(tv, false);
  if (SK && tr.nt > 0) tile_fetch<TU>(smraw, lay, tv, tr, 0);
  pdl_next();
  pdl_wait();
  x = pdl_fresh(x);
  for (int k = 0; k < tr.nt; ++k) {
    TU* v = TileBuf<TU>(smraw, lay, tv, k).v;
    const int64_t r0 = tr.row(k);
    const int rows = tr.rows(k);
    const int la = threadIdx.x, lb = threadIdx.x + 512;
    const bool oka = la < rows, okb = lb < rows;
    const int64_t ia = r0 + la, ib = r0 + lb;
    // rounds of four diagonals (eight for FP32 vectors and values): the loads
    // of a round are all in flight at once, and the registers stay within
    // two CTAs per SM
    constexpr int RU = sizeof(TU) == 4 && sizeof(TA) == 4 && DMAX == 8 ? 8 : 4;
    float sa = 0.f, ta = 0.f, sb = 0.f, tb = 0.f;
    // an interior tile (every x[i + off] of its rows inside 0 .. n-1, the
    // usual case) needs no bounds test: 32-bit offsets from the row pointers
    // (FP32 values or an exact number of diagonals; the other kernels keep one
    // path within their registers)
    const bool interior = (ND > 0 || (DMAX == 8 && sizeof(TA) == 4)) && r0 + offs.lo >= 0 &&
                          r0 + kTileRows + (offs.hi > 0 ? offs.hi : 0) <= n;
    if (interior) {
      const TA* pv = dv + ia;
      const TU* xpa = x + ia;
      constexpr int DE = ND > 0 ? ND : DMAX;
#pragma unroll
      for (int e0 = 0; e0 < DE; e0 += RU) {
        float2 va[RU], vb[RU], xa[RU], xb[RU];
#pragma unroll
        for (int u = 0; u < RU; ++u) {
          const int e = e0 + u;
          if (e >= DE) continue;
          const bool on = ND > 0 || e < D, la_on = ND > 0 || (on && oka), lb_on = ND > 0 || (on && okb);
          const TU* px = xpa + offs.o[e];
          va[u] = la_on ? ldv(pv) : make_float2(0.f, 0.f);
          vb[u] = lb_on ? ldv(pv + 512) : make_float2(0.f, 0.f);
          xa[u] = la_on ? ldv(px) : make_float2(0.f, 0.f);
          xb[u] = lb_on ? ldv(px + 512) : make_float2(0.f, 0.f);
          pv += ldd;
        }
#pragma unroll
        for (int u = 0; u < RU; ++u) {
          if (e0 + u < DE && (ND > 0 || e0 + u < D)) {
            mac_st<TA, TU>(va[u], xa[u], sa, ta);
            mac_st<TA, TU>(vb[u], xb[u], sb, tb);
          }
        }
      }
    } else {
#pragma unroll
      for (int e0 = 0; e0 < DMAX; e0 += RU) {
        float2 va[RU], vb[RU], xa[RU], xb[RU];
#pragma unroll
        for (int u = 0; u < RU; ++u) {
          const int e = e0 + u;
          const bool on = e < D;
          const int64_t ja = ia + offs.o[e], jb = ib + offs.o[e];
          va[u] = (on && oka) ? ldv(dv + e * ldd + ia) : make_float2(0.f, 0.f);
          vb[u] = (on && okb) ? ldv(dv + e * ldd + ib) : make_float2(0.f, 0.f);
          xa[u] = (on && oka && ja >= 0 && ja < n) ? ldv(x + ja) : make_float2(0.f, 0.f);
          xb[u] = (on && okb && jb >= 0 && jb < n) ? ldv(x + jb) : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < RU; ++u) {
          if (e0 + u < D) {
            mac_st<TA, TU>(va[u], xa[u], sa, ta);
            mac_st<TA, TU>(vb[u], xb[u], sb, tb);
          }
        }
      }
    }
    if (oka) tile_put(v + la, stv(w + ia, df_norm(sa, ta)));
    if (okb) tile_put(v + lb, stv(w + ib, df_norm(sb, tb)));
    if (SK && k + 1 < tr.nt && (int)threadIdx.x < D)   // the next tile's diagonals on their way to L2
      prefetch_rows(dv + tr.row(k + 1) + threadIdx.x * ldd, tr.rows(k + 1));
    if (SK) tile_finish<TU>(smraw, lay, tv, tr, k, acc);
  }
  if (SK) tile_write_part(acc, d, part);
}

// Row i's entries into the diagonal copy (dv cleared before)
template <class TV>
__global__ void k_dia_fill(int64_t n, const DiaOffs offs, int D, int64_t ldd, const int32_t* __restrict__ rowptr,
                           const int32_t* __restrict__ colind, const TV* __restrict__ vals, TV* __restrict__ dv) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    for (int p = rowptr[i]; p < rowptr[i + 1]; ++p) {
      const int64_t off = (int64_t)colind[p] - i;
      for (int e = 0; e < D; ++e)
        if (offs.o[e] == off) { dv[e * ldd + i] = vals[p]; break; }
    }
  }
}

// ELLPACK slots of row i (and the padding rows of the last slice)
template <class TV>
__global__ void k_ell_fill(int64_t n, int W, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colind,
                           const TV* __restrict__ vals, int32_t* __restrict__ ecol, TV* __restrict__ evals) {
  const int64_t nrow = (n + 31) / 32 * 32;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nrow; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p0 = i < n ? rowptr[i] : 0;
    const int len = i < n ? (int)(rowptr[i + 1] - p0) : 0;
    const int64_t b = (((i >> 5) * W) << 5) + (i & 31);
    for (int e = 0; e < W; ++e) {
      const int64_t o = b + ((int64_t)e << 5);
      ecol[o] = e < len ? colind[p0 + e] : -1;
      evals[o] = e < len ? vals[p0 + e] : TV();
    }
  }
}

// Vector load of two consecutive rows (i even, ld even): float4 = two pairs,
// float2 = two FP32 values.
__device__ __forceinline__ void ld2(const float2* p, float2& a, float2& b) {
  float4 v = __ldcs(reinterpret_cast<const float4*>(p));
  a = make_float2(v.x, v.y);
  b = make_float2(v.z, v.w);
}
__device__ __forceinline__ void ld2(const float* p, float2& a, float2& b) {
  float2 v = __ldcs(reinterpret_cast<const float2*>(p));
  a = make_float2(v.x, 0.f);
  b = make_float2(v.y, 0.f);
}

// Bytes of the basis that a CTA of the update asks for ahead of the least
// squares in front of it (304 CTAs: 49 MB, 7 us of HBM, within L2 beside w').
// With the launches' overlap: first restart of the 1000 x 1000 problem 11.6 ->
// 11.2 ms, of a power-law matrix 3.42 -> 3.29 ms, 160^3 mixed 12.1 -> 11.8 ms.
constexpr int kPdlPrefetch = 160 * 1024;

// u~ = sj * w' + sum_{col < c} U[:, col] * nrs[col]  (nrs = -b .* scale, DF)
// written to U[:, c]; part[cta] = the CTA's Omega-sums of u~ as stored.
// A thread takes two consecutive rows (tile starts are even and ld is a
// multiple of 32, so the pair load stays aligned and inside the column).
// MODE 1: with the sketch; MODE 0: plain update (Euclidean CGS2); MODE 2:
// plain update, and part[cta] = the CTA's sum of squares of u~ as stored
// (FP64, fixed reduction order).
template <class TU, int UNR, int MINB, int MODE>
__global__ void __launch_bounds__(512, MINB) k_df_update_sketch(
    TU* __restrict__ U, int64_t ldu, int c, const float2* __restrict__ nrs, const float2* __restrict__ sj,
    const SketchTiles tv, double* __restrict__ part) {
  constexpr bool SK = MODE == 1;
  extern __shared__ __align__(16) uint8_t smraw[];
  const int d = tv.d;
  const TileSmem lay = tile_smem_layout(d, tv.L, c, tv.zeta);
  float2* acc = reinterpret_cast<float2*>(smraw + lay.acc);
  float2* rsh = reinterpret_cast<float2*>(smraw + lay.rsh);
  if (SK)
    for (int r = threadIdx.x; r < d; r += blockDim.x) acc[r] = make_float2(0.f, 0.f);
  double ss = 0.0;
  // The second half of the grid takes its tiles last to first: the two CTAs
  // an SM holds (blocks b and b + G/2) then meet their short last tile at
  // different times, and the SM keeps more loads in flight.
  const TileRange tr(tv, blockIdx.x >= gridDim.x / 2);
  if (SK && tr.nt > 0) tile_fetch<TU>(smraw, lay, tv, tr, 0);
  // the first columns of the CTA's first tiles on their way to L2 while the
  // least squares in front of this kernel is still running
  pdl_next();
  if (SK && c > 0) {
    const int k = threadIdx.x / c, col = threadIdx.x - k * c;
    if (k < tr.nt && (int)threadIdx.x < kPdlPrefetch / (int)(kTileRows * sizeof(TU)))
      prefetch_rows(U + tr.row(k) + (int64_t)col * ldu, tr.rows(k));
  }
  pdl_wait();
  nrs = pdl_fresh(nrs);
  sj = pdl_fresh(sj);
  for (int col = threadIdx.x; col < c; col += blockDim.x) rsh[col] = nrs[col];
  __syncthreads();
  const float2 sc = sj[0];
  for (int k = 0; k < tr.nt; ++k) {
    TU* v = TileBuf<TU>(smraw, lay, tv, k).v;
    const int64_t r0 = tr.row(k);
    const int rows = tr.rows(k);
    for (int l = 2 * threadIdx.x; l < rows; l += 2 * blockDim.x) {
      const int64_t i = r0 + l;
      float s0 = 0.f, t0a = 0.f, s1 = 0.f, t1a = 0.f;
      {
        float2 w0, w1;
        ld2(U + i + (int64_t)c * ldu, w0, w1);
        mac_st<TU, float2>(w0, sc, s0, t0a);
        mac_st<TU, float2>(w1, sc, s1, t1a);
      }
      const TU* up = U + i;
      int col = 0;
      for (; col + UNR <= c; col += UNR) {
        float2 a[UNR], bb[UNR];
#pragma unroll
        for (int q = 0; q < UNR; ++q) ld2(up + (int64_t)(col + q) * ldu, a[q], bb[q]);
#pragma unroll
        for (int q = 0; q < UNR; ++q) {
          const float2 r = rsh[col + q];
          mac_st<TU, float2>(a[q], r, s0, t0a);
          mac_st<TU, float2>(bb[q], r, s1, t1a);
        }
      }
      for (; col < c; ++col) {
        float2 a, bb;
        ld2(up + (int64_t)col * ldu, a, bb);
        const float2 r = rsh[col];
        mac_st<TU, float2>(a, r, s0, t0a);
        mac_st<TU, float2>(bb, r, s1, t1a);
      }
      const float2 v0 = stv(U + i + (int64_t)c * ldu, df_norm(s0, t0a));
      tile_put(v + l, v0);
      if (MODE == 2) { const double x = df_to_double(v0); ss = fma(x, x, ss); }
      if (l + 1 < rows) {
        const float2 v1 = stv(U + i + 1 + (int64_t)c * ldu, df_norm(s1, t1a));
        tile_put(v + l + 1, v1);
        if (MODE == 2) { const double x = df_to_double(v1); ss = fma(x, x, ss); }
      }
    }
    // the next tile's first batch of columns on its way to L2 while this
    // tile's sums are formed
    if (SK && k + 1 < tr.nt && (int)threadIdx.x <= min(c, UNR))
      prefetch_rows(U + tr.row(k + 1) + (int64_t)(threadIdx.x == 0 ? c : threadIdx.x - 1) * ldu, tr.rows(k + 1));
    if (SK) tile_finish<TU>(smraw, lay, tv, tr, k, acc);
  }
  if (SK) tile_write_part(acc, d, part);
  if (MODE == 2) {
    __shared__ double red[32];
    for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
      part[blockIdx.x] = s;
    }
  }
}

// Euclidean CGS2 (Krylov-Schur baseline): part[cta * c + l] = the CTA's
// partial of U[:, l]^T U[:, cv] for l < c (DF products, FP64 per CTA, fixed
// order).  Columns go in groups of 8 (U read once); U[:, cv] is re-read per
// group (from L2).
template <class TU>
__global__ void __launch_bounds__(512) k_df_dots(const TU* __restrict__ U, int64_t ldu, int c, int cv,
                                                 const SketchTiles tv, double* __restrict__ part) {
  __shared__ float2 red[16][8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int t0 = tv.ctile[blockIdx.x], t1 = tv.ctile[blockIdx.x + 1];
  const TU* vcol = U + (int64_t)cv * ldu;
  for (int g0 = 0; g0 < c; g0 += 8) {
    const int ng = min(8, c - g0);
    float s[8], e[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) { s[q] = 0.f; e[q] = 0.f; }
    for (int t = t0; t < t1; ++t) {
      const int64_t r0 = tv.row[t];
      const int rows = (int)(tv.row[t + 1] - r0);
      for (int l = 2 * threadIdx.x; l < rows; l += 2 * blockDim.x) {
        const int64_t i = r0 + l;
        float2 x0, x1;
        ld2(vcol + i, x0, x1);
        if (l + 1 >= rows) x1 = make_float2(0.f, 0.f);
        float2 a[8], b[8];
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (q < ng) ld2(U + i + (int64_t)(g0 + q) * ldu, a[q], b[q]);
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (q < ng) {
            df_mac(a[q].x, a[q].y, x0.x, x0.y, s[q], e[q]);
            df_mac(b[q].x, b[q].y, x1.x, x1.y, s[q], e[q]);
          }
      }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      df_warp_sum(s[q], e[q]);
      if (lane == 0) red[warp][q] = df_norm(s[q], e[q]);
    }
    __syncthreads();
    if (threadIdx.x < ng) {
      double v = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += df_to_double(red[w][threadIdx.x]);
      part[(size_t)blockIdx.x * c + g0 + threadIdx.x] = v;
    }
    __syncthreads();
  }
}

// Coefficients of one CGS2 pass from the folded dots g_l = u~_l^T v:
// pass 1 (v = w' = A u~_j): b_l = cs_l cs_j g_l, rprev = b, sj = cs_j;
// pass 2 (v = u~): b_l = cs_l g_l, rprev += b, sj = 1; nrs_l = -b_l cs_l.
// One CTA; the G partials of each l are added in CTA order.
__global__ void __launch_bounds__(256) k_ks_coef(int pass, int j, int c, int G, const double* __restrict__ part,
                                                 const double* __restrict__ colscale, double* __restrict__ rprev,
                                                 float2* __restrict__ nrs, float2* __restrict__ sj) {
  for (int l = threadIdx.x; l < c; l += blockDim.x) {
    double g = 0.0;
    for (int q = 0; q < G; ++q) g += part[(size_t)q * c + l];
    const double b = pass == 1 ? colscale[l] * colscale[j] * g : colscale[l] * g;
    rprev[l] = pass == 1 ? b : rprev[l] + b;
    nrs[l] = df_from_double(-b * colscale[l]);
  }
  if (threadIdx.x == 0) sj[0] = df_from_double(pass == 1 ? colscale[j] : 1.0);
}

// End of a CGS2 step j: beta = ||u~|| from the G sum-of-squares partials,
// colscale[j + 1] = 1/beta, coefficient column j = (rprev_0..j, beta); beta
// <= thr is a breakdown.  With j < 0 only the start vector's scale.
__global__ void k_ks_finish(int j, int G, const double* __restrict__ part, double thr,
                            double* __restrict__ colscale, const double* __restrict__ rprev, double* __restrict__ coef,
                            int ldcoef, int* flag) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double ss = 0.0;
  for (int q = 0; q < G; ++q) ss += part[q];
  const double beta = sqrt(ss);
  const bool finite = isfinite(beta);
  const bool brk = finite && !(beta > thr);
  colscale[j + 1] = (finite && !brk) ? 1.0 / beta : 0.0;
  if (j >= 0) {
    double* cc = coef + (size_t)j * ldcoef;
    for (int i = 0; i <= j; ++i) cc[i] = rprev[i];
    cc[j + 1] = beta;
  }
  if (!finite) atomicOr(flag, RKS_FLAG_NAN);
  else if (brk) atomicOr(flag, RKS_FLAG_BREAKDOWN);
}

// sum over g < G of part[g * d + r] by one warp: lane l adds g = l, l + 32,
// ... in order, then a fixed xor tree adds the 32 lane sums (every lane ends
// with the total).  The same order on every run.
__device__ __forceinline__ double fold_row(const double* __restrict__ part, int d, int G, int r, int lane) {
  double v = 0.0;
#pragma unroll 8
  for (int g = lane; g < G; g += 32) v += part[(size_t)g * d + r];
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// out = the CTA-ordered sum of the sketch kernels' partials (warp per row;
// blockIdx.y: several vectors, G x d partials and d sums each)
__global__ void __launch_bounds__(256) k_df_fold(const double* __restrict__ part, int d, int G,
                                                 double* __restrict__ out) {
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= d) return;
  const double v = fold_row(part + (size_t)blockIdx.y * G * d, d, G, r, lane);
  if (lane == 0) out[(size_t)blockIdx.y * d + r] = v;
}

// Least squares b = S^+ z of one Arnoldi step (Alg. 2, Thm 4.3: against the
// locked and active sketches together), CGS2 in the sketch written through the
// Gram matrix M = S^T S: r1 = S^T z, r = r1 + S^T (z - S r1) = 2 r1 - M r1
// (the same quantity; M is the identity up to rounding).  M is kept on the
// device: the host sets it after every restart, and finishing column j adds
// its row M[:, j] = S^T s_j.  Phases (8 warps per CTA):
//   A  finish column j if requested (beta_j = ||s~_j||, S[:, j] in FP64 and
//      DF, colscale[j] = 1/beta_j, coefficient column j-1, flags: every CTA
//      computes beta_j itself, CTA 0 writes); then per column (one warp)
//      r1 = S^T z and, when finishing, the new row of M;
//   B  per column (one warp) r = 2 r1 - M r1, rprev = r (FP64),
//      nrs = -r .* colscale (DF), sj = colscale[j].
// k_df_ls_coop runs the fold of the sketch partials, A and B in one
// cooperative launch (two grid barriers); k_df_ls1 (A) and k_df_ls_gram (B)
// are the separate-launch form.
// z = z_raw * zscale * colscale[j] (z_raw is the sketch of the unscaled w').

__device__ double block_sum_d(double v, double* red) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (warp == 0) {
    v = lane < nw ? red[lane] : 0.0;
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[32] = v;
  }
  __syncthreads();
  return red[32];
}

// The same sum, known to thread 0 only (one barrier fewer)
__device__ double block_sum_0(double v, double* red) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (warp == 0) {
    v = lane < nw ? red[lane] : 0.0;
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  }
  return v;
}

// Phase A for one column (one warp): r1[col] = S[:, col]^T z (if want_r1)
// and, when column j is being finished (sjd = its DF values), the Gram entries
// M[col, j] = M[j, col] = S[:, col]^T s_j.  Column j itself reads sjd.
__device__ __forceinline__ void ls_phase_a(int col, int j, int d, int finish, int want_r1, const float2* S2,
                                           const float2* zd, const float2* sjd, float2* r1, float2* M2, int ldm,
                                           int lane) {
  const float2* sc = (finish && col == j) ? sjd : S2 + (size_t)col * d;
  float s = 0.f, t = 0.f, g = 0.f, ge = 0.f;
#pragma unroll 4
  for (int r = lane; r < d; r += 32) {
    const float2 a = sc[r];
    if (want_r1) {
      const float2 b = zd[r];
      df_mac(a.x, a.y, b.x, b.y, s, t);
    }
    if (finish) {
      const float2 b = sjd[r];
      df_mac(a.x, a.y, b.x, b.y, g, ge);
    }
  }
  if (want_r1) df_warp_sum(s, t);
  if (finish) df_warp_sum(g, ge);
  if (lane == 0) {
    if (want_r1) r1[col] = df_norm(s, t);
    if (finish) {
      const float2 m = df_norm(g, ge);
      M2[col + (size_t)j * ldm] = m;
      M2[j + (size_t)col * ldm] = m;
    }
  }
}

// Phase B for one column (one warp): r = 2 r1[col] - sum_l M[l, col] r1[l].
__device__ __forceinline__ void ls_phase_b(int col, int c, const float2* M2, int ldm, const float2* r1,
                                           const double* colscale, double* rprev, float2* nrs, int lane) {
  const float2* mc = M2 + (size_t)col * ldm;
  float s = 0.f, t = 0.f;
#pragma unroll 4
  for (int l = lane; l < c; l += 32) {
    const float2 a = mc[l], b = r1[l];
    df_mac(a.x, a.y, b.x, b.y, s, t);
  }
  df_warp_sum(s, t);
  if (lane == 0) {
    const float2 rc = r1[col];
    float hs = 2.f * rc.x, ht = 2.f * rc.y;   // exact doubling
    df_add(-s, -t, hs, ht);
    const double rd = df_to_double(df_norm(hs, ht));
    rprev[col] = rd;
    nrs[col] = df_from_double(-rd * colscale[col]);
  }
}

__global__ void __launch_bounds__(256) k_df_ls1(
    int j, int d, double zscale, int finish, int ls, double* __restrict__ s_raw, const double* __restrict__ z_raw,
    double* __restrict__ S64, float2* __restrict__ S2, double* __restrict__ colscale,
    const double* __restrict__ rprev, double* __restrict__ coef, int ldcoef, double* __restrict__ znorm_prev,
    float2* __restrict__ r1, float2* __restrict__ M2, int ldm, int* flag) {
  extern __shared__ float2 zd[];   // d: z; then d: s_j (when finishing)
  float2* sjd = zd + d;
  __shared__ double red[33];
  const int tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5, lane = tid & 31, nw = nt >> 5;
  double inv = 0.0;
  if (finish) {
    double ss = 0.0;
    for (int r = tid; r < d; r += nt) { double v = s_raw[r] * zscale; ss = fma(v, v, ss); }
    ss = block_sum_d(ss, red);
    const double beta = sqrt(ss);
    const bool finite = isfinite(beta);
    const bool brk = finite && !(beta > 1e-14 * znorm_prev[0]);
    inv = (finite && !brk) ? 1.0 / beta : 0.0;
    for (int r = tid; r < d; r += nt) sjd[r] = df_from_double(s_raw[r] * zscale * inv);
    if (blockIdx.x == 0) {
      for (int r = tid; r < d; r += nt) {
        double v = s_raw[r] * zscale * inv;
        S64[r + (size_t)j * d] = v;
        S2[r + (size_t)j * d] = df_from_double(v);
      }
      if (j >= 1) {
        double* cc = coef + (size_t)(j - 1) * ldcoef;
        for (int i = tid; i < j; i += nt) cc[i] = rprev[i];
        if (tid == 0) cc[j] = beta;
      }
      if (tid == 0) {
        colscale[j] = inv;
        if (!finite) atomicOr(flag, RKS_FLAG_NAN);
        else if (brk) atomicOr(flag, RKS_FLAG_BREAKDOWN);
      }
    }
  }
  if (!ls && !finish) return;
  if (ls) {
    const double scj = finish ? inv : colscale[j];
    double zz = 0.0;
    for (int r = tid; r < d; r += nt) {
      double v = z_raw[r] * zscale * scj;
      zz = fma(v, v, zz);
      zd[r] = df_from_double(v);
    }
    zz = block_sum_d(zz, red);
    if (blockIdx.x == 0 && tid == 0) znorm_prev[0] = sqrt(zz);
  }
  __syncthreads();
  const int c = j + 1;
  for (int col = blockIdx.x * nw + warp; col < c; col += gridDim.x * nw)
    ls_phase_a(col, j, d, finish, ls, S2, zd, sjd, r1, M2, ldm, lane);
}

// Phase B as its own launch (warp per column); CTA 0 also sets sj.
__global__ void __launch_bounds__(256) k_df_ls_gram(int j, const float2* __restrict__ M2, int ldm,
                                                    const float2* __restrict__ r1,
                                                    const double* __restrict__ colscale,
                                                    double* __restrict__ rprev, float2* __restrict__ nrs,
                                                    float2* __restrict__ sj) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int c = j + 1;
  if (blockIdx.x == 0 && threadIdx.x == 0) sj[0] = df_from_double(colscale[j]);
  const int col = blockIdx.x * nw + warp;
  if (col < c) ls_phase_b(col, c, M2, ldm, r1, colscale, rprev, nrs, lane);
}

// Grid-wide barrier of the cooperative least-squares kernel.  bar[0] counts
// arrivals, bar[1] is the generation.  The wait is bounded (about a second of
// clock cycles): on timeout the kernel records RKS_FLAG_TIMEOUT and goes on,
// and the host reports the failure instead of the device hanging.  The
// cooperative launch guarantees that all CTAs are resident, so the bound is
// never reached in a correct run.
__device__ __forceinline__ void grid_barrier(unsigned* bar, unsigned nblocks, int* flag, long long limit) {
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* vgen = bar + 1;
    const unsigned gen = *vgen;
    __threadfence();
    const unsigned arrived = atomicAdd(bar, 1u) + 1u;
    if (arrived == nblocks) {
      bar[0] = 0u;
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      const long long t0 = clock64();
      while (*vgen == gen) {
        if (clock64() - t0 > limit) { atomicOr(flag, RKS_FLAG_TIMEOUT); break; }
        __nanosleep(32);
      }
    }
    __threadfence();
  }
  __syncthreads();
}

// Fold of the sketch partials, phase A and phase B in one cooperative launch.
// The kernel is a chain of L2 round trips, so everything that does not
// depend on the fold is loaded before it: each warp's column of S (phase A)
// and of M (phase B) into registers, z_raw together with s_raw.  The order of
// every sum is that of ls_phase_a / ls_phase_b, so the results are the same
// bits as theirs.
constexpr int kLsPre = 12;          // entries per lane prefetched for phase A (d <= 384 fully)
constexpr int kLsPreB = 4;          // for phase B (c <= 128 fully)
constexpr int kLsStageMax = 2048;   // d up to which z_raw / s_raw are staged in shared memory

__global__ void __launch_bounds__(256) k_df_ls_coop(
    int j, int d, double zscale, int finish, double* __restrict__ s_raw, double* __restrict__ z_raw,
    double* __restrict__ S64, float2* __restrict__ S2, double* __restrict__ colscale, double* __restrict__ rprev,
    double* __restrict__ coef, int ldcoef, double* __restrict__ znorm_prev, float2* __restrict__ nrs,
    float2* __restrict__ sj, float2* __restrict__ r1, float2* __restrict__ M2, int ldm,
    const double* __restrict__ part_z, const double* __restrict__ part_s, int G, unsigned* bar, int* flag,
    int stall) {
  extern __shared__ float2 zd[];   // d: z; d: s_j (when finishing); then 2d doubles: z_raw, s_raw
  float2* sjd = zd + d;
  double* zst = reinterpret_cast<double*>(sjd + d);
  double* sst = zst + d;
  __shared__ double red[33];
  const int tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5, lane = tid & 31, nw = nt >> 5;
  pdl_next();                           // the update's CTAs may come in and fetch what does not depend on this
  const int gw = blockIdx.x * nw + warp, tw = gridDim.x * nw;   // global warp index, warps in grid
  const int c = j + 1;
  // stall (a test hook) waits for one CTA more than the grid holds, so every
  // barrier runs out its short limit and the solve reports RKS_ETIMEOUT
  const unsigned expect = gridDim.x + (stall ? 1u : 0u);
  const long long limit = stall ? 2000000ll : 4000000000ll;
  const bool stage = d <= kLsStageMax;
  // prefetch (independent of the fold): this warp's first column
  const int col0 = gw;
  float2 pa[kLsPre], pb[kLsPreB];
  double cs0 = 0.0;
  const bool pre_a = col0 < c && !(finish && col0 == j);      // column j of S is new when finishing
  const bool pre_b = col0 < c && !(finish && col0 == j);      // so is column j of M
  if (pre_a) {
    const float2* sc = S2 + (size_t)col0 * d;
#pragma unroll
    for (int i = 0; i < kLsPre; ++i) {
      const int r = lane + 32 * i;
      pa[i] = r < d ? sc[r] : make_float2(0.f, 0.f);
    }
  }
  if (pre_b) {
    const float2* mc = M2 + (size_t)col0 * ldm;
#pragma unroll
    for (int i = 0; i < kLsPreB; ++i) {
      const int l = lane + 32 * i;
      pb[i] = (l < c && !(finish && l == j)) ? mc[l] : make_float2(0.f, 0.f);
    }
    cs0 = colscale[col0];
  }
  const double zn_prev = znorm_prev[0];
  // z' and s~_j from the sketch kernels' per-CTA partial sums
  {
    const int nb = finish ? 2 * d : d;
    for (int r = gw; r < nb; r += tw) {
      const bool isz = r < d;
      const double v = fold_row(isz ? part_z : part_s, d, G, isz ? r : r - d, lane);
      if (lane == 0) {
        if (isz) z_raw[r] = v;
        else s_raw[r - d] = v;
      }
    }
    grid_barrier(bar, expect, flag, limit);
  }
  // z_raw and s_raw in one round trip
  const double cs_j = finish ? 0.0 : colscale[j];
  if (stage) {
    for (int r = tid; r < d; r += nt) {
      zst[r] = z_raw[r];
      if (finish) sst[r] = s_raw[r];
    }
    __syncthreads();
  }
  const double* zsrc = stage ? zst : z_raw;
  const double* ssrc = stage ? sst : s_raw;
  // FP64 runs at two lanes a clock: a square root or a division by every
  // thread of the CTA costs thousands of cycles, so thread 0 forms them
  __shared__ double bsh[2];
  double inv = 0.0;
  if (finish) {
    double ss = 0.0;
    for (int r = tid; r < d; r += nt) { double v = ssrc[r] * zscale; ss = fma(v, v, ss); }
    ss = block_sum_0(ss, red);
    if (tid == 0) {
      const double beta = sqrt(ss);
      const bool finite = isfinite(beta);
      const bool brk = finite && !(beta > 1e-14 * zn_prev);
      bsh[0] = (finite && !brk) ? 1.0 / beta : 0.0;
      if (blockIdx.x == 0) {
        bsh[1] = beta;
        colscale[j] = bsh[0];
        if (!finite) atomicOr(flag, RKS_FLAG_NAN);
        else if (brk) atomicOr(flag, RKS_FLAG_BREAKDOWN);
      }
    }
    __syncthreads();
    inv = bsh[0];
    for (int r = tid; r < d; r += nt) {
      const double v = ssrc[r] * zscale * inv;
      const float2 w = df_from_double(v);
      sjd[r] = w;
      if (blockIdx.x == 0) {
        S64[r + (size_t)j * d] = v;
        S2[r + (size_t)j * d] = w;
      }
    }
    if (blockIdx.x == 0 && j >= 1) {
      double* cc = coef + (size_t)(j - 1) * ldcoef;
      for (int i = tid; i < j; i += nt) cc[i] = rprev[i];
      if (tid == 0) cc[j] = bsh[1];
    }
  }
  const double scj = finish ? inv : cs_j;
  double zz = 0.0;
  for (int r = tid; r < d; r += nt) {
    double v = zsrc[r] * zscale * scj;
    if (blockIdx.x == 0) zz = fma(v, v, zz);    // ||z|| is CTA 0's to store
    zd[r] = df_from_double(v);
  }
  if (blockIdx.x == 0) zz = block_sum_0(zz, red);
  __syncthreads();                      // orders the zd and sjd writes before their use
  // phase A: r1[col] = S[:, col]^T z and, when finishing, M[col, j] = S[:, col]^T s_j
  float2 mnew = make_float2(0.f, 0.f);  // M[j, col0] computed here (finishing)
  for (int col = gw; col < c; col += tw) {
    if (col == col0 && pre_a) {
      float s_ = 0.f, t_ = 0.f, g = 0.f, ge = 0.f;
      int i = 0;
#pragma unroll
      for (int ii = 0; ii < kLsPre; ++ii, ++i) {
        const int r = lane + 32 * ii;
        if (r < d) {
          const float2 a = pa[ii], b = zd[r];
          df_mac(a.x, a.y, b.x, b.y, s_, t_);
          if (finish) { const float2 e = sjd[r]; df_mac(a.x, a.y, e.x, e.y, g, ge); }
        }
      }
      for (int r = lane + 32 * kLsPre; r < d; r += 32) {
        const float2 a = S2[(size_t)col * d + r], b = zd[r];
        df_mac(a.x, a.y, b.x, b.y, s_, t_);
        if (finish) { const float2 e = sjd[r]; df_mac(a.x, a.y, e.x, e.y, g, ge); }
      }
      df_warp_sum(s_, t_);
      if (finish) df_warp_sum(g, ge);
      if (lane == 0) r1[col] = df_norm(s_, t_);
      if (finish) {
        mnew = df_norm(g, ge);
        if (lane == 0) {
          M2[col + (size_t)j * ldm] = mnew;
          M2[j + (size_t)col * ldm] = mnew;
        }
      }
    } else {
      ls_phase_a(col, j, d, finish, 1, S2, zd, sjd, r1, M2, ldm, lane);
    }
  }
  grid_barrier(bar, expect, flag, limit);
  // phase B
  if (blockIdx.x == 0 && tid == 0) { sj[0] = df_from_double(scj); znorm_prev[0] = sqrt(zz); }
  for (int col = gw; col < c; col += tw) {
    if (col == col0 && pre_b) {
      float s_ = 0.f, t_ = 0.f;
#pragma unroll
      for (int ii = 0; ii < kLsPreB; ++ii) {
        const int l = lane + 32 * ii;
        if (l < c) {
          const float2 a = (finish && l == j) ? mnew : pb[ii], b = r1[l];
          df_mac(a.x, a.y, b.x, b.y, s_, t_);
        }
      }
      for (int l = lane + 32 * kLsPreB; l < c; l += 32) {
        const float2 a = (finish && l == j) ? mnew : M2[l + (size_t)col * ldm], b = r1[l];
        df_mac(a.x, a.y, b.x, b.y, s_, t_);
      }
      df_warp_sum(s_, t_);
      if (lane == 0) {
        const float2 rc = r1[col];
        float hs = 2.f * rc.x, ht = 2.f * rc.y;   // exact doubling
        df_add(-s_, -t_, hs, ht);
        const double rd = df_to_double(df_norm(hs, ht));
        rprev[col] = rd;
        nrs[col] = df_from_double(-rd * cs0);
      }
    } else {
      ls_phase_b(col, c, M2, ldm, r1, colscale, rprev, nrs, lane);
    }
  }
}

// y = x (FP64) in the storage type
template <class TU>
__global__ void k_d2df(int64_t n, const double* __restrict__ x, TU* __restrict__ y) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    stv(y + i, df_from_double(x[i]));
}

__global__ void k_d2df_cols(int64_t n, const double* __restrict__ x, int64_t ldx, float2* __restrict__ y,
                            int64_t ldy) {
  const int j = blockIdx.y;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    y[i + (int64_t)j * ldy] = df_from_double(x[i + (int64_t)j * ldx]);
}

// stored columns -> FP64 columns (ncols, with leading dimensions)
template <class TU>
__global__ void k_df2d_cols(int64_t n, const TU* __restrict__ x, int64_t ldx, double* __restrict__ y,
                            int64_t ldy, int ncols) {
  const int j = blockIdx.y;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    y[i + (int64_t)j * ldy] = df_to_double(ldv(x + i + (int64_t)j * ldx));
}

// part[cta] = the CTA's Omega-sums of a stored vector (start vector)
template <class TU>
__global__ void __launch_bounds__(512) k_df_sketch_vec(const TU* __restrict__ x, const SketchTiles tv,
                                                       double* __restrict__ part) {
  extern __shared__ __align__(16) uint8_t smraw[];
  const int d = tv.d;
  const TileSmem lay = tile_smem_layout(d, tv.L, 0, tv.zeta);
  float2* acc = reinterpret_cast<float2*>(smraw + lay.acc);
  for (int r = threadIdx.x; r < d; r += blockDim.x) acc[r] = make_float2(0.f, 0.f);
  const TileRange tr(tv, false);
  if (tr.nt > 0) tile_fetch<TU>(smraw, lay, tv, tr, 0);
  pdl_next();
  pdl_wait();
  x = pdl_fresh(x);
  for (int k = 0; k < tr.nt; ++k) {
    TU* v = TileBuf<TU>(smraw, lay, tv, k).v;
    const int64_t r0 = tr.row(k);
    const int rows = tr.rows(k);
    for (int l = threadIdx.x; l < rows; l += blockDim.x) v[l] = x[r0 + l];
    tile_finish<TU>(smraw, lay, tv, tr, k, acc);
  }
  tile_write_part(acc, d, part);
}

// part[col][cta] = the CTA's Omega-sums of column col, for a block of columns
// given in FP64 or double-float; with U, the double-float columns are also
// written there.  A CTA takes up to NC columns (grid.y the others), so that a
// tile's bin lists (16 bytes a row, twice a column's bytes) are staged once
// for NC columns, and FP64 input is converted on the way: a launch, a
// conversion pass and a staging per column took 36 us a column at n = 1e6,
// d = 320; here 14 us.  The next column's values are loaded while one is
// summed; the sums are those of k_df_sketch_vec.
constexpr int kSkCols = kPanelCols;
template <class TS>
__global__ void __launch_bounds__(512, 2) k_df_sketch_cols(const TS* __restrict__ x, int64_t ldx, int ncols, int nc,
                                                           float2* __restrict__ U, int64_t ldu, const SketchTiles tv,
                                                           double* __restrict__ part) {
  extern __shared__ __align__(16) uint8_t smraw[];
  const int d = tv.d, L1 = tv.L + 1;
  float2* vb = reinterpret_cast<float2*>(smraw);                             // two value buffers
  uint16_t* es = reinterpret_cast<uint16_t*>(vb + 2 * kTileRows);
  uint32_t* ms = reinterpret_cast<uint32_t*>(es + (size_t)kTileRows * tv.zeta);
  int* of = reinterpret_cast<int*>(ms + d);
  float2* acc = reinterpret_cast<float2*>(of + L1 + (L1 + d & 1));           // nc x d
  const int q0 = blockIdx.y * nc, nq = min(nc, ncols - q0);
  for (int r = threadIdx.x; r < nq * d; r += blockDim.x) acc[r] = make_float2(0.f, 0.f);
  x += (int64_t)q0 * ldx;
  if (U) U += (int64_t)q0 * ldu;
  const int la = threadIdx.x, lb = threadIdx.x + 512;
  const int t0 = tv.ctile[blockIdx.x], t1 = tv.ctile[blockIdx.x + 1];
  auto as_df = [](TS v) {
    if constexpr (std::is_same<TS, double>::value) return df_from_double(v);
    else return v;
  };
  for (int t = t0; t < t1; ++t) {
    const int64_t r0 = tv.row[t];
    const int rows = (int)(tv.row[t + 1] - r0);
    const TS* xt = x + r0;
    TS a{}, b{};
    if (la < rows) a = xt[la];
    if (lb < rows) b = xt[lb];
    __syncthreads();                               // the last tile's lists and values are read
    tile_stage(tv, t, r0, rows, of, ms, es);
    for (int q = 0; q < nq; ++q) {
      float2* v = vb + (q & 1) * kTileRows;
      const float2 da = as_df(a), db = as_df(b);
      v[la] = da;
      v[lb] = db;
      if (U) {
        if (la < rows) U[(int64_t)q * ldu + r0 + la] = da;
        if (lb < rows) U[(int64_t)q * ldu + r0 + lb] = db;
      }
      if (q + 1 < nq) {
        const TS* xn = xt + (int64_t)(q + 1) * ldx;
        if (la < rows) a = xn[la];
        if (lb < rows) b = xn[lb];
      }
      __syncthreads();
      tile_gather(d, tv.H, v, of, ms, es, acc + (size_t)q * d);
    }
  }
  __syncthreads();
  for (int r = threadIdx.x; r < nq * d; r += blockDim.x) {
    const int q = r / d, i = r - q * d;
    part[((size_t)(q0 + q) * gridDim.x + blockIdx.x) * d + i] = df_to_double(acc[r]);
  }
}

// U[:, p0 + k] += sum_{c < c0} U[:, c] coef[c * kSkCols + k] for k < nb <= kSkCols
// (double-float): a panel of columns updated by all earlier ones in one pass
// over them, where a column at a time read them once per column.  Two rows
// per thread; a column's terms are added in the order of k_df_update_sketch.
// Bound by the FP32 pipes (12 operations per double-float multiply-add).  The
// 80-column RGS at n = 1e6: 5.5 ms of updates -> 1.5 ms here and 2.5 ms of
// updates inside the panels.
__global__ void __launch_bounds__(256, 2) k_df_panel(int64_t n, float2* __restrict__ U, int64_t ldu, int c0, int p0,
                                                     int nb, const float2* __restrict__ coef) {
  extern __shared__ __align__(16) float2 cs[];     // c0 x kSkCols
  for (int t = threadIdx.x; t < c0 * kSkCols; t += blockDim.x) cs[t] = coef[t];
  __syncthreads();
  for (int64_t i = 2 * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x); i < n;
       i += 2 * (int64_t)gridDim.x * blockDim.x) {
    float s[2][kSkCols], t[2][kSkCols];
#pragma unroll
    for (int k = 0; k < kSkCols; ++k) {
      float2 a = make_float2(0.f, 0.f), b = a;
      if (k < nb) ld2(U + i + (int64_t)(p0 + k) * ldu, a, b);
      s[0][k] = a.x; t[0][k] = a.y;
      s[1][k] = b.x; t[1][k] = b.y;
    }
#pragma unroll 4
    for (int c = 0; c < c0; ++c) {
      float2 a, b;
      ld2(U + i + (int64_t)c * ldu, a, b);
#pragma unroll
      for (int k = 0; k < kSkCols; ++k) {
        const float2 r = cs[c * kSkCols + k];
        df_mac(a.x, a.y, r.x, r.y, s[0][k], t[0][k]);
        df_mac(b.x, b.y, r.x, r.y, s[1][k], t[1][k]);
      }
    }
#pragma unroll
    for (int k = 0; k < kSkCols; ++k)
      if (k < nb) {
        float2* p = U + i + (int64_t)(p0 + k) * ldu;
        p[0] = df_norm(s[0][k], t[0][k]);
        if (i + 1 < n) p[1] = df_norm(s[1][k], t[1][k]);
      }
  }
}

// Gram matrix of s double-float columns, upper triangle in 4 x 4 blocks:
// part[cta * npair + p], p = the block's number * 16 + 4 i + j, holds the CTA's
// sum of column (4 bi + i) times column (4 bj + j).  A block reads 8 columns
// for 16 products where a product per column pair read one for one.
__global__ void __launch_bounds__(256) k_df_gram(const float2* __restrict__ U, int64_t ldu, int64_t n, int s,
                                                 double* __restrict__ part, int npair) {
  __shared__ float2 red[8][16];
  int bj = 0, q = blockIdx.y;
  while (q > bj) { q -= bj + 1; ++bj; }            // block (bi = q, bj), bi <= bj
  const int bi = q;
  const float2 *pa[4], *pb[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    pa[u] = U + (int64_t)min(4 * bi + u, s - 1) * ldu;
    pb[u] = U + (int64_t)min(4 * bj + u, s - 1) * ldu;
  }
  float sh[16], sl[16];
#pragma unroll
  for (int u = 0; u < 16; ++u) { sh[u] = 0.f; sl[u] = 0.f; }
  const int64_t per = (n + gridDim.x - 1) / gridDim.x, r0 = blockIdx.x * per, r1 = min(n, r0 + per);
  for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
    float2 a[4], b[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) { a[u] = pa[u][i]; b[u] = pb[u][i]; }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) df_mac(a[u].x, a[u].y, b[v].x, b[v].y, sh[4 * u + v], sl[4 * u + v]);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int u = 0; u < 16; ++u) {
    df_warp_sum(sh[u], sl[u]);
    if (lane == 0) red[warp][u] = df_norm(sh[u], sl[u]);
  }
  __syncthreads();
  if (threadIdx.x < 16) {
    double v = 0.0;
    for (int w = 0; w < 8; ++w) v += df_to_double(red[w][threadIdx.x]);
    part[(size_t)blockIdx.x * npair + blockIdx.y * 16 + threadIdx.x] = v;
  }
}

// U[i, c0 + l] -= coef[l] * U[i, src] for l < ncols (double-float): one
// reflector applied to a block of columns (randomized Householder QR).
__global__ void __launch_bounds__(256) k_df_axpy_cols(int64_t n, float2* __restrict__ U, int64_t ldu, int src,
                                                      int c0, int ncols, const float2* __restrict__ coef) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float2 u = U[i + (int64_t)src * ldu];
    for (int l = 0; l < ncols; ++l) {
      float2* y = U + i + (int64_t)(c0 + l) * ldu;
      const float2 yv = *y, c = coef[l];
      float sh = yv.x, sl = yv.y;
      df_mac(-c.x, -c.y, u.x, u.y, sh, sl);
      *y = df_norm(sh, sl);
    }
  }
}

// Row-blocked DF product, in place: U[i, c0 + o] = sum_l U[i, a0 + l] Q[l, o]
// (Q DF, nin x nout column-major), then U[i, c0 + nout] = U[i, move_src].
template <class TU>
__global__ void __launch_bounds__(128) k_df_rows_gemm(int64_t n, TU* U, int64_t ldu, int a0, int nin,
                                                      const float2* __restrict__ Q, int nout, int c0,
                                                      int move_src) {
  extern __shared__ float2 shq[];
  float2* Qs = shq;
  float2* tmp = shq + (size_t)nin * nout;
  for (int t = threadIdx.x; t < nin * nout; t += blockDim.x) Qs[t] = Q[t];
  __syncthreads();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const TU* up = U + i + (int64_t)a0 * ldu;
  for (int o0 = 0; o0 < nout; o0 += 4) {
    float s[4] = {0.f, 0.f, 0.f, 0.f}, t[4] = {0.f, 0.f, 0.f, 0.f};
    const int no = min(4, nout - o0);
    for (int l = 0; l < nin; ++l) {
      float2 a = ldv(up + (int64_t)l * ldu);
#pragma unroll
      for (int o = 0; o < 4; ++o)
        if (o < no) {
          float2 q = Qs[l + (size_t)(o0 + o) * nin];
          df_mac(a.x, a.y, q.x, q.y, s[o], t[o]);
        }
    }
#pragma unroll
    for (int o = 0; o < 4; ++o)
      if (o < no) tmp[(size_t)(o0 + o) * blockDim.x + threadIdx.x] = df_norm(s[o], t[o]);
  }
  const TU mv = move_src >= 0 ? U[i + (int64_t)move_src * ldu] : TU();
  for (int o = 0; o < nout; ++o) stv(U + i + (int64_t)(c0 + o) * ldu, tmp[(size_t)o * blockDim.x + threadIdx.x]);
  if (move_src >= 0) U[i + (int64_t)(c0 + nout) * ldu] = mv;
}

// y = sum_{j < ncols} U[:, j] (FP32 columns), in FP64
__global__ void k_sum_cols_f32(int64_t n, const float* __restrict__ U, int64_t ldu, int ncols,
                               double* __restrict__ y) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int j = 0; j < ncols; ++j) s += (double)U[i + (int64_t)j * ldu];
    y[i] = s;
  }
}

// Restart product, in place: U[i, c0 + o] = sum_l U[i, a0 + l] Q[l, o] for
// o < nout (<= 4 * MAXOP), then U[i, c0 + nout] = U[i, move_src].  A CTA of
// 256 threads owns 64 rows; the 4 threads of a row split the outputs (up to
// MAXOP DF accumulators each, in registers).  Every read of the CTA's rows
// precedes the barrier, every write follows it, and no other CTA touches
// these rows, so the in-place update is safe.
template <class TU, int MAXOP>
__global__ void __launch_bounds__(256) k_df_restart(int64_t n, TU* U, int64_t ldu, int a0, int nin,
                                                    const float2* __restrict__ Q, int nout, int c0, int move_src) {
  extern __shared__ float2 qs[];                  // nin x nout, column-major
  for (int t = threadIdx.x; t < nin * nout; t += blockDim.x) qs[t] = Q[t];
  __syncthreads();
  const int r = threadIdx.x & 63, g = threadIdx.x >> 6;       // row in tile, output group
  const int64_t i = blockIdx.x * (int64_t)64 + r;
  const int per = (nout + 3) / 4;
  const int o0 = g * per;
  const int no = max(0, min(per, nout - o0));
  float s[MAXOP], t[MAXOP];
#pragma unroll
  for (int o = 0; o < MAXOP; ++o) { s[o] = 0.f; t[o] = 0.f; }
  TU mv{};
  if (i < n) {
    const TU* up = U + i + (int64_t)a0 * ldu;
    int l = 0;
    for (; l + 4 <= nin; l += 4) {          // four loads in flight per thread
      float2 a[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = ldv(up + (int64_t)(l + u) * ldu);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float2* ql = qs + (l + u) + (size_t)o0 * nin;
#pragma unroll
        for (int o = 0; o < MAXOP; ++o)
          if (o < no) {
            const float2 q = ql[(size_t)o * nin];
            df_mac(a[u].x, a[u].y, q.x, q.y, s[o], t[o]);
          }
      }
    }
    for (; l < nin; ++l) {
      const float2 a = ldv(up + (int64_t)l * ldu);
      const float2* ql = qs + l + (size_t)o0 * nin;
#pragma unroll
      for (int o = 0; o < MAXOP; ++o)
        if (o < no) {
          const float2 q = ql[(size_t)o * nin];
          df_mac(a.x, a.y, q.x, q.y, s[o], t[o]);
        }
    }
    if (move_src >= 0 && g == 0) mv = U[i + (int64_t)move_src * ldu];
  }
  __syncthreads();
  if (i < n) {
#pragma unroll
    for (int o = 0; o < MAXOP; ++o)
      if (o < no) stv(U + i + (int64_t)(c0 + o0 + o) * ldu, df_norm(s[o], t[o]));
    if (move_src >= 0 && g == 0) U[i + (int64_t)(c0 + nout) * ldu] = mv;
  }
}

// ---------------------------------------------------------------------------
// Hand-over of the mixed path's FP32 Krylov-Schur decomposition
// A U = U T + u b^T to double-float: the FP32 basis promoted exactly, the
// relation error E = A U - U T - u b^T of the promoted columns, and damped
// Jacobi sweeps on A X - X T = -E for the correction U <- U + X.
// ---------------------------------------------------------------------------

// U2[:, j] = Uf[:, j], j < ncols (exact: the pairs' low words are zero)
__global__ void k_f32_to_df_cols(int64_t n, const float* __restrict__ Uf, int64_t ldu, int ncols,
                                 float2* __restrict__ U2) {
  const int64_t total = (int64_t)ncols * ldu;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = q % ldu;
    if (i < n) U2[q] = make_float2(Uf[q], 0.f);
  }
}

// e = w - v - beta u in double-float, rounded to FP32 (column j of E:
// w = A u_j, v = (U T)_j, beta = b_j times the column scale of u)
__global__ void k_relation_resid(int64_t n, const float2* __restrict__ w, const float2* __restrict__ v,
                                 const float2* __restrict__ u, double beta, float* __restrict__ e) {
  const float2 nb = df_from_double(-beta);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float2 a = w[i], b = v[i], c = u[i];
    float s = a.x, t = a.y;
    df_add(-b.x, -b.y, s, t);
    df_mac(nb.x, nb.y, c.x, c.y, s, t);
    e[i] = s + t;
  }
}

// 1 / a_ii (0 where row i has no diagonal entry or a zero one)
__global__ void k_diag_inv(int64_t n, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colind,
                           const float* __restrict__ vals, float* __restrict__ dinv) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float a = 0.f;
    for (int p = rowptr[i]; p < rowptr[i + 1]; ++p)
      if (colind[p] == i) a += vals[p];
    dinv[i] = a != 0.f ? 1.0f / a : 0.f;
  }
}

// One damped Jacobi sweep on A X - X T = -E for all kk columns:
//   R = E + A X - Y (Y = X T, given),  Xn = X - omega D^{-1} R,
// a thread per row (the row's entries loaded once, up to 16 kept in
// registers), FP32 with FMA.  With part: the per-CTA sums of R^2 per column
// (warp sums by a fixed butterfly, then the warps in order) in
// part[blockIdx.x * kk + j].
constexpr int kJacobiCta = 256;
__global__ void __launch_bounds__(kJacobiCta) k_jacobi_sweep(int64_t n, const int32_t* __restrict__ rowptr,
                                                             const int32_t* __restrict__ colind,
                                                             const float* __restrict__ vals,
                                                             const float* __restrict__ dinv, int kk, int64_t ld,
                                                             const float* __restrict__ X,
                                                             const float* __restrict__ E,
                                                             const float* __restrict__ Y, float omega,
                                                             float* __restrict__ Xn, double* __restrict__ part) {
  constexpr int RM = 16;
  __shared__ double wsum[kJacobiCta / 32];
  const int64_t i = blockIdx.x * (int64_t)kJacobiCta + threadIdx.x;
  const bool on = i < n;
  int p0 = 0, len = 0;
  float di = 0.f;
  int cj[RM];
  float aj[RM];
  if (on) {
    p0 = rowptr[i];
    len = rowptr[i + 1] - p0;
    di = dinv[i];
  }
#pragma unroll
  for (int e = 0; e < RM; ++e) {
    const bool h = e < len;
    cj[e] = h ? colind[p0 + e] : 0;
    aj[e] = h ? vals[p0 + e] : 0.f;
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int j = 0; j < kk; ++j) {
    const int64_t o = (int64_t)j * ld;
    double r2 = 0.0;
    if (on) {
      float acc = E[o + i] - Y[o + i];
#pragma unroll
      for (int e = 0; e < RM; ++e)
        if (e < len) acc = fmaf(aj[e], X[o + cj[e]], acc);
      for (int e = RM; e < len; ++e) acc = fmaf(vals[p0 + e], X[o + colind[p0 + e]], acc);
      Xn[o + i] = fmaf(-omega * di, acc, X[o + i]);
      r2 = (double)acc * (double)acc;
    }
    if (part) {
      for (int s = 16; s; s >>= 1) r2 += __shfl_xor_sync(0xffffffffu, r2, s);
      if (lane == 0) wsum[wid] = r2;
      __syncthreads();
      if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kJacobiCta / 32; ++w) t += wsum[w];
        part[(int64_t)blockIdx.x * kk + j] = t;
      }
      __syncthreads();
    }
  }
}

// U2[:, j] += X[:, j] (double-float + FP32), j < kk
__global__ void k_df_add_f32_cols(int64_t n, float2* __restrict__ U2, int64_t ldu, int kk,
                                  const float* __restrict__ X, int64_t ldx) {
  const int64_t total = (int64_t)kk * n;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = q / n, i = q - j * n;
    const float2 u = U2[j * ldu + i];
    float s = u.x, t = u.y;
    df_add(X[j * ldx + i], 0.f, s, t);
    U2[j * ldu + i] = df_norm(s, t);
  }
}

// ---------------------------------------------------------------------------
// Small problems: the whole expansion in one launch of one cluster
// ---------------------------------------------------------------------------
//
// At a few thousand rows an Arnoldi step is three launches of 6 to 16 us whose
// work would take one (2000 rows, 40 columns: 45 us a step with the gaps).
// Here the CTAs of one thread-block cluster (at most 16) own the row ranges of
// the sketch tiles and run all steps c0 .. m - 1 of Algorithm 2: per step the
// product with A and its sketch, the least squares (by every CTA, from the
// same data), the update and its sketch.  Partial sketches go to every CTA
// through distributed shared memory, so a step has two cluster barriers.
// The bin lists, S and M stay in shared memory, the CTA's rows of the basis too
// where they fit.  The arithmetic and the order of every sum are those of
// k_df_spmv_* / k_df_ls_coop / k_df_update_sketch on the same tiles: the same
// bits.  Sixteen SMs suffice while a step's row work stays below its barriers
// and latencies: kSmallRows.  Measured per step, d = 80, 30 to 40 columns: 12 us
// at 2000 rows (31 with the separate kernels, 45 with their launches queued
// from the host), 18 at 16 000 (24), 24 at 32 000 (24).
struct SmallArgs {
  const int32_t *rowptr, *colind;
  const float2* vals;          // CSR (D = 0)
  const float2* dvals;         // by diagonals (D > 0)
  DiaOffs offs;
  int D;
  int64_t ldd;
  int n, c0, m;
  float2* U;
  int64_t ldu;
  SketchTiles tv;
  double zscale;
  double* S64;
  const float2 *S2, *M2;
  double *colscale, *coef;
  int ldcoef, ldm;
  int* flag;
  int rows_max, tiles_max;     // of a CTA
  int slab;                    // the CTA's basis rows in shared memory
};

__device__ __forceinline__ uint32_t cl_addr(const void* p, int rank) {
  uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void cl_put(uint32_t a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cl_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

struct SmallSmem {
  size_t zx, sx, csc, rp, zd, sjd, acc, v, r1, nrs, mcol, es, ms, of, slab, S, M, total;
};
__host__ __device__ inline SmallSmem small_smem(int G, int d, int m, int rows, int tiles, int L, int zeta,
                                                int slab) {
  SmallSmem s;
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t r = o; o += (bytes + 15) & ~(size_t)15; return r; };
  s.zx = take((size_t)G * d * 8);
  s.sx = take((size_t)G * d * 8);
  s.csc = take((size_t)(m + 1) * 8);
  s.rp = take((size_t)(m + 1) * 8);
  s.zd = take((size_t)d * 8);
  s.sjd = take((size_t)d * 8);
  s.acc = take((size_t)d * 8);
  s.v = take((size_t)rows * 8);
  s.r1 = take((size_t)(m + 1) * 8);
  s.nrs = take((size_t)(m + 1) * 8);
  s.mcol = take((size_t)(m + 1) * 8);
  s.es = take((size_t)rows * zeta * 2);
  s.ms = take((size_t)tiles * d * 4);
  s.of = take((size_t)tiles * (L + 1) * 4);
  s.slab = take(slab ? (size_t)rows * (m + 1) * 8 : 0);
  s.S = take((size_t)d * (m + 1) * 8);
  s.M = take((size_t)(m + 1) * (m + 1) * 8);
  s.total = o;
  return s;
}

// sum over g < G <= 16 of p[g * d] in the tree of fold_row
__device__ __forceinline__ double fold16(const double* p, int d, int G) {
  double v[16];
#pragma unroll
  for (int g = 0; g < 16; ++g) v[g] = g < G ? p[(size_t)g * d] : 0.0;
#pragma unroll
  for (int o = 8; o; o >>= 1)
#pragma unroll
    for (int g = 0; g < o; ++g) v[g] += v[g + o];
  return v[0];
}

__global__ void __launch_bounds__(512) k_df_expand_small(const SmallArgs a) {
  extern __shared__ __align__(16) uint8_t sraw[];
  __shared__ double red[64];
  const SketchTiles& tv = a.tv;
  const int d = tv.d, m = a.m, G = gridDim.x, rank = blockIdx.x, L1 = tv.L + 1;
  const SmallSmem lay = small_smem(G, d, m, a.rows_max, a.tiles_max, tv.L, tv.zeta, a.slab);
  double* zx = reinterpret_cast<double*>(sraw + lay.zx);
  double* sx = reinterpret_cast<double*>(sraw + lay.sx);
  double* csc = reinterpret_cast<double*>(sraw + lay.csc);
  double* rp = reinterpret_cast<double*>(sraw + lay.rp);
  float2* zd = reinterpret_cast<float2*>(sraw + lay.zd);
  float2* sjd = reinterpret_cast<float2*>(sraw + lay.sjd);
  float2* acc = reinterpret_cast<float2*>(sraw + lay.acc);
  float2* v = reinterpret_cast<float2*>(sraw + lay.v);
  float2* r1 = reinterpret_cast<float2*>(sraw + lay.r1);
  float2* nrs = reinterpret_cast<float2*>(sraw + lay.nrs);
  float2* mcol = reinterpret_cast<float2*>(sraw + lay.mcol);
  uint16_t* es = reinterpret_cast<uint16_t*>(sraw + lay.es);
  uint32_t* ms = reinterpret_cast<uint32_t*>(sraw + lay.ms);
  int* of = reinterpret_cast<int*>(sraw + lay.of);
  float2* slab = reinterpret_cast<float2*>(sraw + lay.slab);
  float2* Ss = reinterpret_cast<float2*>(sraw + lay.S);
  float2* Ms = reinterpret_cast<float2*>(sraw + lay.M);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int NT = 512, NW = 16;
  const int t0 = tv.ctile[rank], t1 = tv.ctile[rank + 1];
  const int row0 = (int)tv.row[t0], rows = (int)tv.row[t1] - row0;
  for (int t = t0; t < t1; ++t) {
    const int r0 = (int)tv.row[t];
    tile_stage(tv, t, r0, (int)tv.row[t + 1] - r0, of + (t - t0) * L1, ms + (t - t0) * d,
               es + (size_t)(r0 - row0) * tv.zeta);
  }
  for (int c = tid; c <= a.c0; c += NT) csc[c] = a.colscale[c];
  if (a.slab)
    for (int c = warp; c <= a.c0; c += NW)
      for (int l = lane; l < rows; l += 32) slab[c * a.rows_max + l] = a.U[row0 + l + (int64_t)c * a.ldu];
  for (int t = tid; t < d * (a.c0 + 1); t += NT) Ss[t] = a.S2[t];
  for (int c = warp; c <= a.c0; c += NW)
    for (int l = lane; l <= a.c0; l += 32) Ms[l + c * (m + 1)] = a.M2[l + (size_t)c * a.ldm];
  // the CTA's Omega-sums of its rows' values in v, to every CTA's dst[rank]
  // (tiles last to first when rev: the update kernel's second half of the grid)
  auto sketch_out = [&](double* dst, bool rev) {
    for (int r = tid; r < d; r += NT) acc[r] = make_float2(0.f, 0.f);
    for (int q = 0; q < t1 - t0; ++q) {
      const int t = rev ? t1 - t0 - 1 - q : q;
      __syncthreads();
      tile_gather(d, tv.H, v + t * kTileRows, of + t * L1, ms + t * d, es + (size_t)t * kTileRows * tv.zeta, acc);
    }
    __syncthreads();
    for (int r = tid; r < d; r += NT) {
      const double x = df_to_double(acc[r]);
      const double* p = dst + (size_t)rank * d + r;
      for (int k = 0; k < G; ++k) cl_put(cl_addr(p, k), x);
    }
    cl_sync();
  };
  double zz = 0.0;                 // this thread's part of ||z||^2
  cl_sync();                       // every CTA runs before the first remote store
  for (int j = a.c0; j <= m; ++j) {
    const bool fin = j > a.c0;
    double inv = 0.0;
    if (fin) {                     // column j: beta_j = ||s~_j||, S, scale, coefficients
      double ss = 0.0;
      double sv[2] = {0.0, 0.0};   // this thread's entries r = tid, tid + 512 of s~ (d <= 1024)
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (tid + u * NT < d) sv[u] = fold16(sx + tid + u * NT, d, G) * a.zscale;
      // strands of 256 as in the least-squares kernel: entries through shared memory
      double* st = reinterpret_cast<double*>(acc);   // free until this step's sketches
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (tid + u * NT < d) st[tid + u * NT] = sv[u];
      __syncthreads();
      if (tid < 256)
        for (int r = tid; r < d; r += 256) { const double x = st[r]; ss = fma(x, x, ss); }
      // a warp's sums where it has entries (the others' are zeros); ||z||^2 of
      // the last step goes along.  Roots and quotients by thread 0 only (FP64
      // runs at two lanes a clock)
      if (warp < 8 && warp * 32 < d) {
        for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
      }
      if (warp * 32 < d) {
        for (int o = 16; o; o >>= 1) zz += __shfl_xor_sync(0xffffffffu, zz, o);
      }
      if (lane == 0) { red[warp] = warp < 8 && warp * 32 < d ? ss : 0.0; red[32 + warp] = warp * 32 < d ? zz : 0.0; }
      __syncthreads();
      if (warp == 0) {
        double x = lane < 8 ? red[lane] : 0.0, zq = lane < NW ? red[32 + lane] : 0.0;
        for (int o = 16; o; o >>= 1) {
          x += __shfl_xor_sync(0xffffffffu, x, o);
          zq += __shfl_xor_sync(0xffffffffu, zq, o);
        }
        if (lane == 0) {
          const double beta = sqrt(x);
          const bool finite = isfinite(beta), brk = finite && !(beta > 1e-14 * sqrt(zq));
          const double iv = (finite && !brk) ? 1.0 / beta : 0.0;
          red[60] = iv;
          csc[j] = iv;
          if (rank == 0) {
            a.coef[(size_t)(j - 1) * a.ldcoef + j] = beta;
            a.colscale[j] = iv;
            if (!finite) atomicOr(a.flag, RKS_FLAG_NAN);
            else if (brk) atomicOr(a.flag, RKS_FLAG_BREAKDOWN);
          }
        }
      }
      __syncthreads();
      inv = red[60];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int r = tid + u * NT;
        if (r < d) {
          const double x = sv[u] * inv;
          const float2 w = df_from_double(x);
          sjd[r] = w;
          Ss[r + j * d] = w;
          if (rank == 0) a.S64[r + (size_t)j * d] = x;
        }
      }
      if (rank == 0) {
        double* cc = a.coef + (size_t)(j - 1) * a.ldcoef;
        for (int i = tid; i < j; i += NT) cc[i] = rp[i];
      }
    }
    if (j == m) break;
    // w = A u~_j on the CTA's rows (u~_j was written by all CTAs: from L2)
    const float2* x = a.U + (int64_t)j * a.ldu;
    for (int l = tid; l < rows; l += NT) {
      const int i = row0 + l;
      float sh = 0.f, sl = 0.f;
      if (a.D > 0) {
        for (int e0 = 0; e0 < a.D; e0 += 4) {
          float2 av[4], xv[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int e = e0 + u, jx = e < a.D ? i + a.offs.o[e] : -1;
            const bool on = jx >= 0 && jx < a.n;
            av[u] = e < a.D ? a.dvals[e * a.ldd + i] : make_float2(0.f, 0.f);
            xv[u] = on ? __ldcg(x + jx) : make_float2(0.f, 0.f);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (e0 + u < a.D) df_mac(av[u].x, av[u].y, xv[u].x, xv[u].y, sh, sl);
        }
      } else {
        const int p1 = a.rowptr[i + 1];
#pragma unroll 4
        for (int p = a.rowptr[i]; p < p1; ++p) {
          const float2 av = a.vals[p], xv = __ldcg(x + a.colind[p]);
          df_mac(av.x, av.y, xv.x, xv.y, sh, sl);
        }
      }
      v[l] = df_norm(sh, sl);
    }
    __syncthreads();               // v complete, st (acc) read
    sketch_out(zx, false);
    // z = Omega w / beta_j, r1 = S^T z and the new row of M
    const double scj = fin ? inv : csc[j];
    zz = 0.0;
    for (int r = tid; r < d; r += NT) {
      const double q = fold16(zx + r, d, G) * a.zscale * scj;
      zz = fma(q, q, zz);
      zd[r] = df_from_double(q);
    }
    __syncthreads();
    for (int col = warp; col <= j; col += NW) {
      float s_ = 0.f, t_ = 0.f, g = 0.f, ge = 0.f;
      for (int r = lane; r < d; r += 32) {
        const float2 sc = fin && col == j ? sjd[r] : Ss[r + col * d], b = zd[r];
        df_mac(sc.x, sc.y, b.x, b.y, s_, t_);
        if (fin) { const float2 e = sjd[r]; df_mac(sc.x, sc.y, e.x, e.y, g, ge); }
      }
      df_warp_sum(s_, t_);
      if (fin) df_warp_sum(g, ge);
      if (lane == 0) {
        r1[col] = df_norm(s_, t_);
        if (fin) {
          const float2 mv = df_norm(g, ge);
          mcol[col] = mv;
          Ms[col + j * (m + 1)] = mv;
          Ms[j + col * (m + 1)] = mv;
        }
      }
    }
    __syncthreads();
    // r = 2 r1 - M r1, the update's coefficients
    for (int col = warp; col <= j; col += NW) {
      float s_ = 0.f, t_ = 0.f;
      for (int l = lane; l <= j; l += 32) {
        const float2 mv = fin && l == j ? mcol[col] : (fin && col == j ? mcol[l] : Ms[l + col * (m + 1)]), b = r1[l];
        df_mac(mv.x, mv.y, b.x, b.y, s_, t_);
      }
      df_warp_sum(s_, t_);
      if (lane == 0) {
        const float2 rc = r1[col];
        float hs = 2.f * rc.x, ht = 2.f * rc.y;   // exact doubling
        df_add(-s_, -t_, hs, ht);
        nrs[col] = df_norm(hs, ht);
      }
    }
    __syncthreads();
    for (int col = tid; col <= j; col += NT) {    // FP64 side by side, not one lane a warp
      const double rd = df_to_double(nrs[col]);
      rp[col] = rd;
      nrs[col] = df_from_double(-rd * (col == j ? scj : csc[col]));
    }
    const float2 sj = df_from_double(scj);
    __syncthreads();
    // u~ = w / beta_j - U b on the CTA's rows
    for (int l = tid; l < rows; l += NT) {
      const float2 w = v[l];
      float sh = 0.f, sl = 0.f;
      df_mac(w.x, w.y, sj.x, sj.y, sh, sl);
      if (a.slab) {
#pragma unroll 4
        for (int c = 0; c <= j; ++c) {
          const float2 u = slab[c * a.rows_max + l], r = nrs[c];
          df_mac(u.x, u.y, r.x, r.y, sh, sl);
        }
      } else {
        const float2* up = a.U + row0 + l;
        int c = 0;
        for (; c + 16 <= j + 1; c += 16) {
          float2 u[16];
#pragma unroll
          for (int q = 0; q < 16; ++q) u[q] = __ldcg(up + (int64_t)(c + q) * a.ldu);
#pragma unroll
          for (int q = 0; q < 16; ++q) df_mac(u[q].x, u[q].y, nrs[c + q].x, nrs[c + q].y, sh, sl);
        }
#pragma unroll 4
        for (; c <= j; ++c) {
          const float2 u = __ldcg(up + (int64_t)c * a.ldu), r = nrs[c];
          df_mac(u.x, u.y, r.x, r.y, sh, sl);
        }
      }
      const float2 u = df_norm(sh, sl);
      v[l] = u;
      if (a.slab) slab[(j + 1) * a.rows_max + l] = u;
      a.U[row0 + l + (int64_t)(j + 1) * a.ldu] = u;
    }
    __syncthreads();
    sketch_out(sx, rank >= G / 2);   // its barrier also orders u~'s rows before the next product
  }
}

// CTAs of the fused expansion (0: the separate kernels): a power of two with
// at least 64 rows each.  At most kSmallRows rows, and S, M and the partial
// sketches of all CTAs within one CTA's shared memory: read from L2 instead,
// they cost more than the launches saved (d = 320, 80 columns, 4900 rows: 60
// us a step against 57).
int small_expand_ctas(int64_t n, int d, int m, int zeta) {
  if (n > kSmallRows) return 0;
  int g = 1;
  while (g < 16 && n >= (int64_t)g * 128) g *= 2;
  const int rows = (int)((n + g - 1) / g) + 2;
  return small_smem(g, d, m, rows, 1, 512, zeta, 0).total <= 200 * 1024 ? g : 0;
}

bool launch_df_expand_small(const CsrDF& A, float2* U, int64_t ldu, int c0, int m, const SketchTiles& t, int rows_max,
                            int tiles_max, double zscale, double* S64, float2* S2, float2* M2, int ldm,
                            double* colscale, double* coef, int ldcoef, int* flag, cudaStream_t st) {
  if (t.d > 1024 || A.fmt == kSpmvMerge || A.fmt == kSpmvWarp || A.f32) return false;
  SmallArgs a;
  a.rowptr = A.rowptr; a.colind = A.colind; a.vals = static_cast<const float2*>(A.vals);
  a.dvals = static_cast<const float2*>(A.dvals);
  a.D = A.dvals ? A.D : 0;
  for (int e = 0; e < a.D; ++e) a.offs.o[e] = A.doff[e];
  a.ldd = A.ldd; a.n = (int)A.n; a.c0 = c0; a.m = m; a.U = U; a.ldu = ldu; a.tv = t; a.zscale = zscale;
  a.S64 = S64; a.S2 = S2; a.M2 = M2; a.colscale = colscale; a.coef = coef; a.ldcoef = ldcoef; a.ldm = ldm;
  a.flag = flag; a.rows_max = rows_max; a.tiles_max = tiles_max;
  a.slab = 1;
  auto bytes = [&]() { return small_smem(t.G, t.d, m, rows_max, tiles_max, t.L, t.zeta, a.slab).total; };
  if (bytes() > 200 * 1024) a.slab = 0;
  const size_t sm = bytes();
  if (sm > 200 * 1024) return false;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = t.G;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(t.G);
  cfg.blockDim = dim3(512);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, k_df_expand_small, a) == cudaSuccess) return true;
  (void)cudaGetLastError();     // no room for the cluster on this device: the separate kernels
  return false;
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

static int df_grid(int64_t n, int threads) {
  int64_t g = (n + threads - 1) / threads;
  const int cap = kDfCtas;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return (int)g;
}

static cudaError_t configure_df_kernels_once() {
  const int big = 200 * 1024;
  cudaError_t e = cudaSuccess;
#define RKS_SMEM(f) if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, big)
  RKS_SMEM((k_df_spmv_sketch<float2, float2, true>)); RKS_SMEM((k_df_spmv_sketch<float, float, true>));
  RKS_SMEM((k_df_spmv_sketch<float2, float2, false>));
  RKS_SMEM((k_df_spmv_ell<float2, float2, true, 0>)); RKS_SMEM((k_df_spmv_ell<float, float, true, 0>));
  RKS_SMEM((k_df_spmv_warp<float2, float2, true, 32>)); RKS_SMEM((k_df_spmv_warp<float, float, true, 32>));
  RKS_SMEM((k_df_spmv_warp<float2, float2, false, 32>)); RKS_SMEM((k_df_spmv_warp<float2, float2, true, 8>));
  RKS_SMEM((k_df_spmv_warp<float, float, true, 8>)); RKS_SMEM((k_df_spmv_warp<float2, float2, false, 8>));
  RKS_SMEM((k_df_spmv_dia<float2, float2, true, 8>)); RKS_SMEM((k_df_spmv_dia<float, float, true, 8>));
  RKS_SMEM((k_df_spmv_dia<float2, float2, true, 16>)); RKS_SMEM((k_df_spmv_dia<float, float, true, 16>));
  RKS_SMEM((k_df_spmv_dia<float2, float2, false, 8>)); RKS_SMEM((k_df_spmv_dia<float2, float2, false, 16>));
  RKS_SMEM((k_df_spmv_dia<float2, float, true, 8>)); RKS_SMEM((k_df_spmv_dia<float2, float, false, 8>));
  RKS_SMEM((k_df_spmv_dia<float2, float2, true, 8, 5>)); RKS_SMEM((k_df_spmv_dia<float2, float2, true, 8, 7>));
  RKS_SMEM((k_df_spmv_dia<float2, float2, false, 8, 5>)); RKS_SMEM((k_df_spmv_dia<float2, float2, false, 8, 7>));
  RKS_SMEM((k_df_spmv_dia<float2, float, true, 8, 5>)); RKS_SMEM((k_df_spmv_dia<float2, float, true, 8, 7>));
  RKS_SMEM((k_df_spmv_dia<float2, float, false, 8, 5>)); RKS_SMEM((k_df_spmv_dia<float2, float, false, 8, 7>));
  RKS_SMEM((k_df_spmv_dia<float, float, true, 8, 5>)); RKS_SMEM((k_df_spmv_dia<float, float, true, 8, 7>));
  RKS_SMEM((k_df_spmv_ell<float2, float2, false, 0>)); RKS_SMEM((k_df_spmv_ell<float2, float2, true, 6>));
  RKS_SMEM((k_df_spmv_ell<float, float, true, 6>)); RKS_SMEM((k_df_spmv_ell<float2, float2, false, 6>));
  constexpr int U8 = kDfUpdUnroll, MB = kDfUpdMinBlocks;
  RKS_SMEM((k_df_update_sketch<float2, U8, MB, 1>)); RKS_SMEM((k_df_update_sketch<float, 2 * U8, MB, 1>));
  RKS_SMEM((k_df_update_sketch<float2, U8, MB, 0>)); RKS_SMEM((k_df_update_sketch<float2, U8, MB, 2>));
  RKS_SMEM(k_df_sketch_vec<float2>); RKS_SMEM(k_df_sketch_vec<float>);
  RKS_SMEM(k_df_sketch_cols<float2>); RKS_SMEM(k_df_sketch_cols<double>); RKS_SMEM(k_df_panel);
  RKS_SMEM(k_tiles_count<4>); RKS_SMEM(k_tiles_count<8>); RKS_SMEM(k_tiles_count<16>);
  RKS_SMEM(k_tiles_build<4>); RKS_SMEM(k_tiles_build<8>); RKS_SMEM(k_tiles_build<16>);
  RKS_SMEM(k_df_ls1);
  RKS_SMEM(k_df_ls_coop);
  RKS_SMEM(k_df_expand_small);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_df_expand_small, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  RKS_SMEM(k_df_rows_gemm<float2>);
  RKS_SMEM(k_df_rows_gemm<float>);
  RKS_SMEM((k_df_restart<float2, 4>)); RKS_SMEM((k_df_restart<float2, 8>)); RKS_SMEM((k_df_restart<float2, 16>));
  RKS_SMEM((k_df_restart<float, 4>)); RKS_SMEM((k_df_restart<float, 8>)); RKS_SMEM((k_df_restart<float, 16>));
#undef RKS_SMEM
  return e;
}

cudaError_t configure_df_kernels() { return once_per_device(kCfgDf, configure_df_kernels_once); }

int df_small_smem(int d, int c) { return (int)((size_t)2 * d * sizeof(float2)); }
int df_gemm_smem(int nin, int nout) { return (int)(((size_t)nin * nout + (size_t)128 * nout) * sizeof(float2)); }

void launch_ell_fill(int64_t n, int W, const int32_t* rowptr, const int32_t* colind, const void* vals, bool f32,
                     int32_t* ecol, void* evals, cudaStream_t st) {
  const int g = df_grid((n + 31) / 32 * 32, 256);
  if (f32)
    k_ell_fill<float><<<g, 256, 0, st>>>(n, W, rowptr, colind, static_cast<const float*>(vals), ecol,
                                         static_cast<float*>(evals));
  else
    k_ell_fill<float2><<<g, 256, 0, st>>>(n, W, rowptr, colind, static_cast<const float2*>(vals), ecol,
                                          static_cast<float2*>(evals));
}

void launch_dia_fill(int64_t n, int D, const int* doff, int64_t ldd, const int32_t* rowptr, const int32_t* colind,
                     const void* vals, bool f32, void* dvals, cudaStream_t st) {
  DiaOffs o{};
  for (int e = 0; e < D && e < 16; ++e) o.o[e] = doff[e];
  const int g = df_grid(n, 256);
  cudaMemsetAsync(dvals, 0, (size_t)D * ldd * (f32 ? sizeof(float) : sizeof(float2)), st);
  if (f32)
    k_dia_fill<float><<<g, 256, 0, st>>>(n, o, D, ldd, rowptr, colind, static_cast<const float*>(vals),
                                         static_cast<float*>(dvals));
  else
    k_dia_fill<float2><<<g, 256, 0, st>>>(n, o, D, ldd, rowptr, colind, static_cast<const float2*>(vals),
                                          static_cast<float2*>(dvals));
}

template <class TU, bool SK>
static void launch_dia(const CsrDF& A, const void* x, void* w, const SketchTiles& t, double* part, size_t sm,
                       cudaStream_t st) {
  DiaOffs o{};
  for (int e = 0; e < A.D; ++e) o.o[e] = A.doff[e];
  o.lo = A.D ? A.doff[0] : 0;
  o.hi = A.D ? A.doff[A.D - 1] : 0;
  const TU* xx = static_cast<const TU*>(x);
  TU* ww = static_cast<TU*>(w);
  const TU* dv = static_cast<const TU*>(A.dvals);
  if (A.D > 8) {
    launch_pdl(k_df_spmv_dia<TU, TU, SK, 16>, t.G, 512, sm, st, o, A.D, dv, A.ldd, A.n, xx, ww, t, part);
    return;
  }
  // exact kernels for the 5- and 7-point stencils
  if constexpr (std::is_same<TU, float2>::value) {
    // double-float vectors: the FP32 copy of the diagonals when every value
    // of A is an FP32 number (the pairs' low words are zero: the same bits)
    if (A.dvals_f32) {
      auto k = A.D == 5 ? k_df_spmv_dia<float2, float, SK, 8, 5>
                        : A.D == 7 ? k_df_spmv_dia<float2, float, SK, 8, 7> : k_df_spmv_dia<float2, float, SK, 8>;
      launch_pdl(k, t.G, 512, sm, st, o, A.D, static_cast<const float*>(A.dvals_f32), A.ldd, A.n, xx, ww, t, part);
      return;
    }
  }
  auto k = A.D == 5 ? k_df_spmv_dia<TU, TU, SK, 8, 5>
                    : A.D == 7 ? k_df_spmv_dia<TU, TU, SK, 8, 7> : k_df_spmv_dia<TU, TU, SK, 8>;
  launch_pdl(k, t.G, 512, sm, st, o, A.D, dv, A.ldd, A.n, xx, ww, t, part);
}

// The merge-path partition of A (the first row of every CTA's range), once per
// matrix: it depends on the row pointers only.
void launch_merge_partition(const CsrDF& A, cudaStream_t st) {
  const int64_t nb = (A.mp_threads + kMergeCta - 1) / kMergeCta;
  k_merge_partition<<<df_grid(nb + 1, 256), 256, 0, st>>>(A.n, A.nnz, A.rowptr, nb, A.mp_part);
}

// merge path: w = A x (double-float partials folded), then rounded to FP32 (f32)
static void launch_merge(const CsrDF& A, const void* x, void* w, cudaStream_t st) {
  float2* wd = A.f32 ? A.mp_w : static_cast<float2*>(w);
  const int64_t nb = (A.mp_threads + kMergeCta - 1) / kMergeCta;
  const float2* x2 = A.f32 ? nullptr : static_cast<const float2*>(x);
  const float* x1 = A.f32 ? static_cast<const float*>(x) : nullptr;
  if (A.f32)
    k_df_spmv_merge<float><<<(unsigned)nb, kMergeCta, 0, st>>>(A.n, A.nnz, A.rowptr, A.colind,
                                                              static_cast<const float*>(A.vals), x2, x1, A.mp_part,
                                                              wd, A.mp_row, A.mp_val, A.mp_threads);
  else
    k_df_spmv_merge<float2><<<(unsigned)nb, kMergeCta, 0, st>>>(A.n, A.nnz, A.rowptr, A.colind,
                                                               static_cast<const float2*>(A.vals), x2, x1, A.mp_part,
                                                               wd, A.mp_row, A.mp_val, A.mp_threads);
  k_df_merge_fix<<<df_grid(nb, 256), 256, 0, st>>>(A.mp_row, A.mp_val, nb, wd);
  if (A.f32) k_df_round_f32<<<df_grid(A.n, 256), 256, 0, st>>>(A.n, wd, static_cast<float*>(w));
}

void launch_df_spmv_sketch(const CsrDF& A, const void* x, void* w, const SketchTiles& t, double* part,
                           cudaStream_t st) {
  const size_t sm = tile_smem_bytes(t.d, t.L, 0, t.zeta);
  if (A.fmt == kSpmvMerge) {
    launch_merge(A, x, w, st);
    launch_df_sketch_vec(w, t, part, A.f32, st);
    return;
  }
  if (A.fmt == kSpmvWarp) {
    const bool wide = A.nnz >= 64 * A.n;   // mean row length >= 64: a warp per row, else 8 lanes
    if (A.f32) {
      auto k = wide ? k_df_spmv_warp<float, float, true, 32> : k_df_spmv_warp<float, float, true, 8>;
      launch_pdl(k, t.G, 512, sm, st, A.rowptr, A.colind, static_cast<const float*>(A.vals), static_cast<const float*>(x),
                              static_cast<float*>(w), t, part);
    } else {
      auto k = wide ? k_df_spmv_warp<float2, float2, true, 32> : k_df_spmv_warp<float2, float2, true, 8>;
      launch_pdl(k, t.G, 512, sm, st, A.rowptr, A.colind, static_cast<const float2*>(A.vals), static_cast<const float2*>(x),
                              static_cast<float2*>(w), t, part);
    }
    return;
  }
  if (A.dvals) {
    if (A.f32) launch_dia<float, true>(A, x, w, t, part, sm, st);
    else launch_dia<float2, true>(A, x, w, t, part, sm, st);
    return;
  }
  if (A.ecol) {
    const bool narrow = A.W <= 6;
    if (A.f32) {
      auto k = narrow ? k_df_spmv_ell<float, float, true, 6> : k_df_spmv_ell<float, float, true, 0>;
      launch_pdl(k, t.G, 512, sm, st, A.ecol, static_cast<const float*>(A.evals), A.W, static_cast<const float*>(x),
                              static_cast<float*>(w), t, part);
    } else {
      auto k = narrow ? k_df_spmv_ell<float2, float2, true, 6> : k_df_spmv_ell<float2, float2, true, 0>;
      launch_pdl(k, t.G, 512, sm, st, A.ecol, static_cast<const float2*>(A.evals), A.W, static_cast<const float2*>(x),
                              static_cast<float2*>(w), t, part);
    }
    return;
  }
  if (A.f32)
    launch_pdl(
        k_df_spmv_sketch<float, float, true>, t.G, 512, sm, st, A.rowptr, A.colind, static_cast<const float*>(A.vals), static_cast<const float*>(x), static_cast<float*>(w),
        t, part);
  else
    launch_pdl(
        k_df_spmv_sketch<float2, float2, true>, t.G, 512, sm, st, A.rowptr, A.colind, static_cast<const float2*>(A.vals), static_cast<const float2*>(x),
        static_cast<float2*>(w), t, part);
}

void launch_df_spmv(const CsrDF& A, const void* x, void* w, const SketchTiles& t, cudaStream_t st) {
  const size_t sm = tile_smem_bytes(t.d, t.L, 0, t.zeta);
  if (A.fmt == kSpmvMerge && !A.f32) {
    launch_merge(A, x, w, st);
    return;
  }
  if (A.fmt == kSpmvWarp && !A.f32) {
    auto k = A.nnz >= 64 * A.n ? k_df_spmv_warp<float2, float2, false, 32> : k_df_spmv_warp<float2, float2, false, 8>;
    k<<<t.G, 512, sm, st>>>(A.rowptr, A.colind, static_cast<const float2*>(A.vals), static_cast<const float2*>(x),
                            static_cast<float2*>(w), t, nullptr);
    return;
  }
  if (A.dvals && !A.f32) {
    launch_dia<float2, false>(A, x, w, t, nullptr, sm, st);
    return;
  }
  if (A.ecol && !A.f32) {
    auto k = A.W <= 6 ? k_df_spmv_ell<float2, float2, false, 6> : k_df_spmv_ell<float2, float2, false, 0>;
    k<<<t.G, 512, sm, st>>>(A.ecol, static_cast<const float2*>(A.evals), A.W, static_cast<const float2*>(x),
                            static_cast<float2*>(w), t, nullptr);
    return;
  }
  k_df_spmv_sketch<float2, float2, false><<<t.G, 512, sm, st>>>(
      A.rowptr, A.colind, static_cast<const float2*>(A.vals), static_cast<const float2*>(x), static_cast<float2*>(w),
      t, nullptr);
}

void launch_df_update_plain(void* U, int64_t ldu, int c, const float2* nrs, const float2* sj, const SketchTiles& t,
                            double* norm_part, cudaStream_t st) {
  constexpr int U8 = kDfUpdUnroll, MB = kDfUpdMinBlocks;
  const size_t sm = tile_smem_bytes(t.d, t.L, c, t.zeta);
  float2* u = static_cast<float2*>(U);
  if (norm_part) k_df_update_sketch<float2, U8, MB, 2><<<t.G, 512, sm, st>>>(u, ldu, c, nrs, sj, t, norm_part);
  else k_df_update_sketch<float2, U8, MB, 0><<<t.G, 512, sm, st>>>(u, ldu, c, nrs, sj, t, nullptr);
}

void launch_df_fold(const double* part, int d, int G, double* out, cudaStream_t st, int nvec) {
  k_df_fold<<<dim3((d + 7) / 8, nvec), 256, 0, st>>>(part, d, G, out);
}

template <class TS>
static void sketch_cols_t(const TS* x, int64_t ldx, int ncols, float2* U, int64_t ldu, const SketchTiles& t,
                          double* part, cudaStream_t st) {
  const size_t fixed = (size_t)2 * kTileRows * sizeof(float2) + (size_t)kTileRows * t.zeta * sizeof(uint16_t) +
                       (size_t)(t.d + t.L + 2) * sizeof(int) + 16;
  // columns per CTA: as many accumulators as two CTAs per SM leave room for
  const size_t room = 100 * 1024 > fixed ? 100 * 1024 - fixed : 0;
  const int nc = (int)std::min<size_t>({(size_t)kSkCols, (size_t)ncols,
                                        std::max<size_t>(1, room / ((size_t)t.d * sizeof(float2)))});
  k_df_sketch_cols<TS><<<dim3(t.G, (ncols + nc - 1) / nc), 512, fixed + (size_t)nc * t.d * sizeof(float2), st>>>(
      x, ldx, ncols, nc, U, ldu, t, part);
}
void launch_df_sketch_cols(const float2* x, int64_t ldx, int ncols, const SketchTiles& t, double* part,
                           cudaStream_t st) {
  sketch_cols_t<float2>(x, ldx, ncols, nullptr, 0, t, part, st);
}
void launch_sketch_cols_f64(const double* x, int64_t ldx, int ncols, float2* U, int64_t ldu, const SketchTiles& t,
                            double* part, cudaStream_t st) {
  sketch_cols_t<double>(x, ldx, ncols, U, ldu, t, part, st);
}

void launch_df_panel(int64_t n, float2* U, int64_t ldu, int c0, int p0, int nb, const float2* coef, cudaStream_t st) {
  const int g = (int)std::min<int64_t>((n + 511) / 512, 152 * 2);
  k_df_panel<<<g, 256, (size_t)c0 * kSkCols * sizeof(float2), st>>>(n, U, ldu, c0, p0, nb, coef);
}

int gram_ctas(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>(152, (n + 1023) / 1024)); }
int gram_pairs(int s) { const int b = (s + 3) / 4; return b * (b + 1) / 2 * 16; }
void launch_df_gram(int64_t n, const float2* U, int64_t ldu, int s, double* part, cudaStream_t st) {
  const int npair = gram_pairs(s);
  k_df_gram<<<dim3(gram_ctas(n), npair / 16), 256, 0, st>>>(U, ldu, n, s, part, npair);
}

void launch_df_dots(const void* U, int64_t ldu, int c, int cv, const SketchTiles& t, double* part, cudaStream_t st) {
  k_df_dots<float2><<<t.G, 512, 0, st>>>(static_cast<const float2*>(U), ldu, c, cv, t, part);
}

void launch_ks_coef(int pass, int j, int c, int G, const double* part, const double* colscale, double* rprev,
                    float2* nrs, float2* sj, cudaStream_t st) {
  k_ks_coef<<<1, 256, 0, st>>>(pass, j, c, G, part, colscale, rprev, nrs, sj);
}

void launch_ks_finish(int j, int G, const double* part, double thr, double* colscale,
                      const double* rprev, double* coef, int ldcoef, int* flag, cudaStream_t st) {
  k_ks_finish<<<1, 32, 0, st>>>(j, G, part, thr, colscale, rprev, coef, ldcoef, flag);
}

void launch_df_update_sketch(void* U, int64_t ldu, int c, const float2* nrs, const float2* sj, const SketchTiles& t,
                             double* part, bool f32, cudaStream_t st) {
  constexpr int U8 = kDfUpdUnroll, MB = kDfUpdMinBlocks;
  const size_t sm = tile_smem_bytes(t.d, t.L, c, t.zeta);
  // FP32 basis: twice the columns per batch, so that a thread has as many
  // bytes of loads in flight as with pairs (same order of the sums)
  if (f32)
    launch_pdl(k_df_update_sketch<float, 2 * U8, MB, 1>, t.G, 512, sm, st, static_cast<float*>(U), ldu, c, nrs, sj, t,
               part);
  else
    launch_pdl(k_df_update_sketch<float2, U8, MB, 1>, t.G, 512, sm, st, static_cast<float2*>(U), ldu, c, nrs, sj, t,
               part);
}

int launch_df_small(int j, int d, double zscale, int finish, int ls, double* s_raw, double* z_raw, double* S64,
                    float2* S2, double* colscale, double* rprev, double* coef, int ldcoef, double* znorm_prev,
                    float2* nrs, float2* sj, float2* r1, float2* M2, int ldm, const double* part_z,
                    const double* part_s, int G, int* flag, unsigned* bar, cudaStream_t st, int stall) {
  const size_t sm = (size_t)2 * d * sizeof(float2);
  const size_t sm_coop = sm + (d <= kLsStageMax ? (size_t)2 * d * sizeof(double) : 0);
  const int c = j + 1;
  if (ls && bar) {
    // one cooperative launch: partial-sum fold, phases A and B, two grid
    // barriers; a warp per folded row (the fold's L2 latency dominates, so one
    // row per warp beats fewer CTAs with less barrier traffic)
    const int nb = finish ? 2 * d : d;
    int g = (std::max(c, nb) + 7) / 8;
    g = std::min(g, 96);
    // a small problem (less than one wave of sketch CTAs) shares the GPU with
    // other solves: fewer CTAs are easier to co-schedule for the cooperative
    // launch (the fold of a row is the same whichever warp does it)
    if (G < 152) g = std::min((std::max(c, d) + 7) / 8, 48);
    void* args[] = {&j, &d, &zscale, &finish, &s_raw, &z_raw, &S64, &S2, &colscale, &rprev, &coef, &ldcoef,
                    &znorm_prev, &nrs, &sj, &r1, &M2, &ldm, &part_z, &part_s, &G, &bar, &flag, &stall};
    if (cudaLaunchCooperativeKernel((const void*)k_df_ls_coop, dim3(g), dim3(256), args, sm_coop, st) == cudaSuccess)
      return 1;
    (void)cudaGetLastError();   // not available: fall back to the kernels below
  }
  const int gf = (d + 7) / 8;
  int nl = 0;
  if (finish) { k_df_fold<<<gf, 256, 0, st>>>(part_s, d, G, s_raw); ++nl; }
  if (ls) { k_df_fold<<<gf, 256, 0, st>>>(part_z, d, G, z_raw); ++nl; }
  const int g1 = ls ? (c + 7) / 8 : 1;
  k_df_ls1<<<g1, 256, sm, st>>>(j, d, zscale, finish, ls, s_raw, z_raw, S64, S2, colscale, rprev, coef, ldcoef,
                                znorm_prev, r1, M2, ldm, flag);
  if (!ls) return nl + 1;
  k_df_ls_gram<<<(c + 7) / 8, 256, 0, st>>>(j, M2, ldm, r1, colscale, rprev, nrs, sj);
  return nl + 2;
}

void launch_omega_table(int64_t n, int d, int zeta, uint64_t seed, uint16_t* tab, int* flag, cudaStream_t st) {
  const int g = df_grid(n, 256) * 4;
  if (zeta <= 4) k_omega_table<4><<<g, 256, 0, st>>>(n, d, zeta, seed, tab, flag);
  else if (zeta <= 8) k_omega_table<8><<<g, 256, 0, st>>>(n, d, zeta, seed, tab, flag);
  else k_omega_table<16><<<g, 256, 0, st>>>(n, d, zeta, seed, tab, flag);
}

int omega_slots(int zeta) { return zeta <= 4 ? 4 : (zeta <= 8 ? 8 : 16); }

void launch_sum_cols_f32(int64_t n, const float* U, int64_t ldu, int ncols, double* y, cudaStream_t st) {
  k_sum_cols_f32<<<df_grid(n, 256) * 2, 256, 0, st>>>(n, U, ldu, ncols, y);
}

void launch_d2df(int64_t n, const double* x, void* y, bool f32, cudaStream_t st) {
  if (f32) k_d2df<float><<<df_grid(n, 256) * 2, 256, 0, st>>>(n, x, static_cast<float*>(y));
  else k_d2df<float2><<<df_grid(n, 256) * 2, 256, 0, st>>>(n, x, static_cast<float2*>(y));
}

void launch_d2df_cols(int64_t n, const double* x, int64_t ldx, float2* y, int64_t ldy, int ncols, cudaStream_t st) {
  k_d2df_cols<<<dim3((unsigned)df_grid(n, 256), (unsigned)ncols), 256, 0, st>>>(n, x, ldx, y, ldy);
}

void launch_df2d_cols(int64_t n, const void* x, int64_t ldx, double* y, int64_t ldy, int ncols, bool f32,
                      cudaStream_t st) {
  dim3 grid((unsigned)df_grid(n, 256), (unsigned)ncols);
  if (f32) k_df2d_cols<float><<<grid, 256, 0, st>>>(n, static_cast<const float*>(x), ldx, y, ldy, ncols);
  else k_df2d_cols<float2><<<grid, 256, 0, st>>>(n, static_cast<const float2*>(x), ldx, y, ldy, ncols);
}

void launch_df_axpy_cols(int64_t n, float2* U, int64_t ldu, int src, int c0, int ncols, const float2* coef,
                         cudaStream_t st) {
  if (ncols <= 0) return;
  const int g = (int)std::min<int64_t>((n + 255) / 256, 152 * 8);
  k_df_axpy_cols<<<g, 256, 0, st>>>(n, U, ldu, src, c0, ncols, coef);
}

void launch_df_sketch_vec(const void* x, const SketchTiles& t, double* part, bool f32, cudaStream_t st) {
  const size_t sm = tile_smem_bytes(t.d, t.L, 0, t.zeta);
  if (f32) launch_pdl(k_df_sketch_vec<float>, t.G, 512, sm, st, static_cast<const float*>(x), t, part);
  else launch_pdl(k_df_sketch_vec<float2>, t.G, 512, sm, st, static_cast<const float2*>(x), t, part);
}

// Row ranges: G CTAs (at most kSketchCtas) own contiguous, even-aligned row
// ranges of equal length (to within two rows); each range is cut into tiles
// of at most kTileRows rows.  The partition depends on n (and ctas) only.
int build_sketch_tiles(int64_t n, int d, int zeta, const uint16_t* otab, SketchTiles* out, cudaStream_t st,
                       int ctas) {
  SketchTiles t;
  t.n = n; t.d = d; t.zeta = zeta;
  const int64_t npair = (n + 1) / 2;
  int64_t G = std::min<int64_t>(kSketchCtas, std::max<int64_t>(1, (n + kTileRows - 1) / kTileRows));
  if (ctas > 0) G = ctas;
  G = std::max<int64_t>(1, std::min(G, npair));
  std::vector<int> ctile(G + 1);
  std::vector<int64_t> row;
  for (int64_t g = 0; g < G; ++g) {
    const int64_t a = 2 * (g * npair / G), b = std::min<int64_t>(n, 2 * ((g + 1) * npair / G));
    ctile[g] = (int)row.size();
    for (int64_t r = a; r < b; r += kTileRows) row.push_back(r);
  }
  ctile[G] = (int)row.size();
  row.push_back(n);
  t.G = (int)G;
  for (int64_t g = 0; g < G; ++g) {
    t.tiles_max = std::max(t.tiles_max, ctile[g + 1] - ctile[g]);
    t.rows_max = std::max<int64_t>(t.rows_max, row[ctile[g + 1]] - row[ctile[g]]);
  }
  t.ntile = (int)row.size() - 1;
  t.H = 1;
  while (t.H < 8 && (int64_t)d * t.H * 2 <= 512) t.H *= 2;
  // two device blocks (row bounds, CTA bounds and the longest list; positions,
  // slot offsets and entries): an allocation costs about as much as the
  // kernels that fill them
  const size_t nrow = row.size(), nct = ctile.size();
  row.resize(nrow + (nct + 2) / 2, 0);                 // ctile and a zero behind the rows, in one copy
  std::copy(ctile.begin(), ctile.end(), reinterpret_cast<int*>(row.data() + nrow));
  cudaError_t e = cudaMalloc(&t.row, row.size() * sizeof(int64_t));
  t.ctile = reinterpret_cast<int*>(t.row + nrow);
  int* lmax = t.ctile + nct;
  if (e == cudaSuccess) e = cudaMemcpy(t.row, row.data(), row.size() * sizeof(int64_t), cudaMemcpyHostToDevice);
  const int slots = omega_slots(zeta);
  const size_t smc = (size_t)d * sizeof(int);
  if (e == cudaSuccess) {
    if (slots == 4) k_tiles_count<4><<<t.ntile, 256, smc, st>>>(t.row, d, otab, lmax);
    else if (slots == 8) k_tiles_count<8><<<t.ntile, 256, smc, st>>>(t.row, d, otab, lmax);
    else k_tiles_count<16><<<t.ntile, 256, smc, st>>>(t.row, d, otab, lmax);
    e = cudaGetLastError();
  }
  int L = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&L, lmax, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  t.L = L;
  auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const size_t bm = al((size_t)t.ntile * d * sizeof(uint32_t)), bo = al((size_t)t.ntile * (L + 1) * sizeof(int));
  if (e == cudaSuccess) e = cudaMalloc(&t.meta, bm + bo + (size_t)n * zeta * sizeof(uint16_t));
  if (e == cudaSuccess) {
    t.off = reinterpret_cast<int*>(reinterpret_cast<char*>(t.meta) + bm);
    t.ent = reinterpret_cast<uint16_t*>(reinterpret_cast<char*>(t.meta) + bm + bo);
  }
  const size_t smb = ((size_t)4 * d + L + 1) * sizeof(int);
  if (e == cudaSuccess) {
    if (slots == 4) k_tiles_build<4><<<t.ntile, 256, smb, st>>>(t.row, d, zeta, L, otab, t.meta, t.off, t.ent);
    else if (slots == 8) k_tiles_build<8><<<t.ntile, 256, smb, st>>>(t.row, d, zeta, L, otab, t.meta, t.off, t.ent);
    else k_tiles_build<16><<<t.ntile, 256, smb, st>>>(t.row, d, zeta, L, otab, t.meta, t.off, t.ent);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  *out = t;
  return (int)e;
}

void free_sketch_tiles(SketchTiles* t) {
  cudaFree(t->row);
  cudaFree(t->meta);
  *t = SketchTiles();
}

size_t sketch_tile_smem(const SketchTiles& t, int c) { return tile_smem_bytes(t.d, t.L, c, t.zeta); }

template <class TU>
static void restart_t(int64_t n, TU* U, int64_t ldu, int a0, int nin, const float2* Q, int nout, int c0,
                      int move_src, cudaStream_t st) {
  const size_t sm = (size_t)nin * nout * sizeof(float2);
  const int g = (int)((n + 63) / 64);
  const int per = (nout + 3) / 4;
  if (per <= 4) k_df_restart<TU, 4><<<g, 256, sm, st>>>(n, U, ldu, a0, nin, Q, nout, c0, move_src);
  else if (per <= 8) k_df_restart<TU, 8><<<g, 256, sm, st>>>(n, U, ldu, a0, nin, Q, nout, c0, move_src);
  else k_df_restart<TU, 16><<<g, 256, sm, st>>>(n, U, ldu, a0, nin, Q, nout, c0, move_src);
}

void launch_df_rows_gemm(int64_t n, void* U, int64_t ldu, int a0, int nin, const float2* Q, int nout, int c0,
                         int move_src, bool f32, cudaStream_t st) {
  if (nout <= 64) {        // register-tiled restart product
    if (f32) restart_t<float>(n, static_cast<float*>(U), ldu, a0, nin, Q, nout, c0, move_src, st);
    else restart_t<float2>(n, static_cast<float2*>(U), ldu, a0, nin, Q, nout, c0, move_src, st);
    return;
  }
  const size_t sm = (size_t)df_gemm_smem(nin, nout);
  const int g = (int)((n + 127) / 128);
  if (f32) k_df_rows_gemm<float><<<g, 128, sm, st>>>(n, static_cast<float*>(U), ldu, a0, nin, Q, nout, c0, move_src);
  else k_df_rows_gemm<float2><<<g, 128, sm, st>>>(n, static_cast<float2*>(U), ldu, a0, nin, Q, nout, c0, move_src);
}


void launch_f32_to_df_cols(int64_t n, const float* Uf, int64_t ldu, int ncols, float2* U2, cudaStream_t st) {
  k_f32_to_df_cols<<<df_grid((int64_t)ncols * ldu, 256), 256, 0, st>>>(n, Uf, ldu, ncols, U2);
}

void launch_relation_resid(int64_t n, const float2* w, const float2* v, const float2* u, double beta, float* e,
                           cudaStream_t st) {
  k_relation_resid<<<df_grid(n, 256), 256, 0, st>>>(n, w, v, u, beta, e);
}

void launch_diag_inv(int64_t n, const int32_t* rowptr, const int32_t* colind, const float* vals, float* dinv,
                     cudaStream_t st) {
  k_diag_inv<<<df_grid(n, 256), 256, 0, st>>>(n, rowptr, colind, vals, dinv);
}

int jacobi_sweep_ctas(int64_t n) { return (int)((n + kJacobiCta - 1) / kJacobiCta); }

void launch_jacobi_sweep(int64_t n, const int32_t* rowptr, const int32_t* colind, const float* vals,
                         const float* dinv, int kk, int64_t ld, const float* X, const float* E, const float* Y,
                         float omega, float* Xn, double* part, cudaStream_t st) {
  k_jacobi_sweep<<<jacobi_sweep_ctas(n), kJacobiCta, 0, st>>>(n, rowptr, colind, vals, dinv, kk, ld, X, E, Y, omega,
                                                              Xn, part);
}

void launch_df_add_f32_cols(int64_t n, float2* U2, int64_t ldu, int kk, const float* X, int64_t ldx,
                            cudaStream_t st) {
  k_df_add_f32_cols<<<df_grid((int64_t)kk * n, 256), 256, 0, st>>>(n, U2, ldu, kk, X, ldx);
}

}  // namespace rks
