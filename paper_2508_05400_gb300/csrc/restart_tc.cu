// Restart product U_k = U Q' (Eq. 3.5) of an FP32 basis on the fifth-generation
// tensor cores of sm_103a (tcgen05.mma, accumulators in tensor memory).
//
// Split-BF16: an FP32 value u is the exact sum u1 + u2 + u3 of three bf16
// numbers (u1 = bf16(u), u2 = bf16(u - u1), u3 = bf16(u - u1 - u2); each
// remainder is exact in FP32); Q' is split the same way on the host.  The
// product keeps the six terms u_i q_j with i + j <= 4 (the dropped ones are
// below 2^-32 |u| |q|); every bf16 x bf16 product is exact and the sums are
// FP32 in tensor memory, so the result has FP32-class accuracy.
//
// A CTA owns tiles of 128 rows; per tile the K dimension (the nin input
// columns, padded) streams through shared-memory stages of one K-step of 16
// columns: FP32 loads, coalesced along the rows, three K-steps ahead in
// registers, split into a K-major no-swizzle layout; 6 MMAs of 128 x N x 16
// per stage.  The epilogue reads the 128 x N FP32 accumulator with tcgen05.ld
// and writes the outputs; every read of a tile's rows precedes its writes, so
// the product may be formed in place.  All waits are bounded
// (RKS_FLAG_TIMEOUT).

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "rks_impl.h"

namespace rks {

namespace {

constexpr int kM = 128;           // rows per tile (MMA M)
constexpr int kKc = 32;           // Kp is padded to a multiple of this
constexpr int kThreads = 256;     // splitters of the FP32 product; one more warp issues the MMAs
constexpr int kF32All = kThreads + 32;
constexpr int kF32Stages = 3;
constexpr int kF32Split = kM * 16 * 2;      // bytes of one split of one stage (a K-step of 16 columns)
constexpr int kF32Stage = 3 * kF32Split;
constexpr int kTmemCols = 64;

// Byte offset of element (r, k) of a K-major, no-swizzle tile with `rows`
// rows: K sub-tiles of 16, each of rows/8 groups (stride SBO = 256 B) of two
// 8 x 16-byte core matrices along K (stride LBO = 128 B).
__host__ __device__ inline uint32_t canon_off(int r, int k, int rows) {
  return (uint32_t)((k >> 4) * rows * 32 + (r >> 3) * 256 + ((k >> 3) & 1) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Shared-memory matrix descriptor: start address, LBO, SBO (all >> 4),
// descriptor version 1 (bits 46-48), no swizzle.
__device__ __forceinline__ uint64_t sdesc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(256 >> 4) << 32) |
         (1ull << 46);
}

// Shared-memory matrix descriptor of a K-major, no-swizzle operand whose
// rows lie 16 bytes apart: SBO (next 8 rows) 128 bytes, LBO (next 8 columns) lbo.
__device__ __forceinline__ uint64_t sdesc_rows(uint32_t addr, uint32_t lbo) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(128 >> 4) << 32) |
         (1ull << 46);
}

// Instruction descriptor, kind::f16: D F32 (bits 4-5 = 1), A and B bf16
// (bits 7-9, 10-12 = 1), both K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__device__ __forceinline__ uint32_t idesc_bf16(int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kM >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void mma_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
               : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t mbar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred P1;\n\tmbarrier.try_wait.parity.shared::cta.b64 P1, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, P1;\n\t}\n"
      : "=r"(done)
      : "r"(mbar), "r"(parity)
      : "memory");
  return done != 0;
}
__device__ __noinline__ bool mbar_wait_slow(uint32_t mbar, uint32_t parity, int* flag) {
  const long long t0 = clock64();
  while (!mbar_try(mbar, parity)) {
    if (clock64() - t0 > 2000000000ll) {
      atomicOr(flag, RKS_FLAG_TIMEOUT);
      return false;
    }
  }
  return true;
}
// Bounded wait for the completion of the mbarrier phase with this parity.
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity, int* flag) {
  return mbar_try(mbar, parity) || mbar_wait_slow(mbar, parity, flag);
}

// Aligned instructions: all 32 lanes execute them together.  The lanes come
// here from bounded waits of their own and from stores guarded by the row, so
// they are brought together first.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  __syncwarp();
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(r[j]);
}

__device__ __forceinline__ uint32_t bf16_bits(__nv_bfloat16 h) { return (uint32_t)__bfloat16_as_ushort(h); }

__device__ __forceinline__ void two_sum_f(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// The six split products (i, j) with i + j <= 4, splits numbered 1..3 (0..2 here).
__host__ __device__ constexpr int pair_a(int p) { return p == 2 || p == 4 ? 1 : (p == 5 ? 2 : 0); }
__host__ __device__ constexpr int pair_b(int p) { return p == 1 || p == 4 ? 1 : (p == 3 ? 2 : 0); }

// out[i, o] = sum_l in[i, l] Q'[l, o] for i < n, o < nout; then, when mvsrc
// is given, mvdst[i] = mvsrc[i].  bimg: the three bf16 splits of Q' (Kp x N,
// zero padded) in the canonical layout, split j at byte j * Kp * N * 2.
//
// Warps 0..7 load and split (a thread one row and 8 of a K-step's 16 columns,
// three K-steps ahead, in three sets of registers taken in turn: a set copied
// to another would wait for its loads; one 16-byte store per split) and run
// the epilogue; warp 8 issues the MMAs.  Per stage: full (every splitter arrives)
// and empty (the MMA commit arrives), per tile: done and tfree.  A thread
// whose bounded wait gave up skips its later waits and otherwise goes on, so
// that every barrier keeps its count.
//
// 4 096 000 x 150 -> 51 columns: 1750 us with CTA barriers around every stage
// and one CTA per SM; 1529 us with the MMAs issued by a warp of their own and
// loads three steps ahead; 944 us (3.5 TB/s) with the CTAs an SM has room for
// (two here).  The MMAs of a tile are 60 of 128 x 64 x 16, a seventh of the
// tensor pipe; bound by the split's shared-memory traffic and loads in flight.
__global__ void __launch_bounds__(kF32All, 3) k_tc_restart_f32(int64_t n, const float* in, float* out, int64_t ldu,
                                                                int nin, int Kp, int N, int nout,
                                                                const uint4* __restrict__ bimg, const float* mvsrc,
                                                                float* mvdst, int* flag) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int bbytes = 3 * Kp * N * 2;
  uint8_t* sB = smem;
  uint8_t* sA = smem + ((bbytes + 1023) & ~1023);
  uint64_t* mbar = reinterpret_cast<uint64_t*>(sA + kF32Stages * kF32Stage);   // full[], empty[], done, tfree
  uint32_t* tslot = reinterpret_cast<uint32_t*>(mbar + 2 * kF32Stages + 2);
  const uint32_t full0 = smem_u32(mbar), empty0 = smem_u32(mbar + kF32Stages);
  const uint32_t done_b = smem_u32(mbar + 2 * kF32Stages), tfree_b = smem_u32(mbar + 2 * kF32Stages + 1);

  for (int t = tid; t < bbytes / 16; t += kF32All) reinterpret_cast<uint4*>(sB)[t] = bimg[t];
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int s = 0; s < 2 * kF32Stages + 2; ++s)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar + s)),
                   "r"(s < kF32Stages || s == 2 * kF32Stages + 1 ? kThreads : 1));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  fence_async_smem();
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tslot;
  const int nk = Kp / 16;
  const int64_t ntiles = (n + kM - 1) / kM;
  bool ok = true;

  if (warp == kThreads / 32) {
    // ---- MMA issuer
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16(N);
      const uint32_t sA32 = smem_u32(sA), sB32 = smem_u32(sB);
      int s = 0, tcount = 0;
      uint32_t ph = 0;
      for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++tcount) {
        if (tcount > 0 && ok) ok = mbar_wait(tfree_b, (uint32_t)((tcount - 1) & 1), flag);   // accumulator read
        fence_after();
        for (int ks = 0; ks < nk; ++ks) {
          if (ok) ok = mbar_wait(full0 + 8u * s, ph, flag);
          fence_after();
          if (ok) {
#pragma unroll
            for (int pr = 0; pr < 6; ++pr) {
              const uint64_t a = sdesc_rows(sA32 + s * kF32Stage + pair_a(pr) * kF32Split, 2048);
              const uint64_t b = sdesc(sB32 + pair_b(pr) * Kp * N * 2 + ks * N * 32);
              mma_bf16(tmem, a, b, idesc, (ks | pr) ? 1u : 0u);
            }
          }
          mma_commit(empty0 + 8u * s);
          if (ks == nk - 1) mma_commit(done_b);
          if (++s == kF32Stages) { s = 0; ph ^= 1u; }
        }
      }
      // every issued MMA has completed before the accumulator is freed: the
      // last commit made to each stage's barrier
      const int64_t g = (int64_t)tcount * nk;
      for (int q = 0; q < kF32Stages; ++q) {
        const int64_t c = (g - q + kF32Stages - 1) / kF32Stages;
        if (g > q && c > 0) (void)mbar_wait(empty0 + 8u * q, (uint32_t)((c - 1) & 1), flag);
      }
    }
    __syncwarp();
  } else {
    const int r = tid & (kM - 1), c8 = (tid >> 7) * 8;
    int s = 0, ks = 0, filled = 0;
    uint32_t ph = 1, dpar = 0;             // parity of empty[s]: the first round passes
    int64_t tile = blockIdx.x;
    // the 8 values (one row) of K-step pk of tile pt; then on to the next K-step
    int64_t pt = tile;
    int pk = 0;
    auto load8 = [&](float* v) {
      if (pt < ntiles) {
        const int64_t i = pt * kM + r;
        const int c = pk * 16 + c8;
        const float* p = in + (i < n ? i : n - 1) + (int64_t)c * ldu;
        if (c + 8 <= nin) {
#pragma unroll
          for (int u = 0; u < 8; ++u) v[u] = p[u * ldu];
        } else {
#pragma unroll
          for (int u = 0; u < 8; ++u) v[u] = c + u < nin ? p[u * ldu] : 0.f;
        }
      }
      if (++pk == nk) { pk = 0; pt += gridDim.x; }
    };
    // one K-step: its values to shared memory, then the loads of three
    // K-steps later into the same registers
    auto step = [&](float* v) {
      uint32_t w[3][4];
#pragma unroll
      for (int u = 0; u < 8; u += 2) {
        uint32_t p[3][2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float x = v[u + e];
          const __nv_bfloat16 a = __float2bfloat16_rn(x);
          const float r1 = x - __bfloat162float(a);
          const __nv_bfloat16 b = __float2bfloat16_rn(r1);
          const __nv_bfloat16 c = __float2bfloat16_rn(r1 - __bfloat162float(b));
          p[0][e] = bf16_bits(a);
          p[1][e] = bf16_bits(b);
          p[2][e] = bf16_bits(c);
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) w[q][u >> 1] = p[q][0] | (p[q][1] << 16);
      }
      load8(v);
      if (filled < kF32Stages) ++filled;
      else if (ok) ok = mbar_wait(empty0 + 8u * s, ph, flag);
      uint8_t* st = sA + s * kF32Stage + (c8 >> 3) * 2048 + r * 16;
#pragma unroll
      for (int q = 0; q < 3; ++q)
        *reinterpret_cast<uint4*>(st + q * kF32Split) = make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]);
      fence_async_smem();
      mbar_arrive(full0 + 8u * s);
      if (++s == kF32Stages) { s = 0; ph ^= 1u; }
      if (++ks < nk) return;
      // epilogue
      if (ok) ok = mbar_wait(done_b, dpar, flag);
      dpar ^= 1u;
      fence_after();
      const int q4 = warp & 3;
      const int64_t ir = tile * kM + q4 * 32 + lane;
      float mv = 0.f;
      if (mvsrc && warp < 4 && ir < n) mv = mvsrc[ir];
      for (int cg = warp >> 2; cg < N / 8; cg += 2) {
        float acc[8];
        tmem_ld8(tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(cg * 8), acc);
        if (ir < n) {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int o = cg * 8 + j;
            if (o < nout) out[ir + (int64_t)o * ldu] = acc[j];
          }
        }
      }
      if (mvsrc && warp < 4 && ir < n) mvdst[ir] = mv;
      fence_before();
      mbar_arrive(tfree_b);
      ks = 0;
      tile += gridDim.x;
    };
    float v0[8], v1[8], v2[8];
    load8(v0);
    load8(v1);
    load8(v2);
    while (true) {
      if (tile >= ntiles) break;
      step(v0);
      if (tile >= ntiles) break;
      step(v1);
      if (tile >= ntiles) break;
      step(v2);
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
}

// ---------------------------------------------------------------------------
// Double-float basis: exact split products (Ozaki-type) on the tensor cores
// ---------------------------------------------------------------------------
//
// A value v of row i is written, relative to the row scale 2^e_i
// (|v| < 2^(e_i - 1) for every input column, its column's power of two
// included), as the fixed-point integer V = round(v 2^(48 - e_i)) =
// sum_s d_s 2^(42 - 7s) with seven balanced digits |d_s| <= 64; Q' likewise
// per column with scale 2^f_o (digits c_t, built on the host).  Then
//   sum_l v_l q_l = 2^(e_i + f_o - 12) sum_g 2^(-7g) G_g,
//   G_g = sum_{s + t = g} sum_l d_s(i, l) c_t(l, o),
// with integer G_g.  The 34 digit pairs with s + t <= 7 go to 8 accumulators
// (8 x N tensor-memory columns); the dropped pairs are below 2^-50 of the
// scale.  The bf16 operand holds d_s + 192 (128 .. 256, exact), whose sum
// over l is 192 sum_l c_t(l, o) too large: a constant per group and output
// (corr, from the host) that the epilogue subtracts.  For K <= 192 every group
// of weight above 2^-35 stays below 5 * 192 * 256 * 64 < 2^24, so the
// bf16 MMAs with FP32 accumulation in tensor memory sum it exactly; a lighter
// group may round by a unit or two, far below 2^-48.
//
// The digits cost three FP32 adds each (|d_s| <= 64 holds as the low word of
// v, below 2^-5 of a unit when it enters, cannot push a digit over): with M_s = 2^(-7s) (1.5 2^23 +
// 0x4340), t = x + M_s rounds x to a multiple of 2^(-7s), and the low 16 bits
// of t are the bf16 pattern of d_s + 192; x - (t - M_s) is the exact rest.
// (Cutting a 64-bit integer and converting every digit took three times the
// instructions and bound the kernel.)  Slices of Q' lie side by side, so
// that one MMA multiplies a digit slice of U by all its slices of Q' (up to
// N = 256) where one MMA per pair re-read the U slice 34 times.
// K streams through two shared-memory stages of one K-step (16 input columns
// x 7 digit slices); Q' (7 slices, all K) stays resident.  The row exponents
// of a CTA's next tile are formed while the current one is processed, which
// also brings that tile into L2: HBM sees every input once.
// Measured, n = 1e6, 80 -> 21 columns: see launch_tc_restart_df.

constexpr int kDfDigits = 7;
constexpr int kDfThreads = 256;
constexpr int kDfGroups = 8;
constexpr int kDfStepSplit = kM * 16 * 2;                 // one digit slice of one K-step
constexpr int kDfStage = kDfDigits * kDfStepSplit;        // 28 KB

// What the split needs of a type.  Row exponents are kept biased and clamped
// to [4, 257], so that the row factor 2^(131 - emax) is a float; rows below or
// above lie outside what an FP32 pair resolves.
//   key / key_exp: running maximum over a row and its biased exponent
//   scaled:        v 2^p 2^(6 - e_i) as x + y (x the leading bits,
//                  |y| < 2^-22 |x|, |x| < 32)
template <class T>
struct Split;
template <>
struct Split<float2> {
  typedef float Key;     // |hi| 2^p
  typedef float Probe;   // what a row maximum reads of a value
  static __device__ __forceinline__ Probe probe(const float2* p) { return p->x; }
  static __device__ __forceinline__ Key key(Key k, Probe v, float col) { return fmaxf(k, fabsf(v * col)); }
  static __device__ __forceinline__ int key_exp(Key k) { return min(max((int)(__float_as_uint(k) >> 23), 4), 257); }
  static __device__ __forceinline__ int scale(int emax) { return emax - 125; }   // e_i
  static __device__ __forceinline__ float row(int emax) { return __int_as_float((131 - emax + 127) << 23); }
  static __device__ __forceinline__ void scaled(float2 v, float col, float rowf, float& x, float& y) {
    x = v.x * col * rowf;
    y = v.y * col * rowf;
  }
};
// The FP64 pipe is 60 times slower than the FP32 one, so a double is taken
// apart with integer operations: 24 leading bits, and 23 more rounded.  (No
// column factors: the FP64 product has none.)
template <>
struct Split<double> {
  typedef int Key;       // high word without the sign
  typedef int Probe;
  static __device__ __forceinline__ Probe probe(const double* p) { return reinterpret_cast<const int*>(p)[1]; }
  static __device__ __forceinline__ Key key(Key k, Probe v, float) { return max(k, v & 0x7FFFFFFF); }
  static __device__ __forceinline__ int key_exp(Key k) { return max(k >> 20, 1); }
  static __device__ __forceinline__ int scale(int emax) { return emax - 1021; }
  // k moves a high word to the row's scale; from x0 and y0 on, the moved word
  // gives x and y.  A zero or subnormal value (no leading one to move) lies
  // below x0 in every row: it counts as zero.
  struct Row { int k, x0, y0; };
  static __device__ __forceinline__ Row row(int emax) {
    const int k = (131 - emax) * (1 << 20), x0 = max(k, 0) + (1 << 20);
    return {k, x0, max(x0, 47 << 20)};
  }
  static __device__ __forceinline__ void scaled(double v, float, const Row& r, float& x, float& y) {
    const int hi = __double2hiint(v), lo = __double2loint(v);
    const int d = (hi & 0x7FFFFFFF) + r.k;                  // biased exponent of x, 20 bits of mantissa
    const int xb = __funnelshift_l(lo, d, 3), sg = hi & 0x80000000;
    const float yi = __int_as_float((((lo & 0x1FFFFFFF) + 32) >> 6) + 0x4B000000) - 8388608.0f;
    x = d >= r.x0 ? __int_as_float(xb | sg) : 0.f;
    y = d >= r.y0 ? yi * __int_as_float(((xb & 0x7F800000) - (46 << 23)) | sg) : 0.f;
  }
};

constexpr int kDfAllThreads = kDfThreads + 32;

// Host data of one product, in one device block: column exponents, input
// column powers of two, group corrections, then the digit image.
struct DfBlobHead {
  int fexp[64];
  int pexp[256];
  float corr[kDfGroups * 64];   // [group][output of N]
};
static_assert(sizeof(DfBlobHead) % 16 == 0, "the digit image follows, read in 16-byte pieces");

// out[i, o] = sum_l in[i, l] 2^pexp[l] Q'[l, o] for i < n, o < nout; then,
// when mvsrc is given, mvdst[i] = mvsrc[i].  Input and output in double-float
// or both in FP64.  Every read of a tile's rows precedes its writes (in
// place).
//
// Warp roles: warps 0..7 load and split the digits of one K-step into a
// shared-memory stage and run the epilogue; warp 8 issues the MMAs.  Per
// stage s: full[s] (every splitter arrives once its digits are stored) and
// empty[s] (the MMA commit arrives once they are consumed); per tile: done
// (accumulators complete) and tfree (the epilogue has read them).  Every wait
// is bounded (mbar_wait); a thread whose wait gave up skips its later waits
// and otherwise goes on, so that every barrier keeps its count.
template <class T, int MINB>
__global__ void __launch_bounds__(kDfAllThreads, MINB) k_tc_restart_df(int64_t n, const T* in, T* out, int64_t ldu,
                                                                       int nin, int Kp, int N, int nout,
                                                                       const DfBlobHead* __restrict__ head,
                                                                       const T* mvsrc, T* mvdst, int tcols,
                                                                       int* flag) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int bbytes = kDfDigits * Kp * N * 2;
  uint8_t* sB = smem;
  uint8_t* sA = smem + ((bbytes + 1023) & ~1023);
  uint64_t* mbar = reinterpret_cast<uint64_t*>(sA + 2 * kDfStage);   // full[2], empty[2], done, tfree
  uint32_t* tslot = reinterpret_cast<uint32_t*>(mbar + 6);
  float* colf = reinterpret_cast<float*>(mbar + 8);      // 2^pexp (Kp; the last column repeated)
  short* rowe = reinterpret_cast<short*>(colf + Kp);     // [tile parity][column half][row] largest exponents
  const uint32_t full0 = smem_u32(mbar + 0), empty0 = smem_u32(mbar + 2);
  const uint32_t done_b = smem_u32(mbar + 4), tfree_b = smem_u32(mbar + 5);
  const uint4* bimg = reinterpret_cast<const uint4*>(head + 1);

  for (int t = tid; t < bbytes / 16; t += kDfAllThreads) reinterpret_cast<uint4*>(sB)[t] = bimg[t];
  for (int t = tid; t < Kp; t += kDfAllThreads) colf[t] = __int_as_float((head->pexp[min(t, nin - 1)] + 127) << 23);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(tcols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int s = 0; s < 6; ++s)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar + s)), "r"(s < 2 || s == 5 ? kDfThreads : 1));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  fence_async_smem();
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tslot;
  const int nk = Kp / 16;
  const int64_t ntiles = (n + kM - 1) / kM;
  bool ok = true;

  if (warp == kDfThreads / 32) {
    // ---- MMA issuer (lane 0 of warp 8)
    if (lane == 0) {
      const uint32_t sA32 = smem_u32(sA), sB32 = smem_u32(sB);
      const uint32_t blbo = (uint32_t)(kDfDigits * N * 16);
      const int per = 256 / N;                           // slices of Q' in one MMA
      int g = 0, tcount = 0;
      for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++tcount) {
        if (tcount > 0 && ok) ok = mbar_wait(tfree_b, (uint32_t)((tcount - 1) & 1), flag);   // accumulators read
        fence_after();
        for (int kc = 0; kc < nk; ++kc, ++g) {
          const int s = g & 1;
          if (ok) ok = mbar_wait(full0 + 8u * s, (uint32_t)((g >> 1) & 1), flag);
          fence_after();
          if (ok) {
            const uint32_t b0 = sB32 + (uint32_t)kc * 2u * blbo;
            for (int sa = 0; sa < kDfDigits; ++sa) {
              const uint64_t a = sdesc_rows(sA32 + s * kDfStage + sa * kDfStepSplit, 2048);
              const int t1 = sa <= 1 ? kDfDigits : kDfGroups - sa;   // slices 0 .. t1 - 1: groups sa .. sa + t1 - 1
              for (int t = 0; t < t1;) {
                // the first K-step clears the accumulators: groups 0 .. 6 with
                // digit 0, group 7 with its first pair (digit 1, slice 6)
                const bool last7 = kc == 0 && sa == 1 && t == kDfDigits - 1;
                int cnt = min(per, t1 - t);
                if (kc == 0 && sa == 1 && !last7) cnt = min(cnt, kDfDigits - 1 - t);
                mma_bf16(tmem + (uint32_t)((sa + t) * N), a, sdesc_rows(b0 + (uint32_t)(t * N * 16), blbo),
                         idesc_bf16(cnt * N), (kc == 0 && (sa == 0 || last7)) ? 0u : 1u);
                t += cnt;
              }
            }
          }
          mma_commit(empty0 + 8u * s);
          if (kc == nk - 1) mma_commit(done_b);
        }
      }
      // every issued MMA has completed before the accumulators are freed
      if (g > 0) (void)mbar_wait(empty0 + 8u * ((g - 1) & 1), (uint32_t)(((g - 1) >> 1) & 1), flag);
      if (g > 1) (void)mbar_wait(empty0 + 8u * ((g - 2) & 1), (uint32_t)(((g - 2) >> 1) & 1), flag);
    }
    __syncwarp();
  } else {
    // ---- splitters (warps 0..7) and the epilogue
    int g = 0;                 // stages filled so far (all tiles)
    uint32_t tpar = 0;         // parity of the tile (accumulator-done barrier, row exponents)
    // a thread has one row and 8 of the 16 columns: one 16-byte store per digit
    const int r = tid & (kM - 1), c8 = (tid >> 7) * 8;
    // Rows past n and columns past nin repeat the last one: their outputs are
    // not stored, their rows of Q' are zero.
    typedef Split<T> S;
    auto row_ptr = [&](int64_t tile) {
      const int64_t i = tile * kM + r;
      return in + (i < n ? i : n - 1);
    };
    auto col_off = [&](int c, int u) { return (int64_t)min(c + u, nin - 1) * ldu; };
    auto put_rowe = [&](uint32_t par, typename S::Key key) {
      rowe[(par * 2 + (c8 >> 3)) * kM + r] = (short)S::key_exp(key);
    };
    {
      typename S::Key key = 0;
      const T* p0 = row_ptr(blockIdx.x);
#pragma unroll 2
      for (int kc = 0; kc < nk; ++kc) {
        const int c = kc * 16 + c8;
        typename S::Probe pm[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) pm[u] = S::probe(p0 + col_off(c, u));
#pragma unroll
        for (int u = 0; u < 8; ++u) key = S::key(key, pm[u], colf[c + u]);
      }
      put_rowe(0, key);
    }
    T v[8], vn[8];             // the next K-step's values are loaded during this one's split
    const T* pv = row_ptr(blockIdx.x);
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = pv[col_off(c8, u)];
    asm volatile("bar.sync 1, %0;" ::"n"(kDfThreads) : "memory");
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, tpar ^= 1u) {
      const short* re = rowe + tpar * 2 * kM;
      const auto rowf = S::row(max((int)re[r], (int)re[kM + r]));
      const bool more = tile + gridDim.x < ntiles;
      const T* pnext = row_ptr(more ? tile + gridDim.x : tile);
      typename S::Key key = 0;   // the next tile's row maximum, its loads consumed one K-step later
      typename S::Probe pm[8];
      for (int kc = 0; kc < nk; ++kc, ++g) {
        const int s = g & 1;
        const int c = kc * 16 + c8;
        const int cn = kc + 1 < nk ? c + 16 : c8;
        const T* ps = kc + 1 < nk ? pv : pnext;
        if (cn + 8 <= nin) {
          ps += (int64_t)cn * ldu;
#pragma unroll
          for (int u = 0; u < 8; ++u) vn[u] = ps[u * ldu];
        } else {
#pragma unroll
          for (int u = 0; u < 8; ++u) vn[u] = ps[col_off(cn, u)];
        }
        if (kc > 0) {
#pragma unroll
          for (int u = 0; u < 8; ++u) key = S::key(key, pm[u], colf[c - 16 + u]);
        }
        if (more) {
          if (c + 8 <= nin) {
            const T* pp = pnext + (int64_t)c * ldu;
#pragma unroll
            for (int u = 0; u < 8; ++u) pm[u] = S::probe(pp + u * ldu);
          } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) pm[u] = S::probe(pnext + col_off(c, u));
          }
        }
        // digits of 8 values of one row
        uint32_t w[kDfDigits][4];
#pragma unroll
        for (int u = 0; u < 8; u += 2) {
          float x[2], y[2];
          S::scaled(v[u], colf[c + u], rowf, x[0], y[0]);
          S::scaled(v[u + 1], colf[c + u + 1], rowf, x[1], y[1]);
#pragma unroll
          for (int d = 0; d < kDfDigits; ++d) {
            const float m = __int_as_float(0x4B404340 - ((7 * d) << 23));
            uint32_t b[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              // the low word enters in two parts, each far below a unit of its digit
              if (d == 2) {
                const float z = x[e] + y[e];
                y[e] -= z - x[e];
                x[e] = z;
              }
              if (d == 4) x[e] += y[e];
              const float t = x[e] + m;
              b[e] = __float_as_uint(t);
              x[e] -= t - m;
            }
            w[d][u >> 1] = __byte_perm(b[0], b[1], 0x5410);
          }
        }
        if (ok && g >= 2) ok = mbar_wait(empty0 + 8u * s, (uint32_t)(((g - 2) >> 1) & 1), flag);
        uint8_t* st = sA + s * kDfStage + (c8 >> 3) * 2048 + r * 16;
#pragma unroll
        for (int d = 0; d < kDfDigits; ++d)
          *reinterpret_cast<uint4*>(st + d * kDfStepSplit) = make_uint4(w[d][0], w[d][1], w[d][2], w[d][3]);
        fence_async_smem();
        mbar_arrive(full0 + 8u * s);
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = vn[u];
      }
      pv = pnext;
      if (more) {
#pragma unroll
        for (int u = 0; u < 8; ++u) key = S::key(key, pm[u], colf[(nk - 1) * 16 + c8 + u]);
        put_rowe(tpar ^ 1u, key);
      }
      // epilogue: sum_g 2^(-7g) (G_g - corr_g), times 2^(e_i + f_o - 12)
      if (ok) ok = mbar_wait(done_b, tpar, flag);
      fence_after();
      const int q4 = warp & 3;
      const int64_t ir = tile * kM + q4 * 32 + lane;
      const int em = max((int)re[q4 * 32 + lane], (int)re[kM + q4 * 32 + lane]);
      const int er = S::scale(em) - 12;
      T mv{};
      if (mvsrc && warp < 4 && ir < n) mv = mvsrc[ir];
      for (int cg = warp >> 2; cg < N / 8; cg += kDfThreads / 128) {
        const uint32_t tc = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(cg * 8);
        const float* co = head->corr + cg * 8;
        if constexpr (sizeof(T) == 8 && !std::is_same<T, double>::value) {
          float hs[8], ls[8];
          for (int gg = kDfGroups - 1; gg >= 0; --gg) {
            float gv[8];
            tmem_ld8(tc + (uint32_t)(gg * N), gv);
            const float4 ca = __ldg(reinterpret_cast<const float4*>(co + gg * N));
            const float4 cb = __ldg(reinterpret_cast<const float4*>(co + gg * N) + 1);
            const float cc[8] = {ca.x, ca.y, ca.z, ca.w, cb.x, cb.y, cb.z, cb.w};
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) {
              const float a = gv[jj] - cc[jj];
              if (gg == kDfGroups - 1) {
                hs[jj] = a;
                ls[jj] = 0.f;
              } else {
                const float sh = hs[jj] * 0.0078125f, sl = ls[jj] * 0.0078125f;   // exact scaling by 2^-7
                float s2, e2;
                two_sum_f(a, sh, s2, e2);
                hs[jj] = s2;
                ls[jj] = e2 + sl;
              }
            }
          }
          if (ir < n) {
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) {
              const int o = cg * 8 + jj;
              if (o < nout) {
                const int sc = er + head->fexp[o];
                float hh, ll;
                two_sum_f(hs[jj], ls[jj], hh, ll);
                out[ir + (int64_t)o * ldu] = make_float2(ldexpf(hh, sc), ldexpf(ll, sc));
              }
            }
          }
        } else {
          // FP64: the groups as one 64-bit integer (group 7 rounded to a unit
          // of group 6), converted once
          long long acc[8], top[8];
#pragma unroll
          for (int gg = kDfGroups - 1; gg >= 0; --gg) {
            float gv[8];
            tmem_ld8(tc + (uint32_t)(gg * N), gv);
            const float4 ca = __ldg(reinterpret_cast<const float4*>(co + gg * N));
            const float4 cb = __ldg(reinterpret_cast<const float4*>(co + gg * N) + 1);
            const float cc[8] = {ca.x, ca.y, ca.z, ca.w, cb.x, cb.y, cb.z, cb.w};
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) {
              const float a = gv[jj] - cc[jj];
              if (gg == kDfGroups - 1) acc[jj] = __float2int_rn(a * 0.0078125f);
              else if (gg >= 2) acc[jj] += (long long)__float2int_rn(a) * (1ll << (7 * (kDfGroups - 2 - gg)));
              else if (gg == 1) top[jj] = __float2int_rn(a);
              else acc[jj] += (top[jj] + ((long long)__float2int_rn(a) << 7)) << 35;
            }
          }
          if (ir < n) {
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) {
              const int o = cg * 8 + jj;
              if (o < nout) {
                const int sc = er + head->fexp[o] - 42;
                const double d = __ll2double_rn(acc[jj]);
                const int hi = __double2hiint(d), e = ((hi >> 20) & 0x7FF) + sc;
                // scaling by an exponent add where the result is a normal number;
                // a row with an infinity or a NaN has no digits to add up
                out[ir + (int64_t)o * ldu] = em == 0x7FF             ? __hiloint2double(0x7FF80000, 0)
                                             : (hi & 0x7FF00000) == 0 ? d
                                             : e > 0 && e < 0x7FF   ? __hiloint2double(hi + (sc << 20), __double2loint(d))
                                                                    : scalbn(d, sc);
              }
            }
          }
        }
      }
      if (mvsrc && warp < 4 && ir < n) mvdst[ir] = mv;
      fence_before();
      mbar_arrive(tfree_b);
      __syncwarp();
      asm volatile("bar.sync 1, %0;" ::"n"(kDfThreads) : "memory");   // the next tile's row exponents
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tcols));
}

uint16_t host_bf16(float x) {   // round to nearest even (finite inputs)
  uint32_t u;
  std::memcpy(&u, &x, 4);
  u += 0x7FFFu + ((u >> 16) & 1u);
  return (uint16_t)(u >> 16);
}

double host_bf16_value(uint16_t h) {
  uint32_t u = (uint32_t)h << 16;
  float f;
  std::memcpy(&f, &u, 4);
  return (double)f;
}

}  // namespace

bool tc_restart_supported(int nin, int nout) { return nin >= 1 && nin <= 256 && nout >= 1 && nout <= 64; }

size_t tc_restart_smem(int nin, int nout) {
  const int Kp = (nin + kKc - 1) / kKc * kKc, N = (nout + 15) / 16 * 16;
  return (size_t)((3 * Kp * N * 2 + 1023) & ~1023) + kF32Stages * kF32Stage + 128;
}

// Host image of the three bf16 splits of Q (nin x nout, column-major FP64).
void tc_restart_bimage(int nin, int nout, const double* Q, std::vector<uint16_t>& img) {
  const int Kp = (nin + kKc - 1) / kKc * kKc, N = (nout + 15) / 16 * 16;
  img.assign((size_t)3 * Kp * N, 0);
  for (int o = 0; o < nout; ++o)
    for (int l = 0; l < nin; ++l) {
      double rem = Q[l + (size_t)o * nin];
      for (int s = 0; s < 3; ++s) {
        const uint16_t h = host_bf16((float)rem);
        rem -= host_bf16_value(h);
        img[(size_t)s * Kp * N + canon_off(o, l, N) / 2] = h;
      }
    }
}

// ---- double-float basis ----

static int df_kp(int nin) { return (nin + 15) / 16 * 16; }
static int df_n(int nout) { return (nout + 15) / 16 * 16; }

size_t tc_restart_df_smem(int nin, int nout) {
  const size_t b = (size_t)kDfDigits * df_kp(nin) * df_n(nout) * 2;
  return ((b + 1023) & ~(size_t)1023) + 2 * kDfStage + 64 + (size_t)df_kp(nin) * sizeof(float) +
         (size_t)4 * kM * sizeof(short);
}

bool tc_restart_df_supported(int nin, int nout) {
  return nin >= 1 && nin <= 192 && nout >= 1 && nout <= 64 && tc_restart_df_smem(nin, nout) <= kTcDfSmemMax;
}

// The block a product reads (DfBlobHead, then the digit image of Q, nin x
// nout column-major FP64): |Q[:, o]| < 2^(f_o - 1), W = round(Q 2^(48 - f_o))
// = sum_t c_t 2^(42 - 7t) with balanced digits -64 <= c_t < 64 (t > 0); slice
// t, column l, output o at K-step l / 16: [(l / 8) % 2][t N + o][l % 8].
// pexp: the input columns' powers of two (nullptr: zero).
static_assert(sizeof(DfBlobHead) + (size_t)kDfDigits * 256 * 64 * 2 <= kTcDfBlobBytes, "largest block");
void tc_restart_df_blob(int nin, int nout, const double* Q, const int* pexp, std::vector<uint8_t>& blob) {
  const int Kp = df_kp(nin), N = df_n(nout);
  blob.assign(sizeof(DfBlobHead) + (size_t)kDfDigits * Kp * N * 2, 0);
  DfBlobHead* hd = reinterpret_cast<DfBlobHead*>(blob.data());
  uint16_t* img = reinterpret_cast<uint16_t*>(hd + 1);
  for (int l = 0; l < nin; ++l) hd->pexp[l] = pexp ? pexp[l] : 0;      // -126 .. 126
  for (int o = 0; o < nout; ++o) {
    double mx = 0.0;
    for (int l = 0; l < nin; ++l) mx = std::max(mx, std::fabs(Q[l + (size_t)o * nin]));
    int E2 = 0;
    if (mx > 0.0) std::frexp(mx, &E2);          // mx < 2^E2
    const int f = E2 + 1;
    hd->fexp[o] = f;
    int csum[kDfDigits] = {};
    for (int l = 0; l < nin; ++l) {
      int64_t W = std::llround(std::ldexp(Q[l + (size_t)o * nin], 48 - f));
      for (int t = kDfDigits - 1; t >= 0; --t) {
        const int dgt = t == 0 ? (int)W : (int)(((W + 64) & 127) - 64);
        W = (W - dgt) >> 7;
        csum[t] += dgt;
        img[((size_t)((l >> 4) * 2 + ((l >> 3) & 1)) * kDfDigits * N + (size_t)t * N + o) * 8 + (l & 7)] =
            host_bf16((float)dgt);
      }
    }
    for (int g = 0; g < kDfGroups; ++g) {
      int c = 0;
      for (int t = std::max(0, g - kDfDigits + 1); t <= std::min(g, kDfDigits - 1); ++t) c += csum[t];
      hd->corr[g * N + o] = 192.0f * (float)c;
    }
  }
}

// Two CTAs per SM where the tensor memory holds both (N <= 32) and the
// shared memory too, else one with all its registers.  Measured on the
// GB300, n = 1e6, 80 -> 21 columns (808 MB, 0.12 ms at the copy rate):
// FP64 in and out
// 1.44 ms (with its conversion passes) -> 0.36 ms, bound by the digit split
// (issue 60%, tensor pipe 20%); the whole rks_basis_product_df call 2.52 ->
// 0.42 ms (no allocations, no double-float copies).  A 512-thread form with
// four columns per thread and one store of 8 bytes per digit took 0.56 ms.
template <class T>
static void launch_df_t(int64_t n, const T* in, T* out, int64_t ldu, int nin, int nout, const void* blob,
                        const T* mvsrc, T* mvdst, int* flag, cudaStream_t st) {
  const int Kp = df_kp(nin), N = df_n(nout);
  int tcols = 32;
  while (tcols < kDfGroups * N) tcols *= 2;
  const int64_t ntiles = (n + kM - 1) / kM;
  const size_t sm = tc_restart_df_smem(nin, nout);
  int sms = 152, dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const bool two = tcols <= 256 && 2 * (sm + 1024) <= 228 * 1024;
  const int g = (int)std::min<int64_t>(ntiles, (int64_t)sms * (two ? 2 : 1));
  const DfBlobHead* hd = static_cast<const DfBlobHead*>(blob);
  if (two)
    k_tc_restart_df<T, 2><<<g, kDfAllThreads, sm, st>>>(n, in, out, ldu, nin, Kp, N, nout, hd, mvsrc, mvdst, tcols, flag);
  else
    k_tc_restart_df<T, 1><<<g, kDfAllThreads, sm, st>>>(n, in, out, ldu, nin, Kp, N, nout, hd, mvsrc, mvdst, tcols, flag);
}

void launch_tc_restart_df(int64_t n, const float2* in, float2* out, int64_t ldu, int nin, int nout, const void* blob,
                          const float2* mvsrc, float2* mvdst, int* flag, cudaStream_t st) {
  launch_df_t<float2>(n, in, out, ldu, nin, nout, blob, mvsrc, mvdst, flag, st);
}

void launch_tc_product_f64(int64_t n, const double* in, double* out, int64_t ldu, int nin, int nout, const void* blob,
                           int* flag, cudaStream_t st) {
  launch_df_t<double>(n, in, out, ldu, nin, nout, blob, nullptr, nullptr, flag, st);
}

static cudaError_t configure_tc_kernels_once() {
  cudaError_t e = cudaFuncSetAttribute(k_tc_restart_f32, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  const int df = (int)kTcDfSmemMax;
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_tc_restart_df<float2, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, df);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_tc_restart_df<float2, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, df);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_tc_restart_df<double, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, df);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_tc_restart_df<double, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, df);
  return e;
}

cudaError_t configure_tc_kernels() { return once_per_device(kCfgTc, configure_tc_kernels_once); }

void launch_tc_restart_f32(int64_t n, const float* in, float* out, int64_t ldu, int nin, int nout, const void* bimg,
                           const float* mvsrc, float* mvdst, int* flag, cudaStream_t st) {
  const int Kp = (nin + kKc - 1) / kKc * kKc, N = (nout + 15) / 16 * 16;
  const int64_t ntiles = (n + kM - 1) / kM;
  const size_t sm = tc_restart_smem(nin, nout);
  int sms = 152, dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // CTAs an SM holds: three by registers, the rest by shared memory (the
  // occupancy query counts one for a kernel that allocates tensor memory)
  const int per_sm = (int)std::min<size_t>(3, std::max<size_t>(1, (size_t)228 * 1024 / (sm + 1024)));
  const int g = (int)std::min<int64_t>(ntiles, (int64_t)sms * per_sm);
  k_tc_restart_f32<<<g, kF32All, sm, st>>>(n, in, out, ldu, nin, Kp, N, nout, static_cast<const uint4*>(bimg), mvsrc,
                                           mvdst, flag);
}

}  // namespace rks
