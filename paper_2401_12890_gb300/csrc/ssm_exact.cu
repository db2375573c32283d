// Data projections (Algorithm 2, step 4) as one matrix product with FP64-grade accuracy on
// the tcgen05 tensor cores:
//     out[i][n] = fl32( sum_p A[i][p] m[p][n] ),   A formed in FP64 once per plan
// (low-rank forms: A = rows sigma_i u_i^T, out = S; full-rank forms and Algorithm 1:
// A = (K^T K + beta I)^{-1} K^T, out = h = M g).
//
// Method: error-free slicing into short integers (the splitting of Ozaki, Ogita, Oishi and
// Rump, "Error-free transformations of matrix multiplication", 2012). Every row of A and
// every column of m is scaled by a power of two so that its entries lie in [-1, 1] and cut
// into S slices of 8 bits (slice k a multiple of 2^(-7-8k), |slice| <= 128 units, exact in
// BF16; what is left is at most 2^(-8S)). A product of slices i and j is a 14-bit integer in
// units of 2^(-14-8(i+j)). The products with i + j < S go to one FP32 accumulator per level
// i + j, drained into a 64-bit integer sum that is rounded to FP32 once. What is dropped is
// below (S + 1 + 2^-5) 2^(-8S) of the row's and the column's scale per term, so P times that
// per sum, whatever the size of the terms.
//
// Low-rank forms (S rows, at most 64): S = 7 and a second look, so that the results are those
// of an FP64 accumulation, which S_i had before. 256 entries between drains: level 0 stays
// within 2^22 units and levels up to 3 within 2^24, exact in FP32. A higher level is exact
// unless a partial sum passes 2^24, from where the rest of 256 entries cannot bring it back
// below 2^22. A result is taken if every level above 0 stayed below 2^22 and it is at least
// P 2^-27 of the scales: then it is within 2^-26 of its own size of the exact sum before its
// rounding to FP32. Every other one (a sum that cancels, an outlier in the row and another in
// the column at different p, a column with a NaN or an infinity) is formed again in FP64 from
// the operand itself: at most 3 in 10,000 on data with noise of 1 to 2 %, 3 in 1,000 without
// noise (dictionaries of the solves measured, P = 30 to 1000). With 5 slices and no second
// look 0.3 to 0.5 % of the results were off by more than half an FP32 unit, by up to 8e-6 of
// themselves. It costs (start of a solve, 5 slices before, now) 372 -> 400 us at 96x96x64,
// P = 64, 30 rows; 141 -> 170 at 192x192, P = 1000, 8 rows; 79 -> 84 at P = 200, 20 rows. Where
// every result needs the second look (data orthogonal to every row, P = 1000, 8 rows):
// 1.63 ms, all of it FP64 sums
// Full-rank forms and Algorithm 1 (Q rows): S = 5, 1024 entries between drains (levels above
// 0 could lose their last bit only where every entry is near its row's and column's maximum),
// no second look. What is dropped, 6 P 2^-40 of the scales, replaces the FP32 roundings of
// two products (c = B^T m to FP32, then h = sum_i G_i c_i in FP32), and is smaller than those
// on every input measured (by 18 times with outliers of 1e7 in single samples).
//
// Why: GB300 runs FP64 at about 0.53 TFMA/s, and the projections were bound by it. A solve of
// the 157 x 131 fingerprinting slice (P = 1000, Q = 900, 30 full-rank BF16x3 iterations)
// took 40.4 ms, 35.1 of them in the 18.6 GFMA of FP64 projections and 0.85 in h = Gq c (an
// FP32 product); with this kernel for both it takes 5.0 ms.
//
// Mapping: one CTA per (128 voxels, BN rows of A), row tiles fastest, so that the CTAs
// running together share a tile's data in L2. Eight warps read the data (coalesced along
// the voxels), cut it into the slices and store them K-major in the 64-byte-swizzled
// layout of the MMA's A operand (a slice value is a BF16 whose bits are the upper half of
// its FP32, so packing two is one byte permute). Warp 8 streams the slices of A (cut at
// plan time) by TMA, one thread of warp 9 issues the MMAs. BN = 32 for at most 64 rows, two CTAs
// per SM, which hide each other's start, drain and stores; else 96 (5 x 96 TMEM columns). With
// 7 slices (BN = 32) a CTA has one stage, and as the slices of A lie one after another as rows of
// one operand and the accumulators of the levels side by side, slice i of the data meets
// slices 0 .. 6 - i of A in one instruction of N = 32 (7 - i): 84 us at P = 200, 20 rows, against
// 92 with an instruction per pair (28); one CTA per SM with three stages 85, but 476 instead of
// 400 us at 96x96x64. With 5 slices of 96 rows the wider instructions gave nothing.
#include <algorithm>

#include "ssm_internal.cuh"
#include "ssm_tma.cuh"

namespace ssm {
namespace {

constexpr int XM = 128;                 // voxels per tile (MMA M, TMEM lanes)
constexpr int XK = 32;                  // K per stage: rows of 64 bytes (one swizzle atom)
constexpr int XCONV = 8;                // converting (and draining) warps
constexpr int XNT = 32 * (XCONV + 2);
constexpr int XA_BYTES = XM * XK * 2;   // one slice of the data tile
constexpr int kBad = 1 << 28;           // exponent mark of a column with NaN or infinity,
constexpr int kZero = -(1 << 28);       // of a row or column of zeros

// NSL slices, BN rows of A per CTA
template <int NSL, int BN>
struct XCfg {
  static constexpr bool CHECKED = NSL == 7;    // FP64 where the slices fall short
  static constexpr int DRAIN = (CHECKED ? 256 : 1024) / XK;   // stages between drains
  static constexpr int B_BYTES = BN * XK * 2;
  static constexpr int STAGE = NSL * (XA_BYTES + B_BYTES);
  static constexpr int CTAS = BN == 96 ? 1 : 2;
  static constexpr int NS = CHECKED ? 1 : BN == 96 ? 3 : 2;
  static constexpr int SMEM = NS * STAGE + 1024 + 128;
  static constexpr uint32_t COLS = BN == 96 ? 512 : 256;     // NSL BN columns, a power of two
  // kind::f16 instruction descriptor: D = F32, A = B = BF16, K-major, N, M = 128
  static constexpr uint32_t idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(XM >> 4) << 24);
  }
  static constexpr bool PACKED = CHECKED;      // one MMA for all slices of A that a slice meets
  static_assert(STAGE % 1024 == 0 && B_BYTES % 512 == 0 && BN % 32 == 0, "layout");
  static_assert(NSL * BN <= (int)COLS && SMEM <= 227 * 1024, "size");
};

struct ExactArgs {
  const float* __restrict__ M;       // P x N (row stride ldm)
  const int* __restrict__ vexp;      // column exponents
  const int* __restrict__ rexp;      // row exponents
  float* __restrict__ out;           // rows x N (row stride ldo)
  int* __restrict__ err;
  int64_t ldm, ldo, N;
  int P, rows, rows_pad, ntr;
  // 7 slices: the operand in FP64, A[i][p] = scale_i A64[i sr + p sp]
  const double* __restrict__ A64;
  const double* __restrict__ scale;
  int64_t sr, sp;
  int unit;                          // the integer sums are in units of 2^-unit
  long long least;                   // the smallest sum that is taken as it is (P 2^-27)
};

__device__ __forceinline__ float pow2i(int e) { return __int_as_float((e + 127) << 23); }

// smallest e with |x| <= 2^e for finite x != 0 (any value of e serves for x = 0)
__device__ __forceinline__ int exponent_of(float ax) {
  if (ax == 0.f) return 0;
  int e;
  const float f = frexpf(ax, &e);      // ax = f 2^e, f in [0.5, 1)
  return f == 0.5f ? e - 1 : e;
}

// vexp[n]: the exponent of column n's largest magnitude. A block covers 32 voxels, 8 rows
// in flight per voxel.
__global__ void __launch_bounds__(256) column_exponent_kernel(const float* __restrict__ M,
                                                              int64_t ldm, int64_t N, int P,
                                                              int* __restrict__ vexp) {
  __shared__ float sm[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t n = blockIdx.x * (int64_t)32 + lane;
  float mx = 0.f;
  bool bad = false;
  if (n < N) {
#pragma unroll 4
    for (int p = w; p < P; p += 8) {
      const float v = fabsf(__ldg(M + (int64_t)p * ldm + n));
      bad |= !(v <= 3.402823466e38f);
      mx = fmaxf(mx, v);
    }
  }
  sm[w][lane] = bad ? __int_as_float(0x7f800000) : mx;
  __syncthreads();
  if (w == 0 && n < N) {
    for (int i = 1; i < 8; ++i) mx = fmaxf(mx, sm[i][lane]);
    mx = fmaxf(mx, sm[0][lane]);
    vexp[n] = mx <= 3.402823466e38f ? (mx > 0.f ? exponent_of(mx) : kZero) : kBad;
  }
}

// the FP64 rows of A (A[i][p] = scale_i src[i sr + p sp]) cut into slices
// out[k][i][p] (k < nsl, i < rows_pad, p < Pp; zero past rows and P), one warp per row
__global__ void __launch_bounds__(256) slice_rows_kernel(int nsl, const double* __restrict__ src,
                                                         int64_t sr, int64_t sp,
                                                         const double* __restrict__ scale,
                                                         int rows, int P, int rows_pad, int Pp,
                                                         __nv_bfloat16* __restrict__ out,
                                                         int* __restrict__ rexp) {
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= rows_pad) return;
  const double sc = (i < rows && scale) ? scale[i] : 1.0;
  double mx = 0.0;
  if (i < rows)
    for (int p = lane; p < P; p += 32) mx = fmax(mx, fabs(sc * src[i * sr + p * sp]));
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  int e = 0;
  if (mx > 0.0) {
    const double f = frexp(mx, &e);
    if (f == 0.5) --e;
  }
  if (lane == 0) rexp[i] = mx > 0.0 ? e : kZero;
  for (int p = lane; p < Pp; p += 32) {
    double x = (i < rows && p < P) ? ldexp(sc * src[i * sr + p * sp], -e) : 0.0;
    double unit = 1.0 / 128.0;
    for (int k = 0; k < nsl; ++k) {
      const double sl = rint(x / unit) * unit;
      out[((int64_t)k * rows_pad + i) * Pp + p] = __float2bfloat16_rn((float)sl);
      x -= sl;
      unit *= 1.0 / 256.0;
    }
  }
}

// K-major operand in the 64-byte swizzle layout (atoms of 8 rows x 64 B): stride byte
// offset 512 B, version 1 (bit 46), swizzle mode 4 = 64 B (bits 61-63)
__device__ __forceinline__ uint64_t desc64(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) |
         ((uint64_t)(512 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}

__device__ __forceinline__ void x_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                      uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void x_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void x_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void x_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// 8 FP32 columns of this warp's 32 TMEM lanes at each of the levels' accumulators
template <int NSL, int BN>
__device__ __forceinline__ void ld_levels(uint32_t t, float (*v)[8]) {
  uint32_t r[NSL][8];
#pragma unroll
  for (int l = 0; l < NSL; ++l)
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
        : "=r"(r[l][0]), "=r"(r[l][1]), "=r"(r[l][2]), "=r"(r[l][3]), "=r"(r[l][4]),
          "=r"(r[l][5]), "=r"(r[l][6]), "=r"(r[l][7])
        : "r"(t + l * BN));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int l = 0; l < NSL; ++l)
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      // the value is defined after the wait (the empty statement pins the order)
      asm volatile("" : "+r"(r[l][j]));
      v[l][j] = __uint_as_float(r[l][j]);
    }
}

// One row's FP64 sums for the lanes in `weak` (the others keep f): side by side where many
// need one, else lane by lane with the whole warp on its sum. arow: the row's entries, sp
// apart; mcol: the lane's voxel, ldm apart.
__device__ __noinline__ float sum_fp64(const double* arow, int64_t sp, double scale,
                                       const float* mcol, int64_t ldm, int P, unsigned weak,
                                       float f) {
  const int lane = threadIdx.x & 31;
  if (__popc(weak) > 3) {
    if (weak >> lane & 1) {
      double acc = 0.0;
#pragma unroll 8
      for (int p = 0; p < P; ++p) acc = fma(__ldg(arow + p * sp), (double)__ldg(mcol + p * ldm), acc);
      f = (float)(acc * scale);
    }
    return f;
  }
  for (unsigned w = weak; w; w &= w - 1) {
    const int src = __ffs(w) - 1;
    const float* mc = reinterpret_cast<const float*>(
        __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(mcol), src));
    double acc = 0.0;
#pragma unroll 4
    for (int p = lane; p < P; p += 32)
      acc = fma(__ldg(arow + p * sp), (double)__ldg(mc + p * ldm), acc);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == src) f = (float)(acc * scale);
  }
  return f;
}

// MULTI: the accumulators are drained more than once
template <int NSL, int BN, bool MULTI>
__global__ void __launch_bounds__(XNT, XCfg<NSL, BN>::CTAS)
    exact_product_kernel(const __grid_constant__ CUtensorMap bmap, const ExactArgs a) {
  using C = XCfg<NSL, BN>;
  constexpr int NS = C::NS, XDRAIN = C::DRAIN;
  constexpr int CW = BN / 2;               // columns per draining warp
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + NS * C::STAGE);
  uint64_t* empty = full + NS;
  uint64_t* done = empty + NS;
  uint64_t* drained = done + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drained + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rt = (int)(blockIdx.x % (unsigned)a.ntr);
  const int64_t n0 = (int64_t)(blockIdx.x / (unsigned)a.ntr) * XM;
  const int nk = (a.P + XK - 1) / XK;
  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&full[s], XCONV + 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(done, 1);
    mbar_init(drained, XCONV);
    mbar_fence_init();
  }
  if (warp == XCONV + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(C::COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  x_fence_before();
  __syncthreads();
  x_fence_after();
  const uint32_t tmem = *tmem_slot;
  bool failed = false;
  if (warp == XCONV) {
    // ------------------------------------------------------------ TMA: the slices of A
    if (lane == 0) {
      int c = 0;
      for (; c < nk; ++c) {
        const int s = c % NS;
        if (c >= NS && !mbar_wait_sleep(&empty[s], (c / NS - 1) & 1)) {
          failed = true;
          break;
        }
        unsigned char* b = smem + s * C::STAGE + NSL * XA_BYTES;
        mbar_arrive_expect_tx(&full[s], NSL * C::B_BYTES);
#pragma unroll
        for (int k = 0; k < NSL; ++k)
          tma_load_2d(b + k * C::B_BYTES, &bmap, c * XK, k * a.rows_pad + rt * BN, &full[s]);
      }
      // no copy may be in flight when the CTA exits
      for (int s = 0; s < NS && s < c; ++s)
        mbar_wait_sleep(&full[s], ((s + ((c - 1 - s) / NS) * NS) / NS) & 1);
    }
  } else if (warp == XCONV + 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      for (int c = 0; c < nk; ++c) {
        const int s = c % NS, in_seg = c % XDRAIN;
        if (MULTI && in_seg == 0 && c > 0 &&
            !mbar_wait_sleep(drained, (c / XDRAIN - 1) & 1)) {
          failed = true;
          break;
        }
        if (!mbar_wait_sleep(&full[s], (c / NS) & 1)) {
          failed = true;
          break;
        }
        x_fence_after();
        const uint32_t as = smem_u32(smem + s * C::STAGE);
        const uint32_t bs = as + NSL * XA_BYTES;
#pragma unroll
        for (int kk = 0; kk < XK / 16; ++kk)
#pragma unroll
          for (int i = 0; i < NSL; ++i)
#pragma unroll
            for (int j = 0; j < (C::PACKED ? 1 : NSL - i); ++j)
              x_mma(tmem + (i + j) * BN, desc64(as + i * XA_BYTES + kk * 32),
                    desc64(bs + j * C::B_BYTES + kk * 32),
                    C::idesc(C::PACKED ? (NSL - i) * BN : BN),
                    (in_seg == 0 && kk == 0 && i == 0) ? 0u : 1u);
        x_commit(&empty[s]);
        if (in_seg == XDRAIN - 1 || c == nk - 1) x_commit(done);
      }
      // everything issued completes before the TMEM is freed: the drain waits for `done`
    }
  } else {
    // ------------------------------------------------------------ slice the data, drain
    const int v = tid & 127, ph = tid >> 7;        // voxel of the tile, half of the stage
    const int64_t n = n0 + v;
    const bool in = n < a.N;
    // (a column of zeros takes any scale; the test for it here, among the loads' conditions,
    // made the kernel 14 % slower)
    const int e = in ? max(a.vexp[n], -200) : 0;
    const bool good = in && e != kBad;
    const int eh = good ? e >> 1 : 0;
    const float sc1 = good ? pow2i(-eh) : 0.f, sc2 = good ? pow2i(-(e - eh)) : 0.f;
    const float* mp = a.M + n;
    float x[16];
    auto load = [&](int c) {
      const int p0 = c * XK + ph * 16;
#pragma unroll
      for (int j = 0; j < 16; ++j)
        x[j] = (good && p0 + j < a.P) ? __ldg(mp + (int64_t)(p0 + j) * a.ldm) : 0.f;
    };
    long long sum[MULTI ? CW : 1];
    if constexpr (MULTI) {
#pragma unroll
      for (int j = 0; j < CW; ++j) sum[j] = 0;
    }
    unsigned large = 0;                            // columns of which a lower level was large
    const int quarter = warp & 3, half = warp >> 2;
    const uint32_t tbase = tmem + ((uint32_t)(quarter * 32) << 16) + half * CW;
    const int64_t nd = n0 + quarter * 32 + lane;   // voxel this thread drains
    const int ed = nd < a.N ? a.vexp[nd] : kZero;
    // the levels of 8 columns as one integer each, in units of 2^-unit
    auto drain8 = [&](int j0, long long* t) {
      float lv[NSL][8];
      ld_levels<NSL, BN>(tbase + j0, lv);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if constexpr (C::CHECKED) {
          // Each level is an integer of at most 2^22 (level 0: 256 products of 2^14; the others
          // are checked): adding 1.5 x 2^23 leaves it in the sum's low bits
          int q[NSL];
          unsigned most = 0;
#pragma unroll
          for (int l = 0; l < NSL; ++l) {
            q[l] = __float_as_int(fmaf(lv[l][j], pow2i(14 + 8 * l), 12582912.f)) - 0x4B400000;
            if (l > 0) most = max(most, (unsigned)(q[l] + (1 << 22)));
          }
          if (most >= 1u << 23) large |= 1u << (j0 + j);
          const long long hi = (long long)(q[0] * 256 + q[1]) * 65536 + (q[2] * 256 + q[3]);
          const long long lo = (long long)(q[4] * 256 + q[5]) * 256 + q[6];
          t[j] = (long long)((unsigned long long)hi << (a.unit - 38)) + (lo >> (62 - a.unit));
        } else {
          long long q = 0;
#pragma unroll
          for (int l = 0; l < NSL; ++l)
            q = q * 256 + (long long)__float2int_rn(lv[l][j] * pow2i(14 + 8 * l));
          t[j] = q;
        }
      }
    };
    auto store8 = [&](int j0, const long long* t) {
      const int i0 = rt * BN + half * CW + j0;
      unsigned weak = 0;                           // columns to form again
      float f[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int re = __ldg(a.rexp + i0 + j);     // (there are rows_pad of them)
        const int ex = max(-240, min(240, re + ed - a.unit));
        const int xh = ex >> 1;
        f[j] = __ll2float_rn(t[j]) * pow2i(xh) * pow2i(ex - xh);
        if constexpr (C::CHECKED) {
          const bool taken = re == kZero || ed == kZero ||
                             (ed != kBad && !(large >> (j0 + j) & 1) && llabs(t[j]) >= a.least);
          weak |= taken ? 0u : 1u << j;
        } else if (ed == kBad) {
          f[j] = __int_as_float(0x7fffffff);
        }
      }
      if (C::CHECKED && __any_sync(0xffffffffu, weak != 0)) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const unsigned lanes = __ballot_sync(0xffffffffu, weak >> j & 1);
          if (lanes)                               // (rows past the last are zero: not weak)
            f[j] = sum_fp64(a.A64 + (i0 + j) * a.sr, a.sp, a.scale[i0 + j], a.M + nd, a.ldm, a.P,
                            lanes, f[j]);
        }
      }
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (nd < a.N && i0 + j < a.rows) a.out[(int64_t)(i0 + j) * a.ldo + nd] = f[j];
    };
    // the accumulators' sums of the segment that ends before stage c, once its MMAs are done
    auto drain = [&](int c) {
      if constexpr (MULTI) {
        if (!failed && !mbar_wait_sleep(done, ((c - 1) / XDRAIN) & 1)) failed = true;
        x_fence_after();
#pragma unroll
        for (int j0 = 0; j0 < CW; j0 += 8) {
          long long t[8];
          drain8(j0, t);
#pragma unroll
          for (int j = 0; j < 8; ++j) sum[j0 + j] += t[j];
        }
        x_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(drained);
      }
    };
    load(0);
    for (int c = 0; c < nk; ++c) {
      const int s = c % NS;
      // cut into slices: adding and subtracting 1.5 2^(16-8k) rounds to a multiple of
      // 2^(-7-8k) (round to nearest even); every step is exact
      uint32_t sl[NSL][8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        float2 r = __fmul2_rn(__fmul2_rn(make_float2(x[2 * j], x[2 * j + 1]), make_float2(sc1, sc1)),
                              make_float2(sc2, sc2));
#pragma unroll
        for (int k = 0; k < NSL; ++k) {
          const float m = 1.5f * (float)(1 << 16) / (float)(1ull << (8 * k));
          const float2 t = __fadd2_rn(__fadd2_rn(r, make_float2(m, m)), make_float2(-m, -m));
          r = __fadd2_rn(r, make_float2(-t.x, -t.y));
          sl[k][j] = __byte_perm(__float_as_uint(t.x), __float_as_uint(t.y), 0x7632);
        }
      }
      if (c + 1 < nk) load(c + 1);
      if (c >= NS && !failed && !mbar_wait_sleep(&empty[s], (c / NS - 1) & 1)) failed = true;
      unsigned char* st = smem + s * C::STAGE + v * 64;
      const int key = (v >> 1) & 3;
#pragma unroll
      for (int k = 0; k < NSL; ++k)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          *reinterpret_cast<uint4*>(st + k * XA_BYTES + (((ph * 2 + h) ^ key) << 4)) =
              make_uint4(sl[k][4 * h], sl[k][4 * h + 1], sl[k][4 * h + 2], sl[k][4 * h + 3]);
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[s]);
      // the segment before is drained with the first stage of the next in place, so that the MMAs
      // go on as soon as its sums are read
      if (MULTI && c > 0 && c % XDRAIN == 0) drain(c);
    }
    if constexpr (MULTI) {
      drain(nk);
#pragma unroll
      for (int j0 = 0; j0 < CW; j0 += 8) store8(j0, sum + j0);
    } else {
      if (!failed && !mbar_wait_sleep(done, 0)) failed = true;
      x_fence_after();
#pragma unroll 1
      for (int j0 = 0; j0 < CW; j0 += 8) {
        if (rt * BN + half * CW + j0 >= a.rows) break;   // uniform across the warp
        long long t[8];
        drain8(j0, t);
        store8(j0, t);
      }
    }
  }
  if (failed) atomicExch(a.err, (int)SSM_ETIMEOUT);
  x_fence_before();
  __syncthreads();
  if (warp == XCONV + 1) {
    x_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(C::COLS)
                 : "memory");
  }
}

template <int NSL, int BN, bool MULTI>
ssm_status launch_exact(const CUtensorMap& map, const ExactArgs& a, int64_t ctas, cudaStream_t s) {
  using C = XCfg<NSL, BN>;
  // the attribute is set on every call: it costs about a microsecond once per solve and
  // needs no per-device record
  SSM_CUDA(cudaFuncSetAttribute(exact_product_kernel<NSL, BN, MULTI>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM));
  exact_product_kernel<NSL, BN, MULTI><<<(unsigned)ctas, XNT, C::SMEM, s>>>(map, a);
  SSM_LAUNCHED();
  return SSM_OK;
}

// rows per CTA: 32 up to 64 rows (and wherever the accumulators are drained repeatedly).
// 192x192, P = 64, 96 rows 71.4 us with 32 per CTA, 68.2 with 96; P = 1000, 900 rows, 157x131
// 970 against 657 (the data is cut into slices once per 96 rows instead of once per 32)
int exact_bn(int rows, int P, bool checked) { return checked || rows <= 64 || P > 1024 ? 32 : 96; }

}  // namespace

// slices, padded rows and columns of the sliced operand of `rows` x P
ExactShape exact_shape(int rows, int P, bool checked) {
  ExactShape x;
  const int bn = exact_bn(rows, P, checked);
  x.slices = checked ? 7 : 5;
  x.rows = (rows + bn - 1) / bn * bn;
  x.cols = (P + XK - 1) / XK * XK;
  return x;
}

ssm_status exact_slice(const double* src, int64_t sr, int64_t sp, const double* scale, int rows,
                       int P, bool checked, __nv_bfloat16* slices, int* rexp, cudaStream_t s) {
  const ExactShape x = exact_shape(rows, P, checked);
  slice_rows_kernel<<<(unsigned)((x.rows + 7) / 8), 256, 0, s>>>(
      x.slices, src, sr, sp, scale, rows, P, x.rows, x.cols, slices, rexp);
  SSM_LAUNCHED();
  return SSM_OK;
}

ssm_status exact_product(const double* src, int64_t sr, int64_t sp, const double* scale,
                         const __nv_bfloat16* slices, const int* rexp, int rows, int P, bool checked,
                         const float* M, int64_t ldm, int64_t N, float* out, int64_t ldo,
                         int* vexp, int* err, cudaStream_t s) {
  const ExactShape x = exact_shape(rows, P, checked);
  const int bn = exact_bn(rows, P, checked);
  column_exponent_kernel<<<(unsigned)((N + 31) / 32), 256, 0, s>>>(M, ldm, N, P, vexp);
  SSM_LAUNCHED();
  CUtensorMap map;
  SSM_CUDA(encode_2d(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, slices, (uint64_t)x.cols,
                     (uint64_t)x.slices * x.rows, (uint64_t)x.cols, XK, (unsigned)bn,
                     CU_TENSOR_MAP_SWIZZLE_64B));
  ExactArgs a;
  a.M = M;
  a.vexp = vexp;
  a.rexp = rexp;
  a.out = out;
  a.err = err;
  a.ldm = ldm;
  a.ldo = ldo;
  a.N = N;
  a.P = P;
  a.rows = rows;
  a.rows_pad = x.rows;
  a.ntr = x.rows / bn;
  a.A64 = src;
  a.scale = scale;
  a.sr = sr;
  a.sp = sp;
  a.unit = 46;                       // P 2^46 fits 63 bits
  a.least = 0;
  if (checked) {
    // P 2^unit <= 2^62; P <= 65536
    a.unit = 62;
    while ((int64_t)1 << (62 - a.unit) < P) --a.unit;
    a.least = (long long)P << (a.unit - 27);
  }
  const int64_t ctas = (N + XM - 1) / XM * a.ntr;
  if (ctas > INT32_MAX) {
    set_error("projection grid too large");
    return SSM_EINVAL;
  }
  if (checked)
    return P > XCfg<7, 32>::DRAIN * XK ? launch_exact<7, 32, true>(map, a, ctas, s)
                                       : launch_exact<7, 32, false>(map, a, ctas, s);
  if (bn == 96) return launch_exact<5, 96, false>(map, a, ctas, s);
  return P > XCfg<5, 32>::DRAIN * XK ? launch_exact<5, 32, true>(map, a, ctas, s)
                                     : launch_exact<5, 32, false>(map, a, ctas, s);
}

}  // namespace ssm
