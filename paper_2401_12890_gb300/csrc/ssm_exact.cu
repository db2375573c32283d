// Data projections (Algorithm 2, step 4) as one matrix product with FP64-grade accuracy on
// the tcgen05 tensor cores:
//     out[i][n] = fl32( sum_p A[i][p] m[p][n] ),   A formed in FP64 once per plan
// (low-rank forms: A = rows sigma_i u_i^T, out = S; full-rank forms and Algorithm 1:
// A = (K^T K + beta I)^{-1} K^T, out = h = M g).
//
// Method: error-free slicing into short integers (the splitting of Ozaki, Ogita, Oishi and
// Rump, "Error-free transformations of matrix multiplication", 2012). Every row of A and
// every column of m is scaled by a power of two so that its entries lie in [-1, 1] and cut
// into 5 slices of 8 bits (slice k a multiple of 2^(-7-8k), |slice| <= 128 units, exact in
// BF16). A product of slices i and j is a 14-bit integer in units of 2^(-14-8(i+j)), so
// the tensor core's FP32 accumulation of up to 1024 of them is exact (2^14 * 2^10 = 2^24;
// the levels i + j > 0 sum several products and could lose their last bit only where every
// entry is at its row's and column's maximum). The 15 products with i + j <= 4 go to one
// accumulator per level i + j; the five sums are added as 64-bit integers and rounded to
// FP32 once. What is dropped is below 2^-38 of the largest entries' product per sum: an
// FP64 accumulation's result after its rounding to FP32, except where the sum cancels to
// below 2^-14 of its terms. A column that holds a NaN or an infinity gives NaN.
//
// Why: GB300 runs FP64 at about 0.53 TFMA/s, and the projections were bound by it. A solve of
// the 157 x 131 fingerprinting slice (P = 1000, Q = 900, 30 full-rank BF16x3 iterations)
// took 40.4 ms, 35.1 of them in the 18.6 GFMA of FP64 projections and 0.85 in h = Gq c (an
// FP32 product); with this kernel for both it takes 5.03 ms. The 96 x 96 x 64 volume (P = 64,
// r = 30) spent 2.37 ms of a 74.9 ms solve in them (now 72.7 ms), the 192 x 192
// fingerprinting slice (P = 1000, r = 8) 0.64 of 9.34 ms (now 8.79 ms).
//
// Mapping: one CTA per (128 voxels, BN rows of A), row tiles fastest, so that the CTAs
// running together share a tile's data in L2. Eight warps read the data (coalesced along
// the voxels), cut it into the five slices and store them K-major in the 64-byte-swizzled
// layout of the MMA's A operand (a slice value is a BF16 whose bits are the upper half of
// its FP32, so packing two is one byte permute). Warp 8 streams the slices of A (cut at
// plan time) by TMA, one thread of warp 9 issues the 30 MMAs of a 32-deep stage. BN = 32
// for at most 64 rows (low-rank forms; two CTAs per SM), else 96 (5 x 96 TMEM columns).
// Beyond P = 1024 the accumulators are drained every 1024 entries into 64-bit integers
// held in registers (BN = 32 there, which keeps them to 16 per thread).
#include <algorithm>

#include "ssm_internal.cuh"
#include "ssm_tma.cuh"

namespace ssm {
namespace {

constexpr int XM = 128;                 // voxels per tile (MMA M, TMEM lanes)
constexpr int XK = 32;                  // K per stage: rows of 64 bytes (one swizzle atom)
constexpr int NSL = 5;                  // slices
constexpr int XDRAIN = 1024 / XK;       // stages between drains (exact accumulation)
constexpr int XCONV = 8;                // converting (and draining) warps
constexpr int XNT = 32 * (XCONV + 2);
constexpr int XA_BYTES = XM * XK * 2;   // one slice of the data tile
constexpr int kBadColumn = 1 << 30;     // exponent mark of a column with NaN or infinity

template <int BN>
struct XCfg {
  static constexpr int B_BYTES = BN * XK * 2;
  static constexpr int STAGE = NSL * (XA_BYTES + B_BYTES);
  static constexpr int NS = BN == 96 ? 3 : 2;
  static constexpr int SMEM = NS * STAGE + 1024 + 128;
  static constexpr uint32_t COLS = BN == 96 ? 512 : 256;     // 5 BN columns, a power of two
  static constexpr int CTAS = BN == 96 ? 1 : 2;
  // kind::f16 instruction descriptor: D = F32, A = B = BF16, K-major, N, M = 128
  static constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) |
                                    ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(XM >> 4) << 24);
  static_assert(STAGE % 1024 == 0 && B_BYTES % 512 == 0 && BN % 32 == 0, "layout");
};

struct ExactArgs {
  const float* __restrict__ M;       // P x N (row stride ldm)
  const int* __restrict__ vexp;      // column exponents
  const int* __restrict__ rexp;      // row exponents
  float* __restrict__ out;           // rows x N (row stride ldo)
  int* __restrict__ err;
  int64_t ldm, ldo, N;
  int P, rows, rows_pad, ntr;
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
    vexp[n] = mx <= 3.402823466e38f ? exponent_of(mx) : kBadColumn;
  }
}

// the FP64 rows of A (A[i][p] = scale_i src[i sr + p sp]) cut into slices
// out[k][i][p] (k < 5, i < rows_pad, p < Pp; zero past rows and P), one warp per row
__global__ void __launch_bounds__(256) slice_rows_kernel(const double* __restrict__ src,
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
  if (lane == 0) rexp[i] = e;
  for (int p = lane; p < Pp; p += 32) {
    double x = (i < rows && p < P) ? ldexp(sc * src[i * sr + p * sp], -e) : 0.0;
    double unit = 1.0 / 128.0;
#pragma unroll
    for (int k = 0; k < NSL; ++k) {
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

// 8 FP32 columns of this warp's 32 TMEM lanes at each of the five levels' accumulators
template <int BN>
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

// MULTI: P > 1024, the accumulators are drained more than once
template <int BN, bool MULTI>
__global__ void __launch_bounds__(XNT, XCfg<BN>::CTAS)
    exact_product_kernel(const __grid_constant__ CUtensorMap bmap, const ExactArgs a) {
  using C = XCfg<BN>;
  constexpr int NS = C::NS;
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
            for (int j = 0; j < NSL - i; ++j)
              x_mma(tmem + (i + j) * BN, desc64(as + i * XA_BYTES + kk * 32),
                    desc64(bs + j * C::B_BYTES + kk * 32), C::IDESC,
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
    const int e = in ? a.vexp[n] : 0;
    const bool good = in && e != kBadColumn;
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
    const int quarter = warp & 3, half = warp >> 2;
    const uint32_t tbase = tmem + ((uint32_t)(quarter * 32) << 16) + half * CW;
    const int64_t nd = n0 + quarter * 32 + lane;   // voxel this thread drains
    const int ed = nd < a.N ? a.vexp[nd] : 0;
    // the five levels of 8 columns as integers in units of 2^-46
    auto drain8 = [&](int j0, long long* t) {
      float lv[NSL][8];
      ld_levels<BN>(tbase + j0, lv);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        long long q = 0;
#pragma unroll
        for (int l = 0; l < NSL; ++l)
          q = q * 256 + (long long)__float2int_rn(lv[l][j] * pow2i(14 + 8 * l));
        t[j] = q;
      }
    };
    auto store8 = [&](int j0, const long long* t) {
      if (nd >= a.N) return;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int i = rt * BN + half * CW + j0 + j;
        if (i < a.rows) {
          const int ex = max(-240, min(240, a.rexp[i] + ed - 46));
          const int xh = ex >> 1;
          const float f = __ll2float_rn(t[j]) * pow2i(xh) * pow2i(ex - xh);
          a.out[(int64_t)i * a.ldo + nd] = ed == kBadColumn ? __int_as_float(0x7fffffff) : f;
        }
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
      if constexpr (MULTI) {
        if (c % XDRAIN == XDRAIN - 1 || c == nk - 1) {
          if (!failed && !mbar_wait_sleep(done, (c / XDRAIN) & 1)) failed = true;
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
      }
    }
    if constexpr (MULTI) {
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

template <int BN, bool MULTI>
ssm_status launch_exact(const CUtensorMap& map, const ExactArgs& a, int64_t ctas, cudaStream_t s) {
  // the attribute is set on every call: it costs about a microsecond once per solve and
  // needs no per-device record
  SSM_CUDA(cudaFuncSetAttribute(exact_product_kernel<BN, MULTI>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, XCfg<BN>::SMEM));
  exact_product_kernel<BN, MULTI><<<(unsigned)ctas, XNT, XCfg<BN>::SMEM, s>>>(map, a);
  SSM_LAUNCHED();
  return SSM_OK;
}

// rows per CTA: 32 up to 64 rows (and wherever the accumulators are drained repeatedly).
// 192x192, P = 200, the whole start of a solve: 20 rows 88.9 us (96 per CTA: 98.0), 48 rows 101.0
// (101.8); P = 64, 96 rows 71.4 with 32 per CTA, 68.2 with 96; P = 1000, 900 rows, 157x131 970
// against 657 (the data is cut into slices once per 96 rows instead of once per 32)
int exact_bn(int rows, int P) { return rows <= 64 || P > 1024 ? 32 : 96; }

}  // namespace

// padded rows and columns of the sliced operand of `rows` x P
void exact_shape(int rows, int P, int* rows_pad, int* P_pad) {
  const int bn = exact_bn(rows, P);
  *rows_pad = (rows + bn - 1) / bn * bn;
  *P_pad = (P + XK - 1) / XK * XK;
}

// bytes of the sliced operand and its row exponents
int64_t exact_elems(int rows, int P) {
  int rp, pp;
  exact_shape(rows, P, &rp, &pp);
  return (int64_t)NSL * rp * pp;
}

// the operand from FP64: A[i][p] = scale_i src[i sr + p sp] (scale nullptr: 1)
ssm_status exact_slice(const double* src, int64_t sr, int64_t sp, const double* scale, int rows,
                       int P, __nv_bfloat16* slices, int* rexp, cudaStream_t s) {
  int rp, pp;
  exact_shape(rows, P, &rp, &pp);
  slice_rows_kernel<<<(unsigned)((rp + 7) / 8), 256, 0, s>>>(src, sr, sp, scale, rows, P, rp, pp,
                                                             slices, rexp);
  SSM_LAUNCHED();
  return SSM_OK;
}

// out (rows x ldo) = A m for the data M (P x N, row stride ldm); vexp: N ints of scratch
ssm_status exact_product(const __nv_bfloat16* slices, const int* rexp, int rows, int P,
                         const float* M, int64_t ldm, int64_t N, float* out, int64_t ldo,
                         int* vexp, int* err, cudaStream_t s) {
  int rp, pp;
  exact_shape(rows, P, &rp, &pp);
  const int bn = exact_bn(rows, P);
  column_exponent_kernel<<<(unsigned)((N + 31) / 32), 256, 0, s>>>(M, ldm, N, P, vexp);
  SSM_LAUNCHED();
  CUtensorMap map;
  SSM_CUDA(encode_2d(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, slices, (uint64_t)pp,
                     (uint64_t)NSL * rp, (uint64_t)pp, XK, (unsigned)bn,
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
  a.rows_pad = rp;
  a.ntr = rp / bn;
  const int64_t ctas = (N + XM - 1) / XM * a.ntr;
  if (ctas > INT32_MAX) {
    set_error("projection grid too large");
    return SSM_EINVAL;
  }
  if (bn == 96) return launch_exact<96, false>(map, a, ctas, s);
  if (P > 1024) return launch_exact<32, true>(map, a, ctas, s);
  return launch_exact<32, false>(map, a, ctas, s);
}

}  // namespace ssm
