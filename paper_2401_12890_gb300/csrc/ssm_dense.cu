// Full-rank (Eq. 26) LADMM iteration in plain FP32, plus the kernels shared by every
// form: an FP32 SIMT matrix product, the residual reductions and the objective terms.
//
// Eq. 26 gives f_n = (K^T K + beta I)^{-1} (g_n + beta z_n - d_n). Applied literally in
// FP32 the large, nearly cancelling product M g_n dominates the rounding error, so
// the iteration uses the exact split
//     f = h + M w,   h = M g (formed once per solve),   w = beta z - d,
// and runs the Q x Q by Q x N contraction on w only. The update kernel then applies
// the z-step (Eq. 31 with the nonnegativity projection) and the dual step, and
// writes the next w, so one iteration is: sgemm (M w) -> dense_update.
#include <algorithm>

#include "ssm_internal.cuh"

namespace ssm {
namespace {

// ---------------------------------------------------------------------------
// z-step (Eq. 31 + projection) and dual step for the full-rank form
//   f  = h + acc,  z' = max(0, (xi z - lambda s (deg z - sum_nbr z) + beta f + d)/(xi+beta))
//   d' = d - beta (z' - f),  w' = beta z' - d'
// block: 256 voxels x UQ compartments (loop); residual partials on check iterations.
// ---------------------------------------------------------------------------
constexpr int UV = 256, UQ = 8;

struct UpdateArgs {
  const float* __restrict__ acc;
  const float* __restrict__ H;
  const float* __restrict__ Zin;
  const float* __restrict__ Din;
  float* __restrict__ Zout;
  float* __restrict__ Dout;
  float* __restrict__ Wf;            // w'
  double* __restrict__ partial;
  const uint8_t* __restrict__ mask;  // voxels inside the object (nullptr: every voxel)
  Grid g;
  int Q;
  float beta, xi, lam_s, inv_xb;
};

template <bool CHECK>
__global__ void __launch_bounds__(UV) dense_update_kernel(UpdateArgs a) {
  const int64_t n = (int64_t)blockIdx.x * UV + threadIdx.x;
  const uint8_t* mk = a.mask;
  const bool valid = n < a.g.N && (!mk || mk[n]);   // outside the object: left alone
  const int nx = a.g.nx, ny = a.g.ny, nz = a.g.nz;
  const int64_t sy = nx, sz = (int64_t)nx * ny, ld = a.g.ld;
  int x = 0, y = 0, zc = 0;
  if (valid) {
    x = (int)(n % nx);
    const int64_t t = n / nx;
    y = (int)(t % ny);
    zc = (int)(t / ny);
  }
  const bool hxm = valid && x > 0 && (!mk || mk[n - 1]);
  const bool hxp = valid && x < nx - 1 && (!mk || mk[n + 1]);
  const bool hym = valid && y > 0 && (!mk || mk[n - sy]);
  const bool hyp = valid && y < ny - 1 && (!mk || mk[n + sy]);
  const bool hzm = a.g.zlink && valid && zc > 0 && (!mk || mk[n - sz]);
  const bool hzp = a.g.zlink && valid && zc < nz - 1 && (!mk || mk[n + sz]);
  const float deg = (float)(hxm + hxp + hym + hyp + hzm + hzp);
  float s1 = 0.f, s2 = 0.f, s3 = 0.f;
  const int q0 = blockIdx.y * UQ, q1 = min(a.Q, q0 + UQ);
  if (valid) {
    for (int q = q0; q < q1; ++q) {
      const int64_t o = (int64_t)q * ld + n;
      const float z = __ldg(a.Zin + o), d = __ldg(a.Din + o);
      float nb = 0.f;
      if (hxm) nb += __ldg(a.Zin + o - 1);
      if (hxp) nb += __ldg(a.Zin + o + 1);
      if (hym) nb += __ldg(a.Zin + o - sy);
      if (hyp) nb += __ldg(a.Zin + o + sy);
      if (hzm) nb += __ldg(a.Zin + o - sz);
      if (hzp) nb += __ldg(a.Zin + o + sz);
      const float f = __ldg(a.H + o) + __ldg(a.acc + o);
      const float zn = fmaxf(0.f, (a.xi * z - a.lam_s * (deg * z - nb) + a.beta * f + d) * a.inv_xb);
      const float dn = d - a.beta * (zn - f);
      const float w = a.beta * zn - dn;
      a.Zout[o] = zn;
      a.Dout[o] = dn;
      a.Wf[o] = w;
      if (CHECK) {
        const float e = zn - f, c = zn - z;
        s1 = fmaf(e, e, s1);
        s2 = fmaf(c, c, s2);
        s3 = fmaf(zn, zn, s3);
      }
    }
  }
  if (CHECK) {
    double d1 = s1, d2 = s2, d3 = s3;
    for (int off = 16; off > 0; off >>= 1) {
      d1 += __shfl_xor_sync(0xffffffffu, d1, off);
      d2 += __shfl_xor_sync(0xffffffffu, d2, off);
      d3 += __shfl_xor_sync(0xffffffffu, d3, off);
    }
    __shared__ double sm[UV / 32][3];
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
      sm[w][0] = d1;
      sm[w][1] = d2;
      sm[w][2] = d3;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
      double t = 0.0;
      for (int k = 0; k < UV / 32; ++k) t += sm[k][threadIdx.x];
      a.partial[((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * 4 + threadIdx.x] = t;
    }
  }
}

// sum `nparts` rows of `width` doubles (row stride 4) in a fixed order
__global__ void finish_kernel(const double* __restrict__ part, int nparts, int width,
                              double* __restrict__ out) {
  __shared__ double sm[32][4];
  double acc[4] = {0, 0, 0, 0};
  for (int i = threadIdx.x; i < nparts; i += blockDim.x)
    for (int j = 0; j < width; ++j) acc[j] += part[(int64_t)i * 4 + j];
  for (int j = 0; j < width; ++j)
    for (int off = 16; off > 0; off >>= 1) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], off);
  if ((threadIdx.x & 31) == 0)
    for (int j = 0; j < width; ++j) sm[threadIdx.x >> 5][j] = acc[j];
  __syncthreads();
  if (threadIdx.x < width) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sm[w][threadIdx.x];
    out[threadIdx.x] = t;
  }
}

// B bytes from global to shared memory, of which the first `n` are read and the rest are 0
template <int B>
__device__ __forceinline__ void cp_async(float* dst, const float* src, int n) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if constexpr (B == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(n)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(n)
                 : "memory");
}

struct ProductArgs {
  int M, N, K;
  const float* __restrict__ At;       // A transposed: K x M, row stride lda
  int64_t lda;
  const float* __restrict__ B;        // K x N, row stride ldb
  int64_t ldb;
  float* __restrict__ C;              // A B (store)
  int64_t ldc;
  const float* __restrict__ D;        // residual: sum (D - A B)^2
  int64_t ldd;
  const uint8_t* __restrict__ mask;   // voxels inside the object (nullptr: every voxel)
  double* __restrict__ partial;       // 4 doubles per CTA
};

// s + c (unevaluated) += x, exactly (Knuth's TwoSum)
__device__ __forceinline__ void two_sum(float& s, float& c, float x) {
  const float t = __fadd_rn(s, x);
  const float b = __fsub_rn(t, s);
  c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(x, b)));
  s = t;
}

template <int T>
__device__ __forceinline__ void block_partial(double d1, double d2, double d3, double* out) {
  for (int o = 16; o > 0; o >>= 1) {
    d1 += __shfl_xor_sync(0xffffffffu, d1, o);
    d2 += __shfl_xor_sync(0xffffffffu, d2, o);
    d3 += __shfl_xor_sync(0xffffffffu, d3, o);
  }
  __shared__ double red[T / 32][3];
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    red[w][0] = d1;
    red[w][1] = d2;
    red[w][2] = d3;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    double t = 0.0;
    for (int k = 0; k < T / 32; ++k) t += red[k][threadIdx.x];
    out[threadIdx.x] = t;
  }
}

// sum over a chunk of maps and RT voxels of (F_n - F_m)^2, m the forward neighbours: FP32
// squares (a map's three added in FP32), their sum over the maps in FP64. Eight maps at a time
// are added as a float-float number (its error, seven roundings of the low part, is at most
// 2^-43 of the eight's sum) and that to the FP64 sum: at this chip's FP64 rate an FP64 add per
// element would take 77 us of the 41 M elements of the 128 x 128 slice. Where the FP32 part
// overflows (or is not a number), the eight go to the FP64 sum one by one.
constexpr int RT = 256;
__global__ void __launch_bounds__(RT) roughness_kernel(const float* __restrict__ F, int64_t ldf,
                                                       int Q, int chunk, Grid g,
                                                       const uint8_t* __restrict__ mk,
                                                       double* __restrict__ partial) {
  const int64_t n = blockIdx.x * (int64_t)RT + threadIdx.x;
  const int q0 = (int)blockIdx.y * chunk, q1 = min(Q, q0 + chunk);
  double e2 = 0.0;
  if (n < g.N && (!mk || mk[n])) {
    const int x = (int)(n % g.nx);
    const int64_t t = n / g.nx;
    const int y = (int)(t % g.ny), z = (int)(t / g.ny);
    const int64_t sy = g.nx, sz = (int64_t)g.nx * g.ny;
    const bool hx = x + 1 < g.nx && (!mk || mk[n + 1]);
    const bool hy = y + 1 < g.ny && (!mk || mk[n + sy]);
    const bool hz = g.zlink && z + 1 < g.nz && (!mk || mk[n + sz]);
    // an absent neighbour reads the voxel itself, and its difference is dropped
    const int64_t ox = hx ? 1 : 0, oy = hy ? sy : 0, oz = hz ? sz : 0;
    const float* p = F + (int64_t)q0 * ldf + n;
    const bool z3 = g.zlink && g.nz > 1;
    auto square = [&](float v, float vx, float vy, float vz) {
      const float dx = hx ? __fsub_rn(v, vx) : 0.f, dy = hy ? __fsub_rn(v, vy) : 0.f;
      const float dz = hz ? __fsub_rn(v, vz) : 0.f;
      return fmaf(dz, dz, fmaf(dy, dy, __fmul_rn(dx, dx)));
    };
    // RU maps' loads in flight per thread
    constexpr int RU = 8;
    int q = q0;
    for (; q + RU <= q1; q += RU, p += RU * ldf) {
      float v[RU], vx[RU], vy[RU], vz[RU];
#pragma unroll
      for (int u = 0; u < RU; ++u) {
        v[u] = __ldg(p + u * ldf);
        vx[u] = __ldg(p + u * ldf + ox);
        vy[u] = __ldg(p + u * ldf + oy);
        vz[u] = z3 ? __ldg(p + u * ldf + oz) : v[u];
      }
      float s = 0.f, c = 0.f;
#pragma unroll
      for (int u = 0; u < RU; ++u) {
        v[u] = square(v[u], vx[u], vy[u], vz[u]);
        two_sum(s, c, v[u]);
      }
      if (s <= 3.402823466e38f) {
        e2 += (double)s + (double)c;
      } else {
#pragma unroll
        for (int u = 0; u < RU; ++u) e2 += (double)v[u];
      }
    }
    for (; q < q1; ++q, p += ldf)
      e2 += (double)square(__ldg(p), __ldg(p + ox), __ldg(p + oy), z3 ? __ldg(p + oz) : 0.f);
  }
  block_partial<RT>(0.0, e2, 0.0, partial + ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * 4);
}

// A B for the full-rank FP32 forms (C = A B), or the objective's data term, sum (D - A B)^2
// over the voxels inside the object with squares and sums in FP64. FP32, each product one
// FMA chain over k in ascending order (so the results depend on neither the tile shape nor
// the grid). A is given transposed (K^T, or the symmetric M), so that both operands' k
// slices are rows.
//
// Bound: the FP32 pipe (128 FMA per SM and cycle), and next to it the shared-memory pipe. A
// thread owns 16 rows x 4 columns and a warp 16 rows x 128 columns: the rows' A values are
// the same for every lane (broadcast reads), which takes 8 shared-memory wavefronts per 64
// FMAs of a warp against the 12 of 8 x 8 outputs per thread, whose reads queued behind one
// another. Slices of 8 k come by cp.async into a ring of NST stages, and the fragments of
// slice entry k + 1 are read while those of k are multiplied. Tiles of 64 rows x 128 columns
// (4 warps, three CTAs per SM): CTAs that wait for their own slices only, and a short last
// wave. Per iteration with the update: M = K = 2500, N = 16384 4605 us (tiles of 128 rows and
// two CTAs: 4704), M = K = 300, N = 6048 47.9 us (53.7). The objective with M = 64, K = 1600,
// N = 589824 4011 us (6851: half of a 128-row tile is padding there).
// VEC: the rows of A^T and B are 16-byte aligned (else scalar copies)
constexpr int PM = 64;

template <bool RESIDUAL, bool VEC>
__global__ void __launch_bounds__(2 * PM, 3)
    product_kernel(const ProductArgs a) {
  constexpr int BN = 128;
  constexpr int BM = PM, T = 2 * BM;               // 16 x 4 outputs each
  constexpr int BK = 8;
  constexpr int NST = 4;                           // stages
  constexpr int STAGE = BK * (BM + BN);            // floats per stage: A slice, B slice
  constexpr int LA = BM * BK / 4 / T, LB = BN * BK / 4 / T;   // 16-byte copies per thread
  static_assert(LA >= 1 && LB >= 1, "loader");
  __shared__ __align__(16) float ring[NST * STAGE];
  const int tid = threadIdx.x;
  const int r16 = (tid >> 5) * 16, c4 = (tid & 31) * 4;   // this thread's rows and columns
  const int M = a.M, N = a.N, K = a.K;
  const int mt = (M + BM - 1) / BM;
  const int m0 = ((int)blockIdx.x % mt) * BM, n0 = ((int)blockIdx.x / mt) * BN;
  const int ntile = (K + BK - 1) / BK;
  // k slice kt into stage kt % NST; elements outside the matrices are zero-filled
  auto copy4 = [&](float* d, const float* base, int64_t ldx, int gk, int gc, int lim) {
    const int ok = gk < K ? max(0, min(4, lim - gc)) : 0;
    const float* p = base + (int64_t)gk * ldx + gc;
    if (VEC) {
      cp_async<16>(d, ok > 0 ? p : base, 4 * ok);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) cp_async<4>(d + j, j < ok ? p + j : base, j < ok ? 4 : 0);
    }
  };
  auto load = [&](int kt) {
    float* st = ring + (kt % NST) * STAGE;
#pragma unroll
    for (int i = 0; i < LA; ++i) {
      const int f = tid + i * T, kk = f / (BM / 4), c = (f % (BM / 4)) * 4;
      copy4(st + kk * BM + c, a.At, a.lda, kt * BK + kk, m0 + c, M);
    }
#pragma unroll
    for (int i = 0; i < LB; ++i) {
      const int f = tid + i * T, kk = f / (BN / 4), c = (f % (BN / 4)) * 4;
      copy4(st + BK * BM + kk * BN + c, a.B, a.ldb, kt * BK + kk, n0 + c, N);
    }
  };
  auto commit = [] { asm volatile("cp.async.commit_group;\n" ::: "memory"); };
  float acc[16][4];
#pragma unroll
  for (int i = 0; i < 16; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  float4 fa[2][4], fb[2];
  auto frag = [&](int kt, int k, int buf) {
    const float* st = ring + (kt % NST) * STAGE;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      fa[buf][i] = *reinterpret_cast<const float4*>(st + k * BM + r16 + 4 * i);
    fb[buf] = *reinterpret_cast<const float4*>(st + BK * BM + k * BN + c4);
  };
#pragma unroll
  for (int i = 0; i < NST - 1; ++i) {
    if (i < ntile) load(i);
    commit();
  }
  asm volatile("cp.async.wait_group %0;\n" ::"n"(NST - 2) : "memory");
  __syncthreads();
  frag(0, 0, 0);
#pragma unroll 1
  for (int kt = 0; kt < ntile; ++kt) {
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      if (k == BK - 1) {
        // slice kt + 1 has landed (one group per slice, empty ones past the end)
        asm volatile("cp.async.wait_group %0;\n" ::"n"(NST - 2) : "memory");
        __syncthreads();
        if (kt + 1 < ntile) frag(kt + 1, 0, 0);
      } else {
        frag(kt, k + 1, (k + 1) & 1);
      }
      if (k == 0) {
        // the stage of slice kt - 1, which every thread has left (the barrier above)
        if (kt + NST - 1 < ntile) load(kt + NST - 1);
        commit();
      }
      const float4 y = fb[k & 1];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float4 x4 = fa[k & 1][i / 4];
        const float x = i % 4 == 0 ? x4.x : i % 4 == 1 ? x4.y : i % 4 == 2 ? x4.z : x4.w;
        acc[i][0] = fmaf(x, y.x, acc[i][0]);
        acc[i][1] = fmaf(x, y.y, acc[i][1]);
        acc[i][2] = fmaf(x, y.z, acc[i][2]);
        acc[i][3] = fmaf(x, y.w, acc[i][3]);
      }
    }
  }
  if constexpr (!RESIDUAL) {
    const bool vec = a.ldc % 4 == 0 && n0 + c4 + 3 < N;    // (C is 16-byte aligned)
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int gm = m0 + r16 + i;
      if (gm >= M) break;
      float* c = a.C + (int64_t)gm * a.ldc + n0 + c4;
      if (vec) {
        *reinterpret_cast<float4*>(c) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (n0 + c4 + j < N) c[j] = acc[i][j];
      }
    }
  } else {
    double r2 = 0.0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int gn = n0 + c4 + j;
      if (gn >= N || (a.mask && !a.mask[gn])) continue;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int gm = m0 + r16 + i;
        if (gm >= M) continue;
        const float r = __fsub_rn(__ldg(a.D + (int64_t)gm * a.ldd + gn), acc[i][j]);
        r2 += (double)r * r;
      }
    }
    block_partial<T>(r2, 0.0, 0.0, a.partial + (int64_t)blockIdx.x * 4);
  }
}

int64_t product_ctas(int64_t M, int64_t N) {
  return (M + PM - 1) / PM * ((N + 127) / 128);
}

// Compartment chunks of the roughness sum: about 8 CTAs per SM, at least 16 maps each
int rough_chunks(const ssm_plan_s* pl, int* chunk) {
  const int64_t nb = (pl->g.N + RT - 1) / RT;
  const int64_t c = std::max<int64_t>(1, std::min<int64_t>(8 * (int64_t)sm_count() / nb, pl->Q / 16));
  *chunk = (int)((pl->Q + c - 1) / c);
  return (pl->Q + *chunk - 1) / *chunk;
}

template <bool RESIDUAL>
ssm_status launch_product(const ProductArgs& a, cudaStream_t s) {
  if (a.M <= 0 || a.N <= 0) return SSM_OK;
  const int64_t ctas = product_ctas(a.M, a.N);
  if (ctas > INT32_MAX) {
    set_error("matrix product: too many tiles");
    return SSM_EINVAL;
  }
  const bool vec = a.lda % 4 == 0 && a.ldb % 4 == 0 &&
                   ((reinterpret_cast<uintptr_t>(a.At) | reinterpret_cast<uintptr_t>(a.B)) & 15) == 0;
  const unsigned gr = (unsigned)ctas;
  if (vec) product_kernel<RESIDUAL, true><<<gr, 2 * PM, 0, s>>>(a);
  else product_kernel<RESIDUAL, false><<<gr, 2 * PM, 0, s>>>(a);
  SSM_LAUNCHED();
  return SSM_OK;
}

}  // namespace

// C = A B with A given transposed (K x M)
ssm_status sgemm(int M, int N, int K, const float* At, int64_t lda, const float* B, int64_t ldb,
                 float* C, int64_t ldc, cudaStream_t s) {
  ProductArgs a{};
  a.M = M;
  a.N = N;
  a.K = K;
  a.At = At;
  a.lda = lda;
  a.B = B;
  a.ldb = ldb;
  a.C = C;
  a.ldc = ldc;
  return launch_product<false>(a, s);
}

int dense_max_partials(const ssm_plan_s* pl) {
  return (int)(((pl->g.N + UV - 1) / UV) * ((pl->Q + UQ - 1) / UQ));
}

ssm_status dense_update(ssm_plan_s* pl, int cur, const float* acc, bool check, double* partial,
                        int* nparts, cudaStream_t s) {
  UpdateArgs a;
  a.acc = acc;
  a.H = pl->H;
  a.Zin = pl->Z[cur];
  a.Din = pl->Dl[cur];
  a.Zout = pl->Z[cur ^ 1];
  a.Dout = pl->Dl[cur ^ 1];
  a.Wf = pl->Wf;
  a.partial = partial;
  a.mask = pl->mask;
  a.g = pl->g;
  a.Q = pl->Q;
  a.beta = (float)pl->p.beta;
  a.xi = (float)pl->xi;
  a.lam_s = (float)pl->lam_s;
  a.inv_xb = (float)(1.0 / (pl->xi + pl->p.beta));
  dim3 grid((unsigned)((pl->g.N + UV - 1) / UV), (unsigned)((pl->Q + UQ - 1) / UQ));
  *nparts = (int)(grid.x * grid.y);
  // (ordinary launches: chained by programmatic dependent launch, the next kernel's waiting
  // blocks took the product's places on the SMs: 49 -> 60 us per iteration on the masked
  // 84 x 72 workload)
  if (check)
    dense_update_kernel<true><<<grid, UV, 0, s>>>(a);
  else
    dense_update_kernel<false><<<grid, UV, 0, s>>>(a);
  SSM_LAUNCHED();
  return SSM_OK;
}

ssm_status finish_partials(const double* partial, int nparts, int width, double* out,
                           cudaStream_t s) {
  finish_kernel<<<1, 1024, 0, s>>>(partial, nparts, width, out);
  SSM_LAUNCHED();
  return SSM_OK;
}

int objective_partials(const ssm_plan_s* pl) {
  int chunk;
  const int64_t rough = (pl->g.N + RT - 1) / RT * rough_chunks(pl, &chunk);
  return (int)std::min<int64_t>(INT32_MAX, product_ctas(pl->P, pl->g.N) + rough);
}

// ||M - K F||^2 and the sum over neighbour pairs of the squared differences of F, as
// partial rows (r2, e2, 0): the product's CTAs' first, then the roughness kernel's
ssm_status objective_terms(const ssm_plan_s* pl, const float* Kt, const float* M, int64_t ldm,
                           const float* F, int64_t ldf, double* partial, int* nparts,
                           cudaStream_t s) {
  ProductArgs a{};
  a.M = pl->P;
  a.N = (int)pl->g.N;
  a.K = pl->Q;
  a.At = Kt;
  a.lda = (pl->P + 3) / 4 * 4;
  a.B = F;
  a.ldb = ldf;
  a.D = M;
  a.ldd = ldm;
  a.mask = pl->mask;
  a.partial = partial;
  SSM_TRY(launch_product<true>(a, s));
  const int64_t ctas = product_ctas(pl->P, pl->g.N);
  int chunk;
  const int chunks = rough_chunks(pl, &chunk);
  const dim3 grid((unsigned)((pl->g.N + RT - 1) / RT), (unsigned)chunks);
  roughness_kernel<<<grid, RT, 0, s>>>(F, ldf, pl->Q, chunk, pl->g, pl->mask,
                                       partial + ctas * 4);
  SSM_LAUNCHED();
  *nparts = objective_partials(pl);
  return SSM_OK;
}

}  // namespace ssm
