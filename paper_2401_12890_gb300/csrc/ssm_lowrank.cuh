// One LADMM iteration of Algorithm 2 (rank-r f-step, Eq. 28) fused into one FP32 kernel.
//
// Per voxel n the paper's f-step is
//     c_n = g_n + beta z_n - d_n,   f_n = c_n/beta - sum_i W_i v_i (v_i^T c_n),
// W_i = sigma_i^2 / (beta^2 + beta sigma_i^2). Written literally in FP32, c_n/beta and
// the rank-r correction cancel (both ~ |g|/beta) and rounding is amplified by up to
// sigma_1^2/beta. This kernel evaluates the same f exactly rearranged. With
// g_n = V S_n (S_i = sigma_i u_i^T m_n, formed once in FP64) and V^T V = I,
//     f_n = z_n - d_n/beta + V a_n,
//     a_i = S_i/(beta + sigma_i^2) - W_i u_i,   u = V^T (beta z - d),
// none of whose terms is large against the result. Substituting this f into the
// z-step and the dual step, d cancels from both:
//     beta f + d = beta (z + V a),   d^{k+1} = beta (z^k + V a^k - z^{k+1}),
// so the iteration's state is z and the r-vector u per voxel; d is only
// materialised where the stopping test needs it. One pass over z does the whole
// iteration:
//     t     = z + V a                                                (rank-r product)
//     z'    = max(0, ((xi + beta - lambda s deg) z + lambda s sum_nbr z + beta (V a))
//                    / (xi + beta))                                  (Eq. 31)
//     d'    = beta (t - z')                                          (step 11)
//     u'    = V^T (beta z' - d') = V^T beta (2 z' - t)               (rank-r product)
// D^T D z = s (deg(n) z_n - sum_{m adjacent} z_m): the free-boundary grid Laplacian,
// s = 2 for the literal Eq. 8.
//
// State layout and tiles: z and d are kept blocked, [chunk][voxel][32 compartments], and a
// tile is a patch of bx x by x bz <= 128 voxels (patch_of, as for the tensor-core form in
// ssm_lowrank_tc.cu). A stage is half a chunk: QS = 16 compartments, 64 bytes per voxel. One
// five-dimensional TMA box loads the patch with its halo (64-byte swizzle, zero-filled
// beyond the grid), one 2D box the 16 rows of V; z' is collected in shared memory and
// leaves as a TMA store.
//
// Mapping (persistent). The work units are (segment, tile) pairs, a segment being one of
// the ranges that layout() cuts a tile's stages into; they are dealt round-robin in
// segment-major order to a grid sized to the resident capacity, so the CTAs of one round
// stream the same compartments of neighbouring tiles and the halos are L2 hits. One producer
// warp fills a ring of stages. Four consumer warps own one voxel per lane: four
// compartments at a time they read z and its neighbours with one 128-bit load each, form
// V a and u' from V rows that every lane reads (broadcasts), and keep u' in registers. At
// the end of a unit the partial u' goes to its (tile, segment) slot; the next iteration sums
// a tile's slots in segment order (fixed, hence deterministic) when it forms a.
//
// What bounds it: the FP32 pipe (2 r FMAs per element, packed), the shared-memory pipe (r / 4
// 128-bit reads of a V row per element) and the issue slots around them. With map-major
// tiles of 128 voxels, scalar loads of z and its neighbours and a store per element it
// issued 76 instructions per element and warp at r = 20 (59 at r = 8). Per iteration in a
// solve, before and now:
//   128x128, Q = 2500, r = 20            147.7 -> 125.4 us
//   192x192, Q = 900, r = 8              84.0 -> 62.3 us
//   96x96x64, Q = 1600, r = 30            4543 -> 3871 us
//   84x72, Q = 300, r = 13               12.3 -> 8.2 us
//   32x32, Q = 225, r = 20               12.4 -> 9.5 us
// A dictionary per voxel label (MULTI; ssm_plan_multi): a thread reads its voxel's own rows of
// V through L1, some pairs ahead of their use, instead of staged ones (V [q][dictionary][R]:
// the labels of a patch are mostly neighbours, and so are their rows). Two 128-bit loads per
// element at r = 8 whose lanes differ take 4 passes of L1 each, which is what bounds it.
// 156x156, Q = 900, r = 8, 61 dictionaries: 105.8 us per iteration with the table kernel
// (ssm_table.cu), now 68.8.
// HBM traffic per state element and iteration: read z, write z' (8 B); d is read/written
// only around residual tests. Every mbarrier wait is bounded and reports SSM_ETIMEOUT
// through the plan's device error word.
#pragma once

#include <algorithm>

#include "ssm_internal.cuh"
#include "ssm_tma.cuh"

namespace ssm {

struct LowrankMaps {
  CUtensorMap zi;         // z^k, box {QS, X, Y, Z, 1}
  CUtensorMap zo, di, dd; // z^{k+1}, d^k, d^{k+1}: box {QS, bx, by, bz, 1}
  CUtensorMap v;          // V (Q x R), box {R, QS}
};

struct LowrankArgs {
  const float* __restrict__ S;      // R x ld
  const float* Pin;                 // partial u of the previous iteration [tile][seg][R][TV]
                                    // (which may still run: read after pdl_wait)
  float* __restrict__ Pout;         // partial u of this iteration
  int nst;                          // stages per tile: ceil(Q / QS)
  int coff;                         // added to the chunk of the z loads: past the tensor (all
                                    // zeros, nothing read) in an iteration from z = 0
  int na, nb_seg;                   // segments (and partial-u slots) of tiles [0, fa), of the rest
  int fa;
  int nb, nob;                      // ring stages; z' (and d') buffers, 1 or 2
  const float* __restrict__ coefA;  // R (one row per dictionary)
  const float* __restrict__ coefW;  // R (one row per dictionary)
  const float* __restrict__ V;      // spatially varying dictionaries: V [q][dictionary][R],
  const int32_t* __restrict__ labels;   // each voxel's dictionary, and their number
  int ndict;
  double* __restrict__ partial;     // 4 doubles per block (check iterations)
  const uint8_t* __restrict__ mask; // voxels inside the object (nullptr: every voxel)
  int* __restrict__ err;            // device error word (SSM_ETIMEOUT on a failed wait)
  Grid g;
  Patch p;
  int write_d;                      // store d^{k+1}
  float beta, inv_beta, xi, lam_s, inv_xb;
};

// the launch of rank R with `naxes` axes of smoothness
struct LowrankKernel {
  ssm_status (*launch)(const LowrankMaps&, LowrankArgs, bool check, int64_t grid, bool chained,
                       cudaStream_t);
  int (*blocks_per_sm)(int rows);
};
LowrankKernel lowrank_kernel_small(int R, int naxes);   // R <= 16
LowrankKernel lowrank_kernel_mid(int R, int naxes);     // 20 .. 32
LowrankKernel lowrank_kernel_large(int R, int naxes);   // 40 .. 64
// a dictionary per voxel label, R <= 16
LowrankKernel lowrank_kernel_multi(int R, int naxes);

#ifdef SSM_LOWRANK_KERNEL   // the translation units that instantiate the kernel
namespace {

constexpr int TV = 128;            // lanes per tile (4 consumer warps x 32)
constexpr int NCW = 4;             // consumer warps
constexpr int NT = 32 * (NCW + 1); // + one producer warp
constexpr int QS = 16;             // compartments per stage
constexpr int kMaxNB = 6;          // ring stages at most
constexpr int OUT_BYTES = TV * 64; // one stage of a tile's z' (or d')

// registers are capped for this many resident CTAs per SM
template <int R, bool MULTI> constexpr int min_blocks() {
  return R <= (MULTI ? 12 : 20) ? 3 : (R <= 32 ? 2 : 1);
}
// MULTI: pairs of basis rows a thread has in flight ahead of the one it works on (156x156,
// Q = 900, 61 dictionaries: R = 4 with 2 pairs 67.0 us, 4 pairs 53.9; R = 8 68.8, 71.9;
// R = 16 with 1 pair 176, 2 pairs 144.5; a fourth CTA per SM instead: R = 8 86.8)
template <int R> constexpr int rows_ahead() { return R <= 4 ? 4 : 2; }
// Two compartments are worked on at once where their V rows fit the registers between the
// product with a and the part of u' (2 R, next to 2 R for a and u'), else one (R = 64 with two
// spilled 1 KB per thread: 128x100, Q = 400 125 us per iteration, now 62.7)
template <int R> constexpr bool two_at_once() { return R <= 40; }
constexpr int kMultiNB = 3;        // MULTI: ring stages (the rest of shared memory is L1)

// bytes of one stage: the staged rows and a row of zeros (swizzle atoms of 512 B), V rows, d
__host__ __device__ __forceinline__ int rows_bytes(const Patch& p) {
  return ((p.rows + 1) * 64 + 511) / 512 * 512;
}
__host__ __device__ __forceinline__ int stage_bytes(const Patch& p, int R, bool check) {
  return (rows_bytes(p) + (check ? OUT_BYTES : 0) + QS * R * 4 + 511) / 512 * 512;
}

__device__ __forceinline__ float4 lds4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(a));
  return v;
}
__device__ __forceinline__ void sts4(uint32_t a, float x, float y, float z, float w) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"r"(a), "f"(x), "f"(y), "f"(z),
               "f"(w)
               : "memory");
}

// NAX: neighbour pairs read per element (2 on 1D and 2D grids: an axis that is not there
// reads the row of zeros; 3 on 3D grids)
template <int R, int NAX, bool CHECK, bool MULTI>
__global__ void __launch_bounds__(NT, min_blocks<R, MULTI>())
    lowrank_iter_kernel(const __grid_constant__ LowrankMaps maps, const LowrankArgs a) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  pdl_launch_next();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nb = a.nb, nob = a.nob;
  const int rb = rows_bytes(a.p), stb = stage_bytes(a.p, MULTI ? 0 : R, CHECK);
  const int OB = OUT_BYTES * (a.write_d ? 2 : 1);
  unsigned char* obuf = smem + nb * stb;
  uint64_t* full = reinterpret_cast<uint64_t*>(obuf + nob * OB);
  uint64_t* empty = full + kMaxNB;
  const int nx = a.g.nx, ny = a.g.ny, nz = a.g.nz;
  const int nst = a.nst;
  if (tid == 0) {
    for (int b = 0; b < nb; ++b) {
      mbar_init(&full[b], 1);
      mbar_init(&empty[b], 1);
    }
    mbar_fence_init();
  }
  // the row of zeros after each stage's rows (no copy writes it)
  for (int i = tid; i < nb * 16; i += NT)
    reinterpret_cast<float*>(smem + (i >> 4) * stb + a.p.rows * 64)[i & 15] = 0.f;
  __syncthreads();
  bool failed = false;
  float s1 = 0.f, s2 = 0.f, s3 = 0.f;
  // (plans with a dictionary per voxel label have one segment count. At R = 8 on 2D grids the
  // compiler keeps the basis rows' loads ahead of their use only with this 64-bit arithmetic:
  // 156x156, Q = 900 68 us, else 86. Other ranks are faster with the general one: r = 4 54 -> 46)
  constexpr bool ONE = MULTI && R == 8 && NAX == 2;
  // unit k of this CTA: (segment, tile), dealt round-robin: the first tiles' units, then the
  // others', each segment-major
  auto unit_at = [&](int k, int& tile, int& sg, int& t0, int& t1, int& x0, int& y0,
                     int& z0) -> bool {
    if constexpr (ONE) {
      const int nseg = a.na;
      const int64_t u = blockIdx.x + (int64_t)k * gridDim.x;
      if (u >= a.p.ntiles * nseg) return false;
      sg = nseg > 1 ? (int)(u / a.p.ntiles) : 0;
      tile = (int)(u - sg * a.p.ntiles);
      t0 = (int)((int64_t)sg * nst / nseg);
      t1 = (int)((int64_t)(sg + 1) * nst / nseg);
    } else {
      // (32-bit arithmetic: layout() keeps the units below 2^31)
      const unsigned nf = (unsigned)a.fa * (unsigned)a.na, i = blockIdx.x + (unsigned)k * gridDim.x;
      const bool f = i < nf;
      const unsigned u = f ? i : i - nf, ns = f ? a.na : a.nb_seg;
      const unsigned nt = f ? a.fa : (unsigned)a.p.ntiles - a.fa;
      if (u >= nt * ns) return false;
      sg = ns > 1 ? (int)(u / nt) : 0;
      tile = (int)((f ? 0u : (unsigned)a.fa) + u - (unsigned)sg * nt);
      t0 = (int)((unsigned)(sg * nst) / ns);
      t1 = (int)((unsigned)((sg + 1) * nst) / ns);
    }
    const unsigned t = (unsigned)tile, tx = (unsigned)a.p.tx, ty = (unsigned)a.p.ty;
    x0 = (int)(t % tx) * a.p.bx;
    y0 = (int)(t / tx % ty) * a.p.by;
    z0 = (int)(t / tx / ty) * a.p.bz;
    return true;
  };
  // a tile's first slot of partial u
  auto slot_of = [&](int t) {
    if constexpr (ONE) return (int64_t)t * a.na;
    else return (int64_t)(t < a.fa ? t * a.na : a.fa * a.na + (t - a.fa) * a.nb_seg);
  };
  int tile, sg, t0, t1, x0, y0, z0;
  if (warp == NCW) {
    // ------------------------------- producer warp: one elected lane issues TMA
    if (lane == 0) {
      tma_prefetch_map(&maps.zi);
      if (!MULTI) tma_prefetch_map(&maps.v);
      const unsigned bytes = (unsigned)(a.p.rows * 64 + (MULTI ? 0 : QS * R * 4) +
                                        (CHECK ? a.p.bx * a.p.by * a.p.bz * 64 : 0));
      pdl_wait();
      int c = 0;   // running stage counter over all units
      for (int k = 0; !failed && unit_at(k, tile, sg, t0, t1, x0, y0, z0); ++k)
        for (int t = t0; t < t1; ++t, ++c) {
          const int b = c % nb, kb = c / nb;
          if (kb > 0 && !mbar_wait_sleep(&empty[b], (kb - 1) & 1)) {
            failed = true;
            break;
          }
          unsigned char* st = smem + b * stb;
          mbar_arrive_expect_tx(&full[b], bytes);
          const int q0 = (t & 1) * QS, ch = t >> 1;
          tma_load_5d(st, &maps.zi, q0, x0 - a.p.hx, y0 - a.p.hy, z0 - a.p.hz, ch + a.coff,
                      &full[b]);
          unsigned char* vs = st + rb;
          if (CHECK) {
            tma_load_5d(vs, &maps.di, q0, x0, y0, z0, ch, &full[b]);
            vs += OUT_BYTES;
          }
          if (!MULTI) tma_load_2d(vs, &maps.v, 0, t * QS, &full[b]);
        }
      // no copy may be in flight when the CTA exits
      for (int b = 0; b < nb && b < c; ++b) mbar_wait_sleep(&full[b], ((c - 1 - b) / nb) & 1);
    }
  } else {
    // ------------------------------- consumer warps: one voxel per lane
    const int v = warp * 32 + lane;
    const bool storer = tid == 0;
    const int64_t ld = a.g.ld, plane = (int64_t)nx * ny;
    const bool zl = nz > 1 && a.g.zlink;
    const float c2 = a.lam_s * a.inv_xb;     // weight of the neighbour sum
    const float c3 = a.beta * a.inv_xb;      // weight of V a
    const float2 c2_2 = make_float2(c2, c2), c3_2 = make_float2(c3, c3);
    const float2 m1 = make_float2(-1.f, -1.f), two2 = make_float2(2.f, 2.f);
    const float2 beta2 = make_float2(a.beta, a.beta);
    const int lx = v % a.p.bx, ly = v / a.p.bx % a.p.by, lz = v / (a.p.bx * a.p.by);
    const bool used = lz < a.p.bz;
    // row r of a stage, 64-byte swizzle: 16-byte piece j sits at j ^ ((r >> 1) & 3)
    auto srow = [](int r) { return (uint32_t)(r * 64 + (((r >> 1) & 3) << 4)); };
    const int r0 = ((lz + a.p.hz) * a.p.Y + ly + a.p.hy) * a.p.X + lx + a.p.hx;
    const uint32_t zrow = srow(a.p.rows), vrow = srow(v);
    uint32_t ro[1 + 2 * NAX];                // own row, then minus / plus per axis
    ro[0] = srow(r0);
    {
      int st[3] = {0, 0, 0}, k = 0;
      if (a.p.hx) st[k++] = 1;
      if (a.p.hy) st[k++] = a.p.X;
      if (a.p.hz) st[k++] = a.p.X * a.p.Y;
#pragma unroll
      for (int i = 0; i < NAX; ++i) {
        ro[1 + 2 * i] = i < k ? srow(r0 - st[i]) : zrow;
        ro[2 + 2 * i] = i < k ? srow(r0 + st[i]) : zrow;
      }
    }
    const uint32_t base = smem_u32(smem), ob0 = smem_u32(obuf);
    int c = 0;
    for (int k = 0; unit_at(k, tile, sg, t0, t1, x0, y0, z0); ++k) {
      const int x = x0 + lx, y = y0 + ly, z = z0 + lz;
      const bool valid = used && x < nx && y < ny && z < nz;
      const int64_t n = valid ? x + (int64_t)nx * (y + (int64_t)ny * z) : 0;
      // a voxel outside the object is left alone (its z stays 0) and is nobody's neighbour
      const uint8_t* mk = a.mask;
      const bool in = valid && (!mk || mk[n]);
      int deg = 0;
      if (in) {
        deg = (x > 0 && (!mk || mk[n - 1])) + (x < nx - 1 && (!mk || mk[n + 1])) +
              (y > 0 && (!mk || mk[n - nx])) + (y < ny - 1 && (!mk || mk[n + nx]));
        if (zl)
          deg += (z > 0 && (!mk || mk[n - plane])) + (z < nz - 1 && (!mk || mk[n + plane]));
      }
      const float e1 = (a.xi + a.beta - a.lam_s * (float)deg) * a.inv_xb;   // weight of z
      const float2 e1_2 = make_float2(e1, e1);
      // lanes outside the object read zeros for every row, so that their z', w and d' are 0
      uint32_t rr[1 + 2 * NAX];
#pragma unroll
      for (int i = 0; i < 1 + 2 * NAX; ++i) rr[i] = in ? ro[i] : zrow;
      // a_i = S_i/(beta + sigma_i^2) - W_i u_i, u_i summed over the tile's segment
      // slots of the previous iteration in segment order (R loads of a slot in flight)
      const int lab = MULTI && valid ? __ldg(a.labels + n) : 0;
      const float *cA = a.coefA + lab * R, *cW = a.coefW + lab * R;
      float2 av[R / 2];
      {
        float us[R];
        if (k == 0) pdl_wait();
#pragma unroll
        for (int i = 0; i < R; ++i) us[i] = 0.f;
        if (in) {
          const float* pt = a.Pin + slot_of(tile) * (R * TV) + v;
          int ns = a.na;
          if constexpr (!ONE) ns = tile < a.fa ? a.na : a.nb_seg;
          for (int s = 0; s < ns; ++s) {
#pragma unroll
            for (int i = 0; i < R; ++i) us[i] += pt[(s * R + i) * TV];
          }
        }
#pragma unroll
        for (int i = 0; i < R / 2; ++i) {
          float a0 = 0.f, a1 = 0.f;
          if (in) {
            a0 = __ldg(a.S + (2 * i) * ld + n) * __ldg(cA + 2 * i) - __ldg(cW + 2 * i) * us[2 * i];
            a1 = __ldg(a.S + (2 * i + 1) * ld + n) * __ldg(cA + 2 * i + 1) -
                 __ldg(cW + 2 * i + 1) * us[2 * i + 1];
          }
          av[i] = make_float2(a0, a1);
        }
      }
      float2 uacc[R / 2];
#pragma unroll
      for (int i = 0; i < R / 2; ++i) uacc[i] = make_float2(0.f, 0.f);
      // MULTI: the voxel's own basis rows, read through L1 a few pairs ahead (rows past Q are
      // zero; V has room for the last pairs ahead)
      constexpr int D = MULTI ? rows_ahead<R>() : 1;
      constexpr bool TWO = MULTI || two_at_once<R>();
      const float4* vg = reinterpret_cast<const float4*>(a.V) + lab * (R / 4);
      const int64_t vq1 = MULTI ? (int64_t)a.ndict * (R / 4) : 0;
      if (MULTI) vg += (int64_t)t0 * QS * vq1;
      float4 ahead[D][2][R / 4];
#pragma unroll
      for (int p = 0; MULTI && p < D; ++p) {
#pragma unroll
        for (int i = 0; i < R / 4; ++i) {
          ahead[p][0][i] = __ldg(vg + i);
          ahead[p][1][i] = __ldg(vg + vq1 + i);
        }
        vg += 2 * vq1;
      }
#pragma unroll 1
      for (int t = t0; t < t1; ++t, ++c) {
        const int b = c % nb;
        if (!failed && !mbar_wait_sleep(&full[b], (c / nb) & 1)) failed = true;
        if (nob == 1) {
          // the single z' buffer: the previous store has read it
          if (storer) bulk_wait_read();
          __syncwarp();
          named_barrier(1, 128);
        }
        const uint32_t sb = base + b * stb;
        const uint32_t db = sb + rb + vrow;
        const float4* v4 = reinterpret_cast<const float4*>(smem + b * stb + rb +
                                                           (CHECK ? OUT_BYTES : 0));
        const uint32_t ob = ob0 + (nob == 2 ? (c & 1) * OB : 0) + vrow;
        uint32_t za[1 + 2 * NAX];
#pragma unroll
        for (int q = 0; q < 1 + 2 * NAX; ++q) za[q] = sb + rr[q];
        // MULTI: u' of the stage by itself, then added to the running sum (the shorter chains
        // round less, as the table kernel's quarters of a segment do)
        float2 ust[R / 2];
        if (MULTI) {
#pragma unroll
          for (int i = 0; i < R / 2; ++i) ust[i] = make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int j = 0; j < QS / 4; ++j) {
          const uint32_t jx = (uint32_t)j << 4;
          const float4 z4 = lds4(za[0] ^ jx);
          float4 nb4[2 * NAX];
#pragma unroll
          for (int q = 0; q < 2 * NAX; ++q) nb4[q] = lds4(za[1 + q] ^ jx);
          // e1 z + c2 sum_nbr z needs V a last: e1 z + (c2 nb + c3 (V a))
          float2 s01 = __fadd2_rn(make_float2(nb4[0].x, nb4[0].y), make_float2(nb4[1].x, nb4[1].y));
          float2 s23 = __fadd2_rn(make_float2(nb4[0].z, nb4[0].w), make_float2(nb4[1].z, nb4[1].w));
#pragma unroll
          for (int q = 2; q < 2 * NAX; ++q) {
            s01 = __fadd2_rn(s01, make_float2(nb4[q].x, nb4[q].y));
            s23 = __fadd2_rn(s23, make_float2(nb4[q].z, nb4[q].w));
          }
          float zn[4], dn[4];
          float4 dk = make_float4(0.f, 0.f, 0.f, 0.f);
          if (CHECK) dk = lds4(db ^ jx);
          if constexpr (!TWO) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              // one compartment: its product with a, the z-step and dual step, its part of u'
              const float4* vq = v4 + (4 * j + e) * (R / 4);
              float4 vr[R / 4];
              float2 p0 = make_float2(0.f, 0.f), p1 = make_float2(0.f, 0.f);
#pragma unroll
              for (int i = 0; i < R / 4; ++i) {
                vr[i] = vq[i];
                p0 = __ffma2_rn(make_float2(vr[i].x, vr[i].y), av[2 * i], p0);
                p1 = __ffma2_rn(make_float2(vr[i].z, vr[i].w), av[2 * i + 1], p1);
              }
              auto pick = [&](const float4& f) { return e == 0 ? f.x : e == 1 ? f.y : e == 2 ? f.z : f.w; };
              const float va = (p0.x + p0.y) + (p1.x + p1.y), z = pick(z4);     // (V a)_q
              const float s = e == 0 ? s01.x : e == 1 ? s01.y : e == 2 ? s23.x : s23.y;
              const float n = fmaxf(0.f, fmaf(e1, z, fmaf(c2, s, __fmul_rn(c3, va))));
              const float t = __fadd_rn(z, va);
              const float w = __fmul_rn(a.beta, fmaf(2.f, n, -t));              // beta z' - d'
              const float2 ww = make_float2(w, w);
#pragma unroll
              for (int i = 0; i < R / 4; ++i) {
                uacc[2 * i] = __ffma2_rn(make_float2(vr[i].x, vr[i].y), ww, uacc[2 * i]);
                uacc[2 * i + 1] = __ffma2_rn(make_float2(vr[i].z, vr[i].w), ww, uacc[2 * i + 1]);
              }
              zn[e] = n;
              dn[e] = a.beta * (t - n);
              if (CHECK && in) {
                const float er = n - (t - pick(dk) * a.inv_beta), ch = n - z;
                s1 = fmaf(er, er, s1);
                s2 = fmaf(ch, ch, s2);
                s3 = fmaf(n, n, s3);
              }
            }
          } else {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              // two compartments: their products with a, then the z-step and dual step packed
              float va[2];
              float4 vr[2][R / 4];
              if constexpr (MULTI) {
                const int p = (2 * j + h) % D;
#pragma unroll
                for (int i = 0; i < R / 4; ++i) {
                  vr[0][i] = ahead[p][0][i];
                  vr[1][i] = ahead[p][1][i];
                  ahead[p][0][i] = __ldg(vg + i);
                  ahead[p][1][i] = __ldg(vg + vq1 + i);
                }
                vg += 2 * vq1;
              }
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                float2 p0 = make_float2(0.f, 0.f), p1 = make_float2(0.f, 0.f);
                const float4* vq = v4 + (4 * j + 2 * h + e) * (R / 4);
#pragma unroll
                for (int i = 0; i < R / 4; ++i) {
                  if (!MULTI) vr[e][i] = vq[i];
                  p0 = __ffma2_rn(make_float2(vr[e][i].x, vr[e][i].y), av[2 * i], p0);
                  p1 = __ffma2_rn(make_float2(vr[e][i].z, vr[e][i].w), av[2 * i + 1], p1);
                }
                va[e] = (p0.x + p0.y) + (p1.x + p1.y);     // (V a)_q
              }
              const float2 va2 = make_float2(va[0], va[1]);
              const float2 z2 = h ? make_float2(z4.z, z4.w) : make_float2(z4.x, z4.y);
              const float2 yv = __ffma2_rn(
                  e1_2, z2, __ffma2_rn(c2_2, h ? s23 : s01, __fmul2_rn(c3_2, va2)));
              const float2 n2 = make_float2(fmaxf(0.f, yv.x), fmaxf(0.f, yv.y));
              const float2 t2 = __fadd2_rn(z2, va2);
              const float2 w2 =                                  // beta z' - d'
                  __fmul2_rn(beta2, __ffma2_rn(two2, n2, __fmul2_rn(m1, t2)));
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                const float w = e ? w2.y : w2.x;
                const float2 ww = make_float2(w, w);
#pragma unroll
                for (int i = 0; i < R / 4; ++i) {
                  float2* us = MULTI ? ust : uacc;
                  us[2 * i] = __ffma2_rn(make_float2(vr[e][i].x, vr[e][i].y), ww, us[2 * i]);
                  us[2 * i + 1] = __ffma2_rn(make_float2(vr[e][i].z, vr[e][i].w), ww, us[2 * i + 1]);
                }
              }
              zn[2 * h] = n2.x;
              zn[2 * h + 1] = n2.y;
              dn[2 * h] = a.beta * (t2.x - n2.x);
              dn[2 * h + 1] = a.beta * (t2.y - n2.y);
              if (CHECK && in) {
                // f^{k+1} = t - d^k / beta
                const float f0 = t2.x - (h ? dk.z : dk.x) * a.inv_beta;
                const float f1 = t2.y - (h ? dk.w : dk.y) * a.inv_beta;
                const float ea = n2.x - f0, eb = n2.y - f1;
                const float ca = n2.x - z2.x, cb = n2.y - z2.y;
                s1 = fmaf(eb, eb, fmaf(ea, ea, s1));
                s2 = fmaf(cb, cb, fmaf(ca, ca, s2));
                s3 = fmaf(n2.y, n2.y, fmaf(n2.x, n2.x, s3));
              }
            }
          }
          sts4(ob ^ jx, zn[0], zn[1], zn[2], zn[3]);
          if (a.write_d) sts4((ob + OUT_BYTES) ^ jx, dn[0], dn[1], dn[2], dn[3]);
        }
        if (MULTI) {
#pragma unroll
          for (int i = 0; i < R / 2; ++i) uacc[i] = __fadd2_rn(uacc[i], ust[i]);
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        // the other buffer: its store (of the previous stage) has read it
        if (nob == 2 && storer) bulk_wait_read();
        __syncwarp();
        named_barrier(1, 128);
        if (storer) {
          const unsigned char* o = obuf + (nob == 2 ? (c & 1) * OB : 0);
          const int q0 = (t & 1) * QS, ch = t >> 1;
          tma_store_5d(&maps.zo, o, q0, x0, y0, z0, ch);
          if (a.write_d) tma_store_5d(&maps.dd, o + OUT_BYTES, q0, x0, y0, z0, ch);
          bulk_commit();
          mbar_arrive(&empty[b]);              // the staged rows are no longer read
        }
        __syncwarp();
      }
      // this segment's partial u' (zero for lanes outside the grid or the object)
      float* po = a.Pout + (slot_of(tile) + sg) * (R * TV) + v;
#pragma unroll
      for (int i = 0; i < R / 2; ++i) {
        po[(2 * i) * TV] = in ? uacc[i].x : 0.f;
        po[(2 * i + 1) * TV] = in ? uacc[i].y : 0.f;
      }
    }
    if (storer) bulk_wait_all();
  }
  if (failed) atomicExch(a.err, (int)SSM_ETIMEOUT);
  if (CHECK) {
    double d1 = s1, d2 = s2, d3 = s3;
    for (int o = 16; o > 0; o >>= 1) {
      d1 += __shfl_xor_sync(0xffffffffu, d1, o);
      d2 += __shfl_xor_sync(0xffffffffu, d2, o);
      d3 += __shfl_xor_sync(0xffffffffu, d3, o);
    }
    __shared__ double red[NT / 32][3];
    if (lane == 0) {
      red[warp][0] = d1;
      red[warp][1] = d2;
      red[warp][2] = d3;
    }
    __syncthreads();
    if (tid < 3) {
      double t = 0.0;
      for (int w = 0; w < NT / 32; ++w) t += red[w][tid];
      a.partial[(int64_t)blockIdx.x * 4 + tid] = t;
    }
  }
}

// shared memory for `blocks` resident CTAs per SM (228 KB per SM, 1 KB of it taken per CTA;
// at most 227 KB per CTA); the residual variant's static array comes out of it too
constexpr int smem_budget(int blocks) {
  const int b = 228 * 1024 / blocks - 1024 - 256;
  return b > 226 * 1024 ? 226 * 1024 : b / 128 * 128;
}
constexpr int kFixed = 1024 + 128;   // alignment slack, barriers

// ring stages and z' buffers: two buffers where three stages fit beside them
template <int R, bool MULTI>
bool ring(const Patch& p, bool check, bool write_d, int* nb, int* nob, int* bytes) {
  const int st = stage_bytes(p, MULTI ? 0 : R, check), ob = OUT_BYTES * (write_d ? 2 : 1);
  for (int blocks = min_blocks<R, MULTI>(); blocks >= 1; --blocks) {
    const int room = smem_budget(blocks) - kFixed;
    *nob = (room - 2 * ob) / st >= 3 ? 2 : 1;
    *nb = std::min(MULTI ? kMultiNB : kMaxNB, (room - *nob * ob) / st);
    if (*nb >= 2) {
      *bytes = kFixed + *nb * st + *nob * ob;
      return true;
    }
  }
  return false;
}

template <int R, int NAX, bool CHECK, bool MULTI>
cudaError_t allow_smem() {
  return cudaFuncSetAttribute(lowrank_iter_kernel<R, NAX, CHECK, MULTI>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
}

template <int R, int NAX, bool MULTI>
ssm_status launch_r(const LowrankMaps& maps, LowrankArgs args, bool check, int64_t grid,
                    bool chained, cudaStream_t s) {
  int bytes;
  if (!ring<R, MULTI>(args.p, check, args.write_d != 0, &args.nb, &args.nob, &bytes)) {
    set_error("low-rank form: two ring stages do not fit");
    return SSM_EUNSUPPORTED;
  }
  return check ? launch_chained(lowrank_iter_kernel<R, NAX, true, MULTI>, (unsigned)grid, NT, bytes, s,
                                chained, maps, args)
               : launch_chained(lowrank_iter_kernel<R, NAX, false, MULTI>, (unsigned)grid, NT, bytes, s,
                                chained, maps, args);
}

// resident CTAs per SM of a plain iteration with patches of `rows` staged rows (also sets the
// kernels' shared-memory limits)
template <int R, int NAX, bool MULTI>
int blocks_per_sm(int rows) {
  std::lock_guard<std::mutex> lock(attr_mutex());
  if (allow_smem<R, NAX, true, MULTI>() != cudaSuccess ||
      allow_smem<R, NAX, false, MULTI>() != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  Patch p{};
  p.rows = rows;
  int nb, nob, bytes, b = 0;
  if (!ring<R, MULTI>(p, false, false, &nb, &nob, &bytes)) return 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, lowrank_iter_kernel<R, NAX, false, MULTI>, NT, bytes);
  return std::max(1, b);
}

template <int R, bool MULTI = false>
LowrankKernel kernel_of(int naxes) {
  if (naxes == 3) return LowrankKernel{launch_r<R, 3, MULTI>, blocks_per_sm<R, 3, MULTI>};
  return LowrankKernel{launch_r<R, 2, MULTI>, blocks_per_sm<R, 2, MULTI>};
}

}  // namespace
#endif

}  // namespace ssm
