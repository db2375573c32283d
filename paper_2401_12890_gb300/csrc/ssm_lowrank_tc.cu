// One LADMM iteration of Algorithm 2 (rank-r f-step, Eq. 28) with its two rank-r products
// on the tcgen05 tensor cores ("TF32x3").
//
// The iteration is the d-free recurrence of ssm_lowrank.cu (the algebra is derived there):
// with a_i = S_i/(beta + sigma_i^2) - W_i u_i per voxel (u summed from the previous
// iteration's partial products),
//     t  = z + V a                                            (rank-r product 1)
//     z' = max(0, e1 z + c2 sum_nbr z + c3 (V a))               (Eq. 31)
//     d' = beta (t - z')                                        (step 11)
//     w  = beta (2 z' - t)            (= beta z' - d')
//     u' = V^T w                                                (rank-r product 2)
// For a tile of up to 128 voxels and a chunk of QC = 32 compartments both products are
// matrix products with the voxels as the M dimension:
//     VA [128 x 32] = A [128 x RP] . V_c^T [RP x 32]      (K = rank, padded to RP = 32/64)
//     U  [128 x RP] = W [128 x 32] . V_c   [32 x RP]      (K = the chunk's compartments)
// Both run as tcgen05.mma kind::tf32 with FP32 accumulation in tensor memory (TMEM). The
// A operands live in TMEM too: the epilogue warps own one voxel (= one TMEM lane) per thread
// and write a (once per tile segment) and w (per chunk) with tcgen05.st; the B operands
// (the chunk's rows of V and of V^T) are TMA boxes in the 128-byte-swizzled K-major layout.
//
// Precision (TF32x3): each operand x is split as x_hi = tf32(x), x_lo = tf32(x - x_hi)
// (round to nearest), and each product is formed as hi.hi + (hi.lo + lo.hi) (the dropped
// lo.lo term is ~2^-22 relative). The tensor core's FP32 accumulation does not round to
// nearest, so every chain of MMAs into one accumulator is kept short and the two parts
// go to separate accumulators: the main term hi.hi (one MMA per K step of 8) and the
// correction hi.lo + lo.hi (~2^-11 smaller, so its own accumulation error is negligible),
// added in FP32 registers with round-to-nearest. Product 2 starts from zero for every
// chunk and its 32-compartment partial sums are added into registers the same way (a
// chain over all Q compartments would bias u').
//
// State layout: z and d are kept blocked, [chunk][voxel][32 compartments], 128 bytes per
// voxel and chunk (the compartments past Q are zero and stay zero). A tile is a patch of
// bx x by x bz <= 128 voxels of the grid; one five-dimensional TMA box loads it with its
// halo as 128-byte-swizzled rows, zero-filled beyond the grid, and another stores it. What
// this buys over map-major rows of 128 voxels (the layout of F, used here before):
//   - a 16 x 8 patch of a 2D grid loads 180 rows per chunk instead of 3 x 128 and their
//     alignment slack, an 8 x 4 x 4 patch 360 instead of 5 x 128: about half the traffic
//     between L2 and the SMs, and room for more stages;
//   - a thread reads 4 compartments of a voxel (and of each neighbour) with one 128-bit
//     shared-memory load, straight into the register pairs of the packed FP32x2
//     arithmetic, and neighbours beyond the grid (or outside the object, whose z is 0)
//     read as zeros: no neighbour flags in the loop;
//   - z' leaves by TMA: no global address arithmetic and no store instructions.
// Measured per iteration in a solve, map-major tiles and one MMA warp before, now:
//   128x128, Q = 2500, r = 20            110.6 -> 74 us
//   256x256, Q = 2500, r = 20            446.9 -> 286 us (4.6 TB/s of 8 Q N bytes)
//   96x96x64, Q = 1600, r = 30            3300 -> 1833 us (4.1 TB/s)
//   192x192, Q = 900, r = 8              85.4 -> 61.3 us
//   40 slices of 37x29, Q = 225, r = 20  44.9 -> 33.4 us
//   32x32, Q = 225, r = 20               10.3 -> 6.5 us
// What bounds it now: HBM and the L2 behind it on large grids (0.6-0.7 of the measured copy
// rate), on small ones a unit's start (a-vector, filling the pipeline: about 6 chunks).
// Measured and not kept: the patch of the next chunks prefetched into L2 (256x256 -4 %, the
// others +0 to +4 %); the a-vector of the next unit formed while the last chunk of this
// one is processed, from a second TMEM buffer (128x128 -2 %, the others +2 to +12 %).
//
// Schedule (one CTA per SM): the work units are (segment, tile) pairs, segment-major,
// dealt round-robin to the CTAs; a segment is a contiguous run of a tile's chunks (one
// segment per tile when there are at least as many tiles as CTAs, several otherwise).
// CTAs running together therefore hold the same chunks of neighbouring tiles, and the
// halos are L2 hits. With between half as many tiles as CTAs and as many, each tile is one
// main unit and one tail unit instead, the tails going to the CTAs that would otherwise
// idle (see layout()). Each segment writes its partial u' to its own slot; the next
// iteration sums a tile's slots in segment order (fixed, hence deterministic). Warp roles:
//   warp 0      TMA: per chunk, the patch of z with its halo (and of d on residual-test
//               iterations)
//   warp 3      TMA: the chunk's V rows and V^T rows (hi and lo), in rings of their own: V is
//               free again when product 1 is done, well before product 2 (one ring for both
//               held product 1 back until product 2 of NSV chunks before had completed)
//   warp 1      product 1, up to NVA - 1 chunks ahead of product 2
//   warp 2      product 2 as soon as a chunk's w is complete. Two warps, because an MMA takes
//               62 cycles to issue whatever its N (measured, N <= 128): issued by one
//               thread in turn with its waits, 21 MMAs per chunk (N = 32 each) bounded the
//               whole kernel at 2900 cycles per chunk. The hi and lo rows of V lie side by
//               side as one operand of N = 64 (2 RP), which takes 14
//   warps 4-11  epilogue: two groups of four (one per TMEM lane quarter), which take the
//               chunks alternately, so that one group's waits and TMEM round trips overlap
//               the other's arithmetic: tcgen05.ld of V a, the z-step and dual step, z' (and
//               d') to shared memory, w split into TMEM, and the running sum of its chunks'
//               product 2 in registers. One thread per group issues the TMA stores.
// Waiting warps sleep in mbarrier.try_wait (with a suspend-time hint) instead of polling.
// TMEM: NVA slots of 64 columns, each holding a chunk's V a (main, correction) and then,
// column by column once read, its w (hi, lo), until product 2 of the chunk has completed. a
// (hi, lo) is per segment; U (main, correction) is double-buffered for RP = 32 and single
// for 64.
// Consecutive iterations are chained by programmatic dependent launch: a CTA of the next one
// starts on an SM as soon as it is free, initialises, loads V and S, and waits for this
// iteration to complete before it reads z and u.
// HBM traffic per state element and iteration: read z, write z' (8 B); per voxel and rank:
// S, the partial u in and out. Every mbarrier wait is bounded and reports SSM_ETIMEOUT
// through the plan's device error word; the TMA warp waits (bounded) for its last copies,
// the storing threads for their stores and the MMA warp for its last products before the
// CTA frees its TMEM and exits.
#include <algorithm>
#include <cstdlib>

#include "ssm_internal.cuh"
#include "ssm_tma.cuh"

namespace ssm {
namespace {

constexpr int TV = 128;              // lanes per tile: MMA M, TMEM lanes
constexpr int QC = 32;               // compartments per chunk
constexpr int NG = 2;                // epilogue groups of four warps
constexpr int NT = 128 + 128 * NG;
constexpr int NVA = 4;               // V a / w slots in TMEM: even, so that a slot's chunks all
                                     // belong to one group (its phases complete in the order
                                     // that group waits for them)
constexpr int kMaxNSZ = 8;           // z stages (as many as fit, at most)
constexpr int OUT_BYTES = TV * 128;  // one chunk of a tile's z' (or d')
constexpr uint32_t TMEM_COLS = 512;
constexpr int kSmemLimit = 227 * 1024;
constexpr int kReserve = 1024 + 1024 + 512 + 1024;   // alignment, the residual variant's static
                                                     // array, barriers, weights and zero row

template <int RP, int NAX>
struct Lay {
  // stages of the V ring (product 1) and of the V^T ring (product 2)
  static constexpr int NSV = RP == 32 && NAX < 3 ? NVA : NVA - 1;
  static constexpr int UB = RP == 32 ? 2 : 1;
  // V stage: per 32 ranks the chunk's rows of V_hi, then those of V_lo (one B operand of
  // N = 64); V^T stage: the rows of V_hi^T, then those of V_lo^T (one of N = 2 RP)
  static constexpr int v1(int at, int part) { return (2 * at + part) * QC * 128; }
  static constexpr int VST = RP * 256;           // bytes of either
  static constexpr uint32_t T_VA = 0;                     // slot b: 64 b (main / hi, +32)
  static constexpr uint32_t T_A = 64 * NVA;               // hi, lo at + RP
  static constexpr uint32_t T_U = T_A + 2 * RP;           // buffer b: main 2 RP b, corr + RP
  // kind::tf32 instruction descriptors: D = F32 (bits 4-5 = 1), A = B = TF32 (bits 7-9,
  // 10-12 = 2), both K-major, N >> 3 at bits 17-22, M >> 4 at bits 24-28
  static constexpr uint32_t idesc(int n) {
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(TV >> 4) << 24);
  }
  static_assert(VST == RP / 32 * 2 * QC * 128 && VST % 1024 == 0, "layout");
  static_assert(T_U + 2 * RP * UB <= TMEM_COLS, "tensor memory");
};

struct LrtcMaps {
  CUtensorMap v1h, v1l;   // V (Q x RP), box {32, QC}, 128-byte swizzle
  CUtensorMap v2h, v2l;   // V^T (RP x Qs), box {QC, RP}, 128-byte swizzle
  CUtensorMap zi;         // z^k, box {32, X, Y, Z, 1}
  CUtensorMap zo, di, dd; // z^{k+1}, d^k, d^{k+1}: box {32, bx, by, bz, 1}
};

struct LrtcArgs {
  const float* __restrict__ S;      // RP x ld
  const float* Pin;                 // partial u of the previous iteration [tile][slot][RP][TV]
                                    // (which may still run: read after pdl_wait)
  float* __restrict__ Pout;         // partial u of this iteration
  int nch;                          // compartment chunks per tile
  int full;                         // tiles [0, full) are one unit and one slot each, the others
  int spc;                          // are spc segments (contiguous runs of chunks) and slots
  int split;                        // > 0: main/tail layout, the chunk where tails start
  int kr;                           // K steps of 8 ranks holding the rank r (<= RP / 8)
  int coff;                         // added to the chunk of the z loads: past the tensor (all
                                    // zeros, nothing read) in an iteration from z = 0
  int nsz, nob;                     // z stages; z' (and d') buffers per group, 1 or 2
  const float* __restrict__ coefA;  // RP
  const float* __restrict__ coefW;  // RP
  double* __restrict__ partial;     // 4 doubles per block (check iterations)
  const uint8_t* __restrict__ mask; // voxels inside the object (nullptr: every voxel)
  int* __restrict__ err;            // device error word
  Grid g;
  Patch p;
  float beta, inv_beta, xi, lam_s, inv_xb;
};

// x rounded to TF32 (10 stored mantissa bits), to nearest with ties away from zero: add
// half a unit of the last kept place to the magnitude bits and clear the 13 bits below
// (a carry into the exponent is the correct rounding up; finite inputs of magnitude
// below 2^128 (1 - 2^-12) stay finite)
__device__ __forceinline__ float tf32_rna(float x) {
  return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u);
}

// shared-memory descriptor, K-major operand in the 128-byte swizzle layout (8 rows x
// 128 B atoms, 1024 B apart): start >> 4, leading byte offset 16 B (unused here),
// stride byte offset 1024 B, version 1 (bit 46), swizzle mode 2 = 128 B (bits 61-63)
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) |
         ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// D (TMEM) (+)= A (TMEM) . B (shared memory), kind::tf32
__device__ __forceinline__ void mma_tf32(uint32_t d_tmem, uint32_t a_tmem, uint64_t b,
                                         uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tst8(uint32_t taddr, const float* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"r"(
          taddr),
      "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
      "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
      "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7]))
      : "memory");
}
__device__ __forceinline__ void tst_wait() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// C consecutive 32-bit columns of this warp's TMEM lanes; the values are defined after the
// next tld_wait on the same registers
template <int C>
__device__ __forceinline__ void tld(uint32_t t, uint32_t* r) {
  static_assert(C == 8 || C == 16, "columns per load");
  if constexpr (C == 8)
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7])
        : "r"(t)
        : "memory");
  else
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(t)
        : "memory");
}
template <int C>
__device__ __forceinline__ void tld_wait(uint32_t* r) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < C; ++i) asm volatile("" : "+r"(r[i]));   // no use moves above the wait
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
// NAX: axes with smoothness (neighbour pairs per element)
template <int RP, int NAX, bool CHECK, bool WD>
__global__ void __launch_bounds__(NT, 1) lrtc_kernel(const __grid_constant__ LrtcMaps maps,
                                                     const LrtcArgs a) {
  using L = Lay<RP, NAX>;
  constexpr int UB = L::UB, NSV = L::NSV;
  constexpr int RQ = RP / NG;         // ranks of a per epilogue group
  constexpr int UC = RP == 64 ? 8 : 16;   // columns of u' read at once (registers)
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  // aligned by an offset from the shared array itself (not through an integer), so that
  // the compiler keeps the shared address space of every pointer derived from it
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int nsz = a.nsz, nob = a.nob;
  const int zst = a.p.zst + (CHECK ? OUT_BYTES : 0);      // z rows, then d^k
  unsigned char* v1ring = smem;
  unsigned char* v2ring = smem + NSV * L::VST;
  unsigned char* obuf = smem + 2 * NSV * L::VST;          // [group][buffer]: z', then d'
  // a residual test that also stores d writes it over the staged d^k
  constexpr bool OWN_D = WD && !CHECK;
  constexpr int OB = OUT_BYTES * (OWN_D ? 2 : 1);
  unsigned char* zring = obuf + NG * nob * OB;
  unsigned char* tail = zring + nsz * zst;
  float* zero_row = reinterpret_cast<float*>(tail);       // 128 bytes of zeros (128-aligned)
  float* cAW = zero_row + 32;                             // coefA, coefW (RP each)
  uint64_t* v1full = reinterpret_cast<uint64_t*>(cAW + 2 * RP);
  uint64_t* v2full = v1full + NSV;
  uint64_t* v1empty = v2full + NSV;
  uint64_t* v2empty = v1empty + NSV;
  uint64_t* zfull = v2empty + NSV;
  uint64_t* zempty = zfull + 2 * kMaxNSZ;
  uint64_t* va_full = zempty + kMaxNSZ;
  uint64_t* w_full = va_full + NVA;
  uint64_t* p2_done = w_full + NVA;       // product 2 of a slot's chunk has completed
  uint64_t* u_free = p2_done + NVA;
  uint64_t* a_ready = u_free + 2;
  uint64_t* a_free = a_ready + 1;
  uint64_t* fin = a_free + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(fin + 2);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // the next iteration's CTAs may take the SMs that this one leaves (or does not use) and
  // set up; what they read of this iteration they wait for (pdl_wait)
  pdl_launch_next();
  const int nch = a.nch, spc = a.spc;

  if (tid == 0) {
    for (int s = 0; s < NSV; ++s) {
      mbar_init(&v1full[s], 1);
      mbar_init(&v2full[s], 1);
      mbar_init(&v1empty[s], 1);
      mbar_init(&v2empty[s], 1);
    }
    for (int s = 0; s < nsz; ++s) {
      mbar_init(&zfull[2 * s], 1);
      mbar_init(&zfull[2 * s + 1], 1);
      mbar_init(&zempty[s], 1);
    }
    for (int i = 0; i < NVA; ++i) {
      mbar_init(&va_full[i], 1);
      mbar_init(&w_full[i], 4);
      mbar_init(&p2_done[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&u_free[i], 4);
    }
    mbar_init(a_ready, 4 * NG);
    mbar_init(a_free, 1);
    mbar_init(&fin[0], 1);
    mbar_init(&fin[1], 1);
    mbar_fence_init();
  }
  if (tid < 32) zero_row[tid] = 0.f;
  if (tid < RP) {
    cAW[tid] = a.coefA[tid];
    cAW[RP + tid] = a.coefW[tid];
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;
  bool failed = false;
  float s1 = 0.f, s2 = 0.f, s3 = 0.f;

  // the k-th unit of this CTA. Main/tail layout (a.split > 0, fewer tiles than CTAs but
  // more than half as many): CTA j < ntiles owns chunks [0, split) of tile j; the other
  // CTAs take the tails [split, nch) of tiles j - ntiles, j - ntiles + (G - ntiles), ...
  // (concurrent tails are of consecutive tiles too). Otherwise units are dealt round-robin,
  // the whole tiles first, then the segments of the others in segment-major order, so that the
  // CTAs running together hold the same chunks of consecutive tiles.
  // (32-bit division: only fewer tiles than CTAs are split into segments)
  auto unit_at = [&](int k, int& tile, int& c0, int& c1, int& sg) -> bool {
    const unsigned nt = (unsigned)a.p.ntiles, G = gridDim.x, j = blockIdx.x;
    if (a.split > 0) {
      if (j < nt) {
        if (k > 0) return false;
        tile = (int)j;
        sg = 0;
        c0 = 0;
        c1 = a.split;
        return true;
      }
      const unsigned t = j - nt + (unsigned)k * (G - nt);
      if (t >= nt) return false;
      tile = (int)t;
      sg = 1;
      c0 = a.split;
      c1 = nch;
      return true;
    }
    const int64_t u = j + (int64_t)k * G;
    if (u < a.full) {
      tile = (int)u;
      sg = 0;
      c0 = 0;
      c1 = nch;
      return true;
    }
    const unsigned rest = nt - (unsigned)a.full, v = (unsigned)(u - a.full);
    if (u - a.full >= (int64_t)rest * spc) return false;
    sg = (int)(v / rest);
    tile = a.full + (int)(v - (unsigned)sg * rest);
    c0 = sg * nch / spc;
    c1 = (sg + 1) * nch / spc;
    return true;
  };
  // a tile's first slot of partial u
  auto slot_of = [&](int t) { return t < a.full ? (int64_t)t : a.full + (int64_t)(t - a.full) * spc; };
  // first voxel of a tile
  auto origin = [&](int tile, int& x0, int& y0, int& z0) {
    const unsigned t = (unsigned)tile, tx = (unsigned)a.p.tx, ty = (unsigned)a.p.ty;
    x0 = (int)(t % tx) * a.p.bx;
    y0 = (int)(t / tx % ty) * a.p.by;
    z0 = (int)(t / tx / ty) * a.p.bz;
  };

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA: z (and d)
    if (lane == 0) {
      tma_prefetch_map(&maps.zi);
      pdl_wait();
      const unsigned zbytes = (unsigned)a.p.rows * 128u +
                              (CHECK ? (unsigned)(a.p.bx * a.p.by * a.p.bz) * 128u : 0u);
      int g = 0;
      int tile, c0, c1, sg;
      for (int k = 0; !failed && unit_at(k, tile, c0, c1, sg); ++k) {
        int x0, y0, z0;
        origin(tile, x0, y0, z0);
        for (int c = c0; c < c1; ++c, ++g) {
          const int sz = g % nsz, kz = g / nsz;
          if (kz > 0 && !mbar_wait_sleep(&zempty[sz], (kz - 1) & 1)) {
            failed = true;
            break;
          }
          // a stage's loads complete on two barriers in turn: with an odd number of stages
          // the groups alternate on a stage, and a group waiting for its load must not take
          // the one before last (of the same parity on a single barrier) for it
          unsigned char* zs = zring + sz * zst;
          uint64_t* bar = &zfull[2 * sz + (kz & 1)];
          mbar_arrive_expect_tx(bar, zbytes);
          tma_load_5d(zs, &maps.zi, 0, x0 - a.p.hx, y0 - a.p.hy, z0 - a.p.hz, c + a.coff, bar);
          if (CHECK) tma_load_5d(zs + a.p.zst, &maps.di, 0, x0, y0, z0, c, bar);
        }
      }
      // no copy may still be in flight when the CTA exits: wait (bounded) for the last
      // phase issued into every stage
      for (int s = 0; s < nsz && s < g; ++s) {
        const int kz = (g - 1 - s) / nsz;            // the stage's last round
        mbar_wait_sleep(&zfull[2 * s + (kz & 1)], (kz >> 1) & 1);
      }
    }
  } else if (warp == 3) {
    // ------------------------------------------------------------------ TMA: V and V^T
    if (lane == 0) {
      tma_prefetch_map(&maps.v1h);
      tma_prefetch_map(&maps.v2h);
      int g = 0, g2 = 0;
      int tile, c0, c1, sg;
      for (int k = 0; !failed && unit_at(k, tile, c0, c1, sg); ++k)
        for (int c = c0; c < c1; ++c, ++g) {
          const int sv = g % NSV, kv = g / NSV, q0 = c * QC;
          // a stage is free once its product has completed (where there are as many stages
          // as slots, the slot's barrier says so)
          if (kv > 0 &&
              !mbar_wait_sleep(NSV == NVA ? &va_full[sv] : &v1empty[sv], (kv - 1) & 1)) {
            failed = true;
            break;
          }
          unsigned char* vs = v1ring + sv * L::VST;
          mbar_arrive_expect_tx(&v1full[sv], (unsigned)L::VST);
#pragma unroll
          for (int at = 0; at < RP / 32; ++at) {
            tma_load_2d(vs + L::v1(at, 0), &maps.v1h, at * 32, q0, &v1full[sv]);
            tma_load_2d(vs + L::v1(at, 1), &maps.v1l, at * 32, q0, &v1full[sv]);
          }
          if (kv > 0 &&
              !mbar_wait_sleep(NSV == NVA ? &p2_done[sv] : &v2empty[sv], (kv - 1) & 1)) {
            failed = true;
            ++g;          // the V copies of this chunk were issued
            break;
          }
          vs = v2ring + sv * L::VST;
          mbar_arrive_expect_tx(&v2full[sv], (unsigned)L::VST);
          tma_load_2d(vs, &maps.v2h, q0, 0, &v2full[sv]);
          tma_load_2d(vs + L::VST / 2, &maps.v2l, q0, 0, &v2full[sv]);
          g2 = g + 1;
        }
      for (int s = 0; s < NSV && s < g; ++s)
        mbar_wait_sleep(&v1full[s], ((g - 1 - s) / NSV) & 1);
      for (int s = 0; s < NSV && s < g2; ++s)
        mbar_wait_sleep(&v2full[s], ((g2 - 1 - s) / NSV) & 1);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ product 1
    if (lane == 0) {
      const uint32_t a_hi = tmem + L::T_A, a_lo = tmem + L::T_A + RP;
      int g = 0, si = 0;
      int tile, c0, c1, sg;
      for (int k = 0; !failed && unit_at(k, tile, c0, c1, sg); ++k) {
        const int nchk = c1 - c0;
        if (!mbar_wait_sleep(a_ready, si & 1)) {
          failed = true;
          break;
        }
        fence_after();
        for (int i = 0; i < nchk; ++i) {
          // V a (main, correction) of chunk gg: a_hi . [V_hi | V_lo]^T into both, then
          // a_lo . V_hi^T into the correction; its slot's previous w has been read
          const int gg = g + i, b = gg % NVA;
          if (!mbar_wait_sleep(&v1full[gg % NSV], (gg / NSV) & 1)) failed = true;
          if (!failed && gg >= NVA && !mbar_wait_sleep(&p2_done[b], (gg / NVA - 1) & 1))
            failed = true;
          if (failed) break;
          fence_after();
          const uint32_t vs = smem_u32(v1ring + (gg % NSV) * L::VST);
          const uint32_t dm = tmem + L::T_VA + 64 * b, dc = dm + 32;
          // the padding ranks beyond r carry zero a: their K steps are skipped
#pragma unroll 4
          for (int k8 = 0; k8 < a.kr; ++k8) {
            const uint64_t bh = sdesc(vs + L::v1(k8 / 4, 0) + (k8 % 4) * 32);
            mma_tf32(dm, a_hi + 8 * k8, bh, L::idesc(2 * QC), k8 > 0 ? 1u : 0u);
            mma_tf32(dc, a_lo + 8 * k8, bh, L::idesc(QC), 1u);
          }
          commit(&va_full[b]);
          if (NSV != NVA) commit(&v1empty[gg % NSV]);
          if (i == nchk - 1) commit(a_free);     // a may be rewritten once these complete
        }
        g += nchk;
        ++si;
      }
      // every product issued has completed before the TMEM is freed
      commit(&fin[0]);
      mbar_wait_sleep(&fin[0], 0);
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------------ product 2
    if (lane == 0) {
      int g = 0;
      int tile, c0, c1, sg;
      for (int k = 0; !failed && unit_at(k, tile, c0, c1, sg); ++k) {
        for (int c = c0; c < c1; ++c, ++g) {
          // U (main, correction) of chunk g: w_hi . [V_hi | V_lo] into both, then w_lo . V_hi
          // into the correction
          const int b = g % NVA, gp = g - UB;
          if (!mbar_wait_sleep(&v2full[g % NSV], (g / NSV) & 1)) failed = true;
          if (!failed && !mbar_wait_sleep(&w_full[b], (g / NVA) & 1)) failed = true;
          // the U buffer is free once the epilogue has read chunk g - UB's
          if (!failed && gp >= 0 && !mbar_wait_sleep(&u_free[gp & 1], (gp >> 1) & 1))
            failed = true;
          if (failed) break;
          fence_after();
          const uint32_t vs = smem_u32(v2ring + (g % NSV) * L::VST);
          const uint32_t dm = tmem + L::T_U + 2 * RP * (g % UB), dc = dm + RP;
          const uint32_t w_hi = tmem + L::T_VA + 64 * b, w_lo = w_hi + 32;
#pragma unroll
          for (int k8 = 0; k8 < QC / 8; ++k8) {
            const uint64_t bh = sdesc(vs + k8 * 32);
            mma_tf32(dm, w_hi + 8 * k8, bh, L::idesc(2 * RP), k8 > 0 ? 1u : 0u);
            mma_tf32(dc, w_lo + 8 * k8, bh, L::idesc(RP), 1u);
          }
          commit(&p2_done[b]);
          if (NSV != NVA) commit(&v2empty[g % NSV]);
        }
      }
      commit(&fin[1]);
      mbar_wait_sleep(&fin[1], 0);
    }
  } else if (warp >= 4) {
    // ------------------------------------------------------------------ epilogue warps
    const int quarter = warp & 3;
    const int grp = (warp - 4) >> 2;                 // takes the chunks gg with gg % NG == grp
    const int v = quarter * 32 + lane;               // lane of the tile = TMEM lane
    const bool storer = quarter == 0 && lane == 0;   // issues the group's TMA stores
    const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
    const int64_t ld = a.g.ld;
    const int nx = a.g.nx, ny = a.g.ny, nz = a.g.nz;
    const int64_t plane = (int64_t)nx * ny;
    const bool zl = nz > 1 && a.g.zlink;
    const float c2 = a.lam_s * a.inv_xb;             // weight of the neighbour sum
    const float c3 = a.beta * a.inv_xb;              // weight of V a
    const float beta = a.beta;
    const float2 c2_2 = make_float2(c2, c2), c3_2 = make_float2(-c3, -c3);   // (of -V a)
    const float2 beta2 = make_float2(beta, beta), two2 = make_float2(2.f, 2.f);
    const float2 m1 = make_float2(-1.f, -1.f);
    // this lane's voxel within a patch, and its row among the staged rows (swizzled: the
    // 16-byte piece j of row r sits at piece j ^ (r & 7))
    const int lx = v % a.p.bx, ly = v / a.p.bx % a.p.by, lz = v / (a.p.bx * a.p.by);
    const bool used = lz < a.p.bz;
    auto srow = [](int r) { return (uint32_t)(r * 128 + ((r & 7) << 4)); };
    const int r0 = ((lz + a.p.hz) * a.p.Y + ly + a.p.hy) * a.p.X + lx + a.p.hx;
    uint32_t ro[1 + 2 * NAX];                        // own row, then minus / plus per axis
    ro[0] = srow(r0);
    {
      // strides of the axes with smoothness, in the order x, y, z
      int st[3] = {0, 0, 0}, k = 0;
      if (a.p.hx) st[k++] = 1;
      if (a.p.hy) st[k++] = a.p.X;
      if (a.p.hz) st[k++] = a.p.X * a.p.Y;
#pragma unroll
      for (int i = 0; i < NAX; ++i) {
        ro[1 + 2 * i] = srow(r0 - st[i]);
        ro[2 + 2 * i] = srow(r0 + st[i]);
      }
    }
    const uint32_t vrow = srow(v);                   // own row of an unhaloed buffer
    const uint32_t zero = smem_u32(zero_row), ring = smem_u32(zring);
    const uint32_t ob0 = smem_u32(obuf) + grp * nob * OB;

    int64_t n = 0;
    int tile = 0, c0 = 0, c1 = 0, sg = 0;
    bool in = false;
    float e1 = 0.f;
    float us[RQ], sv[RQ];
    // unit k: its voxel, and the loads of its a-vector (S and the u slots of the previous
    // iteration, in slot order)
    auto begin = [&](int k) -> bool {
      if (!unit_at(k, tile, c0, c1, sg)) return false;
      int x0, y0, z0;
      origin(tile, x0, y0, z0);
      const int x = x0 + lx, y = y0 + ly, z = z0 + lz;
      const bool valid = used && x < nx && y < ny && z < nz;
      n = valid ? x + (int64_t)nx * (y + (int64_t)ny * z) : 0;
      // a voxel outside the object is left alone (its z stays 0) and is nobody's neighbour
      const uint8_t* mk = a.mask;
      in = valid && (!mk || mk[n]);
      int deg = 0;
      if (in) {
        deg = (x > 0 && (!mk || mk[n - 1])) + (x < nx - 1 && (!mk || mk[n + 1])) +
              (y > 0 && (!mk || mk[n - nx])) + (y < ny - 1 && (!mk || mk[n + nx]));
        if (zl)
          deg += (z > 0 && (!mk || mk[n - plane])) + (z < nz - 1 && (!mk || mk[n + plane]));
      }
      e1 = (a.xi + a.beta - a.lam_s * (float)deg) * a.inv_xb;   // weight of z
      const float* pt = a.Pin + slot_of(tile) * (RP * TV) + grp * RQ * TV + v;
      const float* sp = a.S + (int64_t)(grp * RQ) * ld + n;
#pragma unroll
      for (int i = 0; i < RQ; ++i) sv[i] = in ? __ldg(sp + i * ld) : 0.f;
      if (k == 0) pdl_wait();     // S is the solve's; u is the previous iteration's
#pragma unroll
      for (int i = 0; i < RQ; ++i) us[i] = pt[i * TV];
      // the next unit's come from HBM: into L2 ahead
      {
        int t1, d0, d1, d2, x1, y1, z1;
        if (unit_at(k + 1, t1, d0, d1, d2)) {
          origin(t1, x1, y1, z1);
          const int64_t n1 = min(x1 + lx, nx - 1) +
                             (int64_t)nx * (min(y1 + ly, ny - 1) + (int64_t)ny * min(z1 + lz, nz - 1));
          const float* p1 = a.Pin + (slot_of(t1) * RP + grp * RQ) * TV + v;
          const float* s1p = a.S + (int64_t)(grp * RQ) * ld + n1;
#pragma unroll 4
          for (int i = 0; i < RQ; ++i) {
            asm volatile("prefetch.global.L2 [%0];" ::"l"(s1p + i * ld));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p1 + i * TV));
          }
        }
      }
      // (SB slots' loads in flight together; a slot past the last reads the last with weight 0)
      constexpr int SB = RQ <= 16 ? 3 : 1;
#pragma unroll 1
      for (int s = 1; tile >= a.full && s < spc; s += SB) {
        float u1[SB][RQ];
#pragma unroll
        for (int t = 0; t < SB; ++t)
#pragma unroll
          for (int i = 0; i < RQ; ++i) u1[t][i] = pt[(min(s + t, spc - 1) * RP + i) * TV];
#pragma unroll
        for (int t = 0; t < SB; ++t)
#pragma unroll
          for (int i = 0; i < RQ; ++i) us[i] += s + t < spc ? u1[t][i] : 0.f;
      }
      return true;
    };
    int g = 0, si = 0, own = 0;                      // own: chunks this group has processed
    bool more = begin(0);
    for (int k = 0; more; ++k) {
      const int nchk = c1 - c0;
      // a_i = S_i/(beta + sigma_i^2) - W_i u_i for this group's ranks
      if (si > 0 && !failed && !mbar_wait_sleep(a_free, (si - 1) & 1)) failed = true;
      fence_after();
#pragma unroll
      for (int i = 0; i < RQ; i += 8) {
        float ah[8], al[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int r = grp * RQ + i + j;
          // negated, so that -t = (-V a) - z needs no sign flips below
          const float av = in ? cAW[RP + r] * us[i + j] - sv[i + j] * cAW[r] : 0.f;
          ah[j] = tf32_rna(av);
          al[j] = tf32_rna(av - ah[j]);
        }
        tst8(tmem + lane_base + L::T_A + grp * RQ + i, ah);
        tst8(tmem + lane_base + L::T_A + RP + grp * RQ + i, al);
      }
      tst_wait();
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(a_ready);
      // lanes outside the object read zeros for every row, so that their z', w and d' are 0
      uint32_t rr[1 + 2 * NAX];
#pragma unroll
      for (int i = 0; i < 1 + 2 * NAX; ++i) rr[i] = in ? ro[i] : 0u;
      const uint32_t dro = in ? vrow : 0u;
      const float2 e1_2 = make_float2(e1, e1);
      float uacc[RP];
#pragma unroll
      for (int i = 0; i < RP; ++i) uacc[i] = 0.f;
      // product 2's sums of chunk gg (main + correction, rounded to nearest in registers)
      auto consume_u = [&](int gg) {
        if (!failed && !mbar_wait_sleep(&p2_done[gg % NVA], (gg / NVA) & 1)) failed = true;
        fence_after();
        const uint32_t ub = tmem + lane_base + L::T_U + 2 * RP * (gg % UB);
#pragma unroll
        for (int j0 = 0; j0 < RP; j0 += UC) {
          uint32_t um[2 * UC];
          tld<UC>(ub + j0, um);
          tld<UC>(ub + RP + j0, um + UC);
          tld_wait<2 * UC>(um);
#pragma unroll
          for (int j = 0; j < UC; j += 2) {
            const float2 t2 = __fadd2_rn(
                make_float2(__uint_as_float(um[j]), __uint_as_float(um[j + 1])),
                make_float2(__uint_as_float(um[UC + j]), __uint_as_float(um[UC + 1 + j])));
            const float2 s2 = __fadd2_rn(make_float2(uacc[j0 + j], uacc[j0 + j + 1]), t2);
            uacc[j0 + j] = s2.x;
            uacc[j0 + j + 1] = s2.y;
          }
        }
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&u_free[gg & 1]);
      };
      int x0, y0, z0;
      origin(tile, x0, y0, z0);
      int pend = -1;                                 // own chunk whose u is not yet summed
#pragma unroll 1
      for (int i = (g ^ grp) & 1; i < nchk; i += NG) {
        const int gg = g + i, sz = gg % nsz, b = gg % NVA;
        const int kz = gg / nsz;
        if (!failed && !mbar_wait_sleep(&zfull[2 * sz + (kz & 1)], (kz >> 1) & 1)) failed = true;
        if (!failed && !mbar_wait_sleep(&va_full[b], (gg / NVA) & 1)) failed = true;
        fence_after();
        const uint32_t tb = tmem + lane_base + L::T_VA + 64 * b;
        uint32_t vr[16];
        tld<8>(tb, vr);
        tld<8>(tb + 32, vr + 8);
        if (nob == 1) {
          // the group's single buffer: the previous store has read it
          if (storer) bulk_wait_read();
          __syncwarp();
          named_barrier(1 + grp, 128);
        }
        // (the stages are 1024-byte-aligned: the piece index only flips bits 4-6)
        const uint32_t zb = in ? ring + sz * zst : zero;
        uint32_t za[1 + 2 * NAX];
#pragma unroll
        for (int q = 0; q < 1 + 2 * NAX; ++q) za[q] = zb + rr[q];
        const uint32_t db = in ? ring + sz * zst + a.p.zst : zero;
        const uint32_t ob = ob0 + (nob == 2 ? (own & 1) * OB : 0) + vrow;
#pragma unroll
        for (int sb = 0; sb < 4; ++sb) {
          // 8 compartments: V a (the next 8's TMEM loads issued ahead), the staged rows, the
          // z-step and dual step in packed FP32x2 arithmetic (each half rounds as the scalar
          // operation)
          tld_wait<16>(vr);
          float2 va2[4];
#pragma unroll
          for (int j = 0; j < 4; ++j)
            va2[j] = __fadd2_rn(
                make_float2(__uint_as_float(vr[2 * j]), __uint_as_float(vr[2 * j + 1])),
                make_float2(__uint_as_float(vr[8 + 2 * j]), __uint_as_float(vr[9 + 2 * j])));
          if (sb < 3) {
            tld<8>(tb + 8 * (sb + 1), vr);
            tld<8>(tb + 32 + 8 * (sb + 1), vr + 8);
          }
          // (with 64 ranks 4 at a time, which leaves registers for the running u')
          constexpr int HB = RP == 64 ? 1 : 2;
          float4 zz[2], nb[2 * NAX][2], dk[2];
          float zn[8], w[8], dn[8];
#pragma unroll
          for (int h0 = 0; h0 < 2; h0 += HB) {
#pragma unroll
            for (int h = h0; h < h0 + HB; ++h) {
              const uint32_t jx = (uint32_t)(2 * sb + h) << 4;
              zz[h] = lds4(za[0] ^ jx);
#pragma unroll
              for (int q = 0; q < 2 * NAX; ++q) nb[q][h] = lds4(za[1 + q] ^ jx);
            }
            if constexpr (CHECK) {
#pragma unroll
              for (int h = h0; h < h0 + HB; ++h)
                dk[h] = lds4((db + dro) ^ ((uint32_t)(2 * sb + h) << 4));
            }
#pragma unroll
            for (int j = 2 * h0; j < 2 * (h0 + HB); ++j) {
              const int h = j >> 1;
              auto pr = [&](const float4& f) {
                return (j & 1) ? make_float2(f.z, f.w) : make_float2(f.x, f.y);
              };
              const float2 z2 = pr(zz[h]);
              float2 s = __fadd2_rn(pr(nb[0][h]), pr(nb[1][h]));
#pragma unroll
              for (int q = 2; q < 2 * NAX; ++q) s = __fadd2_rn(s, pr(nb[q][h]));
              const float2 y = __ffma2_rn(e1_2, z2, __ffma2_rn(c2_2, s, __fmul2_rn(c3_2, va2[j])));
              const float2 n2 = make_float2(fmaxf(0.f, y.x), fmaxf(0.f, y.y));
              const float2 mt = __ffma2_rn(m1, z2, va2[j]);                       // -t
              const float2 w2 = __fmul2_rn(beta2, __ffma2_rn(two2, n2, mt));
              zn[2 * j] = n2.x;
              zn[2 * j + 1] = n2.y;
              w[2 * j] = w2.x;
              w[2 * j + 1] = w2.y;
              if constexpr (WD) {
                dn[2 * j] = -beta * (mt.x + n2.x);
                dn[2 * j + 1] = -beta * (mt.y + n2.y);
              }
              if constexpr (CHECK) {
                // f^{k+1} = t - d^k / beta
                const float2 d2 = pr(dk[h]);
                const float f0 = -(mt.x + d2.x * a.inv_beta), f1 = -(mt.y + d2.y * a.inv_beta);
                const float ea = n2.x - f0, eb = n2.y - f1;
                const float ca = n2.x - z2.x, cb = n2.y - z2.y;
                s1 = fmaf(eb, eb, fmaf(ea, ea, s1));
                s2 = fmaf(cb, cb, fmaf(ca, ca, s2));
                s3 = fmaf(n2.y, n2.y, fmaf(n2.x, n2.x, s3));
              }
            }
#pragma unroll
            for (int h = h0; h < h0 + HB; ++h) {
              const uint32_t jx = (uint32_t)(2 * sb + h) << 4;
              sts4(ob ^ jx, zn[4 * h], zn[4 * h + 1], zn[4 * h + 2], zn[4 * h + 3]);
              if constexpr (OWN_D)
                sts4((ob + OUT_BYTES) ^ jx, dn[4 * h], dn[4 * h + 1], dn[4 * h + 2], dn[4 * h + 3]);
              else if constexpr (WD)
                sts4((ring + sz * zst + a.p.zst + vrow) ^ jx, dn[4 * h], dn[4 * h + 1], dn[4 * h + 2],
                     dn[4 * h + 3]);
            }
          }
          float wh[8], wl[8];
#pragma unroll
          for (int j = 0; j < 8; j += 2) {
            wh[j] = tf32_rna(w[j]);
            wh[j + 1] = tf32_rna(w[j + 1]);
            const float2 l2 =
                __ffma2_rn(m1, make_float2(wh[j], wh[j + 1]), make_float2(w[j], w[j + 1]));
            wl[j] = tf32_rna(l2.x);
            wl[j + 1] = tf32_rna(l2.y);
          }
          tst8(tb + 8 * sb, wh);
          tst8(tb + 32 + 8 * sb, wl);
          // the sums of this group's previous chunk join the running u'
          if (sb == 1 && pend >= 0) consume_u(pend);
        }
        pend = gg;
        tst_wait();
        fence_before();
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&w_full[b]);
        // the other buffer: its store (of the previous chunk) has read it, so the group may
        // write it after the barrier
        if (nob == 2 && storer) bulk_wait_read();
        __syncwarp();
        named_barrier(1 + grp, 128);
        if (storer) {
          const unsigned char* ob_ = obuf + grp * nob * OB + (nob == 2 ? (own & 1) * OB : 0);
          tma_store_5d(&maps.zo, ob_, 0, x0, y0, z0, c0 + i);
          if constexpr (OWN_D)
            tma_store_5d(&maps.dd, ob_ + OUT_BYTES, 0, x0, y0, z0, c0 + i);
          else if constexpr (WD)
            tma_store_5d(&maps.dd, zring + sz * zst + a.p.zst, 0, x0, y0, z0, c0 + i);
          bulk_commit();
          // the staged rows are no longer read (d' over the staged d^k is, by its store)
          if constexpr (WD && CHECK) bulk_wait_read();
          mbar_arrive(&zempty[sz]);
        }
        __syncwarp();
        ++own;
      }
      // the next unit's loads go out before this one's last sums are waited for (64 ranks: after
      // the sums are stored, as their registers hold both only by spilling 450 bytes per thread)
      float* po = a.Pout + (slot_of(tile) + sg) * (RP * TV) + v;
      const bool in0 = in;
      const int gl = g + nchk - 1;                   // the unit's last chunk
      if (RP == 32) more = begin(k + 1);
      if (pend >= 0) consume_u(pend);
      // the unit's partial u': the second group hands its sums over in the TMEM slot of its
      // last chunk (read by product 2, and not written by product 1 before both groups have
      // arrived for the next unit), the first adds and stores them (zero for lanes outside
      // the grid or the object). A unit of one chunk has one group's sums only
      if (nchk > 1) {
        const uint32_t xt =
            tmem + lane_base + L::T_VA + 64 * (((gl & 1) == 1 ? gl : gl - 1) % NVA);
        if (grp == 1) {
#pragma unroll
          for (int i = 0; i < RP; i += 8) tst8(xt + i, uacc + i);
          tst_wait();
          fence_before();
          asm volatile("bar.arrive 3, 256;\n" ::: "memory");
        } else {
          asm volatile("bar.sync 3, 256;\n" ::: "memory");
          fence_after();
#pragma unroll
          for (int j0 = 0; j0 < RP; j0 += 16) {
            uint32_t x[16];
            tld<16>(xt + j0, x);
            tld_wait<16>(x);
#pragma unroll
            for (int j = 0; j < 16; ++j) uacc[j0 + j] += __uint_as_float(x[j]);
          }
          fence_before();
        }
      }
      if (nchk > 1 ? grp == 0 : (gl & 1) == grp) {
#pragma unroll
        for (int i = 0; i < RP; ++i) po[i * TV] = in0 ? uacc[i] : 0.f;
      }
      if (RP == 64) more = begin(k + 1);
      g += nchk;
      ++si;
    }
    if (storer) bulk_wait_all();
  }
  if (failed) atomicExch(a.err, (int)SSM_ETIMEOUT);
  if constexpr (CHECK) {
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
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(TMEM_COLS)
                 : "memory");
  }
}

// V (Q x RP) and V^T (RP x Qs), each split into TF32 hi/lo parts (round to nearest)
__global__ void split_basis_kernel(const float* __restrict__ V32, int Q, int RP, int Qs,
                                   float* __restrict__ v1h, float* __restrict__ v1l,
                                   float* __restrict__ v2h, float* __restrict__ v2l) {
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= (int64_t)RP * Qs) return;
  const int i = (int)(idx / Qs), q = (int)(idx % Qs);
  const float x = q < Q ? V32[(int64_t)q * RP + i] : 0.f;
  const float h = tf32_rna(x);
  const float l = tf32_rna(x - h);
  v2h[idx] = h;
  v2l[idx] = l;
  if (q < Q) {
    v1h[(int64_t)q * RP + i] = h;
    v1l[(int64_t)q * RP + i] = l;
  }
}

template <int RP, int NAX, bool CHECK, bool WD>
ssm_status set_attr() {
  return cudaFuncSetAttribute(lrtc_kernel<RP, NAX, CHECK, WD>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                              kSmemLimit - (CHECK ? 1024 : 0)) == cudaSuccess
             ? SSM_OK
             : SSM_ECUDA;
}

template <int RP, int NAX>
ssm_status prepare_rn() {
  SSM_TRY((set_attr<RP, NAX, false, false>()));
  SSM_TRY((set_attr<RP, NAX, false, true>()));
  SSM_TRY((set_attr<RP, NAX, true, false>()));
  SSM_TRY((set_attr<RP, NAX, true, true>()));
  return SSM_OK;
}

// shared memory of one variant for patches of `z_bytes` bytes of staged rows: ring stages, z'
// (and d') buffers per group, dynamic bytes
struct Ring {
  int nsz, nob;
  size_t shm;
};
template <int RP, int NAX, bool CHECK, bool WD>
constexpr Ring ring_of(int z_bytes) {
  const int zst = z_bytes + (CHECK ? OUT_BYTES : 0);
  const int ob = OUT_BYTES * (WD && !CHECK ? 2 : 1);
  const int vbytes = 2 * Lay<RP, NAX>::NSV * Lay<RP, NAX>::VST;
  const int room = kSmemLimit - kReserve - vbytes;
  // two z' buffers per group spare a barrier per chunk, where three z stages still fit
  const int nob = (room - NG * 2 * ob) / zst >= 3 ? 2 : 1;
  const int fit = (room - NG * nob * ob) / zst, nsz = fit < kMaxNSZ ? fit : kMaxNSZ;
  return Ring{nsz, nob, (size_t)(kReserve - 1024) + vbytes + (size_t)(NG * nob * ob) +
                            (size_t)nsz * zst};
}

// staged rows at most: every variant has two ring stages, and 400 (3D grids) or 260 rows pack
// 128 voxels well enough. At RP = 64 the V rings leave room for 248 (2D: 260 otherwise, taken
// by patches two voxels wide and by stacks of very small slices)
template <int RP, int NAX>
constexpr int max_rows() {
  int rows = NAX == 3 ? 400 : 260;
  for (; rows > 0; --rows) {
    const int z = (rows * 128 + 1023) / 1024 * 1024;
    if (ring_of<RP, NAX, false, false>(z).nsz >= 2 && ring_of<RP, NAX, false, true>(z).nsz >= 2 &&
        ring_of<RP, NAX, true, false>(z).nsz >= 2 && ring_of<RP, NAX, true, true>(z).nsz >= 2)
      break;
  }
  return rows;
}
// (a patch of one voxel has 3, 9 or 27 rows)
static_assert(max_rows<32, 1>() == 260 && max_rows<32, 2>() == 260 && max_rows<32, 3>() == 400 &&
                  max_rows<64, 1>() == 248 && max_rows<64, 2>() == 248,
              "rows of a patch");

template <int RP, int NAX, bool CHECK, bool WD>
ssm_status launch_one(const LrtcMaps& maps, LrtcArgs args, int64_t grid, bool chained,
                      cudaStream_t s) {
  const Ring ring = ring_of<RP, NAX, CHECK, WD>(args.p.zst);
  args.nob = ring.nob;
  args.nsz = ring.nsz;
  const size_t shm = ring.shm;
  return launch_chained(lrtc_kernel<RP, NAX, CHECK, WD>, (unsigned)grid, NT, shm, s, chained, maps,
                        args);
}

template <int RP, int NAX>
ssm_status launch_rn(const LrtcMaps& maps, const LrtcArgs& args, bool check, bool write_d,
                     int64_t grid, bool chained, cudaStream_t s) {
  if (check && write_d) return launch_one<RP, NAX, true, true>(maps, args, grid, chained, s);
  if (check) return launch_one<RP, NAX, true, false>(maps, args, grid, chained, s);
  if (write_d) return launch_one<RP, NAX, false, true>(maps, args, grid, chained, s);
  return launch_one<RP, NAX, false, false>(maps, args, grid, chained, s);
}

int64_t chunks_of(const ssm_plan_s* pl) { return (pl->Q + QC - 1) / QC; }

// Launch layout: the CTAs' budget G0 (one per SM per launch wave).
//  - At least G0 tiles: whole tiles (one unit each, its whole Q range), the grid the fewest CTAs
//    that keep the rounds of G tiles equal. Where the last round has few tiles, these are split
//    into spc segments each instead, which all G0 CTAs take.
//  - Between G0/2 and G0 tiles (the 128x128 slice: 128 tiles, 152 SMs): one segment per
//    tile would leave G0 - ntiles SMs idle, two would give some CTAs two whole-Q-halves
//    of work; instead CTA j < ntiles takes chunks [0, split) of tile j and the spare
//    CTAs take the tails, `split` chosen so that both kinds finish together, a unit's start
//    counting as kStart chunks. Where the few spare CTAs would take longer over their tails
//    than a whole tile takes (many tails each, few chunks), every tile is one unit instead
//    (13 slices of 36x29, Q = 225, 130 tiles, 46 iterations: 1466 us with tails, 693
//    without; 177x74, 38 iterations 849, 571).
//  - Fewer tiles: each tile is split into spc equal segments so that all CTAs have work.
// chunks a unit's start (a-vector, filling the pipeline) takes as long as. On 128x128, Q = 2500
// (79 chunks) 6 gives split = 72: 75 us per iteration; split 70 78, 74 75, 76 77. Twice the
// ranks take twice as long (128x100, Q = 400, r = 64: 26.1 us with 6, 24.9 with 12)
constexpr int start_chunks(int R) { return R == 64 ? 12 : 6; }
struct Layout {
  int64_t cost, grid;        // (cost: chunks, starts included, one after another)
  int full, spc, split;
};
// `wanted`: the chunk where tails start (sweeps), 0 no tails, -1 by the rule
Layout layout(int64_t ntiles, int64_t nch, int64_t g0, int kStart, int64_t wanted) {
  const int64_t whole = nch + kStart;
  if (ntiles >= g0) {
    const int64_t base = ntiles / g0, rest = ntiles % g0;
    int64_t best = 1, cost = rest > 0 ? whole : 0;    // of the last round
    for (int64_t c = 2; rest > 0 && c <= nch; ++c) {
      const int64_t t = (rest * c + g0 - 1) / g0 * ((nch + c - 1) / c + kStart);
      if (t < cost) {
        cost = t;
        best = c;
      }
    }
    cost += base * whole;
    if (best > 1) return Layout{cost, g0, (int)(base * g0), (int)best, 0};
    const int64_t rounds = base + (rest > 0);
    return Layout{cost, (ntiles + rounds - 1) / rounds, (int)ntiles, 1, 0};
  }
  if (2 * ntiles > g0 && nch >= 4 && wanted != 0) {
    const int64_t spare = g0 - ntiles;
    const int64_t per = (ntiles + spare - 1) / spare;   // tails per spare CTA
    int64_t best = 1, cost = INT64_MAX;
    for (int64_t c = 1; c < nch; ++c) {
      const int64_t t = std::max(c + kStart, per * (nch - c + kStart));
      if (t < cost) {
        cost = t;
        best = c;
      }
    }
    if (wanted > 0) best = wanted;
    if (wanted < 0 && cost >= whole) return Layout{whole, ntiles, (int)ntiles, 1, 0};
    return Layout{cost, ntiles + (ntiles + per - 1) / per, 0, 2, (int)best};
  }
  const int64_t spc = std::max<int64_t>(1, std::min(nch, g0 / ntiles));
  return Layout{(nch + spc - 1) / spc + kStart, ntiles * spc, 0, (int)spc, 0};
}
Layout layout(const ssm_plan_s* pl, int64_t ntiles) {
  const int64_t nch = chunks_of(pl);
  int64_t g0 = (int64_t)sm_count() * std::max(1, pl->waves), wanted = -1;
  if (const char* env = getenv("SSM_LRTC_GRID")) {   // launch-shape override for sweeps
    const long v = atol(env);
    if (v >= 1 && v <= 65536) g0 = v;
  }
  if (const char* env = getenv("SSM_LRTC_SPLIT")) {
    const long v = atol(env);
    if (v >= 0 && v < nch) wanted = v;
  }
  return layout(ntiles, nch, g0, start_chunks(pl->R), wanted);
}

// The plan's tiles. A staged row adds 0.1 % to a tile's time, a run of them along x 0.5 % and an
// extra pass of the quarter warps' reads 1.1 %; on 3D grids 0.3, 0 and 2.7 %. (Fitted over 13
// grids and stacks, to 4 %; the patches so chosen are within 1.2 % of the best on average)
Patch tiles_of(const ssm_plan_s* pl) {
  const bool cube = grid_axes(pl->g) == 3;
  const int rows = pl->R == 64 ? max_rows<64, 2>() : cube ? max_rows<32, 3>() : max_rows<32, 2>();
  return patch_of(pl->g, PatchRule{rows, cube ? 3e-3 : 1.1e-3, cube ? 0.0 : 5e-3,
                                   cube ? 2.7e-2 : 1.06e-2,
                                   [=](int64_t nt) { return layout(pl, nt).cost; }});
}

// what a plan of this form keeps: its tiles and launch layout, and the tensor maps of both
// ping-pong halves
struct LrtcState {
  Patch p;
  Layout l;
  LrtcMaps maps[2];
  // units, and slots of partial u: one per unit
  int64_t units() const { return l.full + (p.ntiles - l.full) * l.spc; }
};

LrtcState shape_of(const ssm_plan_s* pl) {
  if (pl->lr_state) return *static_cast<const LrtcState*>(pl->lr_state);
  LrtcState st{};
  st.p = tiles_of(pl);
  st.l = layout(pl, st.p.ntiles);
  return st;
}

}  // namespace

// padded rank of the tensor-core low-rank form: 32 or 64 (0: not supported)
int lrtc_padded_rank(int r, bool three_d) {
  if (r <= 32) return 32;
  if (r <= 64 && !three_d) return 64;
  return 0;
}

int64_t lrtc_grid(const ssm_plan_s* pl) { return shape_of(pl).l.grid; }

int64_t lrtc_partial_floats(const ssm_plan_s* pl, int64_t grid) {
  (void)grid;
  return shape_of(pl).units() * (int64_t)pl->R * TV;
}

// the kernels' shared-memory limits, and the plan's tiles and tensor maps (the state
// buffers are allocated)
ssm_status lrtc_prepare(ssm_plan_s* pl) {
  {
    std::lock_guard<std::mutex> lock(attr_mutex());
    SSM_TRY((prepare_rn<32, 1>()));
    SSM_TRY((prepare_rn<32, 2>()));
    SSM_TRY((prepare_rn<32, 3>()));
    SSM_TRY((prepare_rn<64, 1>()));
    SSM_TRY((prepare_rn<64, 2>()));
  }
  auto* st = new LrtcState(shape_of(pl));
  pl->lr_state = st;
  pl->lr_grid = st->l.grid;
  const Patch& p = st->p;
  const uint64_t Q = (uint64_t)pl->Q, RP = (uint64_t)pl->R, Qs = (uint64_t)pl->lrtc_qs;
  const auto SW = CU_TENSOR_MAP_SWIZZLE_128B;
  const auto F32 = CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
  const uint64_t nx = (uint64_t)pl->g.nx, ny = (uint64_t)pl->g.ny, nz = (uint64_t)pl->g.nz;
  const uint64_t dims[5] = {QC, nx, ny, nz, (uint64_t)chunks_of(pl)};
  const uint64_t strides[4] = {128, 128 * nx, 128 * nx * ny, 128 * nx * ny * nz};
  const unsigned halo[5] = {QC, (unsigned)p.X, (unsigned)p.Y, (unsigned)p.Z, 1};
  const unsigned patch[5] = {QC, (unsigned)p.bx, (unsigned)p.by, (unsigned)p.bz, 1};
  for (int cur = 0; cur < 2; ++cur) {
    LrtcMaps& m = st->maps[cur];
    SSM_CUDA(encode_2d(&m.v1h, F32, 4, pl->V1h, RP, Q, RP, 32, QC, SW));
    SSM_CUDA(encode_2d(&m.v1l, F32, 4, pl->V1l, RP, Q, RP, 32, QC, SW));
    SSM_CUDA(encode_2d(&m.v2h, F32, 4, pl->V2h, Q, RP, Qs, QC, (unsigned)RP, SW));
    SSM_CUDA(encode_2d(&m.v2l, F32, 4, pl->V2l, Q, RP, Qs, QC, (unsigned)RP, SW));
    SSM_CUDA(encode_nd(&m.zi, F32, 5, pl->Z[cur], dims, strides, halo, SW));
    SSM_CUDA(encode_nd(&m.zo, F32, 5, pl->Z[cur ^ 1], dims, strides, patch, SW));
    SSM_CUDA(encode_nd(&m.di, F32, 5, pl->Dl[cur], dims, strides, patch, SW));
    SSM_CUDA(encode_nd(&m.dd, F32, 5, pl->Dl[cur ^ 1], dims, strides, patch, SW));
  }
  return SSM_OK;
}

void lrtc_release(ssm_plan_s* pl) {
  delete static_cast<LrtcState*>(pl->lr_state);
  pl->lr_state = nullptr;
}

// the TF32 hi/lo parts of V and V^T from the plan's FP32 basis V32 (Q x R)
ssm_status lrtc_split_basis(ssm_plan_s* pl, cudaStream_t s) {
  const int Qs = pl->lrtc_qs;
  const int64_t cnt = (int64_t)pl->R * Qs;
  split_basis_kernel<<<(unsigned)((cnt + 255) / 256), 256, 0, s>>>(
      pl->V32, pl->Q, pl->R, Qs, pl->V1h, pl->V1l, pl->V2h, pl->V2l);
  SSM_LAUNCHED();
  return SSM_OK;
}

ssm_status lrtc_iteration(ssm_plan_s* pl, int cur, bool check, bool write_d, double* partial,
                          int* nparts, cudaStream_t s) {
  const LrtcState& st = *static_cast<const LrtcState*>(pl->lr_state);
  const int64_t grid = pl->lr_grid;
  LrtcArgs a;
  a.S = pl->S;
  a.Pin = pl->U[cur];
  a.Pout = pl->U[cur ^ 1];
  a.nch = (int)chunks_of(pl);
  a.full = st.l.full;
  a.spc = st.l.spc;
  a.split = st.l.split;
  a.kr = std::max(1, std::min(pl->R / 8, (pl->r + 7) / 8));
  a.nsz = a.nob = 0;                 // set per variant (launch_one)
  a.coff = pl->from_zero ? a.nch : 0;
  a.coefA = pl->coefA;
  a.coefW = pl->coefW;
  a.partial = partial;
  a.mask = pl->mask;
  a.err = pl->dev_err;
  a.g = pl->g;
  a.p = st.p;
  a.beta = (float)pl->p.beta;
  a.inv_beta = (float)(1.0 / pl->p.beta);
  a.xi = (float)pl->xi;
  a.lam_s = (float)pl->lam_s;
  a.inv_xb = (float)(1.0 / (pl->xi + pl->p.beta));
  *nparts = (int)grid;
  const LrtcMaps& m = st.maps[cur];
  // Chained launches spare the launch gap and the set-up (32x32: 10.4 -> 7.2 us per
  // iteration; 192x192, Q = 900, two units per CTA: 65.0 -> 60.4), but let the CTAs of an
  // iteration start as the last one's leave, out of step with the tiles next to them, whose
  // halo rows they then find in L2 less often: with 31 units per CTA (96x96x64) 1877 ->
  // 1979 us. With few units per CTA the gap weighs more (256x256, 3.4 units: 273 -> 269)
  const bool chained = pl->chained && st.units() <= 8 * grid;
  if (pl->R == 32) {
    if (st.p.naxes == 1) return launch_rn<32, 1>(m, a, check, write_d, grid, chained, s);
    if (st.p.naxes == 2) return launch_rn<32, 2>(m, a, check, write_d, grid, chained, s);
    return launch_rn<32, 3>(m, a, check, write_d, grid, chained, s);
  }
  if (pl->R == 64) {
    if (st.p.naxes == 1) return launch_rn<64, 1>(m, a, check, write_d, grid, chained, s);
    if (st.p.naxes == 2) return launch_rn<64, 2>(m, a, check, write_d, grid, chained, s);
    set_error("tensor-core low-rank form: this rank is not offered on 3D grids (r <= 32)");
    return SSM_EUNSUPPORTED;
  }
  set_error("tensor-core low-rank form: unsupported padded rank");
  return SSM_EUNSUPPORTED;
}

}  // namespace ssm
