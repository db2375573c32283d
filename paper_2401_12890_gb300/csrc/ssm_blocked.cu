// The blocked state of the low-rank forms, [chunk][voxel][32 compartments], and its tiles.
#include <algorithm>

#include "ssm_internal.cuh"

namespace ssm {
namespace {

constexpr int QC = 32;               // compartments per chunk
constexpr int TV = 128;              // lanes per tile

// F (Q x ldf, map-major) from the blocked z: a block transposes 128 voxels of a chunk
// through shared memory (both sides coalesced; bound by memory)
__global__ void __launch_bounds__(256) unblock_kernel(const float* __restrict__ Z, int64_t N,
                                                      int Q, float* __restrict__ F,
                                                      int64_t ldf) {
  __shared__ float sm[QC][129];
  const int64_t n0 = blockIdx.x * (int64_t)128;
  const int c = blockIdx.y;
  const float4* src = reinterpret_cast<const float4*>(Z) + ((int64_t)c * N + n0) * (QC / 4);
  const int nv = (int)min((int64_t)128, N - n0);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int t = threadIdx.x + i * 256, n = t >> 3, j = t & 7;
    if (n < nv) {
      const float4 f = __ldg(src + t);
      sm[4 * j][n] = f.x;
      sm[4 * j + 1][n] = f.y;
      sm[4 * j + 2][n] = f.z;
      sm[4 * j + 3][n] = f.w;
    }
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int r = w; r < QC; r += 8) {
    const int q = c * QC + r;
    if (q >= Q) break;
    float* dst = F + (int64_t)q * ldf + n0;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (lane + 32 * i < nv) dst[lane + 32 * i] = sm[r][lane + 32 * i];
  }
}

}  // namespace

// axes with smoothness (at least 1: see patch_of)
int grid_axes(const Grid& g) {
  return std::max(1, (g.nx > 1) + (g.ny > 1) + (g.nz > 1 && g.zlink));
}

// The patch of a grid's tiles: among all bx x by x bz <= 128 with at most max_rows staged
// rows (halo included; what the kernel's ring has room for), the one with the least tiles x (a tile's fixed work + its staged rows). The
// weight of the fixed work (300 rows) and the penalty for rows that do not start on
// multiples of 8 (a quarter warp's 128-bit loads then meet in the same banks) only break
// near-ties: 16 x 8 (2D) and 8 x 4 x 4 (3D) where the grid divides. An axis without
// smoothness (one voxel, or the stacking axis of a batch) needs no halo; a single voxel
// takes one on x (zero-filled rows), so that there is always a neighbour pair to read.
Patch patch_of(const Grid& g, int max_rows) {
  Patch best{};
  double cost = 1e300;
  const int hy = g.ny > 1, hz = g.nz > 1 && g.zlink;
  const int hx = g.nx > 1 || (!hy && !hz);
  for (int bz = 1; bz <= std::min(g.nz, TV); ++bz)
    for (int by = 1; by <= std::min(g.ny, TV / bz); ++by)
      for (int bx = 1; bx <= std::min(g.nx, TV / (bz * by)); ++bx) {
        const int X = bx + 2 * hx, Y = by + 2 * hy, Z = bz + 2 * hz, rows = X * Y * Z;
        if (rows > max_rows) continue;
        const int64_t tx = (g.nx + bx - 1) / bx, ty = (g.ny + by - 1) / by, tz = (g.nz + bz - 1) / bz;
        const double c = (double)tx * ty * tz * (300 + rows + (bx % 8 ? 60 : 0));
        if (c < cost) {
          cost = c;
          best = Patch{bx, by, bz, hx, hy, hz, X, Y, Z, rows, (int)tx, (int)ty, (int)tz,
                       tx * ty * tz, hx + hy + hz, (rows * 128 + 1023) / 1024 * 1024};
        }
      }
  return best;
}

int64_t blocked_floats(const Grid& g, int Q) { return (int64_t)((Q + QC - 1) / QC) * QC * g.N; }

// F = z of ping-pong half `cur`
ssm_status blocked_output(const ssm_plan_s* pl, int cur, float* F, int64_t ldf, cudaStream_t s) {
  const dim3 grid((unsigned)((pl->g.N + 127) / 128), (unsigned)((pl->Q + QC - 1) / QC));
  unblock_kernel<<<grid, 256, 0, s>>>(pl->Z[cur], pl->g.N, pl->Q, F, ldf);
  SSM_LAUNCHED();
  return SSM_OK;
}

}  // namespace ssm
