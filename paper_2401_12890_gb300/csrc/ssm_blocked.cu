// The blocked state of the low-rank forms, [chunk][voxel][32 compartments], and its tiles.
#include <algorithm>
#include <map>

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

namespace {

// Extra shared-memory passes of a read of every lane's own row, 16 bytes each: the lanes of a
// quarter warp whose rows are equal mod 8 meet in the same banks (rows of 64 or 128 bytes in
// their swizzles)
int conflicts(int bx, int by, int bz, int hx, int hy, int hz) {
  const int X = bx + 2 * hx, Y = by + 2 * hy;
  int extra = 0;
  for (int q = 0; q < TV; q += 8) {
    int n[8] = {0}, most = 1;
    for (int v = q; v < q + 8 && v < bx * by * bz; ++v) {
      const int lx = v % bx, ly = v / bx % by, lz = v / (bx * by);
      most = std::max(most, ++n[(((lz + hz) * Y + ly + hy) * X + lx + hx) % 8]);
    }
    extra += most - 1;
  }
  return extra;
}

}  // namespace

// The patch of a grid's tiles, among all bx x by x bz <= 128 with at most max_rows staged rows
// (halo included; what the kernel's ring has room for). First choice: the least tiles x (300 +
// staged rows + 60 for rows that do not start on multiples of 8): 16 x 8 (2D) and 8 x 4 x 4 (3D)
// where the grid divides. It knows nothing of the rounds that its tiles take: 56 slices of 39x26
// would be 560 patches of 8x13, four rounds of 152 CTAs, instead of 504 of 13x9. So another one is
// taken if it is 3 % better (about the model's error) by
//     rounds(tiles) (1 + row x staged rows + line x runs of them along x + conflict x extra passes)
// and few tiles, rounds() the time of the launch layout that so many tiles get, the weights
// fitted to the times of 370 (grid, patch) pairs (see PatchRule's users). An axis without
// smoothness (one voxel, or the stacking axis of a batch) needs no halo; a single voxel takes
// one on x (zero-filled rows), so that there is always a neighbour pair to read.
Patch patch_of(const Grid& g, const PatchRule& rule) {
  const int hy = g.ny > 1, hz = g.nz > 1 && g.zlink;
  const int hx = g.nx > 1 || (!hy && !hz);
  auto candidates = [&](auto&& f) {
    for (int bz = 1; bz <= std::min(g.nz, TV); ++bz)
      for (int by = 1; by <= std::min(g.ny, TV / bz); ++by)
        for (int bx = 1; bx <= std::min(g.nx, TV / (bz * by)); ++bx) {
          const int X = bx + 2 * hx, Y = by + 2 * hy, Z = bz + 2 * hz;
          if (X * Y * Z > rule.max_rows) continue;
          const int64_t tx = (g.nx + bx - 1) / bx, ty = (g.ny + by - 1) / by, tz = (g.nz + bz - 1) / bz;
          f(Patch{bx, by, bz, hx, hy, hz, X, Y, Z, X * Y * Z, (int)tx, (int)ty, (int)tz, tx * ty * tz,
                  hx + hy + hz, (X * Y * Z * 128 + 1023) / 1024 * 1024});
        }
  };
  int64_t least = INT64_MAX;
  Patch best{};
  double cost = 1e300;
  candidates([&](const Patch& p) {
    least = std::min(least, p.ntiles);
    const double c = (double)p.ntiles * (300 + p.rows + (p.bx % 8 ? 60 : 0));
    if (c < cost) {
      cost = c;
      best = p;
    }
  });
  if (!rule.rounds) return best;
  // (a small grid's segments could take any number of tiles in one round, but every tile costs
  // a unit's whole work)
  std::map<int64_t, int64_t> rounds;          // (the candidates share few tile counts)
  auto time = [&](const Patch& p) {
    auto r = rounds.find(p.ntiles);
    if (r == rounds.end()) r = rounds.emplace(p.ntiles, rule.rounds(p.ntiles)).first;
    return (double)r->second * (1 + 0.3 * ((double)p.ntiles / least - 1)) *
           (1 + rule.row * p.rows + rule.line * p.Y * p.Z +
            rule.conflict * conflicts(p.bx, p.by, p.bz, hx, hy, hz));
  };
  cost = 0.97 * time(best);
  candidates([&](const Patch& p) {
    if (4 * p.ntiles > 5 * least) return;
    const double c = time(p);
    if (c < cost) {
      cost = c;
      best = p;
    }
  });
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
