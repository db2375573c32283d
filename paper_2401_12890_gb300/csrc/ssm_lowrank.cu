// Host side of the low-rank FP32 form: launch layout, tensor maps, launches (the kernel and
// its derivation are in ssm_lowrank.cuh, instantiated in ssm_lowrank_small/mid/large.cu).
#include <algorithm>
#include <cstdlib>

#include "ssm_lowrank.cuh"

namespace ssm {
namespace {

constexpr int TV = 128, QS = 16;

// the plan's tiles: at most 400 staged rows on 3D grids, else 260 (the ring of every rank has
// room for two such stages: ring())
Patch tiles_of(const ssm_plan_s* pl) {
  return patch_of(pl->g, grid_axes(pl->g) == 3 ? 400 : 260);
}

// a unit's start (the a-vector from the segment slots, the partial u' at its end) costs
// about as much as this many compartment rows (8, 24 and 64 give the same times within 1 % on
// 32x32 .. 192x192)
constexpr int kUnitRows = 24;

LowrankKernel kernel_for(const ssm_plan_s* pl, int naxes) {
  const int R = pl->R;
  if (pl->ndict > 0) return lowrank_kernel_multi(R, naxes);
  if (R <= 16) return lowrank_kernel_small(R, naxes);
  if (R <= 32) return lowrank_kernel_mid(R, naxes);
  return lowrank_kernel_large(R, naxes);
}

// Launch layout: G CTAs (every resident slot, times the launch waves) and nseg segments
// per tile, the units (segment, tile) dealt round-robin. nseg minimises rounds x (rows
// per unit + a unit's start), rounds = ceil(ntiles nseg / G).
void layout(const ssm_plan_s* pl, const Patch& p, int64_t* grid, int* nseg) {
  const LowrankKernel k = kernel_for(pl, p.naxes);
  int64_t g0 = (int64_t)sm_count() * (k.blocks_per_sm ? k.blocks_per_sm(p) : 1) *
               std::max(1, pl->waves);
  if (const char* env = getenv("SSM_LOWRANK_GRID")) {   // launch-shape override for sweeps
    const long v = atol(env);
    if (v >= 1 && v <= 65536) g0 = v;
  }
  const int nst = (pl->Q + QS - 1) / QS;
  const int smax = std::max(1, std::min(64, nst / 2));   // at least two stages a unit
  int best = 1;
  int64_t cost = INT64_MAX;
  for (int sg = 1; sg <= smax; ++sg) {
    const int64_t rounds = (p.ntiles * sg + g0 - 1) / g0;
    const int64_t c = rounds * ((nst + sg - 1) / sg * QS + kUnitRows);
    if (c < cost) {
      cost = c;
      best = sg;
    }
  }
  *nseg = best;
  *grid = std::max<int64_t>(1, std::min<int64_t>(g0, p.ntiles * best));
}

// what a plan of this form keeps: tiles, tensor maps of both ping-pong halves, layout
struct LowrankState {
  Patch p;
  LowrankMaps maps[2];
  int nseg = 1;
};

}  // namespace

// A dictionary per voxel label: patch tiles up to rank 16 from 1600 voxels on, else the work
// table. Per iteration, table kernel -> this one: 156x156, Q = 900, 61 dictionaries,
// r = 4 88.1 -> 53.9 us, r = 8 105.8 -> 68.8 (random labels 134.7 -> 117.7), r = 16
// 159.4 -> 144.5, but r = 24 198.8 -> 212.2 and r = 32 355.8 -> 408.3 (the basis rows of
// the resident CTAs no longer fit L1, and fewer threads wait for them); 40x40, Q = 300, r = 8
// 8.1 -> 8.0, but 1000 voxels 6.6 -> 6.8 and 16x16 6.2 -> 6.4 (two to eight tiles of 128
// voxels, in at most 10 segments each, leave most SMs idle; the table's tiles are 32).
bool lowrank_multi_patches(const ssm_plan_s* pl) { return pl->R <= 16 && pl->g.N >= 1600; }

int64_t lowrank_grid(const ssm_plan_s* pl) {
  int64_t grid;
  int nseg;
  layout(pl, tiles_of(pl), &grid, &nseg);
  return grid;
}

int64_t lowrank_partial_floats(const ssm_plan_s* pl, int64_t grid) {
  (void)grid;
  int64_t g;
  int nseg;
  const Patch p = tiles_of(pl);
  layout(pl, p, &g, &nseg);
  return p.ntiles * nseg * (int64_t)pl->R * TV;
}

int lowrank_max_partials(const ssm_plan_s* pl) { return (int)lowrank_grid(pl); }

// the plan's tiles, launch layout and tensor maps (the state buffers are allocated)
ssm_status lowrank_prepare(ssm_plan_s* pl) {
  auto* st = new LowrankState();
  pl->lr_state = st;
  st->p = tiles_of(pl);
  layout(pl, st->p, &pl->lr_grid, &st->nseg);
  const Patch& p = st->p;
  const auto F32 = CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
  const auto SW = CU_TENSOR_MAP_SWIZZLE_64B;
  const uint64_t nx = (uint64_t)pl->g.nx, ny = (uint64_t)pl->g.ny, nz = (uint64_t)pl->g.nz;
  const uint64_t dims[5] = {32, nx, ny, nz, ((uint64_t)pl->Q + 31) / 32};
  const uint64_t strides[4] = {128, 128 * nx, 128 * nx * ny, 128 * nx * ny * nz};
  const unsigned halo[5] = {QS, (unsigned)p.X, (unsigned)p.Y, (unsigned)p.Z, 1};
  const unsigned patch[5] = {QS, (unsigned)p.bx, (unsigned)p.by, (unsigned)p.bz, 1};
  for (int cur = 0; cur < 2; ++cur) {
    LowrankMaps& m = st->maps[cur];
    SSM_CUDA(encode_nd(&m.zi, F32, 5, pl->Z[cur], dims, strides, halo, SW));
    SSM_CUDA(encode_nd(&m.zo, F32, 5, pl->Z[cur ^ 1], dims, strides, patch, SW));
    SSM_CUDA(encode_nd(&m.di, F32, 5, pl->Dl[cur], dims, strides, patch, SW));
    SSM_CUDA(encode_nd(&m.dd, F32, 5, pl->Dl[cur ^ 1], dims, strides, patch, SW));
    if (pl->ndict > 0) continue;     // their rows are not staged
    SSM_CUDA(encode_2d(&m.v, F32, 4, pl->V32, (uint64_t)pl->R, (uint64_t)pl->Q, (uint64_t)pl->R,
                       (unsigned)pl->R, QS));
  }
  return SSM_OK;
}

void lowrank_release(ssm_plan_s* pl) {
  delete static_cast<LowrankState*>(pl->lr_state);
  pl->lr_state = nullptr;
}

ssm_status lowrank_iteration(ssm_plan_s* pl, int cur, bool check, bool write_d, double* partial,
                             int* nparts, cudaStream_t s) {
  const LowrankState& st = *static_cast<const LowrankState*>(pl->lr_state);
  const LowrankKernel k = kernel_for(pl, st.p.naxes);
  if (!k.launch) {
    set_error("low-rank kernel: unsupported padded rank");
    return SSM_EUNSUPPORTED;
  }
  const int64_t grid = pl->lr_grid;
  LowrankArgs a;
  a.S = pl->S;
  a.Pin = pl->U[cur];
  a.Pout = pl->U[cur ^ 1];
  a.nst = (pl->Q + QS - 1) / QS;
  a.nseg = st.nseg;
  a.coff = pl->from_zero ? (pl->Q + 31) / 32 : 0;
  a.nb = a.nob = 0;                  // set per variant (the launch)
  a.coefA = pl->coefA;
  a.coefW = pl->coefW;
  a.V = pl->V32;
  a.labels = pl->labels;
  a.ndict = pl->ndict;
  a.partial = partial;
  a.mask = pl->mask;
  a.err = pl->dev_err;
  a.g = pl->g;
  a.p = st.p;
  a.write_d = write_d ? 1 : 0;
  a.beta = (float)pl->p.beta;
  a.inv_beta = (float)(1.0 / pl->p.beta);
  a.xi = (float)pl->xi;
  a.lam_s = (float)pl->lam_s;
  a.inv_xb = (float)(1.0 / (pl->xi + pl->p.beta));
  *nparts = (int)grid;
  // Chained where the launch gap weighs: 32x32 12.3 -> 9.2 us per iteration, 192x192 at
  // Q = 900 65.7 -> 62.4, 128x128 at Q = 2500 129.7 -> 126.1; with more units per CTA it gives
  // nothing (256x256 510.7 -> 508.1, 96x96x64 3893 -> 3893)
  const bool chained = pl->chained && st.p.ntiles * st.nseg <= 8 * grid;
  return k.launch(st.maps[cur], a, check, grid, chained, s);
}

}  // namespace ssm
