// Host side of the low-rank FP32 form: launch layout, tensor maps, launches (the kernel and
// its derivation are in ssm_lowrank.cuh, instantiated in ssm_lowrank_small/mid/large.cu).
#include <algorithm>
#include <cstdlib>

#include "ssm_lowrank.cuh"

namespace ssm {
namespace {

constexpr int TV = 128, QS = 16;

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

// staged rows at most: the ring of every rank has room for two such stages (ring())
int max_rows(const ssm_plan_s* pl) { return grid_axes(pl->g) == 3 ? 400 : 260; }

// CTAs of a plan with patches of `rows` staged rows: every resident slot, times the launch waves
int64_t resident_ctas(const ssm_plan_s* pl, int rows) {
  const LowrankKernel k = kernel_for(pl, grid_axes(pl->g));
  // (which also sets the kernels' shared-memory limits)
  const int64_t g = (int64_t)sm_count() * (k.blocks_per_sm ? k.blocks_per_sm(rows) : 1) *
                    std::max(1, pl->waves);
  if (const char* env = getenv("SSM_LOWRANK_GRID")) {   // launch-shape override for sweeps
    const long v = atol(env);
    if (v >= 1 && v <= 65536) return v;
  }
  return g;
}

// Launch layout: up to G CTAs, the units (segment, tile) dealt round-robin. As many tiles as
// fill whole rounds of G units are cut into na segments each, the rest into nb, so that their
// last round is short; na and nb minimise the rounds x (rows per unit + a unit's start). One
// segment count for all tiles left the last round nearly empty where the tiles are just past
// whole rounds. (128-voxel tiles that ignore the grid, patches with one count, now):
//   56 slices of 39x26, Q = 225, r = 20  53.3  80.2  57.6 us per iteration
//   55 of 38x34                          83.9  99.4  67.5
//   27 of 24x30                          22.6  25.5  23.6
//   61x50x11, Q = 400, r = 30            84.0  129.3  87.0
//   33x27x19, Q = 400, r = 30            43.0  61.4  43.1
// Equal shares of all tiles' stages for all CTAs instead (a CTA's share then straddles tiles):
// 128x128, Q = 2500 124.3 -> 126.3, 157x131 36.6 -> 38.2 us, and a larger rounding error of u'.
struct Layout {
  int64_t cost, fa;          // (cost: a sixteenth of a row)
  int na, nb;
};
// `two_counts`: na and nb may differ (a dictionary per voxel label: one)
Layout layout(int64_t ntiles, int nst, int64_t G, int R, bool two_counts) {
  // at least two stages a unit, fewer than 2^31 units
  const int smax =
      (int)std::max<int64_t>(1, std::min<int64_t>({64, nst / 2, INT32_MAX / (2 * ntiles)}));
  // every further slot of partial u that a unit's start sums: 1.5 rows at R = 20, less where
  // R is small (97x218, r = 4 15.2 us with five segments in two rounds, 16.7 with two in one;
  // 27 slices of 24x30, r = 20 25.7 and 23.6)
  const int slot = 29 * R / (R + 4);
  auto unit = [&](int n) -> int64_t {
    return 16 * ((nst + n - 1) / n * QS + kUnitRows) + (n - 1) * slot;
  };
  Layout best{INT64_MAX, ntiles, 1, 1}, two = best;
  for (int na = 1; na <= smax; ++na) {
    const int64_t c1 = (ntiles * na + G - 1) / G * unit(na);
    if (c1 < best.cost) best = Layout{c1, ntiles, na, 1};
    const int64_t k = ntiles * na / G, fa = std::min(ntiles, k * G / na), rest = ntiles - fa;
    const int64_t ca = k * unit(na);
    for (int nb = 1; two_counts && rest > 0 && nb <= smax && ca < two.cost; ++nb) {
      const int64_t c = ca + (rest * nb + G - 1) / G * unit(nb);
      if (c < two.cost) two = Layout{c, fa, na, nb};
    }
  }
  // (a unit's start may cost more than modelled: not for less than 5 %)
  return 20 * two.cost < 19 * best.cost ? two : best;
}

// a plan's tiles and launch layout
struct Shape {
  Patch p;
  Layout l;
  int64_t G;                 // CTAs at most
  // units, and slots of partial u: one per unit
  int64_t units() const { return l.fa * l.na + (p.ntiles - l.fa) * l.nb; }
  int64_t grid() const { return std::max<int64_t>(1, std::min(G, units())); }
};

// The FP32 pipe bounds a tile's stage (2 R FMAs per element), and a tile's time hardly depends on
// its shape: at R = 20 0.03 % per staged row and 0.6 % per extra pass of the quarter warps'
// reads, more where R is small (fitted over 14 grids and stacks, to 3 %). With a dictionary per
// voxel label the first choice of patch stays (a warp's labels differ least in square patches:
// 156x156, 61 dictionaries, r = 8: 16x8 68 us per iteration, 32x4 76)
Shape shape_of(const ssm_plan_s* pl) {
  const int nst = (pl->Q + QS - 1) / QS, R = pl->R;
  const int64_t g = resident_ctas(pl, max_rows(pl));
  const bool two = pl->ndict == 0;
  PatchRule rule{max_rows(pl), 7.2e-3 / (R + 4), 0.0, 0.144 / (R + 4), nullptr};
  if (two) rule.rounds = [=](int64_t nt) { return layout(nt, nst, g, R, true).cost; };
  Shape s;
  s.p = patch_of(pl->g, rule);
  s.G = resident_ctas(pl, s.p.rows);
  s.l = layout(s.p.ntiles, nst, s.G, R, two);
  return s;
}

// what a plan of this form keeps: tiles, tensor maps of both ping-pong halves, layout
struct LowrankState {
  Shape s;
  LowrankMaps maps[2];
};

Shape plan_shape(const ssm_plan_s* pl) {
  return pl->lr_state ? static_cast<const LowrankState*>(pl->lr_state)->s : shape_of(pl);
}

}  // namespace

// A dictionary per voxel label: patch tiles up to rank 16 from 1600 voxels on, else the work
// table. Per iteration, table kernel -> this one: 156x156, Q = 900, 61 dictionaries,
// r = 4 88.1 -> 53.9 us, r = 8 105.8 -> 68.8 (random labels 134.7 -> 117.7), r = 16
// 159.4 -> 144.5, but r = 24 198.8 -> 212.2 and r = 32 355.8 -> 408.3 (the basis rows of
// the resident CTAs no longer fit L1, and fewer threads wait for them); 40x40, Q = 300, r = 8
// 8.1 -> 8.0, but 1000 voxels 6.6 -> 6.8 and 16x16 6.2 -> 6.4 (two to eight tiles of 128
// voxels, in at most 10 segments each, leave most SMs idle; the table's tiles are 32).
bool lowrank_multi_patches(const ssm_plan_s* pl) { return pl->R <= 16 && pl->g.N >= 1600; }

int64_t lowrank_grid(const ssm_plan_s* pl) { return plan_shape(pl).grid(); }

int64_t lowrank_partial_floats(const ssm_plan_s* pl, int64_t grid) {
  (void)grid;
  return plan_shape(pl).units() * (int64_t)pl->R * TV;
}

// the plan's tiles, launch layout and tensor maps (the state buffers are allocated)
ssm_status lowrank_prepare(ssm_plan_s* pl) {
  auto* st = new LowrankState{shape_of(pl), {}};
  pl->lr_state = st;
  const Patch& p = st->s.p;
  pl->lr_grid = st->s.grid();
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
  const LowrankKernel k = kernel_for(pl, st.s.p.naxes);
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
  a.fa = (int)st.s.l.fa;
  a.na = st.s.l.na;
  a.nb_seg = st.s.l.nb;
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
  a.p = st.s.p;
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
  const bool chained = pl->chained && st.s.units() <= 8 * grid;
  return k.launch(st.maps[cur], a, check, grid, chained, s);
}

}  // namespace ssm
