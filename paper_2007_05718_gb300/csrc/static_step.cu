// Host side of the static step: tile plans, the persistent grid, tensor maps
// and the dispatch to the translation unit of a plan (static_step.h).
#include "static_step.h"

#include <algorithm>
#include <numeric>

#include "tma_common.cuh"

namespace lbrt {

// Tile plans: directions per warp, planes the grid must have, most warps; in
// order of preference.  A scheduler holds floor(16384 / (32 x registers))
// warps, counted in groups of four per CTA: 96 registers allow 5 per scheduler
// (two CTAs of 9 warps, ico-42 with 45 internal directions, or one of 17), 128
// allow 4 (one CTA of 16 warps, ico-162 with 176 internal directions).  The
// plan fixes the direction grouping, and with it the layout of the populations
// and the order of every sum.
namespace {
constexpr TilePlan kPlansF32[] = {{5, 2, 10}, {11, 1, 16}, {10, 1, 17}, {8, 2, 12}, {4, 2, 16}, {4, 1, 20}};
constexpr TilePlan kPlans16Small[] = {{5, 1, 9}, {4, 1, 16}};
constexpr TilePlan kPlans16[] = {{5, 1, 10}, {11, 1, 16}, {10, 1, 17}, {8, 1, 16}, {4, 1, 20}};
}  // namespace

int static_plan_lists(int storage, const TilePlan* lists[2], int counts[2]) {
  if (storage == ST_F32) {
    lists[0] = kPlansF32;
    counts[0] = sizeof(kPlansF32) / sizeof(kPlansF32[0]);
    return 1;
  }
  lists[0] = kPlans16Small;
  counts[0] = sizeof(kPlans16Small) / sizeof(kPlans16Small[0]);
  lists[1] = kPlans16;
  counts[1] = sizeof(kPlans16) / sizeof(kPlans16[0]);
  return 2;
}

// Planes per batch of the plan's kernel.  5 directions per warp work two
// planes a batch, which halves the per-batch work of a warp (128^3 x 42
// sphere, float16: 0.228 -> 0.175 ms a step).  The flux terms leave no
// registers for that (128^3 x 42 float32 with kappa_1: two planes 308 to 329 us a
// step, one plane 228), and a 2D grid has one plane.
int static_zc(int dpt, const Grid& g) { return dpt == 5 && g.dims == 3 && g.nz >= 2 ? 2 : 1; }
int static_flux_zc(int) { return 1; }

// Planes per batch of the alternative batched kernel (same memory layout,
// other registers; the batch autotuner times it against the plan's own), or 0.
int batch_alt_zc(int dpt, int zc) { return dpt == 5 && zc == 2 ? 1 : 0; }

namespace {

cudaError_t run(int storage, StaticCall c) {
  static const CUtensorMap no_map{};
  static const ProblemDesc no_problem{};
  static const DirTable no_dirs{};
  if (!c.tmap) c.tmap = &no_map;
  if (!c.emap) c.emap = &no_map;
  if (!c.one) c.one = &no_problem;
  if (!c.dirs) c.dirs = &no_dirs;
  typedef cudaError_t (*Fn)(const StaticCall&);
  static const Fn fns[3][4] = {{static_f32_d5, static_f32_d11, static_f32_d10, static_f32_d84},
                               {static_f16_d5, static_f16_d11, static_f16_d10, static_f16_d84},
                               {static_bf16_d5, static_bf16_d11, static_bf16_d10, static_bf16_d84}};
  const int p = c.dpt == 5 ? 0 : c.dpt == 11 ? 1 : c.dpt == 10 ? 2 : c.dpt == 8 || c.dpt == 4 ? 3 : -1;
  if (p < 0 || storage < 0 || storage > 2) return cudaErrorInvalidValue;
  return fns[storage][p](c);
}

cudaError_t run_pair(int storage, const StaticPairCall& c) {
  if (storage == ST_F32) return static_f32_pair(c);
  if (storage == ST_F16) return static_f16_pair(c);
  if (storage == ST_BF16) return static_bf16_pair(c);
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_step_static(const StepLaunch& L, const StaticCoef& c, const DirTable& t, int storage,
                               cudaStream_t s, int* nblocks) {
  const bool f32 = storage == ST_F32;
  if (!L.tmap_in || (!f32 && (!L.tmap_e || !L.e_out)) || L.nzc < 1 || L.nzc > march_length(L.g) || L.ctas < 1 ||
      L.nzc_flux < 1 || L.nzc_flux > march_length(L.g) || L.ctas_flux < 1)
    return cudaErrorInvalidValue;
  ProblemDesc one{};
  one.g = L.g;
  one.out = L.out;
  one.e_out = L.e_out;
  one.cf = c;
  one.dt = L.dt;
  one.collision = L.collision;
  one.lambda_iters = L.lambda_iters;
  one.nzc = L.nzc;
  one.ntiles = static_tiles(L.g, L.nzc);
  one.budget_partials = L.budget_partials;
  one.mom_E = f32 ? L.mom_E : nullptr;
  one.mom_F = f32 ? L.mom_F : nullptr;
  StaticCall k;
  k.mode = one.mom_E || one.mom_F ? 2 : 0;
  k.flux = has_flux(c);
  k.budget = L.budget_partials != nullptr;
  k.dpt = L.dpt;
  k.zc = L.zc;
  k.N = L.N;
  k.ntiles = one.ntiles;
  k.ctas = L.ctas;
  const bool fl = k.flux || k.mode == 2;
  k.tmap = fl && L.tmap_flux ? L.tmap_flux : L.tmap_in;
  k.emap = fl && L.tmap_flux ? L.tmap_e_flux : L.tmap_e;
  if (fl) k.ctas = L.ctas_flux, one.nzc = L.nzc_flux, one.ntiles = k.ntiles = static_tiles(L.g, L.nzc_flux);
  k.one = &one;
  k.nprob = 1;
  // energy budget: a partial sum per 32 sites of a row, stored by the unit that
  // owns them, so that its order does not depend on who ran which tile
  const long long nslots = (long long)((L.g.nx + 31) / 32) * L.g.ny * L.g.nz;
  if (L.budget_partials && nslots > L.partials_cap) return cudaErrorInvalidValue;
  if (nblocks) *nblocks = (int)nslots;
  k.err = L.err;
  k.sched = L.sched;
  k.dirs = &t;
  k.stream = s;
  return run(storage, k);
}

cudaError_t launch_static_batch(const BatchLaunch& B, const DirTable& t, cudaStream_t s) {
  if (!B.table || B.nprob < 1) return cudaErrorInvalidValue;
  StaticCall k;
  k.mode = 1;
  k.flux = B.flux;
  k.alt = B.alt;
  k.dpt = B.dpt;
  k.zc = B.zc;
  k.N = B.N;
  k.table = B.table;
  k.nprob = B.nprob;
  k.ntiles = B.ntiles;
  k.ctas = B.ctas;
  k.err = B.err;
  k.sched = B.sched;
  k.dirs = &t;
  k.stream = s;
  return run(B.storage, k);
}

// Resident CTAs per SM of the kernel that such a launch takes.  The kernels with
// and without the flux terms, and the alternative one of a plan, differ: 45
// float32 directions in a batch are 2, 2 and 3 CTAs of 9 warps.
static cudaError_t occupancy(int storage, int mode, int dpt, int zc, int Ni, int alt, bool flux, int* per_sm) {
  StaticCall k;
  k.mode = mode;
  k.flux = flux;
  k.alt = alt;
  k.dpt = dpt;
  k.zc = zc;
  k.N = Ni;
  k.per_sm = per_sm;
  return run(storage, k);
}

cudaError_t occupancy_static(int storage, int dpt, int zc, int Ni, bool flux, int* per_sm) {
  return occupancy(storage, 0, dpt, zc, Ni, 0, flux, per_sm);
}

cudaError_t occupancy_static_batch(int storage, int dpt, int zc, int Ni, int alt, bool flux, int* per_sm) {
  return occupancy(storage, 1, dpt, zc, Ni, alt, flux, per_sm);
}

bool static_batch_pair_supported(int dpt_a, int zc_a, int dpt_b, int zc_b) {
  return dpt_a == 5 && zc_a == 2 && dpt_b == 11 && zc_b == 1;
}

cudaError_t launch_static_batch_pair(const BatchLaunch& A, const DirTable& ta, const BatchLaunch& B,
                                     const DirTable& tb, int ctas_a, int ctas, cudaStream_t s) {
  if (A.storage != B.storage || !static_batch_pair_supported(A.dpt, A.zc, B.dpt, B.zc))
    return cudaErrorInvalidValue;
  StaticPairCall k;
  k.flux = A.flux || B.flux;
  k.a = A;
  k.b = B;
  k.dirs_a = &ta;
  k.dirs_b = &tb;
  k.ctas_a = ctas_a;
  k.ctas = ctas;
  k.stream = s;
  return run_pair(A.storage, k);
}

cudaError_t occupancy_static_batch_pair(int storage, int dpt_a, int zc_a, int Na, int dpt_b, int zc_b, int Nb,
                                        bool flux, int* per_sm) {
  if (!static_batch_pair_supported(dpt_a, zc_a, dpt_b, zc_b)) return cudaErrorInvalidValue;
  static const DirTable no_dirs{};
  StaticPairCall k;
  k.flux = flux;
  k.a.N = Na;
  k.b.N = Nb;
  k.dirs_a = k.dirs_b = &no_dirs;
  k.per_sm = per_sm;
  return run_pair(storage, k);
}

// Persistent grid of the tiled kernels: CTAs = resident CTAs per SM x SMs (at
// most one per tile), and the number of chunks nzc of the march axis.
//
// Static step: tiles are taken from a counter as CTAs come free, so the time
// is about the mean of the evenly shared work and of the busiest SM's whole
// tiles, plus half a tile for the end of the launch.  A tile's work is its
// batches (a 3D tile of l planes loads l + 1, rounded up to whole batches).
// Kernels with the flux terms, and those of three or more small CTAs an SM, go
// by the busiest CTA instead: they are bound by the latency of a batch's chain,
// which the CTAs of an SM go through side by side, and want shorter tiles (us a
// step: 64^3 x 12 with the flux terms 37 -> 29, 64^3 x 42 48 -> 46, 93x61x47 x 72
// 98 -> 91, 100^3 x 12 110 -> 95).  For two CTAs an SM without the flux terms that
// would be faster alone (64^3 x 42 51 -> 42) but slower beside the steps of other
// handles, which fill the ends of a launch (three 128^3 x 42 spheres 2.5 %, three
// 96x49x33 x 42 bfloat16 problems 13 %): the planes read twice are work.
//
// Moving step: tiles cta, cta + ncta, ...; the count minimises the busiest
// CTA's share of plane loads.
cudaError_t plan_static_grid(const Grid& g, int Ni, int dpt, int zc, int storage, int* nzc,
                             int* ctas, bool moving, bool flux) {
  const int G = Ni / dpt;
  int per_sm = 0;
  cudaError_t e = cudaErrorInvalidValue;
  if (moving) {
    e = storage == ST_F32 ? occupancy_tma_moving(dpt, G, &per_sm)
                          : occupancy_tma16_moving(storage, dpt, G, &per_sm);
  } else {
    e = occupancy_static(storage, dpt, zc, Ni, flux, &per_sm);
  }
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  int dev = 0, sms = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const long long slots = (long long)per_sm * sms;
  const int nxb = (g.nx + 63) / 64;
  if (!moving) {
    const bool flat = marches_in_y(g);
    const int march = march_length(g);
    const long long columns = (long long)nxb * march_rows(g);
    // A tile is at most about 720 KB of populations per SM long (16 planes of
    // 176 float32 directions): CTAs drift apart within a tile, and the second
    // reader of an upwind row must find it in L2.  256^3 x 162 float32, four
    // boards, ms a step: 16 planes 5.1 - 5.8, 64 planes 5.3 - 8.1.
    const long long plane = 64LL * Ni * (storage == ST_F32 ? 4 : 2) * per_sm;
    const int longest = (int)std::max(8LL, (720LL << 10) / plane);
    const int fewest = flat ? 1 : std::min((march + longest - 1) / longest, 512);
    const long long share = flux || per_sm >= 3 ? slots : sms;
    double best = 1e300;
    *nzc = 1;
    for (int c = fewest; c <= std::min(march, 512) && columns * c <= (1LL << 24); ++c) {
      const int base = march / c, rem = march % c;
      auto items = [&](int len) { return flat ? len : (len + 1 + zc - 1) / zc; };
      const double most = items(base + (rem ? 1 : 0));
      const double total = (double)columns * ((double)rem * items(base + 1) + (double)(c - rem) * items(base));
      const double whole = (double)((columns * c + share - 1) / share) * (total / ((double)columns * c));
      const double cost = 0.5 * (total / share + whole) + 0.5 * most;
      if (cost < best * 0.999) {
        best = cost;
        *nzc = c;
      }
    }
    *ctas = (int)std::min(columns * *nzc, slots);
    return cudaSuccess;
  }
  const long long txy = (long long)nxb * g.ny;
  // With a periodic x axis the tiles of the first and last x-block also write
  // the ghost columns.  Tiles are numbered x-block fastest and CTA b takes
  // tiles b, b + C, ...: when C is a multiple of the x-blocks per row, every
  // CTA keeps one x-block and the ghost-writing CTAs fall behind the others
  // for the whole step.  A CTA count coprime to the x-blocks rotates every CTA
  // through all x-blocks (measured with two CTAs per SM, 256^3 x 42 periodic:
  // 2.09 -> 1.78 ms).  With one CTA per SM an idle SM costs more than it
  // saves; those grids keep every SM.
  const bool rotate = g.periodic[0] && per_sm >= 2 && nxb > 1;
  auto grid_ctas = [&](long long nt) {
    long long nc = std::min(nt, slots);
    if (rotate)
      while (nc > 1 && std::gcd(nc, (long long)nxb) > 1) --nc;
    return nc;
  };
  double best = 1e300;
  int best_c = 1;
  const int cmax = std::min(g.nz, 64);
  for (int c = 1; c <= cmax; ++c) {
    const long long nt = txy * c;
    if (nt > (1LL << 24)) break;
    const long long nc = grid_ctas(nt);
    const int base = g.nz / c, rem = g.nz % c;
    auto cost = [&](long long ti) {
      const long long ch = ti / txy;
      const int zlen = base + (ch < rem ? 1 : 0);
      return (double)((zlen + 1 + zc - 1) / zc * zc) + 0.5;
    };
    double worst = 0.0;  // the busiest CTA of the round-robin order
    for (long long b = 0; b < nc; ++b) {
      double sum = 0.0;
      for (long long ti = b; ti < nt; ti += nc) sum += cost(ti);
      worst = std::max(worst, sum);
    }
    if (worst < best * 0.999) {
      best = worst;
      best_c = c;
    }
  }
  *nzc = best_c;
  *ctas = (int)grid_ctas(txy * best_c);
  return cudaSuccess;
}

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder(std::string& err) {
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  if (!encode) {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn) {
      err = "cuTensorMapEncodeTiled is not available from the driver";
      return nullptr;
    }
    encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
  return encode;
}

bool make_pop_tensor_map(CUtensorMap* map, const Grid& g, int Ni, void* base, int dpt, int zc,
                         std::string& err) {
  auto encode = tensor_map_encoder(err);
  if (!encode) return false;
  const cuuint64_t dims[4] = {(cuuint64_t)g.PX, (cuuint64_t)Ni, (cuuint64_t)g.PY,
                              (cuuint64_t)g.PZ};
  const cuuint64_t strides[3] = {(cuuint64_t)g.si * 4, (cuuint64_t)g.sy * 4,
                                 (cuuint64_t)g.sz * 4};
  const cuuint32_t box[4] = {(cuuint32_t)tma::BOXX, (cuuint32_t)dpt, 2, (cuuint32_t)zc};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, base, dims, strides, box,
                            estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    err = "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")";
    return false;
  }
  return true;
}

constexpr int kBox16 = 72;  // columns of a 16-bit population box and of an E box

// TMA descriptors of a padded 16-bit population buffer ([PZ][PY][Ni][PX],
// box 72 x dpt x 2 x zc) and of a padded float32 E buffer ([PZ][PY][PX],
// box 72 x 3 x (zc + 1)).
bool make_pop16_tensor_map(CUtensorMap* map, const Grid& g, int Ni, void* base, int storage, int dpt,
                           int zc, std::string& err) {
  auto encode = tensor_map_encoder(err);
  if (!encode) return false;
  const cuuint64_t dims[4] = {(cuuint64_t)g.PX, (cuuint64_t)Ni, (cuuint64_t)g.PY, (cuuint64_t)g.PZ};
  const cuuint64_t strides[3] = {(cuuint64_t)g.si * 2, (cuuint64_t)g.sy * 2, (cuuint64_t)g.sz * 2};
  const cuuint32_t box[4] = {(cuuint32_t)kBox16, (cuuint32_t)dpt, 2, (cuuint32_t)zc};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  const CUresult r = encode(map, storage == ST_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                    : CU_TENSOR_MAP_DATA_TYPE_FLOAT16,
                            4, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                            CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    err = "cuTensorMapEncodeTiled (16-bit populations) failed (" + std::to_string((int)r) + ")";
    return false;
  }
  return true;
}

bool make_e_tensor_map(CUtensorMap* map, const Grid& g, float* base, int zc, std::string& err) {
  auto encode = tensor_map_encoder(err);
  if (!encode) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)g.PX, (cuuint64_t)g.PY, (cuuint64_t)g.PZ};
  const cuuint64_t strides[2] = {(cuuint64_t)g.PX * 4, (cuuint64_t)g.PX * g.PY * 4};
  const cuuint32_t box[3] = {(cuuint32_t)kBox16, 3, (cuuint32_t)(zc + 1)};
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, base, dims, strides, box, estr,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    err = "cuTensorMapEncodeTiled (E) failed (" + std::to_string((int)r) + ")";
    return false;
  }
  return true;
}

}  // namespace lbrt
