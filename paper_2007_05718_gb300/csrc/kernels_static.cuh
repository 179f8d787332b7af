// Fused stream + collide step for a static fluid: one kernel body for float32
// and 16-bit population storage, single problems and batches.  Weih et al.
// 2020: Sec. 3.3, Eqs. (interp), (rte_implicit), (collision-step).
//
// Storage.  float32: I_i.  16 bits: per site E in float32 (padded array, same
// ghost layer) and per direction the relative deviation q_i of
//   f_i = I_i / w_i = E^ (1 + q_i),   E^ = max(E, 1e-30);
// all arithmetic is float32, the stream works on f_i (w_i factors out of Eq.
// interp) and the output is encoded straight from the collision scalars.
//
// Tiles.  A CTA owns 64 consecutive x sites of one row over a chunk of planes
// (3D), or of a chunk of rows (2D: no direction leaves the plane, so the march
// is along y, no seed plane is loaded and the mirror planes of a periodic z
// axis, which no pull reads, are not written: two thirds of the stores); each
// lane owns an x-pair (packed float32 x 2 arithmetic).  Warp g owns the DPT
// directions g DPT .. of the internal order, all of one upwind (row, plane)
// class; per batch of ZC planes one TMA box brings its directions x own and
// upwind row x ZC planes.  The bilinear value of a plane is lerped in z against
// the one carried in registers from the plane before, so every plane is loaded
// once per tile.
//
// Who waits for whom.  The collision of a site needs the sum over all
// directions, that is over all warps.  A warp does not wait for the sum of the
// batch it has just streamed: it first streams the leading H directions of the
// next batch into spare registers,
//   warp, batch q: wait TMA(q); stream directions 0 .. HU - 1 of q
//                  [unit of batch q - 1: wait P(q - 1); sum the warps' partial
//                   moments; collision scalars -> coef; arrive C(q - 1)]
//                  stream directions HU .. H - 1 of q
//                  wait C(q - 1); store batch q - 1
//                  stream directions H .. DPT - 1 of q; issue TMA(q + 2) into
//                  the slot just read; write partials(q); arrive P(q)
// A unit is half a row of one plane (32 sites); the units of a batch go to the
// warps in turn, so that no warp carries the reduction alone.  P and C are
// mbarriers in shared memory.  The phases cannot run ahead: a warp arrives at
// P(q) after it has waited for C(q - 1), which needs P(q - 1).  So one buffer
// of partial moments and two of collision scalars are enough.  The loop body
// exists once (two copies with the register buffers swapped cost 120 KB of
// code, and instruction fetch was the largest stall).
//
// Flux.  With lambda == 0 (no kappa_1 scattering) the collision does not
// depend on the flux: c1 = dt kappa_0 lambda F = 0.  FLUX == false leaves out
// the flux partials and the n . c1 terms (exact zeros, see unit()), about a third
// of the packed arithmetic and most of the direction constants.
//
// What bounds it.  float32, 256 x 256 x 64 periodic, 162 directions: 1.24 ms,
// 3.6 GB read and 2.9 GB written in DRAM, 5.2 TB/s; 64 instructions per
// direction and 64-site plane, issue slots 49 % busy.  Behind DRAM the
// shared-memory wavefronts of the stream (48 of 59 cycles per direction-plane
// with resident boxes) are the next limit.  16 bits: the decode and the lerps,
// 84 instructions, issue slots 70 % busy, 1.16 ms.  Waiting takes no issue slots
// worth naming: a launch repeats about 12000 tries of its barriers and queue, in
// 0.7 to 1.0e9 warp instructions (the hardware suspends a waiting warp).  Before
// (partials and scalars between two CTA barriers per plane, tiles dealt out in
// advance) the same grid took 2.0 and 2.2 ms.  Times in ms:
//   a step, 256^3 x 162, float32 7.5 -> 4.74, float16 8.8 -> 4.30
//   a step, 128^3 x 42 sphere, float32 0.21 -> 0.15, float16 0.24 -> 0.18
//   a step of eight 512^2 x 120 float32 problems in a batch 3.63 -> 0.62 (1.32
//   before the mirror planes went)
//
// Every wait is bounded (about 2 s).  A warp whose wait gives up sets the error
// word and leaves its loop, after the copies it has in flight have landed; what
// is left of its tiles is not written.  It no longer arrives at P and C, so the
// other warps of the CTA run into their own limit and leave likewise.
#pragma once

#include <algorithm>
#include <type_traits>

#include "lb_rt_internal.h"
#include "tma_common.cuh"

namespace lbrt {
namespace {

using namespace tma;

constexpr float kEpsE = 1e-30f;
constexpr int kRing = 2;   // population boxes per warp
constexpr int kEring = 3;  // E boxes per CTA (16-bit storage)

template <class ST> struct SV;
template <> struct SV<float> {
  static constexpr int BOX = BOXX;  // box columns
  static constexpr bool F32 = true;
};
template <> struct SV<__half> {
  static constexpr int BOX = 72;
  static constexpr bool F32 = false;
  using T2 = __half2;
  static __device__ __forceinline__ float2 to2(T2 v) { return __half22float2(v); }
  static __device__ __forceinline__ float to1(__half v) { return __half2float(v); }
  static __device__ __forceinline__ T2 from2(float2 v) { return __float22half2_rn(v); }
  static __device__ __forceinline__ __half from1(float v) { return __float2half_rn(v); }
};
template <> struct SV<__nv_bfloat16> {
  static constexpr int BOX = 72;
  static constexpr bool F32 = false;
  using T2 = __nv_bfloat162;
  static __device__ __forceinline__ float2 to2(T2 v) { return __bfloat1622float2(v); }
  static __device__ __forceinline__ float to1(__nv_bfloat16 v) { return __bfloat162float(v); }
  static __device__ __forceinline__ T2 from2(float2 v) { return __float22bfloat162_rn(v); }
  static __device__ __forceinline__ __nv_bfloat16 from1(float v) { return __float2bfloat16_rn(v); }
};
constexpr int kBoxE = 72;  // columns of an E box

// Per-direction constants as pre-broadcast pairs: a = (a_x, a_x, a_y, a_y),
// b = (a_z', a_z', w, w) (a_z' the weight of the carried plane); with the
// flux terms n0 = (n_x, n_x, n_y, n_y), n1 = (n_z, n_z, w n_x, w n_x),
// n2 = (w n_y, w n_y, w n_z, w n_z).
template <bool FLUX> struct DirC;
template <> struct DirC<false> {
  float4 a, b;
};
template <> struct DirC<true> {
  float4 a, b, n0, n1, n2;
};

template <class ST, int DPT, int ZC>
__host__ __device__ constexpr int st_slot_bytes() {
  return ((SV<ST>::BOX * DPT * 2 * ZC * (int)sizeof(ST) + 127) / 128) * 128;
}
template <int ZC>
__host__ __device__ constexpr int st_eslot_floats() {
  return ((kBoxE * 3 * (ZC + 1) * 4 + 127) / 128) * 32;
}
// A tile in the queue: column, row and padded plane of item 0, planes (2D: minus
// the rows; 0: no such tile), flag bits 2, 8 and 16 of BatchCtx.
struct TileInfo {
  int x0, y, z, len, flags;
};

// Shared memory (bytes), every offset known at compile time (GM = the plan's
// largest warp count; run-time offsets were recomputed all over the loop):
// TMA barriers [GM][2] | E barriers [3] | P, C | tile queue | coef
// [2][ZC][NC][64] f32 | site fields of two batches [2][2 ZC][3 or 4][32] f32 |
// descriptors of 4 tiles (batch) | E ring [3][ESLOT] | partials [GM][ZC][1 or 4][64] f32 |
// directions [GM DPT] | ring [G][2][SLOT]
template <class ST, bool BATCH, bool FLUX, int DPT, int ZC, int GM>
struct StLayout {
  static constexpr int EBAR = 8 * GM * kRing;
  static constexpr int PBAR = EBAR + 8 * kEring;
  static constexpr int CBAR = PBAR + 8;
  static constexpr int TILEQ = CBAR + 8;  // 4 TileInfo, the count published
  static constexpr int COEF = (TILEQ + 4 * (int)sizeof(TileInfo) + 4 + 127) / 128 * 128;
  static constexpr int FIELDS = COEF + 2 * ZC * (FLUX ? 5 : 2) * 256;
  static constexpr int DESC = FIELDS + 2 * (2 * ZC) * (FLUX ? 4 : 3) * 128;
  static constexpr int ERING = (DESC + (BATCH ? 4 * (int)sizeof(ProblemDesc) : 0) + 127) / 128 * 128;
  static constexpr int PART = ERING + (SV<ST>::F32 ? 0 : kEring * st_eslot_floats<ZC>() * 4);
  static constexpr int DIRS = PART + GM * ZC * (FLUX ? 4 : 1) * 256;
  static constexpr int RING = (DIRS + (int)sizeof(DirC<FLUX>) * GM * DPT + 127) / 128 * 128;
  static constexpr size_t bytes(int G) { return RING + (size_t)G * kRing * st_slot_bytes<ST, DPT, ZC>(); }
};

// What the store and the units of a batch need once the warp has moved on.
template <class ST>
struct BatchCtx {
  ST* base;      // the lane's pair in direction i0, first plane of the batch
  int m;         // item of its tile
  int flags;     // 1: all planes inside, no periodic y / z face; 2: ragged row;
                 // 4: row on a periodic y face; 8: periodic y or z; 16: an x
                 // ghost column; 256 << j: plane j inside; 65536 << j: periodic
                 // z face; bits 24, 25: slot of the tile queue
};

template <class ST, int MODE, bool FLUX, int DPT, int ZC, int HU, int H, int GM, bool PART>
__device__ __forceinline__ void static_body(const CUtensorMap& tmap1, const CUtensorMap& emap1,
                                            const ProblemDesc& one,
                                            const ProblemDesc* __restrict__ table, int nprob,
                                            int ntiles, unsigned* err, const DirTable& t,
                                            unsigned* __restrict__ sched, const int cta, const int ncta,
                                            const int G) {
  constexpr bool F32 = SV<ST>::F32;
  constexpr bool BATCH = MODE == 1;
  constexpr bool MOM = (MODE & 3) == 2;
  // the energy budget has kernels of its own: tested at run time it cost the
  // step without it 1 % (256^3 x 162 float32, 4.74 against 4.78 ms)
  constexpr bool BUDGET = MODE & 4;
  static_assert(!MOM || (FLUX && F32), "the moments epilogue needs the flux and float32 storage");
  constexpr int BOX = SV<ST>::BOX;
  constexpr int SLOT = st_slot_bytes<ST, DPT, ZC>();
  constexpr int ESLOT = st_eslot_floats<ZC>();
  constexpr int NC = FLUX ? 5 : 2;
  constexpr int NP = FLUX ? 4 : 1;
  constexpr int NU = 2 * ZC;  // units of a batch: (plane, half row)
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int lane = threadIdx.x;
  const int g = __shfl_sync(0xffffffffu, (int)threadIdx.y, 0);
  using L = StLayout<ST, BATCH, FLUX, DPT, ZC, GM>;
  const uint32_t smem0 = smem_u32(smem_raw);
  unsigned char* const ring = smem_raw + L::RING;
  float* const ering = reinterpret_cast<float*>(smem_raw + L::ERING);
  float* const part = reinterpret_cast<float*>(smem_raw + L::PART);
  float* const coef = reinterpret_cast<float*>(smem_raw + L::COEF);
  DirC<FLUX>* const dirs = reinterpret_cast<DirC<FLUX>*>(smem_raw + L::DIRS);
  const uint32_t e_bar = smem0 + L::EBAR, p_bar = smem0 + L::PBAR, c_bar = smem0 + L::CBAR;

  const int i0 = g * DPT;
  const int oct0 = __float_as_int(t.au[i0].w);
  const bool yneg = oct0 & 2;
  const int zs = (oct0 & 4) ? 1 : 0;
  const int row_own = yneg ? 0 : 1, row_up = yneg ? 1 : 0;  // rows of a population box
  const int erow_up = yneg ? 2 : 0;                          // rows of the E box: y-1, y, y+1

  for (int i = g * 32 + lane; i < G * DPT; i += G * 32) {
    const float4 au = t.au[i], nw = t.nw[i];
    const int oct = __float_as_int(au.w);
    const float azw = (oct & 4) ? 1.f - au.z : au.z;
    DirC<FLUX> d;
    d.a = make_float4(au.x, au.x, au.y, au.y);
    d.b = make_float4(azw, azw, nw.w, nw.w);
    if constexpr (FLUX) {
      const float wx = nw.w * nw.x, wy = nw.w * nw.y, wz = nw.w * nw.z;
      d.n0 = make_float4(nw.x, nw.x, nw.y, nw.y);
      d.n1 = make_float4(nw.z, nw.z, wx, wx);
      d.n2 = make_float4(wy, wy, wz, wz);
    }
    dirs[i] = d;
  }
  if (lane == 0) {
    for (int r = 0; r < kRing; ++r) mbar_init(smem0 + 8 * (g * kRing + r), 1);
    if (g == 0) {
      for (int r = 0; r < kEring; ++r) mbar_init(e_bar + 8 * r, 1);
      mbar_init(p_bar, G);
      mbar_init(c_bar, NU);
      *reinterpret_cast<volatile int*>(smem_raw + L::TILEQ + 4 * sizeof(TileInfo)) = 0;
    }
  }
  // x-negative directions of the warp, and the number of its directions that
  // are not padding (which follows them); from votes, so that branches on them
  // are known to be uniform
  const int oct_l = lane < DPT ? __float_as_int(t.au[i0 + lane].w) : 8;
  const unsigned xneg_mask = __ballot_sync(0xffffffffu, oct_l & 1);
  const int nreal = __popc(__ballot_sync(0xffffffffu, !(oct_l & 8)));
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  cta_sync<PART>(32 * G);

  unsigned char* const my_ring = ring + (size_t)g * kRing * SLOT;
  const uint32_t my_bar = smem0 + 8 * kRing * g;
  // false: the wait gave up (error word set); the warp then leaves its loop,
  // and so do the warps that wait for it
  auto wait = [&](uint32_t bar, int phase) { return mbar_wait_warp(bar, (uint32_t)(phase & 1), err); };
  auto arrive = [&](uint32_t bar) {
    __syncwarp();
    if (lane == 0)
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
  };

  auto flat_of = [&](const ProblemDesc& D) { return ZC == 1 && D.g.dims == 2; };

  // byte offsets of the lane's data in shared memory, kept in registers (left
  // to itself the compiler forms them again for every batch)
  int off_own = L::RING + g * kRing * SLOT + (row_own * DPT * BOX + 2 + 2 * lane) * (int)sizeof(ST);
  int off_up = L::RING + g * kRing * SLOT + (row_up * DPT * BOX + 2 + 2 * lane) * (int)sizeof(ST);
  int off_dirs = L::DIRS + i0 * (int)sizeof(DirC<FLUX>);
  int off_eo = L::ERING + ((zs * 3 + 1) * kBoxE + 2 + 2 * lane) * 4;
  int off_eu = L::ERING + ((zs * 3 + erow_up) * kBoxE + 2 + 2 * lane) * 4;
  asm volatile("" : "+r"(off_own), "+r"(off_up), "+r"(off_dirs), "+r"(off_eo), "+r"(off_eu));
  const DirC<FLUX>* const my_dirs = reinterpret_cast<const DirC<FLUX>*>(smem_raw + off_dirs);

  // ---- tiles of this CTA ------------------------------------------------------
  // Tile number 0 is tile `cta` of the list; the next ones are taken from a
  // counter (sched[0]) as the CTA comes to them, so that at any time the tiles
  // in flight are neighbours in the list and rows that share an upwind row
  // start within a fraction of a plane of each other: the second CTA to read a
  // row finds it in L2.  (With tiles dealt out in advance CTAs drift apart, and
  // on some boards the upwind rows came from DRAM a second time: the 256^3 x
  // 162 float32 step took 8.0 ms there against 5.3 ms.)  Which CTA runs a tile
  // does not change its arithmetic, nor the energy budget, which has a partial
  // sum per unit.
  // Warp 0 takes tile n + 1 when it opens tile n and publishes its geometry in
  // the queue (slot n + 1 mod 4) while it works on the tile's first item.
  volatile TileInfo* const tq = reinterpret_cast<volatile TileInfo*>(smem_raw + L::TILEQ);
  const uint32_t tq_count = smem0 + L::TILEQ + 4 * (int)sizeof(TileInfo);
  ProblemDesc* const pd = reinterpret_cast<ProblemDesc*>(smem_raw + L::DESC);
  auto desc = [&](int slot) -> const ProblemDesc& { return BATCH ? pd[slot] : one; };
  int w_prob = 0;  // warp 0: problem of the tile published last
  auto publish = [&](int n, int tl) {
    int x0 = 0, y = 0, z = 0, len = 0, p = w_prob, fl = 0;
    if (tl < ntiles) {
      if constexpr (BATCH) {
        while (p < nprob && tl >= table[p].tile_start + table[p].ntiles) ++p;
        if (p >= nprob) {  // the tile counts do not add up
          if (lane == 0) atomicOr(err, 4u);
        }
        w_prob = p;
      }
      if (p < nprob) {
        const ProblemDesc& D = BATCH ? table[p] : one;
        const Grid& gr = D.g;
        const bool flat = flat_of(D);
        const int nxb = (gr.nx + 63) / 64, rel = (int)tl - (BATCH ? D.tile_start : 0);
        const TileGeom tg = tile_geom(rel, nxb, flat ? 1 : gr.ny, flat ? gr.ny : gr.nz, D.nzc);
        x0 = tg.x0;
        y = flat ? tg.zbeg : tg.y;
        z = flat ? 1 : tg.zbeg;
        len = flat ? -tg.zlen : tg.zlen;
        fl = (x0 + 64 <= gr.nx ? 0 : 2) | (gr.periodic[1] || (gr.periodic[2] && !flat) ? 8 : 0) |
             (gr.periodic[0] && (x0 == 0 || x0 + 64 >= gr.nx) ? 16 : 0);
        if constexpr (BATCH) {
          const int* src = reinterpret_cast<const int*>(&D);
          int* dst = reinterpret_cast<int*>(&pd[n & 3]);
          for (int w = lane; w < (int)(sizeof(ProblemDesc) / 4); w += 32) dst[w] = src[w];
          __syncwarp();  // orders the lanes' copies before lane 0's release
        }
      }
    }
    if (lane == 0) {
      volatile TileInfo& e = tq[n & 3];
      e.x0 = x0;
      e.y = y;
      e.z = z;
      e.len = len;
      e.flags = fl;
      st_release(tq_count, n + 1);
    }
    __syncwarp();
  };
  // wait until tile number n is published (bounded like every wait).  The count
  // is released after the tile's slot and descriptor and acquired here by every
  // lane, so plain reads of both may follow.
  auto published = [&](int n) {
    if (__all_sync(0xffffffffu, ld_acquire(tq_count) > n)) return true;
    const long long t0 = clock64();
    while (__any_sync(0xffffffffu, ld_acquire(tq_count) <= n)) {
      if (__any_sync(0xffffffffu, clock64() - t0 > WAIT_CYCLES)) {
        atomicOr(err, 1u);
        return false;
      }
    }
    return true;
  };
  auto items_of = [&](int len) { return len < 0 ? -len : tile_items<ZC>(len); };
  int my_tile = cta;        // warp 0: the tile published last
  unsigned grabbed = 0;     // warp 0, lane 0: counter value of the tile to publish
  bool to_publish = false;

  // ---- stream cursor: item m of M of tile number tn -------------------------
  int tn = -1, m = 0, M = 0;
  int t_x0 = 0, t_y = 0, t_z = 0, t_len = 0, t_fl = 0;  // its TileInfo
  int t_zf0 = -9, t_zf1 = -9;  // items' planes (3D: m ZC + j) on a periodic z face
  ST* t_base = nullptr;  // the lane's pair in direction i0, first plane of the item
  auto publish_next = [&]() {  // warp 0
    // as late as the copies issued ahead allow: the counter's answer queues
    // behind the stores in flight
    if (!to_publish || (m < 2 && m + kRing + 1 < M)) return;
    to_publish = false;
    // (the test of `sched`, never null, is for the compiler, which otherwise
    // makes other choices all over the batched kernels: ten float16 problems of
    // 32^3 to 128^3, 40 steps, 51.1 instead of 50.3 ms; in float32 the test
    // costs 1 %)
    if (BATCH && !F32 && !sched) my_tile += ncta;
    else my_tile = ncta + (int)__shfl_sync(0xffffffffu, grabbed, 0);
    publish(tn + 1, my_tile);
  };
  auto open_tile = [&]() {  // false: no tile left
    ++tn;
    M = m = 0;
    if (!published(tn)) return false;
    const volatile TileInfo& e = tq[tn & 3];
    t_len = e.len;
    if (t_len == 0) return false;
    t_x0 = e.x0;
    t_y = e.y;
    t_z = e.z;
    t_fl = e.flags;
    M = items_of(t_len);
    const ProblemDesc& D = desc(tn & 3);
    t_zf0 = t_zf1 = -9;
    if (t_fl & 8) {  // some axis of y, z is periodic: faces have mirrors
      if (t_len > 0 && D.g.periodic[2]) t_zf0 = 1 - t_z, t_zf1 = D.g.nz - t_z;
      if (t_len > 0 && D.g.periodic[1] && (t_y == 0 || t_y == D.g.ny - 1)) t_fl |= 4;
    }
    t_base = static_cast<ST*>(D.out) + (long long)i0 * D.g.si + (long long)t_z * D.g.sz +
             (long long)(t_y + 1) * D.g.sy + (t_x0 + 2 * lane + GL);
    if (g == 0) {
      // (the same here: without the test up to 186 bytes are spilled, and the
      // 128^3 x 42 float32 step took 2.4 times as long)
      if (sched && lane == 0) grabbed = atomicAdd(sched, 1u);
      to_publish = true;
    }
    return true;
  };

  // issue the copies of batch number `issued`, the item issued - q items after
  // item m of the current tile (batch q); it may lie in the next tile, and one
  // after that is not known yet
  int q = 0, issued = 0, waited = 0;
  auto issue = [&]() {
    int im = m + issued - q, n = tn, x0 = t_x0, y = t_y, zp = t_z, len = t_len;
    if (im >= M) {
      im -= M;
      if (!published(++n)) return false;
      const volatile TileInfo& e = tq[n & 3];
      len = e.len;
      if (len == 0 || im >= items_of(len)) return false;
      x0 = e.x0;
      y = e.y;
      zp = e.z;
    }
    if (len < 0) y += im;
    else zp += im * ZC;
    __syncwarp();
    if (lane == 0) {
      const CUtensorMap* map = BATCH ? pd[n & 3].tmap : &tmap1;
      const uint32_t bar = my_bar + 8 * (issued % kRing);
      mbar_arrive_tx(bar, BOX * DPT * 2 * ZC * (int)sizeof(ST));
      tma_load_4d(smem_u32(my_ring + (size_t)(issued % kRing) * SLOT), map, x0, i0, y + (yneg ? 1 : 0),
                  zp + zs, bar);
      if (!F32 && g == 0) {
        // the E box of the same item, shared by the CTA's warps
        const CUtensorMap* em = BATCH ? pd[n & 3].emap : &emap1;
        const uint32_t eb = e_bar + 8 * (issued % kEring);
        mbar_arrive_tx(eb, kBoxE * 3 * (ZC + 1) * 4);
        tma_load_3d(smem_u32(ering + (size_t)(issued % kEring) * ESLOT), em, x0, y, zp, eb);
      }
    }
    ++issued;
    return true;
  };
  // context of item m of the open tile
  auto item_ctx = [&]() {
    const int len = t_len;
    BatchCtx<ST> c;
    c.base = t_base;
    c.m = m;
    int fl = t_fl;
    if (len < 0 && (fl & 8)) {  // 2D: the row moves with m
      const Grid& gr = desc(tn & 3).g;
      if (gr.periodic[1] && (t_y + m == 0 || t_y + m == gr.ny - 1)) fl |= 4;
    }
    bool plain = !(fl & 4);
#pragma unroll
    for (int j = 0; j < ZC; ++j) {
      const int rel = len < 0 ? 0 : m * ZC + j;  // 3D: rel 0 only seeds the carried plane
      const bool ok = len < 0 || (rel >= 1 && rel <= len);
      const bool zf = rel == t_zf0 || rel == t_zf1;
      fl |= (ok ? 256 << j : 0) | (zf ? 65536 << j : 0);
      plain = plain && ok && !zf;
    }
    c.flags = fl | (plain ? 1 : 0) | (tn & 3) << 24;
    return c;
  };
  // row and plane of j = 0 of a batch
  auto row_of = [&](const BatchCtx<ST>& c) {
    const volatile TileInfo& e = tq[c.flags >> 24];
    return e.y + (e.len < 0 ? c.m : 0);
  };
  auto plane_of = [&](const BatchCtx<ST>& c) {
    const volatile TileInfo& e = tq[c.flags >> 24];
    return e.z - 1 + (e.len < 0 ? 0 : c.m * ZC);
  };

  // ---- a unit: collision scalars of 32 sites of one plane ------------------
  // Its site fields come in asynchronously (one group per batch and warp), a
  // batch ahead: their loads queue behind the boxes and stores in flight.
  constexpr int NF = FLUX ? 4 : 3;
  float* const fields = reinterpret_cast<float*>(smem_raw + L::FIELDS);
  auto unit_fields = [&](const BatchCtx<ST>& c, int qb, int u) {
    const ProblemDesc& D = desc(c.flags >> 24);
    const int j = u >> 1, x = tq[c.flags >> 24].x0 + ((u & 1) << 5) + lane;
    if (x < D.g.nx && (c.flags >> (8 + j) & 1)) {
      const long long st = ((long long)(plane_of(c) + j) * D.g.ny + row_of(c)) * D.g.nx + x;
      float* f = fields + ((qb & 1) * NU + u) * NF * 32 + lane;
      if (D.cf.ka) cp_async4(f, D.cf.ka + st);
      if (D.cf.k0) cp_async4(f + 32, D.cf.k0 + st);
      if (D.cf.eta) cp_async4(f + 64, D.cf.eta + st);
      if (FLUX && D.cf.lam) cp_async4(f + 96, D.cf.lam + st);
    }
  };
  auto unit = [&](const BatchCtx<ST>& c, int qb, int u) {
    const ProblemDesc& D = desc(c.flags >> 24);
    const Grid& gr = D.g;
    const int j = u >> 1, fx = ((u & 1) << 5) + lane;
    const int x = tq[c.flags >> 24].x0 + fx, y = row_of(c), z = plane_of(c) + j;
    const float* f = fields + ((qb & 1) * NU + u) * NF * 32 + lane;
    const float ka = D.cf.ka ? f[0] : D.cf.ka_s, k0 = D.cf.k0 ? f[32] : D.cf.k0_s;
    const float eta = D.cf.eta ? f[64] : D.cf.eta_s;
    float lam = 0.f;
    if constexpr (FLUX) lam = D.cf.lam ? f[96] : D.cf.lam_s;
    const bool v = x < gr.nx && (c.flags >> (8 + j) & 1);
    const float inv_d = 1.f / (float)gr.dims;
    float E = 0.f, Fx = 0.f, Fy = 0.f, Fz = 0.f;
    const float* p = part + j * NP * 64 + fx;
#pragma unroll 4
    for (int w = 0; w < G; ++w, p += ZC * NP * 64) {
      E += p[0];
      if constexpr (FLUX) {
        Fx += p[64];
        Fy += p[128];
        Fz += p[192];
      }
    }
    Coef cc = collide_scalars(D.collision, D.lambda_iters, D.dt, inv_d, ka, k0, lam, eta, E, Fx, Fy, Fz);
    // lambda == 0: c1 = 0 x F, which is an exact zero, or the NaN of an infinite
    // opacity, which c0 then takes, or of an infinite F, that is of an infinite E:
    // the Lambda iteration alone would keep Inf (the others form Inf - Inf).  (The
    // test for it is faster than 0 x E for all: 128^3 x 42 float16 sphere 7.43
    // against 7.57 ms.)
    if constexpr (!FLUX) {
      cc.c0 += cc.c1x;
      if (D.collision == LB_RT_LAMBDA_K) cc.c0 = fmaf(0.f, E, cc.c0);
    }
    float* o = coef + ((size_t)(qb & 1) * ZC + j) * NC * 64 + fx;
    float Eh = 0.f;
    if constexpr (F32) {
      o[0] = cc.alpha;
      o[64] = cc.c0;
      if constexpr (FLUX) {
        o[128] = cc.c1x;
        o[192] = cc.c1y;
        o[256] = cc.c1z;
      }
    } else {
      // q' = f' / E^' - 1 with E^' = max(E', eps): the float32 scalars over E^'
      Eh = fmaxf(cc.Enew, kEpsE);
      const float ri = __fdividef(1.f, Eh);
      o[0] = cc.alpha * ri;
      o[64] = fmaf(cc.c0, ri, -1.f);
      if constexpr (FLUX) {
        o[128] = cc.c1x * ri;
        o[192] = cc.c1y * ri;
        o[256] = cc.c1z * ri;
      }
    }
    arrive(c_bar);
    if constexpr (BUDGET) {
      // Sums over the 32 sites in FP64, whose additions are slow here (two a
      // cycle and SM): lanes 0 - 15 go on with E*, lanes 16 - 31 with E'.
      const double a = v ? (double)E : 0.0, b = v ? (double)cc.Enew : 0.0;
      double r = (lane < 16 ? a : b) + __shfl_xor_sync(0xffffffffu, lane < 16 ? b : a, 16);
      for (int s = 8; s > 0; s >>= 1) r += __shfl_xor_sync(0xffffffffu, r, s);
      const int x32 = tq[c.flags >> 24].x0 + ((u & 1) << 5);
      if (!(lane & 15) && x32 < gr.nx && (c.flags >> (8 + j) & 1))
        one.budget_partials[2 * (((long long)z * gr.ny + y) * ((gr.nx + 31) / 32) + x32 / 32) + lane / 16] = r;
    }
    if (v) {
      if constexpr (MOM) {
        // moments of I' = alpha I* + w (c0 + n . c1) for an isotropic table
        // (sum w = 1, sum w n = 0, sum w n n = Id / d): E' = alpha E* + c0,
        // F' = alpha F* + c1 / d
        const long long st = ((long long)z * gr.ny + y) * gr.nx + x;
        if (one.mom_E) one.mom_E[st] = cc.Enew;
        if (one.mom_F) {
          one.mom_F[st] = fmaf(cc.alpha, Fx, cc.c1x * inv_d);
          one.mom_F[gr.sites + st] = fmaf(cc.alpha, Fy, cc.c1y * inv_d);
          one.mom_F[2 * gr.sites + st] = fmaf(cc.alpha, Fz, cc.c1z * inv_d);
        }
      }
      if constexpr (!F32) {
        {
          float* e = D.e_out;
          const int pz = gr.periodic[2] && !flat_of(D);
          if ((gr.periodic[0] && (x == 0 || x == gr.nx - 1)) || (gr.periodic[1] && (y == 0 || y == gr.ny - 1)) ||
              (pz && (z == 0 || z == gr.nz - 1))) {
            int xs[3], ys[3], zs_[3];
            const int nxs = mirrors(x, gr.nx, gr.periodic[0], GL, xs);
            const int nys = mirrors(y, gr.ny, gr.periodic[1], 1, ys);
            const int nzs = mirrors(z, gr.nz, pz, 1, zs_);
            for (int a = 0; a < nzs; ++a)
              for (int b = 0; b < nys; ++b)
                for (int cx = 0; cx < nxs; ++cx)
                  e[((long long)zs_[a] * gr.PY + ys[b]) * gr.PX + xs[cx]] = Eh;
          } else {
            e[((long long)(z + 1) * gr.PY + (y + 1)) * gr.PX + x + GL] = Eh;
          }
        }
      }
    }
  };

  // ---- the store of a batch ------------------------------------------------
  auto store = [&](const float2 (&Is)[DPT][ZC], const BatchCtx<ST>& c, int par) {
    float2 al[ZC], c0[ZC], c1x[ZC], c1y[ZC], c1z[ZC];
#pragma unroll
    for (int j = 0; j < ZC; ++j) {
      const float2* p = reinterpret_cast<const float2*>(coef + ((size_t)par * ZC + j) * NC * 64) + lane;
      al[j] = p[0];
      c0[j] = p[32];
      if constexpr (FLUX) {
        c1x[j] = p[64];
        c1y[j] = p[96];
        c1z[j] = p[128];
      }
    }
    // float32: I' = alpha I* + w c0 + (w n) . c1; 16 bits: q' = A' f* + c0' + n . c1'
    auto value = [&](int k, int j) -> float2 {
      const DirC<FLUX>& d = my_dirs[k];
      float2 eq;
      if constexpr (F32) {
        const float4 b = d.b;
        eq = f2mul(make_float2(b.z, b.w), c0[j]);
        if constexpr (FLUX) {
          const float4 n1 = d.n1, n2 = d.n2;
          eq = f2fma(make_float2(n1.z, n1.w), c1x[j], eq);
          eq = f2fma(make_float2(n2.x, n2.y), c1y[j], eq);
          eq = f2fma(make_float2(n2.z, n2.w), c1z[j], eq);
        }
      } else {
        eq = c0[j];
        if constexpr (FLUX) {
          const float4 n0 = d.n0, n1 = d.n1;
          eq = f2fma(make_float2(n0.x, n0.y), c1x[j], eq);
          eq = f2fma(make_float2(n0.z, n0.w), c1y[j], eq);
          eq = f2fma(make_float2(n1.x, n1.y), c1z[j], eq);
        }
      }
      return f2fma(al[j], Is[k][j], eq);
    };
    auto put2 = [&](ST* p, float2 o) {
      if constexpr (F32) *reinterpret_cast<float2*>(p) = o;
      else *reinterpret_cast<typename SV<ST>::T2*>(p) = SV<ST>::from2(o);
    };
    auto put1 = [&](ST* p, float o) {
      if constexpr (F32) *p = o;
      else *p = SV<ST>::from1(o);
    };
    const ProblemDesc& D = desc(c.flags >> 24);
    const int si = (int)D.g.si;
    const long long sz = D.g.sz;
    if ((c.flags & 3) == 1) {
      // interior rows and planes, full pairs: one pair store per value
      ST* p = c.base;
      if (!(c.flags & 16)) {
#pragma unroll
        for (int k = 0; k < DPT; ++k) {
#pragma unroll
          for (int j = 0; j < ZC; ++j) {
            const float2 o = value(k, j);
            if (k < nreal) put2(p + j * sz, o);
          }
          p += si;
        }
        return;
      }
      // and the ghost column of a periodic x axis as one predicated store (the
      // lane of x = nx - 1 mirrors into column GL - 1, the lane of x = 0 into
      // column nx + GL; full rows, so no lane holds both)
      const int nx = D.g.nx, xa = tq[c.flags >> 24].x0 + 2 * lane;
      const bool gx_y = xa + 1 == nx - 1;
      const bool gx = gx_y || xa == 0;
      const int og = gx_y ? GL - 1 - (xa + GL) : nx - xa;
#pragma unroll
      for (int k = 0; k < DPT; ++k) {
#pragma unroll
        for (int j = 0; j < ZC; ++j) {
          const float2 o = value(k, j);
          if (k < nreal) put2(p + j * sz, o);
          if (k < nreal && gx) put1(p + j * sz + og, gx_y ? o.y : o.x);
        }
        p += si;
      }
      return;
    }
    // x edges (ragged rows, the ghost columns of a periodic x axis) and
    // periodic y / z faces (every row / plane image)
    const int nx = D.g.nx, ny = D.g.ny, nz = D.g.nz;
    const int xa = tq[c.flags >> 24].x0 + 2 * lane, y = row_of(c);
    if (xa >= nx) return;
    const bool in1 = xa + 1 < nx;
    const bool perx = D.g.periodic[0];
    const bool gx_lo = perx && (xa == nx - 1 || xa + 1 == nx - 1);
    const bool gx_hi = perx && xa == 0;
    const bool lo_y = xa + 1 == nx - 1;
    const int off_lo = GL - 1 - (xa + GL), off_hi = nx - xa;
#pragma unroll
    for (int j = 0; j < ZC; ++j) {
      if (!(c.flags >> (8 + j) & 1)) continue;
      const int z = plane_of(c) + j;
      const bool yf = c.flags & 4, zf = c.flags >> (16 + j) & 1;
      // the site and its mirrors: rows (own, below, above) x planes
#pragma unroll 1
      for (int im = 0; im < ((yf || zf) ? 9 : 1); ++im) {
        const int iy = im % 3, iz = im / 3;
        if ((iy == 1 && !(yf && y == ny - 1)) || (iy == 2 && !(yf && y == 0)) ||
            (iz == 1 && !(zf && z == nz - 1)) || (iz == 2 && !(zf && z == 0)))
          continue;
        const long long oy = iy == 0 ? 0 : (iy == 1 ? -(long long)ny : (long long)ny) * D.g.sy;
        const long long oz = iz == 0 ? 0 : (iz == 1 ? -(long long)nz : (long long)nz) * D.g.sz;
        ST* p = c.base + j * sz + oy + oz;
#pragma unroll
        for (int k = 0; k < DPT; ++k) {
          const float2 o = value(k, j);
          if (k < nreal) {
            if (in1) put2(p, o);
            else put1(p, o.x);
            if (gx_lo) put1(p + off_lo, lo_y ? o.y : o.x);
            if (gx_hi) put1(p + off_hi, o.x);
          }
          p += si;
        }
      }
    }
  };

  float2 carry[DPT];
#pragma unroll
  for (int k = 0; k < DPT; ++k) carry[k] = make_float2(0.f, 0.f);
  BatchCtx<ST> ctx{};  // batch whose store is pending

  // stream directions K0 .. K1 - 1 of batch q into dst[0 ..], adding to the
  // partial moments
  auto stream = [&](auto K0_, auto K1_, int q, float2 (*dst)[ZC], float2 (&aE)[ZC], float2 (&aX)[ZC],
                    float2 (&aY)[ZC], float2 (&aZ)[ZC]) {
    constexpr int K0 = decltype(K0_)::value, K1 = decltype(K1_)::value;
    const ST* own = reinterpret_cast<const ST*>(smem_raw + off_own + q % kRing * SLOT);
    const ST* up = reinterpret_cast<const ST*>(smem_raw + off_up + q % kRing * SLOT);
    // 16-bit storage: E^ of the lane's pair and its x-neighbours, both rows
    float2 EPo[ZC], EPu[ZC];
    float Emo[ZC], Epo[ZC], Emu[ZC], Epu[ZC];
    if constexpr (!F32) {
#pragma unroll
      for (int j = 0; j < ZC; ++j) {
        const float* eo = reinterpret_cast<const float*>(smem_raw + off_eo + q % kEring * (ESLOT * 4)) + j * 3 * kBoxE;
        const float* eu = reinterpret_cast<const float*>(smem_raw + off_eu + q % kEring * (ESLOT * 4)) + j * 3 * kBoxE;
        EPo[j] = *reinterpret_cast<const float2*>(eo);
        EPu[j] = *reinterpret_cast<const float2*>(eu);
        Emo[j] = eo[-1];
        Epo[j] = eo[2];
        Emu[j] = eu[-1];
        Epu[j] = eu[2];
      }
    }
#pragma unroll
    for (int k = K0; k < K1; ++k) {
      const DirC<FLUX>& d = my_dirs[k];
      const float4 ca = d.a, cb = d.b;
      const float2 ax = make_float2(ca.x, ca.y), ay = make_float2(ca.z, ca.w);
      const float2 az = make_float2(cb.x, cb.y), w2 = make_float2(cb.z, cb.w);
      const bool xneg = xneg_mask >> k & 1u;
      // Eq. (interp) as nested lerps: x on both rows, then y, then z against
      // the carried plane (B(z - 1) for sgn n^z = +1, B(z + 1) otherwise, the
      // box being shifted by one plane for the latter).  The x-upwind pair
      // shares one value with the lane's own pair.
      float2 Po[ZC], Pu[ZC], So[ZC], Su[ZC];
      if constexpr (F32) {
#pragma unroll
        for (int j = 0; j < ZC; ++j) {
          Po[j] = *reinterpret_cast<const float2*>(own + (j * 2 * DPT + k) * BOX);
          Pu[j] = *reinterpret_cast<const float2*>(up + (j * 2 * DPT + k) * BOX);
        }
        if (xneg) {
#pragma unroll
          for (int j = 0; j < ZC; ++j) {
            So[j] = make_float2(Po[j].y - Po[j].x, own[(j * 2 * DPT + k) * BOX + 2] - Po[j].y);
            Su[j] = make_float2(Pu[j].y - Pu[j].x, up[(j * 2 * DPT + k) * BOX + 2] - Pu[j].y);
          }
        } else {
#pragma unroll
          for (int j = 0; j < ZC; ++j) {
            So[j] = make_float2(own[(j * 2 * DPT + k) * BOX - 1] - Po[j].x, Po[j].x - Po[j].y);
            Su[j] = make_float2(up[(j * 2 * DPT + k) * BOX - 1] - Pu[j].x, Pu[j].x - Pu[j].y);
          }
        }
      } else {
        using T2 = typename SV<ST>::T2;
#pragma unroll
        for (int j = 0; j < ZC; ++j) {
          const ST* po = own + (j * 2 * DPT + k) * BOX;
          const ST* pu = up + (j * 2 * DPT + k) * BOX;
          Po[j] = f2fma(EPo[j], SV<ST>::to2(*reinterpret_cast<const T2*>(po)), EPo[j]);
          Pu[j] = f2fma(EPu[j], SV<ST>::to2(*reinterpret_cast<const T2*>(pu)), EPu[j]);
        }
        if (xneg) {
#pragma unroll
          for (int j = 0; j < ZC; ++j) {
            const ST* po = own + (j * 2 * DPT + k) * BOX;
            const ST* pu = up + (j * 2 * DPT + k) * BOX;
            So[j] = make_float2(Po[j].y - Po[j].x, fmaf(Epo[j], SV<ST>::to1(po[2]), Epo[j]) - Po[j].y);
            Su[j] = make_float2(Pu[j].y - Pu[j].x, fmaf(Epu[j], SV<ST>::to1(pu[2]), Epu[j]) - Pu[j].y);
          }
        } else {
#pragma unroll
          for (int j = 0; j < ZC; ++j) {
            const ST* po = own + (j * 2 * DPT + k) * BOX;
            const ST* pu = up + (j * 2 * DPT + k) * BOX;
            So[j] = make_float2(fmaf(Emo[j], SV<ST>::to1(po[-1]), Emo[j]) - Po[j].x, Po[j].x - Po[j].y);
            Su[j] = make_float2(fmaf(Emu[j], SV<ST>::to1(pu[-1]), Emu[j]) - Pu[j].x, Pu[j].x - Pu[j].y);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < ZC; ++j) {
        const float2 X0 = f2fma(ax, So[j], Po[j]);
        const float2 X1 = f2fma(ax, Su[j], Pu[j]);
        const float2 Bn = f2fma(ay, f2sub(X1, X0), X0);
        const float2 r = f2fma(az, f2sub(carry[k], Bn), Bn);
        carry[k] = Bn;
        dst[k - K0][j] = r;
        if constexpr (F32) {
          aE[j] = f2add(aE[j], r);
          if constexpr (FLUX) {
            const float4 n0 = d.n0, n1 = d.n1;
            aX[j] = f2fma(make_float2(n0.x, n0.y), r, aX[j]);
            aY[j] = f2fma(make_float2(n0.z, n0.w), r, aY[j]);
            aZ[j] = f2fma(make_float2(n1.x, n1.y), r, aZ[j]);
          }
        } else {
          aE[j] = f2fma(w2, r, aE[j]);
          if constexpr (FLUX) {
            const float4 n1 = d.n1, n2 = d.n2;
            aX[j] = f2fma(make_float2(n1.z, n1.w), r, aX[j]);
            aY[j] = f2fma(make_float2(n2.x, n2.y), r, aY[j]);
            aZ[j] = f2fma(make_float2(n2.z, n2.w), r, aZ[j]);
          }
        }
      }
    }
  };

  if (g == 0) publish(0, cta);
  bool more = open_tile();
  if (more) {
    if (M < kRing) publish_next();
#pragma unroll 1
    for (int r = 0; r < kRing; ++r)
      if (!issue()) break;
  }
  // units of a batch go to warps ub, ub + 1, ...; u: this warp's unit of the
  // pending batch (none: >= NU), un: of the batch being streamed
  const int nu_mod = NU % G;
  int u = 0, un = g;
  float2 Is[DPT][ZC];   // streamed values of the batch to store
#pragma unroll 1
  while (more || q > 0) {
    float2 T[H > 0 ? H : 1][ZC];
    float2 aE[ZC], aX[ZC], aY[ZC], aZ[ZC];
#pragma unroll
    for (int j = 0; j < ZC; ++j) aE[j] = aX[j] = aY[j] = aZ[j] = make_float2(0.f, 0.f);
    if (more) {
      if constexpr (ZC == 1) {
        // 2D: the march is along y and nothing is carried.  The lerp, of weight
        // 0 there, must not see the row before, which may be of another tile or
        // another problem: 0 x Inf and 0 x NaN are NaN.  (Cleared here, where
        // it costs a 3D step 0.2 to 0.4 % and a 2D one 1 %; at the end of the
        // loop body it cost 3D steps 3 to 8 %.)
        if (t_len < 0) {
#pragma unroll
          for (int k = 0; k < DPT; ++k) carry[k] = make_float2(0.f, 0.f);
        }
      }
      if (un < NU) {
        const BatchCtx<ST> c = item_ctx();
#pragma unroll 1
        for (int v = un; v < NU; v += G) unit_fields(c, q, v);
      }
      cp_async_commit();
      if (!wait(my_bar + 8 * (q % kRing), q / kRing)) break;
      if (!F32 && !wait(e_bar + 8 * (q % kEring), q / kEring)) break;
      waited = q + 1;
      if constexpr (HU > 0)
        stream(std::integral_constant<int, 0>(), std::integral_constant<int, HU>(), q, T, aE, aX, aY, aZ);
    }
    if (q > 0 && u < NU) {
      if (!wait(p_bar, q - 1)) break;
      if (more) cp_async_wait<1>();
      else cp_async_wait<0>();
#pragma unroll 1
      for (; u < NU; u += G) unit(ctx, q - 1, u);
    }
    if constexpr (H > HU) {
      if (more)
        stream(std::integral_constant<int, HU>(), std::integral_constant<int, H>(), q, T + HU, aE, aX, aY, aZ);
    }
    if (q > 0) {
      if (!wait(c_bar, q - 1)) break;  // coef(q - 1) ready, partials(q - 1) read
      store(Is, ctx, (q - 1) & 1);
      if (!more) break;
    }
#pragma unroll
    for (int k = 0; k < H; ++k)
#pragma unroll
      for (int j = 0; j < ZC; ++j) Is[k][j] = T[k][j];
    if constexpr (H < DPT)
      stream(std::integral_constant<int, H>(), std::integral_constant<int, DPT>(), q, Is + H, aE, aX, aY, aZ);
    // the slot has been read: the box after next goes there.  Warp 0 also
    // issues the E box, into the slot of batch q - 1, which every warp has
    // left: C(q - 1) is complete
    publish_next();
#pragma unroll 1
    while (issued <= q + kRing && issue()) {
    }
    float2* pw = reinterpret_cast<float2*>(part + (size_t)g * ZC * NP * 64) + lane;
#pragma unroll
    for (int j = 0; j < ZC; ++j) {
      pw[j * NP * 32] = aE[j];
      if constexpr (FLUX) {
        pw[j * 128 + 32] = aX[j];
        pw[j * 128 + 64] = aY[j];
        pw[j * 128 + 96] = aZ[j];
      }
    }
    arrive(p_bar);
    ctx = item_ctx();
    u = un;
    un -= nu_mod;
    if (un < 0) un += G;
    ++q;
    if (++m == M) {
      more = open_tile();
    } else {
      const Grid& gr = desc(tn & 3).g;
      t_base += t_len < 0 ? gr.sy : ZC * gr.sz;
    }
  }
  // the last CTA to leave puts the tile counter back
  if (g == 0 && lane == 0 && atomicAdd(sched + 1, 1u) == (unsigned)ncta - 1) {
    sched[0] = 0;
    sched[1] = 0;
  }
  // copies still in flight (only after a failed wait) land before the CTA's
  // shared memory is released; each slot has at most one outstanding
  for (int qq = waited; qq < issued; ++qq)
    mbar_wait(my_bar + 8 * (qq % kRing), (uint32_t)((qq / kRing) & 1), err);
  if constexpr (!F32) {
    if (g == 0)
      for (int qq = waited; qq < issued; ++qq)
        mbar_wait(e_bar + 8 * (qq % kEring), (uint32_t)((qq / kEring) & 1), err);
  }
}

template <class ST, int MODE, bool FLUX, int DPT, int ZC, int HU, int H, int MAXT, int REGS>
__global__ void __launch_bounds__(MAXT) __maxnreg__(REGS)
k_static(const __grid_constant__ CUtensorMap tmap1, const __grid_constant__ CUtensorMap emap1,
         const __grid_constant__ ProblemDesc one, const ProblemDesc* __restrict__ table, int nprob,
         int ntiles, unsigned* err, unsigned* sched, const __grid_constant__ DirTable t) {
  static_body<ST, MODE, FLUX, DPT, ZC, HU, H, MAXT / 32, false>(tmap1, emap1, one, table, nprob, ntiles, err,
                                                                 t, sched, blockIdx.x, gridDim.x, blockDim.y);
}

// One batched launch over the problems of two groups with different tile
// plans (the 42- and 162-direction icosahedral sets): CTAs 0 .. ctas_a - 1
// walk group A's tiles with GA warps, the others group B's with GB warps;
// the warps a plan does not use leave at once.  Per tile the arithmetic is
// that of k_static, so every problem gives the same bits as in its own
// group's launch.
template <class ST, bool FLUX, int DA, int ZA, int UA, int HA, int DB, int ZB, int UB, int HB, int MAXT, int REGS>
__global__ void __launch_bounds__(MAXT) __maxnreg__(REGS)
k_static_pair(const __grid_constant__ CUtensorMap unused, const __grid_constant__ ProblemDesc none,
              const ProblemDesc* __restrict__ table_a, int nprob_a, int ntiles_a, int ga, int ctas_a,
              const ProblemDesc* __restrict__ table_b, int nprob_b, int ntiles_b, int gb, unsigned* err,
              unsigned* sched,
              const __grid_constant__ DirTable ta, const __grid_constant__ DirTable tb) {
  if ((int)blockIdx.x < ctas_a) {
    if ((int)threadIdx.y >= ga) return;
    static_body<ST, 1, FLUX, DA, ZA, UA, HA, MAXT / 32, true>(unused, unused, none, table_a, nprob_a, ntiles_a, err,
                                                 ta, sched, blockIdx.x, ctas_a, ga);
  } else {
    if ((int)threadIdx.y >= gb) return;
    // (the test of `sched` as in static_body: without it the ten float16 problems
    // take 65.4 instead of 53.8 ms)
    static_body<ST, 1, FLUX, DB, ZB, UB, HB, MAXT / 32, true>(unused, unused, none, table_b, nprob_b, ntiles_b, err,
                                                 tb, sched ? sched + 2 : nullptr, blockIdx.x - ctas_a, gridDim.x - ctas_a, gb);
  }
}

}  // namespace
}  // namespace lbrt
