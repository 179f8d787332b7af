// Auxiliary kernels on the padded population layout: initial populations,
// moments (Eqs. moments_discrete, higher_moments), decoding to dense
// float32, frozen-cell overwrite and the FP64 energy-budget reductions.
// Every population write also writes the site's periodic ghost mirrors.
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "lb_rt_internal.h"

namespace lbrt {

namespace {

constexpr int BLK = 256;

__device__ __forceinline__ void site_xyz(const Grid& g, long long s, int& x, int& y, int& z) {
  x = (int)(s % g.nx);
  const long long r = s / g.nx;
  y = (int)(r % g.ny);
  z = (int)(r / g.ny);
}

__device__ __forceinline__ float load_pop(const void* pop, const Grid& g, int i, int z, int y,
                                          int x) {
  return static_cast<const float*>(pop)[pidx(g, i, z, y, x)];
}

// kind: populations (data [Next][sites] in the external order), isotropic
// (I_i = w_i E0) or P1 (I_i = w_i (E0 + d n_i.F0)).  Inert padding directions
// (w = 0, n = 0) get 0.
__global__ void k_init_state(Grid g, int Ni, int Next, const int* __restrict__ int_of_ext,
                             const float* __restrict__ data, int kind, float* __restrict__ pop,
                             DirTable t) {
  const long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (s >= g.sites) return;
  int x, y, z;
  site_xyz(g, s, x, y, z);
  const float d = (float)g.dims;
  if (kind == LB_RT_STATE_POPULATIONS) {
    for (int e = 0; e < Next; ++e)
      store_pop(pop, g, int_of_ext[e], z, y, x, data[(size_t)e * g.sites + s]);
    return;
  }
  for (int i = 0; i < Ni; ++i) {
    const float4 nw = t.nw[i];
    float v;
    if (kind == LB_RT_STATE_ISOTROPIC) {
      v = nw.w * data[s];
    } else {
      v = nw.w * (data[s] + d * (nw.x * data[g.sites + s] + nw.y * data[2 * g.sites + s] +
                                 nw.z * data[3 * g.sites + s]));
    }
    store_pop(pop, g, i, z, y, x, v);
  }
}

// Dense [Next][sites] float32 copy in the external direction order.
__global__ void k_decode(Grid g, int Next, const int* __restrict__ int_of_ext,
                         const void* __restrict__ pop, float* __restrict__ out) {
  const long long total = g.sites * (long long)Next;
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < total;
       k += (long long)gridDim.x * blockDim.x) {
    const int e = (int)(k / g.sites);
    int x, y, z;
    site_xyz(g, k % g.sites, x, y, z);
    out[k] = load_pop(pop, g, int_of_ext[e], z, y, x);
  }
}

// Frozen cells: overwrite, and add (prescribed - collided) energy to the
// FP64 injection accumulator.  One warp per cell, lanes over the directions:
// the cells are few, so what counts is the chain of dependent accesses (one
// thread per cell walked its directions one after the other: 18.6 us for 32
// cells x 16 directions).
__global__ void k_frozen(Grid g, int Next, const int* __restrict__ int_of_ext, int ncells,
                         const int64_t* __restrict__ cells, const float* __restrict__ vals,
                         float* __restrict__ pop, double* injection) {
  // 32 threads a cell: their number passes 2^32 before ncells passes an int
  const long long c = (blockIdx.x * (long long)blockDim.x + threadIdx.x) / 32;
  const int lane = threadIdx.x % 32;
  if (c >= ncells) return;
  int x, y, z;
  site_xyz(g, cells[c], x, y, z);
  double add = 0.0;
  for (int e = lane; e < Next; e += 32) {
    const int i = int_of_ext[e];
    const float v = vals[(size_t)c * Next + e];
    if (injection) add += (double)v - (double)pop[pidx(g, i, z, y, x)];
    store_pop(pop, g, i, z, y, x, v);
  }
  if (injection) {
    for (int s = 16; s > 0; s >>= 1) add += __shfl_xor_sync(0xffffffffu, add, s);
    if (lane == 0) atomicAdd(injection, add);
  }
}

// acc layout: [0] total, [1] initial, [2] outflow, [3] source, [4] injection,
// [5] steps, [6] injection of the current step (added by the frozen kernel).
// partials: [nblocks][2] = (sum E*, sum E_collided) of the step just taken.
// A block sums kFinSlots of them; where there are more, every block leaves its
// sum in its first slot and the last one to finish adds those up in their order
// (a slot per 32 sites: 17 blocks at 93x61x47, 1024 at 256^3).  The rate of FP64
// additions (two a cycle and SM) is what counts: hence many blocks, and a tree in
// shared memory instead of shuffles, which add in every lane.
constexpr int kFinSlots = 2 * BLK;
__global__ void k_budget_finalize(double* partials, int nblocks, double* acc, unsigned* done) {
  __shared__ double2 sh[BLK];
  __shared__ bool last;
  double2* const slots = reinterpret_cast<double2*>(partials);
  // sum of slots k0, k0 + stride .. < k1, in sh[0]
  auto block_sum = [&](long long k0, long long k1, int stride) {
    double2 a = make_double2(0.0, 0.0);
    long long k = k0 + (long long)threadIdx.x * stride;
    if (k < k1) a = __ldcg(slots + k);
    while ((k += BLK * stride) < k1) {
      const double2 v = __ldcg(slots + k);
      a.x += v.x;
      a.y += v.y;
    }
    sh[threadIdx.x] = a;
    __syncthreads();
    for (int w = BLK / 2; w > 0; w >>= 1) {
      if (threadIdx.x < w) {
        sh[threadIdx.x].x += sh[threadIdx.x + w].x;
        sh[threadIdx.x].y += sh[threadIdx.x + w].y;
      }
      __syncthreads();
    }
  };
  const long long first = (long long)blockIdx.x * kFinSlots;
  block_sum(first, min((long long)nblocks, first + kFinSlots), 1);
  if (gridDim.x > 1) {
    if (threadIdx.x == 0) {
      __stcg(slots + first, sh[0]);
      __threadfence();
      last = atomicAdd(done, 1u) == gridDim.x - 1;
      if (last) {
        *done = 0;
        __threadfence();
      }
    }
    __syncthreads();
    if (!last) return;
    block_sum(0, (long long)gridDim.x * kFinSlots, kFinSlots);
  }
  if (threadIdx.x == 0) {
    const double estar = sh[0].x, ecoll = sh[0].y;
    const double inj = acc[6];
    acc[2] += acc[0] - estar;   // outflow through vacuum faces
    acc[3] += ecoll - estar;    // collision source
    acc[4] += inj;
    acc[0] = ecoll + inj;
    acc[5] += 1.0;
    acc[6] = 0.0;
  }
}

// sum over sites of sum_i I_i in FP64: per-block partials, then one block.
__global__ void k_total_partials(Grid g, int N, const void* __restrict__ pop,
                                 double* __restrict__ partials) {
  __shared__ double sh[BLK];
  double acc = 0.0;
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < g.sites;
       s += (long long)gridDim.x * blockDim.x) {
    int x, y, z;
    site_xyz(g, s, x, y, z);
    float e = 0.f;
    for (int i = 0; i < N; ++i) e += load_pop(pop, g, i, z, y, x);
    acc += (double)e;
  }
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) partials[blockIdx.x] = sh[0];
}

__global__ void k_sum_partials(const double* __restrict__ partials, int n, double* out) {
  __shared__ double sh[BLK];
  double a = 0.0;
  for (int k = threadIdx.x; k < n; k += blockDim.x) a += partials[k];
  sh[threadIdx.x] = a;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = sh[0];
}

// ---- 16-bit storage: f_i = I_i / w_i = E^ (1 + q_i), E^ = max(E, 1e-30) --

constexpr float EPS_E = 1e-30f;

__device__ __forceinline__ long long eidx(const Grid& g, int z, int y, int x) {
  return (long long)(z + 1) * g.PX * g.PY + (long long)(y + 1) * g.PX + x + GL;
}

template <class ST> __device__ __forceinline__ float to_f(ST v);
template <> __device__ __forceinline__ float to_f<__half>(__half v) { return __half2float(v); }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) {
  return __bfloat162float(v);
}
template <class ST> __device__ __forceinline__ ST from_f(float v);
template <> __device__ __forceinline__ __half from_f<__half>(float v) { return __float2half_rn(v); }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) {
  return __float2bfloat16_rn(v);
}

// E^ of a site and every periodic mirror.
__device__ __forceinline__ void store_e_site(float* e, const Grid& g, int z, int y, int x, float v) {
  int xs[3], ys[3], zs[3];
  const int nxs = mirrors(x, g.nx, g.periodic[0], GL, xs);
  const int nys = mirrors(y, g.ny, g.periodic[1], 1, ys);
  const int nzs = mirrors(z, g.nz, g.periodic[2], 1, zs);
  for (int a = 0; a < nzs; ++a)
    for (int b = 0; b < nys; ++b)
      for (int c = 0; c < nxs; ++c)
        e[(long long)zs[a] * g.PX * g.PY + (long long)ys[b] * g.PX + xs[c]] = v;
}

// Encode f_i (per internal direction, from `kind` and `data` as in
// k_init_state) into q_i and E^.  Inert padding directions keep q = 0.
template <class ST>
__global__ void k_init_state16(Grid g, int Ni, int Next, const int* __restrict__ int_of_ext,
                               const float* __restrict__ data, int kind, ST* __restrict__ pop,
                               float* __restrict__ e, DirTable t) {
  const long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (s >= g.sites) return;
  int x, y, z;
  site_xyz(g, s, x, y, z);
  const float d = (float)g.dims;
  // f_i of internal direction i; E = sum_i w_i f_i
  auto f_of = [&](int i) -> float {
    const float4 nw = t.nw[i];
    if (kind == LB_RT_STATE_ISOTROPIC) return data[s];
    return data[s] + d * (nw.x * data[g.sites + s] + nw.y * data[2 * g.sites + s] +
                          nw.z * data[3 * g.sites + s]);
  };
  float E = 0.f;
  if (kind == LB_RT_STATE_POPULATIONS) {
    for (int ex = 0; ex < Next; ++ex) E += data[(size_t)ex * g.sites + s];
  } else if (kind == LB_RT_STATE_ISOTROPIC) {
    E = data[s];
  } else {
    for (int i = 0; i < Ni; ++i) E = fmaf(t.nw[i].w, f_of(i), E);
  }
  const float Eh = fmaxf(E, EPS_E);
  const float ri = 1.f / Eh;
  store_e_site(e, g, z, y, x, Eh);
  if (kind == LB_RT_STATE_POPULATIONS) {
    for (int ex = 0; ex < Next; ++ex) {
      const int i = int_of_ext[ex];
      const float f = data[(size_t)ex * g.sites + s] / t.nw[i].w;
      store_pop(pop, g, i, z, y, x, from_f<ST>(fmaf(f, ri, -1.f)));
    }
    return;
  }
  for (int i = 0; i < Ni; ++i) {
    const bool inert = __float_as_int(t.au[i].w) & 8;
    store_pop(pop, g, i, z, y, x, from_f<ST>(inert ? 0.f : fmaf(f_of(i), ri, -1.f)));
  }
}

template <class ST>
__device__ __forceinline__ float f_at(const ST* pop, const float* e, const Grid& g, int i, int z,
                                      int y, int x) {
  const float Eh = e[eidx(g, z, y, x)];
  return fmaf(Eh, to_f<ST>(pop[pidx(g, i, z, y, x)]), Eh);
}

// The site pair (x, x + 1), x even, of thread `p`: row base and coordinates.
struct SitePair {
  int x, y, z;
  bool in1;      // x + 1 inside
  long long s;   // site of x
};
__device__ __forceinline__ bool site_pair(const Grid& g, long long p, SitePair& q) {
  const unsigned npx = (unsigned)(g.nx + 1) / 2;  // sites < 2^31, so pairs and rows fit 32 bits
  const unsigned r = (unsigned)p / npx;
  if (p >= (long long)npx * g.ny * g.nz) return false;
  q.x = 2 * (int)((unsigned)p - r * npx);
  q.y = (int)(r % (unsigned)g.ny);
  q.z = (int)(r / (unsigned)g.ny);
  q.in1 = q.x + 1 < g.nx;
  q.s = (long long)r * g.nx + q.x;
  return true;
}

// Populations (x, x + 1) of a direction row, as stored and as a float32 pair;
// 16-bit storage: I = w E^ (1 + q).
template <class ST>
using RawPair = std::conditional_t<std::is_same<ST, float>::value, float2, unsigned>;
template <class ST>
__device__ __forceinline__ float2 decode_pair(RawPair<ST> v, float2 Eh, float w) {
  if constexpr (std::is_same<ST, float>::value) {
    return v;
  } else {
    ST lo, hi;
    const unsigned short a = (unsigned short)v, b = (unsigned short)(v >> 16);
    memcpy(&lo, &a, 2);
    memcpy(&hi, &b, 2);
    return make_float2(w * fmaf(Eh.x, to_f<ST>(lo), Eh.x), w * fmaf(Eh.y, to_f<ST>(hi), Eh.y));
  }
}

// Moments of a site pair: sums over directions in the table order.  The rows
// of padding and, past the end of an odd row, the ghost column are read and
// not used.  U > 1: U directions are loaded before any is added up (left to
// itself the compiler keeps too few loads in flight where there are ten sums).
struct Moments {
  float e = 0, fx = 0, fy = 0, fz = 0, pxx = 0, pxy = 0, pxz = 0, pyy = 0, pyz = 0, pzz = 0;
  template <bool WITH_P>
  __device__ __forceinline__ void add(float4 nw, float v) {
    e += v;
    fx = fmaf(nw.x, v, fx);
    fy = fmaf(nw.y, v, fy);
    fz = fmaf(nw.z, v, fz);
    if constexpr (WITH_P) {
      pxx = fmaf(nw.x * nw.x, v, pxx);
      pxy = fmaf(nw.x * nw.y, v, pxy);
      pxz = fmaf(nw.x * nw.z, v, pxz);
      pyy = fmaf(nw.y * nw.y, v, pyy);
      pyz = fmaf(nw.y * nw.z, v, pyz);
      pzz = fmaf(nw.z * nw.z, v, pzz);
    }
  }
};

template <class ST, bool WITH_P, int U>
__device__ __forceinline__ void pair_moments(const Grid& g, int N, const ST* __restrict__ pop,
                                             const float* __restrict__ e, const DirTable& t, const SitePair& q,
                                             Moments& a, Moments& b) {
  float2 Eh = make_float2(0.f, 0.f);
  if constexpr (!std::is_same<ST, float>::value)
    Eh = *reinterpret_cast<const float2*>(e + eidx(g, q.z, q.y, q.x));
  const ST* p = pop + pidx(g, 0, q.z, q.y, q.x);
  auto add = [&](RawPair<ST> v, int i) {
    const float4 nw = t.nw[i];
    const float2 f = decode_pair<ST>(v, Eh, nw.w);
    a.add<WITH_P>(nw, f.x);
    b.add<WITH_P>(nw, f.y);
  };
  int i = 0;
  if constexpr (U > 1) {
#pragma unroll 1
    for (; i + U <= N; i += U) {
      RawPair<ST> v[U];
#pragma unroll
      for (int u = 0; u < U; ++u, p += g.si) v[u] = *reinterpret_cast<const RawPair<ST>*>(p);
#pragma unroll
      for (int u = 0; u < U; ++u) add(v[u], i + u);
    }
  }
#pragma unroll 4
  for (; i < N; ++i, p += g.si) add(*reinterpret_cast<const RawPair<ST>*>(p), i);
}

// E, F, P of the current populations, two sites a thread: 8-byte (4-byte) loads
// bring whole sectors, and E and F alone (no P) leave out six of ten sums.
// 128^3 x 162 float16: 0.42 -> 0.14 ms (5.3 TB/s); 256^3 x 162 float32: 2.4 ->
// 1.78 ms (6.7 TB/s), the rate of a plain copy.  With P, eight directions loaded
// ahead: 128^3 x 162 float16 0.43 -> 0.24 ms, 64^3 67 -> 46 us (four, as the
// compiler places them: 0.41 ms and 87 us).
template <class ST, bool WITH_P>
__global__ void k_moments(Grid g, int N, const ST* __restrict__ pop, const float* __restrict__ e,
                          float* __restrict__ E, float* __restrict__ F, float* __restrict__ P,
                          const __grid_constant__ DirTable t) {
  SitePair q;
  if (!site_pair(g, blockIdx.x * (long long)blockDim.x + threadIdx.x, q)) return;
  Moments m[2];
  pair_moments<ST, WITH_P, WITH_P ? 8 : 1>(g, N, pop, e, t, q, m[0], m[1]);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    if (k && !q.in1) return;
    const long long s = q.s + k;
    if (E) E[s] = m[k].e;
    if (F) {
      F[s] = m[k].fx;
      F[g.sites + s] = m[k].fy;
      F[2 * g.sites + s] = m[k].fz;
    }
    if (WITH_P && P) {
      P[s] = m[k].pxx;
      P[g.sites + s] = m[k].pxy;
      P[2 * g.sites + s] = m[k].pxz;
      P[3 * g.sites + s] = m[k].pyy;
      P[4 * g.sites + s] = m[k].pyz;
      P[5 * g.sites + s] = m[k].pzz;
    }
  }
}

template <class ST>
__global__ void k_decode16(Grid g, int Next, const int* __restrict__ int_of_ext,
                           const ST* __restrict__ pop, const float* __restrict__ e,
                           float* __restrict__ out, DirTable t) {
  const long long total = g.sites * (long long)Next;
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < total;
       k += (long long)gridDim.x * blockDim.x) {
    const int ex = (int)(k / g.sites);
    int x, y, z;
    site_xyz(g, k % g.sites, x, y, z);
    const int i = int_of_ext[ex];
    out[k] = t.nw[i].w * f_at(pop, e, g, i, z, y, x);
  }
}

// Frozen cells in 16-bit storage: the site's E^ becomes the sum of the
// prescribed values and every direction is re-encoded against it.
template <class ST>
__global__ void k_frozen16(Grid g, int Ni, int Next, const int* __restrict__ int_of_ext, int ncells,
                           const int64_t* __restrict__ cells, const float* __restrict__ vals,
                           ST* __restrict__ pop, float* __restrict__ e, double* injection,
                           DirTable t) {
  // 32 threads a cell: their number passes 2^32 before ncells passes an int
  const long long c = (blockIdx.x * (long long)blockDim.x + threadIdx.x) / 32;
  const int lane = threadIdx.x % 32;
  if (c >= ncells) return;
  int x, y, z;
  site_xyz(g, cells[c], x, y, z);
  float E = 0.f;  // every lane the whole sum, in the order of the directions
#pragma unroll 8
  for (int ex = 0; ex < Next; ++ex) E += vals[(size_t)c * Next + ex];
  const float Eh = fmaxf(E, EPS_E);
  const float ri = 1.f / Eh;
  if (injection) {
    double d = 0.0;  // prescribed - collided
    for (int i = lane; i < Ni; i += 32) d -= (double)(t.nw[i].w * f_at(pop, e, g, i, z, y, x));
    for (int ex = lane; ex < Next; ex += 32) d += (double)vals[(size_t)c * Next + ex];
    for (int s = 16; s > 0; s >>= 1) d += __shfl_xor_sync(0xffffffffu, d, s);
    if (lane == 0) atomicAdd(injection, d);
  }
  for (int ex = lane; ex < Next; ex += 32) {
    const int i = int_of_ext[ex];
    const float f = vals[(size_t)c * Next + ex] / t.nw[i].w;
    store_pop(pop, g, i, z, y, x, from_f<ST>(fmaf(f, ri, -1.f)));
  }
  if (lane == 0) store_e_site(e, g, z, y, x, Eh);
}

template <class ST>
__global__ void k_total_partials16(Grid g, int N, const ST* __restrict__ pop,
                                   const float* __restrict__ e, double* __restrict__ partials,
                                   DirTable t) {
  __shared__ double sh[BLK];
  double acc = 0.0;
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < g.sites;
       s += (long long)gridDim.x * blockDim.x) {
    int x, y, z;
    site_xyz(g, s, x, y, z);
    float v = 0.f;
    for (int i = 0; i < N; ++i) v = fmaf(t.nw[i].w, f_at(pop, e, g, i, z, y, x), v);
    acc += (double)v;
  }
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) partials[blockIdx.x] = sh[0];
}

// Coupling outputs (Sec. 5, coupling step 4): from the site's E, F, P and
// the fluid velocity v, the comoving J = W^2 (E - 2 F.v + P:vv) (Eq. J),
// H_j = W^3 (F.v - E) v_j + W h_ji F^i - W h_ji v_k P^ik with
// h_ij = W^2 v_i v_j + delta_ij, and S_0 = W (kt_a J - eta_t) + kt H^0,
// S_j = W (kt_a J - eta_t) v_j + kt H_j with kt = kt_a + kt_0 (kt_1 = 0):
// the lab components of the four-vector (kt_a J - eta_t) u^mu + kt H^mu, with
// H^0 = v.H the time component of the comoving flux (H^mu u_mu = 0,
// signature -+++).  ST = float: populations; 16-bit types: the deviation
// form against the E array `e`.  Two sites a thread, bound by the latency of
// the loads at small grids: 64^3 x 42 float32, 16.7 -> 12.7 us.  Eight directions
// loaded ahead pay from about a hundred directions on: 64^3 x 162 float16 48 ->
// 42 us, but 128^3 x 42 float32 94 -> 101.
template <class ST>
__global__ void k_coupling(Grid g, int N, const ST* __restrict__ pop, const float* __restrict__ e,
                           const __grid_constant__ DirTable t, MovingCoef c, float* __restrict__ Jo,
                           float* __restrict__ Ho, float* __restrict__ So) {
  SitePair q;
  if (!site_pair(g, blockIdx.x * (long long)blockDim.x + threadIdx.x, q)) return;
  Moments mm[2];
  if (N >= 96) pair_moments<ST, true, 8>(g, N, pop, e, t, q, mm[0], mm[1]);
  else pair_moments<ST, true, 1>(g, N, pop, e, t, q, mm[0], mm[1]);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    if (k && !q.in1) return;
    const long long s = q.s + k;
    const float E = mm[k].e, Fx = mm[k].fx, Fy = mm[k].fy, Fz = mm[k].fz, Pxx = mm[k].pxx, Pxy = mm[k].pxy,
                Pxz = mm[k].pxz, Pyy = mm[k].pyy, Pyz = mm[k].pyz, Pzz = mm[k].pzz;
    const float vx = c.v ? c.v[s] : 0.f, vy = c.v ? c.v[g.sites + s] : 0.f,
                vz = c.v ? c.v[2 * g.sites + s] : 0.f;
    const float W2 = 1.f / (1.f - (vx * vx + vy * vy + vz * vz));
    const float W = sqrtf(W2);
    const float Fv = Fx * vx + Fy * vy + Fz * vz;
    // Pv_i = P^ik v_k
    const float Pvx = Pxx * vx + Pxy * vy + Pxz * vz;
    const float Pvy = Pxy * vx + Pyy * vy + Pyz * vz;
    const float Pvz = Pxz * vx + Pyz * vy + Pzz * vz;
    const float Pvv = Pvx * vx + Pvy * vy + Pvz * vz;
    const float J = W2 * (E - 2.f * Fv + Pvv);
    // h_ji a^i = a_j + W^2 v_j (v.a) for a = F - Pv
    const float ax = Fx - Pvx, ay = Fy - Pvy, az = Fz - Pvz;
    const float va = vx * ax + vy * ay + vz * az;
    const float c1 = W * W2 * (Fv - E), c2 = W * W2 * va;
    const float Hx = c1 * vx + W * ax + c2 * vx;
    const float Hy = c1 * vy + W * ay + c2 * vy;
    const float Hz = c1 * vz + W * az + c2 * vz;
    if (Jo) Jo[s] = J;
    if (Ho) {
      Ho[s] = Hx;
      Ho[g.sites + s] = Hy;
      Ho[2 * g.sites + s] = Hz;
    }
    if (So) {
      const float kta = c.kta ? c.kta[s] : c.kta_s, kt0 = c.kt0 ? c.kt0[s] : c.kt0_s;
      const float etat = c.etat ? c.etat[s] : c.etat_s;
      const float kt = kta + kt0;
      // time component of the comoving flux four-vector, H^mu u_mu = 0
      const float H0 = vx * Hx + vy * Hy + vz * Hz;
      const float emit = W * (kta * J - etat);
      So[s] = fmaf(kt, H0, emit);
      So[g.sites + s] = fmaf(kt, Hx, emit * vx);
      So[2 * g.sites + s] = fmaf(kt, Hy, emit * vy);
      So[3 * g.sites + s] = fmaf(kt, Hz, emit * vz);
    }
  }
}

unsigned grid1d(long long n) { return (unsigned)((n + BLK - 1) / BLK); }
// blocks of the kernels that take two sites a thread; of 128 threads, so that a
// small grid still reaches every SM (31^3 x 42: coupling 8.4 -> 7.6 us)
constexpr int PAIR_BLK = 128;
unsigned pair_grid(const Grid& g) {
  return (unsigned)(((long long)((g.nx + 1) / 2) * g.ny * g.nz + PAIR_BLK - 1) / PAIR_BLK);
}

}  // namespace

cudaError_t launch_init_state(const Grid& g, int Ni, int Next, const int* int_of_ext,
                              const float* data, int kind, void* pop, float* e, int storage,
                              const DirTable& t, cudaStream_t s) {
  if (storage == ST_F32)
    k_init_state<<<grid1d(g.sites), BLK, 0, s>>>(g, Ni, Next, int_of_ext, data, kind,
                                                 static_cast<float*>(pop), t);
  else if (storage == ST_F16)
    k_init_state16<__half><<<grid1d(g.sites), BLK, 0, s>>>(g, Ni, Next, int_of_ext, data, kind,
                                                           static_cast<__half*>(pop), e, t);
  else
    k_init_state16<__nv_bfloat16><<<grid1d(g.sites), BLK, 0, s>>>(
        g, Ni, Next, int_of_ext, data, kind, static_cast<__nv_bfloat16*>(pop), e, t);
  return cudaGetLastError();
}

cudaError_t launch_moments(const Grid& g, int N, const void* pop, const float* e, int storage,
                           const DirTable& t, float* E, float* F, float* P, cudaStream_t s) {
  auto go = [&](auto tag) {
    using ST = decltype(tag);
    const ST* p = static_cast<const ST*>(pop);
    if (P) k_moments<ST, true><<<pair_grid(g), PAIR_BLK, 0, s>>>(g, N, p, e, E, F, P, t);
    else k_moments<ST, false><<<pair_grid(g), PAIR_BLK, 0, s>>>(g, N, p, e, E, F, P, t);
  };
  if (storage == ST_F32) go(float());
  else if (storage == ST_F16) go(__half());
  else go(__nv_bfloat16());
  return cudaGetLastError();
}

cudaError_t launch_decode(const Grid& g, int Next, const int* int_of_ext, const void* pop,
                          const float* e, int storage, const DirTable& t, float* out,
                          cudaStream_t s) {
  if (storage == ST_F32)
    k_decode<<<1024, BLK, 0, s>>>(g, Next, int_of_ext, pop, out);
  else if (storage == ST_F16)
    k_decode16<__half><<<1024, BLK, 0, s>>>(g, Next, int_of_ext, static_cast<const __half*>(pop),
                                            e, out, t);
  else
    k_decode16<__nv_bfloat16><<<1024, BLK, 0, s>>>(
        g, Next, int_of_ext, static_cast<const __nv_bfloat16*>(pop), e, out, t);
  return cudaGetLastError();
}

cudaError_t launch_frozen(const Grid& g, int Ni, int Next, const int* int_of_ext, int ncells,
                          const int64_t* cells, const float* vals, void* pop, float* e,
                          int storage, const DirTable& t, double* injection_acc, cudaStream_t s) {
  if (ncells <= 0) return cudaSuccess;
  const int nb = (int)((ncells + BLK / 32 - 1LL) / (BLK / 32));  // a warp per cell
  if (storage == ST_F32)
    k_frozen<<<nb, BLK, 0, s>>>(g, Next, int_of_ext, ncells, cells, vals,
                                static_cast<float*>(pop), injection_acc);
  else if (storage == ST_F16)
    k_frozen16<__half><<<nb, BLK, 0, s>>>(g, Ni, Next, int_of_ext, ncells, cells, vals,
                                          static_cast<__half*>(pop), e, injection_acc, t);
  else
    k_frozen16<__nv_bfloat16><<<nb, BLK, 0, s>>>(g, Ni, Next, int_of_ext, ncells, cells, vals,
                                                 static_cast<__nv_bfloat16*>(pop), e,
                                                 injection_acc, t);
  return cudaGetLastError();
}

cudaError_t launch_coupling(const Grid& g, int N, const void* pop, const float* e, int storage,
                            const DirTable& t, const MovingCoef& c, float* J, float* H, float* S,
                            cudaStream_t s) {
  if (storage == ST_F32)
    k_coupling<float><<<pair_grid(g), PAIR_BLK, 0, s>>>(g, N, static_cast<const float*>(pop), e, t,
                                                      c, J, H, S);
  else if (storage == ST_F16)
    k_coupling<__half><<<pair_grid(g), PAIR_BLK, 0, s>>>(g, N, static_cast<const __half*>(pop), e,
                                                       t, c, J, H, S);
  else
    k_coupling<__nv_bfloat16><<<pair_grid(g), PAIR_BLK, 0, s>>>(
        g, N, static_cast<const __nv_bfloat16*>(pop), e, t, c, J, H, S);
  return cudaGetLastError();
}

cudaError_t launch_budget_finalize(double* partials, int nblocks, double* acc, unsigned* done,
                                   cudaStream_t s) {
  const int blocks = std::max(1, (int)((nblocks + (long long)kFinSlots - 1) / kFinSlots));
  k_budget_finalize<<<blocks, BLK, 0, s>>>(partials, nblocks, acc, done);
  return cudaGetLastError();
}

cudaError_t launch_total_energy(const Grid& g, int N, const void* pop, const float* e, int storage,
                                const DirTable& t, double* partials, int max_blocks, double* out,
                                cudaStream_t s) {
  int nb = (int)std::min<long long>((long long)max_blocks, (long long)grid1d(g.sites));
  if (nb < 1) nb = 1;
  if (storage == ST_F32)
    k_total_partials<<<nb, BLK, 0, s>>>(g, N, pop, partials);
  else if (storage == ST_F16)
    k_total_partials16<__half><<<nb, BLK, 0, s>>>(g, N, static_cast<const __half*>(pop), e,
                                                  partials, t);
  else
    k_total_partials16<__nv_bfloat16><<<nb, BLK, 0, s>>>(
        g, N, static_cast<const __nv_bfloat16*>(pop), e, partials, t);
  k_sum_partials<<<1, BLK, 0, s>>>(partials, nb, out);
  return cudaGetLastError();
}

}  // namespace lbrt
