// lb_sites.cuh -- passes over the sites of a lattice, one thread per site, joined by small
// per-site arrays in device memory: the observables and fields of every storage layout,
// and the FP64 step (arXiv:2003.11069, "Materials and Methods").
//
//   site_moments_kernel   psi, (rho_1, rho_2) and, for the fields, the momentum j of the
//                         streamed populations: the only pass that reads the state
//   site_normals_kernel   (n, |grad psi|) from psi
//   site_fields_kernel    the near-contact ray over (n, |grad psi|), u, the outputs and
//                         the block sums of the observables
//   site_collide64_kernel the near-contact ray, the totals f_i^1 + f_i^2 and the FP64
//                         collision (Guo forcing)
//   site_collide2d_kernel the near-contact ray and the D2Q9 collision in FP32 arithmetic
//                         (FP32 and FP16-deviation storage, either forcing)
//
// Measured on GB300 (lb_observables with psi and u on the device, before -> after): FP16-dev
// duct 512 x 128 x 128 3.8 -> 0.82 ms, FP16-dev channel 8192 x 1024 1.40 -> 0.43 ms. The
// kernels it replaces there (psi, then tiled_kernel) staged 27.6 psi cells per site and
// spent 100 additions per site of the narrow FP64 pipe on their block sums. FP64 steps: a 128
// x 128 box 117 -> 23 us, a 128 x 48 x 48 duct 1.40 -> 0.64 ms. FP32 steps with the exact
// difference forcing of a 1030 x 131 channel: 16.4 -> 12.7 us.
//
// Every quantity is computed once per site, by the expressions (and in the order) of the
// kernels that recompute it over halos (lb_fused2d.cuh, lb_march3d.cuh, tiled_kernel): the
// passes give the same bits.
#pragma once

#include "lb_launch.h"
#include "lb_march3d.cuh"

namespace lbnci {

// Vectors of per-site scratch in the arithmetic type.
template <typename T> struct alignas(2 * sizeof(T)) Pair { T x, y; };
template <typename T> struct alignas(16) Quad { T x, y, z, w; };

// Scratch of the passes, carved from one block: (rho_1, rho_2), (n, |grad psi|) and, for the
// fields, j.
template <typename T> struct SiteScratch {
  Pair<T>* rho;
  Quad<T>* ng;
  T* j;  // [D][N]
};
inline size_t site_align(size_t v) { return (v + 255) & ~(size_t)255; }
template <int LAT, typename T>
size_t site_scratch_bytes(size_t N, bool with_j) {
  return site_align(N * sizeof(Pair<T>)) + site_align(N * sizeof(Quad<T>)) +
         (with_j ? site_align(N * Lattice<LAT>::D * sizeof(T)) : 0);
}
template <int LAT, typename T>
SiteScratch<T> site_scratch(void* base, size_t N) {
  unsigned char* b = (unsigned char*)base;
  SiteScratch<T> s;
  s.rho = (Pair<T>*)b;
  b += site_align(N * sizeof(Pair<T>));
  s.ng = (Quad<T>*)b;
  b += site_align(N * sizeof(Quad<T>));
  s.j = (T*)b;
  return s;
}

// Blocks are 32 sites along x by blockDim.y rows, one plane.
struct SiteIdx {
  int x, y, z;
  unsigned i;
};
template <typename T>
__device__ __forceinline__ SiteIdx site_of(const StepT<T>& p) {
  SiteIdx s;
  s.x = blockIdx.x * 32 + threadIdx.x;
  s.y = blockIdx.y * blockDim.y + threadIdx.y;
  s.z = blockIdx.z;
  s.i = (unsigned)s.x + (unsigned)p.nx * ((unsigned)s.y + (unsigned)p.ny * (unsigned)s.z);
  return s;
}

// ------------------------------------------------------------------ moments
template <int LAT, typename ST, bool WITHJ>
__global__ void __launch_bounds__(256) site_moments_kernel(typename ST::Reader f,
                                                           typename ST::Compute* __restrict__ psi,
                                                           SiteScratch<typename ST::Compute> sc,
                                                           StepT<typename ST::Compute> p) {
  using T = typename ST::Compute;
  pdl_enter();
  const SiteIdx s = site_of(p);
  if (s.x >= p.nx || s.y >= p.ny) return;
  T fin[2][Lattice<LAT>::Q];
  pull_any<LAT, T>(f, s.x, s.y, s.z, p, fin);
  T r1, r2;
  psi[s.i] = psi_of<Lattice<LAT>::Q, T>(fin, &r1, &r2);
  sc.rho[s.i] = Pair<T>{r1, r2};
  if constexpr (WITHJ) {
    T j[3];
    momentum<LAT, T>(fin, j);
#pragma unroll
    for (int a = 0; a < Lattice<LAT>::D; ++a) sc.j[(unsigned)a * (unsigned)p.N + s.i] = j[a];
  }
}

// ------------------------------------------------------------------ normals
// Isotropic gradient of psi at a site from the psi array (beyond a wall the mirror site),
// summed in direction order as grad_smem does. FP64 forms each w_i psi once and adds it
// with the sign of c_i (the same bits: the product's sign is exact), which leaves one
// multiplication per direction on the narrow FP64 pipe instead of up to three.
template <int LAT, typename T>
__device__ __forceinline__ void grad_site(const T* __restrict__ psi, const SiteIdx& s, const StepT<T>& p, T g[3]) {
  constexpr bool D3 = Lattice<LAT>::D == 3;
  int xs[3], ys[3], zs[3] = {0, 0, 0};  // coordinate of neighbour digit 0, +1, -1, as row offsets
  xs[0] = s.x;
  xs[1] = s.x == p.nx - 1 ? 0 : s.x + 1;
  xs[2] = s.x == 0 ? p.nx - 1 : s.x - 1;
  ys[0] = s.y;
  ys[1] = s.y == p.ny - 1 ? (p.wall_y ? s.y : 0) : s.y + 1;
  ys[2] = s.y == 0 ? (p.wall_y ? 0 : p.ny - 1) : s.y - 1;
  if (D3) {
    zs[0] = s.z;
    zs[1] = s.z == p.nz - 1 ? (p.wall_z ? s.z : 0) : s.z + 1;
    zs[2] = s.z == 0 ? (p.wall_z ? 0 : p.nz - 1) : s.z - 1;
  }
  g[0] = T(0); g[1] = T(0); g[2] = T(0);
  static_for<Lattice<LAT>::Q>([&](auto I) {
    constexpr int i = decltype(I)::value;
    if constexpr (i > 0) {
      constexpr int cx = cc(i, 0), cy = cc(i, 1), cz = D3 ? cc(i, 2) : 0;
      const T v = psi[(unsigned)xs[i % 3] + (unsigned)p.nx * ((unsigned)ys[(i / 3) % 3] +
                                                               (unsigned)p.ny * (unsigned)zs[D3 ? i / 9 : 0])];
      if constexpr (std::is_same<T, double>::value) {
        const T q = T(Lattice<LAT>::w(i)) * v;
        if constexpr (cx != 0) g[0] = cx > 0 ? g[0] + q : g[0] - q;
        if constexpr (cy != 0) g[1] = cy > 0 ? g[1] + q : g[1] - q;
        if constexpr (cz != 0) g[2] = cz > 0 ? g[2] + q : g[2] - q;
      } else {
        if constexpr (cx != 0) g[0] += T(Lattice<LAT>::w(i) * cx) * v;
        if constexpr (cy != 0) g[1] += T(Lattice<LAT>::w(i) * cy) * v;
        if constexpr (cz != 0) g[2] += T(Lattice<LAT>::w(i) * cz) * v;
      }
    }
  });
  g[0] = T(3) * g[0];
  g[1] = T(3) * g[1];
  g[2] = T(3) * g[2];
}

// |g| and -g/|g| of a D-component gradient (M<T>::unit; on D2Q9 without the z component's
// operations, which add 0 and divide 0).
template <int LAT, typename T>
__device__ __forceinline__ T unit_site(const T g[3], T n[3]) {
  if constexpr (std::is_same<T, double>::value && Lattice<LAT>::D == 2) {
    const T gn = ::sqrt(g[0] * g[0] + g[1] * g[1]);
    const bool in = gn > 0.0;
    n[0] = in ? -g[0] / gn : 0.0;
    n[1] = in ? -g[1] / gn : 0.0;
    n[2] = 0.0;
    return gn;
  } else {
    return M<T>::unit(g, n);
  }
}

template <int LAT, typename T>
__global__ void __launch_bounds__(256) site_normals_kernel(const T* __restrict__ psi, Quad<T>* __restrict__ ng,
                                                           StepT<T> p) {
  pdl_enter();
  const SiteIdx s = site_of(p);
  if (s.x >= p.nx || s.y >= p.ny) return;
  T g[3], n[3];
  grad_site<LAT, T>(psi, s, p, g);
  const T gn = unit_site<LAT, T>(g, n);
  ng[s.i] = Quad<T>{n[0], n[1], n[2], gn};
}

// (n, |grad psi|) of a 32 x 8 column's sites on kN3Z consecutive planes from the psi
// array: the block keeps psi of its 34 x 10 cells (beyond a wall the mirror cell, along
// periodic axes the image) in a shared-memory ring of four planes; the loads of plane z + 2
// are issued before plane z is computed and stored after it, into the slot plane z - 2
// held, so their latency overlaps the arithmetic and one barrier per plane suffices (62 us
// per duct step against 65 us with three slots and two barriers). Every site sums its 26
// neighbours in direction order.
constexpr int kN3Z = 16;
// FIELDS: the roundings of tiled_kernel's fields, whose |grad psi|^2 is x^2 rounded, then y^2
// and z^2 added by fused multiply-adds (so that the ray of lb_fields decides its ties as it
// always did); the step's normals keep M<T>::unit.
template <typename T, bool FIELDS>
__device__ __forceinline__ T unit3_site(const T g[3], T n[3]) {
  if constexpr (!FIELDS || sizeof(T) == 8) return M<T>::unit(g, n);
  else {
    const float g2 = fmaf(g[2], g[2], fmaf(g[1], g[1], __fmul_rn(g[0], g[0])));
    const bool in = g2 > 0.0f;
    const float inv = in ? rsqrtf(g2) : 0.0f;
#pragma unroll
    for (int a = 0; a < 3; ++a) n[a] = in ? -g[a] * inv : 0.0f;
    return in ? g2 * inv : 0.0f;
  }
}
template <typename T, bool FIELDS>
__global__ void __launch_bounds__(256) normals3d_kernel(const T* __restrict__ psi, Quad<T>* __restrict__ ng,
                                                        StepT<T> p) {
  constexpr int RX = 34, RXY = RX * 10, PER = (RXY + 255) / 256;
  __shared__ T s_psi[4 * RXY];
  pdl_enter();
  const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 8, z0 = blockIdx.z * kN3Z;
  const int nx = p.nx, ny = p.ny, nz = p.nz;
  const int tid = threadIdx.x + 32 * threadIdx.y;
  const int z1 = min(nz, z0 + kN3Z);
  auto load = [&](int q, T v[PER]) {  // plane q (wrapped or mirrored) into registers
    const int gz = p.wall_z ? clampc(q, nz) : wrapn(q, nz);
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int c = tid + 256 * k;
      if (c < RXY) {
        const int ly = c / RX, lx = c - ly * RX;
        const int gx = wrapn(x0 - 1 + lx, nx);
        const int gy = p.wall_y ? clampc(y0 - 1 + ly, ny) : wrapn(y0 - 1 + ly, ny);
        v[k] = psi[(unsigned)gx + (unsigned)nx * ((unsigned)gy + (unsigned)ny * (unsigned)gz)];
      }
    }
  };
  auto store = [&](int q, const T v[PER]) {  // into ring slot q mod 4
    T* dst = s_psi + ((q + 4) & 3) * RXY;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int c = tid + 256 * k;
      if (c < RXY) dst[c] = v[k];
    }
  };
  {
    T v[PER];
    load(z0 - 1, v);
    store(z0 - 1, v);
    load(z0, v);
    store(z0, v);
    load(z0 + 1, v);
    store(z0 + 1, v);
  }
  __syncthreads();
  const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
  const int cxy = (threadIdx.x + 1) + RX * (threadIdx.y + 1);
  const bool in = x < nx && y < ny;
  for (int z = z0; z < z1; ++z) {
    T vn[PER];
    const bool more = z + 1 < z1;  // plane z + 2 is needed by the next iteration
    if (more) load(z + 2, vn);
    const T* pm = s_psi + ((z + 3) & 3) * RXY;
    const T* p0 = s_psi + (z & 3) * RXY;
    const T* pp = s_psi + ((z + 1) & 3) * RXY;
    T g[3];
    grad_ring<T>(pm, p0, pp, RX, cxy, g);
    T n[3];
    const T gn = unit3_site<T, FIELDS>(g, n);
    if (in)  // columns at the edge of a lattice of no whole 32 x 8 columns
      ng[(unsigned)x + (unsigned)nx * ((unsigned)y + (unsigned)ny * (unsigned)z)] = Quad<T>{n[0], n[1], n[2], gn};
    // plane z + 2 goes to the fourth slot, the one plane z - 2 held: every thread finished
    // reading it before the barrier that ended the previous plane
    if (more) store(z + 2, vn);
    __syncthreads();
  }
}

template <typename T, bool FIELDS = false>
cudaError_t launch_normals3d(const T* psi, Quad<T>* ng, const StepT<T>& p, cudaStream_t s, bool chained = true) {
  const dim3 grid((unsigned)((p.nx + 31) / 32), (unsigned)((p.ny + 7) / 8), (unsigned)((p.nz + kN3Z - 1) / kN3Z));
  if (chained) return launch_pdl(normals3d_kernel<T, FIELDS>, grid, dim3(32, 8), 0, s, psi, ng, p);
  normals3d_kernel<T, FIELDS><<<grid, dim3(32, 8), 0, s>>>(psi, ng, p);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ near-contact ray
// Distance h of the facing interface along n (0: none), over the stored (n, |grad psi|).
template <int LAT, typename T>
__device__ __forceinline__ int ray_site(const Quad<T>* __restrict__ ng, const Quad<T>& v, const SiteIdx& s,
                                        const StepT<T>& p) {
  constexpr bool D3 = Lattice<LAT>::D == 3;
  if (p.smax == 0 || !(v.w > p.g_th)) return 0;
  int hit = 0;
  static_for<kMaxProbe>([&](auto I) {
    constexpr int st = decltype(I)::value + 1;
    if (hit != 0 || st > p.smax) return;
    int px = s.x + round_probe<st, T>(T(st) * v.x);
    int py = s.y + round_probe<st, T>(T(st) * v.y);
    int pz = D3 ? s.z + round_probe<st, T>(T(st) * v.z) : 0;
    if ((p.wall_y && (py < 0 || py >= p.ny)) || (D3 && p.wall_z && (pz < 0 || pz >= p.nz))) {
      hit = -1;  // the ray left the fluid through a wall
      return;
    }
    px = wrapn(px, p.nx);
    if (!p.wall_y) py = wrapn(py, p.ny);
    if (D3 && !p.wall_z) pz = wrapn(pz, p.nz);
    const Quad<T> w = ng[(unsigned)px + (unsigned)p.nx * ((unsigned)py + (unsigned)p.ny * (unsigned)pz)];
    if (!(w.w > p.g_th)) return;
    T dot = w.x * v.x + w.y * v.y;
    if (D3) dot += w.z * v.z;
    if (dot < T(0)) hit = st;
  });
  return hit < 0 ? 0 : hit;
}

// A_h(h) of a hit, indexed at compile time (a run-time index would put the parameters on the
// stack).
template <typename T>
__device__ __forceinline__ T ah_of(const StepT<T>& p, int hit) {
  T A = T(0);
  static_for<kMaxProbe>([&](auto I) {
    constexpr int st = decltype(I)::value + 1;
    if (hit == st) A = p.Ah[st];
  });
  return A;
}

// ------------------------------------------------------------------ fields and observables
// FP32 -> FP64 by integer operations where the value is zero or normal: the FP64 pipe,
// which also carries conversions, has 1/64 of the FP32 rate and bounds this pass.
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(float v) {
  const unsigned b = __float_as_uint(v), m = b & 0x7FFFFFFFu;
  if (m - 0x00800000u < 0x7F000000u)
    return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(b << 29));
  if (m == 0u) return __hiloint2double((int)b, 0);
  return (double)v;  // subnormal, infinite or NaN
}

// A rounded sum that the compiler does not fuse with the product it adds (G + F_rep).
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return a + b; }

constexpr int kFieldThreads = 256;

// Each thread takes the sites t, t + threads, ... of the lattice and adds their share of the
// observables in FP64 registers (six additions a site on D3Q27, five on D2Q9; the counts
// are integers), so that the block's tree is paid once per block instead of once per 256
// sites. Block sums go to partials[block][kRedSlots] in the slots of tiled_kernel.
template <int LAT, typename T>
__global__ void __launch_bounds__(kFieldThreads) site_fields_kernel(const T* __restrict__ psi, SiteScratch<T> sc,
                                                                    StepT<T> p, FieldOut fo) {
  constexpr int D = Lattice<LAT>::D;
  pdl_enter();
  const unsigned N = (unsigned)p.N, nx = (unsigned)p.nx, ny = (unsigned)p.ny;
  double m1 = 0.0, m2 = 0.0, P[3] = {0.0, 0.0, 0.0}, qd = 0.0;
  unsigned nif = 0, nnci = 0, nbad = 0;
  const unsigned stride = gridDim.x * (unsigned)kFieldThreads;
  for (unsigned i = blockIdx.x * (unsigned)kFieldThreads + threadIdx.x; i < N; i += stride) {
    SiteIdx s;
    const unsigned row = i / nx;
    s.x = (int)(i - row * nx);
    s.z = D == 3 ? (int)(row / ny) : 0;
    s.y = (int)(row - (unsigned)s.z * ny);
    s.i = i;
    const Quad<T> v = sc.ng[i];
    const Pair<T> r = sc.rho[i];
    const T rho = r.x + r.y;
    const int hit = ray_site<LAT, T>(sc.ng, v, s, p);
    T frep[3] = {T(0), T(0), T(0)};
    if (hit) {
      const T A = ah_of(p, hit);
      const T deltaI = T(0.5) * v.w;
      frep[0] = -A * v.x * deltaI;
      frep[1] = -A * v.y * deltaI;
      if (D == 3) frep[2] = -A * v.z * deltaI;
    }
    T u[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int a = 0; a < D; ++a) u[a] = M<T>::div(sc.j[(unsigned)a * N + i] + T(0.5) * add_rn(p.G[a], frep[a]), rho);
    const double r1 = widen(r.x), r2 = widen(r.y), rr = widen(rho);
    double ud[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int a = 0; a < D; ++a) ud[a] = widen(u[a]);
    if (fo.rho1) fo.rho1[i] = r1;
    if (fo.rho2) fo.rho2[i] = r2;
    if (fo.psi) fo.psi[i] = widen(psi[i]);
    if (fo.u) {
      fo.u[i] = ud[0];
      fo.u[(size_t)N + i] = ud[1];
      fo.u[2 * (size_t)N + i] = ud[2];
    }
    if (fo.frep)
      for (int a = 0; a < 3; ++a) fo.frep[(size_t)a * N + i] = widen(frep[a]);
    if (fo.hit) fo.hit[i] = hit;
    if (fo.grad) {
      T g[3];
      grad_site<LAT, T>(psi, s, p, g);
      for (int a = 0; a < 3; ++a) fo.grad[(size_t)a * N + i] = widen(g[a]);
    }
    m1 += r1;
    m2 += r2;
#pragma unroll
    for (int a = 0; a < D; ++a) P[a] += rr * ud[a];
    qd += r1 * ud[0];
    nif += v.w > p.g_th;
    nnci += hit != 0;
    nbad += !(isfinite(r.x) && isfinite(r.y) && rho > T(0)) || !(isfinite(u[0]) && isfinite(u[1]) && isfinite(u[2]));
  }
  // block sums: warp shuffles, then one warp over the warp sums
  __shared__ double wsum[kFieldThreads / 32][6];
  __shared__ unsigned wcnt[kFieldThreads / 32][3];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double red[6] = {m1, m2, P[0], P[1], P[2], qd};
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    if (D == 2 && q == 4) continue;
    for (int o = 16; o > 0; o >>= 1) red[q] += __shfl_down_sync(0xffffffffu, red[q], o);
    if (lane == 0) wsum[warp][q] = red[q];
  }
  nif = __reduce_add_sync(0xffffffffu, nif);
  nnci = __reduce_add_sync(0xffffffffu, nnci);
  nbad = __reduce_add_sync(0xffffffffu, nbad);
  if (lane == 0) {
    wcnt[warp][0] = nif;
    wcnt[warp][1] = nnci;
    wcnt[warp][2] = nbad;
  }
  __syncthreads();
  if (threadIdx.x < kRedSlots) {
    // slots: mass1, mass2, P_x, P_y, P_z, flux (= P_x), flux_disp, n_if, n_nci, n_bad
    const int q = threadIdx.x;
    double v = 0.0;
    if (q < 7) {
      const int k = q == 5 ? 2 : (q == 6 ? 5 : q);
      if (!(D == 2 && k == 4))
        for (int w = 0; w < kFieldThreads / 32; ++w) v += wsum[w][k];
    } else {
      unsigned c = 0;
      for (int w = 0; w < kFieldThreads / 32; ++w) c += wcnt[w][q - 7];
      v = (double)c;
    }
    fo.partials[(size_t)blockIdx.x * kRedSlots + q] = v;
  }
  if (!fo.out) return;
  // the block that draws the last ticket adds the blocks' sums: thread t the elements t, t +
  // 250, ... of the flat array (all of slot t mod 10), then each slot's 25 sums in order
  static_assert(kRedSlots == 10 && kFieldThreads >= 250, "25 threads to each slot");
  __shared__ unsigned last;
  __shared__ double fin[250];
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicInc(fo.ticket, gridDim.x - 1) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (threadIdx.x < 250) {
    const unsigned n = gridDim.x * kRedSlots;
    double v = 0.0;
#pragma unroll 8
    for (unsigned e = threadIdx.x; e < n; e += 250) v += __ldcg(fo.partials + e);
    fin[threadIdx.x] = v;
  }
  __syncthreads();
  if (threadIdx.x < kRedSlots) {
    double v = 0.0;
#pragma unroll
    for (int k = 0; k < 25; ++k) v += fin[threadIdx.x + k * kRedSlots];
    fo.out[threadIdx.x] = v;
  }
  if (threadIdx.x == 32)
    *reinterpret_cast<int*>(fo.out + kErrSlot) = (fo.err ? *fo.err : 0) | (fo.ens ? *fo.ens : 0);
}

// ------------------------------------------------------------------ FP64 collision
// collide_exact with Guo forcing on the totals t_i = f_i^1 + f_i^2, the same roundings with
// fewer operations on the FP64 pipe, which bounds the FP64 step (1/64 of the FP32 rate):
// products with c_i = 0 and 1 are left out (they are exact), and a pair of opposite
// directions shares what only changes its sign (c.u, c.F, c.m and the products odd in
// them) or nothing at all (the products even in them).
template <int LAT, typename WR>
__device__ __forceinline__ void collide64(const double t[Lattice<LAT>::Q], double rho1, double rho2, const double u[3],
                                          const double F[3], double g, const double m[3], const StepT<double>& p,
                                          const WR& fout, unsigned idx) {
  constexpr int Q = Lattice<LAT>::Q;
  constexpr bool D3 = Lattice<LAT>::D == 3;
  const double rho = rho1 + rho2;
  double uF = u[0] * F[0] + u[1] * F[1], uu = u[0] * u[0] + u[1] * u[1];
  if (D3) {
    uF = uF + u[2] * F[2];
    uu = uu + u[2] * u[2];
  }
  const double seg = (p.beta * rho1 * rho2) / rho;
  const double pamp = p.pamp * g;
  const double c1 = rho1 / rho, c2 = rho2 / rho;
  const double u15 = 1.5 * uu;
  static_for<Q>([&](auto I) {
    constexpr int i = decltype(I)::value;
    constexpr int o = opposite(i);
    constexpr double w = Lattice<LAT>::w(i);
    constexpr double w3 = w / 3.0;
    const double wr = w * rho, gw = p.guo * w;
    auto put = [&](auto J, double cuF, double cu3, double cu45, double pert, double rc) {
      constexpr int d = decltype(J)::value;
      const double feq = wr * (((1.0 + cu3) + cu45) - u15);
      const double S = gw * cuF;
      double fs = (t[d] - p.omega * (t[d] - feq)) + S;
      fs = fs + pert;
      fout.template put_step<d>(idx, c1 * fs + rc, c2 * fs - rc, rho1, rho2, 0u);
    };
    if constexpr (i == 0) {
      put(I, 3.0 * (0.0 - uF), 0.0, 0.0, pamp * (0.0 - w3), 0.0);
    } else if constexpr (i < o) {
      constexpr double inv_len = 1.0 / (speed2(i) == 1 ? 1.0 : (speed2(i) == 2 ? 1.4142135623730951
                                                                                : 1.7320508075688772));
      auto dotc = [&](const double v[3]) {  // c.v in x, y, z order, zero components left out
        constexpr int ix = cc(i, 0), iy = cc(i, 1), iz = D3 ? cc(i, 2) : 0;
        double r = 0.0;
        if constexpr (ix != 0) r = ix > 0 ? v[0] : -v[0];
        if constexpr (iy != 0) {
          const double b = iy > 0 ? v[1] : -v[1];
          r = ix != 0 ? r + b : b;
        }
        if constexpr (iz != 0) {
          const double b = iz > 0 ? v[2] : -v[2];
          r = (ix != 0 || iy != 0) ? r + b : b;
        }
        return r;
      };
      const double cu = dotc(u), cF = dotc(F), cm = dotc(m);
      const double cu3 = 3.0 * cu, cu45 = (4.5 * cu) * cu, cuF9 = (9.0 * cu) * cF;
      const double pert = pamp * ((w * cm) * cm - w3);
      const double rc = (seg * w) * (cm * inv_len);
      put(std::integral_constant<int, i>{}, 3.0 * (cF - uF) + cuF9, cu3, cu45, pert, rc);
      put(std::integral_constant<int, o>{}, 3.0 * (-cF - uF) + cuF9, -cu3, cu45, pert, -rc);
    }
  });
}

// One site of the FP64 step with Guo forcing. (rho_1, rho_2) come from the moments pass, so
// the collision needs only the 9 or 27 totals of the pulled populations (their sums over i
// are not formed twice).
template <int LAT>
__global__ void __launch_bounds__(256) site_collide64_kernel(typename Plain<LAT, double>::Reader f,
                                                             typename Plain<LAT, double>::Writer fout,
                                                             SiteScratch<double> sc, StepT<double> p) {
  constexpr int Q = Lattice<LAT>::Q;
  constexpr int D = Lattice<LAT>::D;
  pdl_enter();
  const SiteIdx s = site_of(p);
  if (s.x >= p.nx || s.y >= p.ny) return;
  double fin[2][Q];
  pull_any<LAT, double>(f, s.x, s.y, s.z, p, fin);
#pragma unroll
  for (int i = 0; i < Q; ++i) fin[0][i] = fin[0][i] + fin[1][i];
  const double* t = fin[0];
  const Quad<double> v = sc.ng[s.i];
  const Pair<double> r = sc.rho[s.i];
  const double rho = r.x + r.y;
  const int hit = ray_site<LAT, double>(sc.ng, v, s, p);
  double F[3] = {p.G[0], p.G[1], p.G[2]};
  if (hit) {
    const double A = ah_of(p, hit);
    const double deltaI = 0.5 * v.w;
    F[0] = p.G[0] + -A * v.x * deltaI;
    F[1] = p.G[1] + -A * v.y * deltaI;
    if (D == 3) F[2] = p.G[2] + -A * v.z * deltaI;
  }
  double j[3] = {0.0, 0.0, 0.0};
  static_for<Q>([&](auto I) {
    constexpr int i = decltype(I)::value;
    if constexpr (cc(i, 0) != 0) j[0] = cc(i, 0) > 0 ? j[0] + t[i] : j[0] - t[i];
    if constexpr (cc(i, 1) != 0) j[1] = cc(i, 1) > 0 ? j[1] + t[i] : j[1] - t[i];
    if constexpr (D == 3 && cc(i, 2) != 0) j[2] = cc(i, 2) > 0 ? j[2] + t[i] : j[2] - t[i];
  });
  double u[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int a = 0; a < D; ++a) u[a] = (j[a] + 0.5 * F[a]) / rho;
  const double m[3] = {-v.x, -v.y, -v.z};
  collide64<LAT>(t, r.x, r.y, u, F, v.w, m, p, fout, s.i);
}

// ------------------------------------------------------------------ FP32 collision, D2Q9
// One site of the D2Q9 step in FP32 arithmetic (FP32 and FP16-deviation storage, either
// forcing): the near-contact ray over the stored (n, |grad psi|), then the collision of
// fused2d_kernel by the same expressions. Against that kernel, whose 32 x 16 tiles pull twice
// as many sites again for their halos and run three barriers one after the other, the passes
// read the populations twice, from L2 on lattices that fit there, and wait on each other's
// launches, which the chain hides (us per step, passes against fused): 37 x 19 7.2 / 9.8, 515 x
// 131 9.1 / 10.3, 1030 x 131 10.4 / 13.6, 2050 x 515 52 / 59, 8190 x 1024 374 / 407; FP16
// deviations 1030 x 131 11.8 / 14.4, 8190 x 1024 355 / 477.
template <typename ST, bool EDM>
__global__ void __launch_bounds__(256) site_collide2d_kernel(typename ST::Reader f, typename ST::Writer fout,
                                                             SiteScratch<float> sc, StepT<float> p) {
  pdl_enter();
  const SiteIdx s = site_of(p);
  if constexpr (ST::kHalf)
    fout.seed = step_seed(p, p.parity, blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && threadIdx.y == 0);
  if (s.x >= p.nx || s.y >= p.ny) return;
  float fin[2][9];
  pull_any<0, float>(f, s.x, s.y, 0, p, fin);
  const Quad<float> v = sc.ng[s.i];
  const Pair<float> r = sc.rho[s.i];
  const float rho = r.x + r.y;
  const int hit = ray_site<0, float>(sc.ng, v, s, p);
  float frep[3] = {0.f, 0.f, 0.f};
  if (hit) {
    const float A = ah_of(p, hit);
    const float deltaI = 0.5f * v.w;
    frep[0] = -A * v.x * deltaI;
    frep[1] = -A * v.y * deltaI;
  }
  float j[3], F[3], u[3];
  momentum<0, float>(fin, j);
#pragma unroll
  for (int a = 0; a < 3; ++a) F[a] = add_rn(p.G[a], frep[a]);
#pragma unroll
  for (int a = 0; a < 3; ++a) u[a] = M<float>::div(j[a] + 0.5f * F[a], rho);
  const float m[3] = {-v.x, -v.y, 0.f};
  collide_store<0, float, typename ST::Writer, EDM>(fin, r.x, r.y, j, u, F, v.w, m, p, fout, (int)s.i);
}

// ------------------------------------------------------------------ launches
// Rows of a block: eight (256 sites) where the lattice then still gives every multiprocessor
// several blocks, fewer on small lattices, so that their few warps spread over all of them
// (the FP64 pipe of a multiprocessor is the bound there, not its occupancy).
template <typename T>
dim3 site_block(const HostParams& h) {
  const long long rows = (long long)((h.nx + 31) / 32) * h.ny * h.nz;  // warps of the launch
  const int ry = rows >= 32LL * h.num_sms ? 8 : (rows >= 8LL * h.num_sms ? 4 : 1);
  return dim3(32, ry);
}
inline dim3 site_grid(const HostParams& h, dim3 b) {
  return dim3((h.nx + 31) / 32, (h.ny + b.y - 1) / b.y, h.nz);
}
// Blocks of the fields pass: up to eight per multiprocessor, no more than its partial sums
// have rows (one per tile of tiled_kernel).
inline unsigned site_field_blocks(const HostParams& h, long long rows) {
  long long b = (h.N + kFieldThreads - 1) / kFieldThreads;
  const long long cap = 8LL * h.num_sms;
  if (b > cap) b = cap;
  if (b > rows) b = rows;
  return (unsigned)(b < 1 ? 1 : b);
}

// (n, |grad psi|) of every site by the lattice's normals pass.
template <int LAT, typename T>
cudaError_t launch_site_normals(const T* psi, Quad<T>* ng, const HostParams& h, const StepT<T>& p, cudaStream_t s) {
  const dim3 b = site_block<T>(h);
  return launch_pdl(site_normals_kernel<LAT, T>, site_grid(h, b), b, 0, s, psi, ng, p);
}

// The FP64 step with Guo forcing: moments, normals, collision, each launched programmatically.
template <int LAT>
cudaError_t site_step64(const void* fa, void* fb, double* psi, void* scratch, const HostParams& h,
                        const StepT<double>& p, int* nk, cudaStream_t s) {
  using ST = Plain<LAT, double>;
  const SiteScratch<double> sc = site_scratch<LAT, double>(scratch, (size_t)p.N);
  const dim3 b = site_block<double>(h), g = site_grid(h, b);
  const unsigned N = (unsigned)p.N;
  *nk = 3;
  cudaError_t e = launch_pdl(site_moments_kernel<LAT, ST, false>, g, b, 0, s, ST::reader(fa, N), psi, sc, p);
  if (e == cudaSuccess) e = launch_pdl(site_normals_kernel<LAT, double>, g, b, 0, s, (const double*)psi, sc.ng, p);
  if (e != cudaSuccess) return e;
  return launch_pdl(site_collide64_kernel<LAT>, g, b, 0, s, ST::reader(fa, N), ST::writer(fb, N), sc, p);
}

// The D2Q9 step in FP32 arithmetic: moments, normals, collision, each launched programmatically.
template <typename ST>
cudaError_t site_step2d(const void* fa, void* fb, float* psi, void* scratch, const HostParams& h,
                        const StepT<float>& p, int* nk, cudaStream_t s) {
  const SiteScratch<float> sc = site_scratch<0, float>(scratch, (size_t)p.N);
  const dim3 b = site_block<float>(h), g = site_grid(h, b);
  const unsigned N = (unsigned)p.N;
  *nk = 3;
  cudaError_t e = launch_pdl(site_moments_kernel<0, ST, false>, g, b, 0, s, ST::reader(fa, N), psi, sc, p);
  if (e == cudaSuccess) e = launch_pdl(site_normals_kernel<0, float>, g, b, 0, s, (const float*)psi, sc.ng, p);
  if (e != cudaSuccess) return e;
  return p.edm ? launch_pdl(site_collide2d_kernel<ST, true>, g, b, 0, s, ST::reader(fa, N), ST::writer(fb, N), sc, p)
               : launch_pdl(site_collide2d_kernel<ST, false>, g, b, 0, s, ST::reader(fa, N), ST::writer(fb, N), sc, p);
}

// The observables and fields of a state: three passes, launched programmatically: on a small
// lattice the launches are most of the time. ng is filled by `normals` (the lattice's own
// normals pass). rows: partial sums the caller has room for; *used: written.
template <int LAT, typename ST, typename Normals>
cudaError_t site_fields(typename ST::Reader f, typename ST::Compute* psi, void* scratch, const HostParams& h,
                        const StepT<typename ST::Compute>& p, const FieldOut& fo, long long rows, long long* used,
                        int* nk, cudaStream_t s, Normals&& normals) {
  using T = typename ST::Compute;
  const SiteScratch<T> sc = site_scratch<LAT, T>(scratch, (size_t)p.N);
  const dim3 b = site_block<T>(h);
  cudaError_t e = launch_pdl(site_moments_kernel<LAT, ST, true>, site_grid(h, b), b, 0, s, f, psi, sc, p);
  if (e == cudaSuccess) e = normals(psi, sc.ng);
  if (e != cudaSuccess) return e;
  const unsigned nb = site_field_blocks(h, rows);
  *used = nb;
  *nk = 3;
  return launch_pdl(site_fields_kernel<LAT, T>, dim3(nb), dim3(kFieldThreads), 0, s, (const T*)psi, sc, p, fo);
}

}  // namespace lbnci
