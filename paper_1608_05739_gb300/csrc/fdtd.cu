// fdtd.cu -- Yee and Cole-Karkkainen (CKC) FDTD steps on a periodic grid
// (Sec. III.A; Table 1 rows "Yee" and "CKC"), the comparators of the PSATD step.
//
// Staggering (index [k][j][i] of each component):
//   Ex (i+1/2, j, k)  Ey (i, j+1/2, k)  Ez (i, j, k+1/2)
//   Bx (i, j+1/2, k+1/2)  By (i+1/2, j, k+1/2)  Bz (i+1/2, j+1/2, k); J with E.
// A step advances co-temporal (E, B): B -= (dt/2) curl E; E += dt (c^2 curl B
// - J/eps0); B -= (dt/2) curl E.  Faraday uses forward differences of E,
// Ampere backward differences of B.  CKC (2D only, beta = 1/4): each Faraday
// difference along one axis is averaged over the transverse neighbour rows
// with weights (beta/2, 1 - beta, beta/2).  An absent component (NULL) is
// identically zero.
//
// Bound: HBM (2D grids up to 2048^2: L2).  A thread takes V cells of a row (16 bytes
// where the rows are whole 16-byte blocks, else one cell) and marches M rows (2D)
// or planes (3D), keeping what the next row needs in registers.  Between two steps
// of a call the second half step of B and the first of the next use the same E:
// one pass subtracts the half step twice (the same two roundings), 2 N + 1 passes
// for N steps instead of 3 N.  Against one cell per thread and 3 N passes: CKC TE 2048^2
// with J, 8 steps 705 -> 161 us; Yee 256^3 with J, one step 549 -> 303 us (2.0 GB moved,
// 6.6 TB/s).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "launch.h"

namespace psatd {

struct FdtdGrid {
  int nx, ny, nz;
  int64_t plane;  // nx * ny
  int M;          // rows (2D) or planes (3D) a thread marches
};

template <typename R>
struct FdtdCoef {
  R h, dt, c2, dt_eps0, idx, idy, idz;
};

// V consecutive values of a row
template <typename R, int V>
struct Cells {
  R v[V];
};
template <typename R, int V>
__device__ __forceinline__ Cells<R, V> ldv(const R* p) {
  Cells<R, V> c;
  if constexpr (V == 4) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    c.v[0] = q.x; c.v[1] = q.y; c.v[2] = q.z; c.v[3] = q.w;
  } else if constexpr (V == 2) {
    const double2 q = *reinterpret_cast<const double2*>(p);
    c.v[0] = q.x; c.v[1] = q.y;
  } else {
    c.v[0] = *p;
  }
  return c;
}
template <typename R, int V>
__device__ __forceinline__ void stv(R* p, const Cells<R, V>& c) {
  if constexpr (V == 4) *reinterpret_cast<float4*>(p) = make_float4(c.v[0], c.v[1], c.v[2], c.v[3]);
  else if constexpr (V == 2) *reinterpret_cast<double2*>(p) = make_double2(c.v[0], c.v[1]);
  else *p = c.v[0];
}
template <typename R, int V>
__device__ __forceinline__ Cells<R, V> zerov() {
  Cells<R, V> c;
#pragma unroll
  for (int q = 0; q < V; ++q) c.v[q] = R(0);
  return c;
}

// A row's cells i0 .. i0 + V - 1 with their left and right neighbours (offsets l, r
// of the neighbours relative to i0, periodic)
template <typename R, int V>
struct Wide {
  Cells<R, V> c;
  R l, r;
  __device__ __forceinline__ R at(int q) const { return q < 0 ? l : q < V ? c.v[q] : r; }
};
template <typename R, int V, bool LEFT, bool RIGHT>
__device__ __forceinline__ Wide<R, V> ldw(const R* p, int lo, int ro) {
  Wide<R, V> w;
  w.c = ldv<R, V>(p);
  w.l = LEFT ? p[lo] : R(0);
  w.r = RIGHT ? p[ro] : R(0);
  return w;
}

// b -= h curl, once or twice
template <typename R, bool TWICE>
__device__ __forceinline__ R half_step(R b, R h, R curl) {
  b = b - h * curl;
  if constexpr (TWICE) b = b - h * curl;
  return b;
}

// ---- 2D: rows along x, marching along y.  Bx, By from Ez; Bz from Ex, Ey.
template <typename R, int V, bool CKC, bool TWICE>
__global__ void __launch_bounds__(128) k_faraday2(FdtdGrid g, R* Bx, R* By, R* Bz, const R* Ex, const R* Ey,
                                                  const R* Ez, FdtdCoef<R> f) {
  pass_begin();
  const int i0 = (blockIdx.x * blockDim.x + threadIdx.x) * V;
  const int j0 = (blockIdx.y * blockDim.y + threadIdx.y) * g.M;
  if (i0 >= g.nx || j0 >= g.ny) return;
  const int lo = i0 == 0 ? g.nx - 1 : -1, ro = i0 + V == g.nx ? -i0 : V;  // the neighbours' offsets from i0
  const int j1 = j0 + g.M < g.ny ? j0 + g.M : g.ny;
  auto row = [&](int j) { return (int64_t)(j < 0 ? j + g.ny : j >= g.ny ? j - g.ny : j) * g.nx + i0; };
  typedef Wide<R, V> W;
  // difference along x of a row, at cell q
  auto dx = [&](const W& w, int q) { return (w.at(q + 1) - w.at(q)) * f.idx; };
  // x difference averaged over the rows below and above (CKC)
  auto dx_s = [&](const W& dn, const W& w, const W& up, int q) {
    if constexpr (!CKC) return dx(w, q);
    else return R(0.75) * dx(w, q) + R(0.125) * (dx(dn, q) + dx(up, q));
  };
  auto dy_s = [&](const W& w, const W& up, int q) {
    auto d = [&](int s) { return (up.at(s) - w.at(s)) * f.idy; };
    if constexpr (!CKC) return d(q);
    else return R(0.75) * d(q) + R(0.125) * (d(q - 1) + d(q + 1));
  };
  if (Bz) {
    W x = ldw<R, V, CKC, CKC>(Ex + row(j0), lo, ro), y = ldw<R, V, false, true>(Ey + row(j0), lo, ro), yd{}, yu{};
    if constexpr (CKC) {
      yd = ldw<R, V, false, true>(Ey + row(j0 - 1), lo, ro);
    }
    for (int j = j0; j < j1; ++j) {
      const int64_t c = row(j), cu = row(j + 1);
      const W xu = ldw<R, V, CKC, CKC>(Ex + cu, lo, ro);
      if (CKC || j + 1 < j1) yu = ldw<R, V, false, true>(Ey + cu, lo, ro);
      Cells<R, V> b = ldv<R, V>(Bz + c);
#pragma unroll
      for (int q = 0; q < V; ++q)
        b.v[q] = half_step<R, TWICE>(b.v[q], f.h, dx_s(yd, y, yu, q) - dy_s(x, xu, q));
      stv<R, V>(Bz + c, b);
      x = xu;
      yd = y;
      y = yu;
    }
  }
  if (Bx) {  // TM: By present too
    W e = ldw<R, V, CKC, true>(Ez + row(j0), lo, ro), ed{};
    if constexpr (CKC) ed = ldw<R, V, false, true>(Ez + row(j0 - 1), lo, ro);
    for (int j = j0; j < j1; ++j) {
      const int64_t c = row(j);
      const W eu = ldw<R, V, CKC, true>(Ez + row(j + 1), lo, ro);
      Cells<R, V> bx = ldv<R, V>(Bx + c), by = ldv<R, V>(By + c);
#pragma unroll
      for (int q = 0; q < V; ++q) {
        bx.v[q] = half_step<R, TWICE>(bx.v[q], f.h, dy_s(e, eu, q) - R(0));
        by.v[q] = half_step<R, TWICE>(by.v[q], f.h, R(0) - dx_s(ed, e, eu, q));
      }
      stv<R, V>(Bx + c, bx);
      stv<R, V>(By + c, by);
      ed = e;
      e = eu;
    }
  }
}

template <typename R, int V>
__global__ void __launch_bounds__(128) k_ampere2(FdtdGrid g, R* Ex, R* Ey, R* Ez, const R* Bx, const R* By,
                                                 const R* Bz, const R* Jx, const R* Jy, const R* Jz, FdtdCoef<R> f) {
  pass_begin();
  const int i0 = (blockIdx.x * blockDim.x + threadIdx.x) * V;
  const int j0 = (blockIdx.y * blockDim.y + threadIdx.y) * g.M;
  if (i0 >= g.nx || j0 >= g.ny) return;
  const int lo = i0 == 0 ? g.nx - 1 : -1;
  const int j1 = j0 + g.M < g.ny ? j0 + g.M : g.ny;
  const int64_t first = (int64_t)j0 * g.nx + i0;
  const int64_t below = (int64_t)(j0 == 0 ? g.ny - 1 : j0 - 1) * g.nx + i0;
  typedef Wide<R, V> W;
  auto update = [&](R e, R curl, const R* J, R j) {
    e = e + f.dt * (f.c2 * curl);
    return J ? e - f.dt_eps0 * j : e;
  };
  if (Ex) {  // TE: Ey present too
    Cells<R, V> d = ldv<R, V>(Bz + below);
    int64_t c = first;
    for (int j = j0; j < j1; ++j, c += g.nx) {
      const W b = ldw<R, V, true, false>(Bz + c, lo, 0);
      Cells<R, V> ex = ldv<R, V>(Ex + c), ey = ldv<R, V>(Ey + c);
      const Cells<R, V> jx = Jx ? ldv<R, V>(Jx + c) : zerov<R, V>(), jy = Jy ? ldv<R, V>(Jy + c) : zerov<R, V>();
#pragma unroll
      for (int q = 0; q < V; ++q) {
        ex.v[q] = update(ex.v[q], (b.at(q) - d.v[q]) * f.idy - R(0), Jx, jx.v[q]);
        ey.v[q] = update(ey.v[q], R(0) - (b.at(q) - b.at(q - 1)) * f.idx, Jy, jy.v[q]);
      }
      stv<R, V>(Ex + c, ex);
      stv<R, V>(Ey + c, ey);
      d = b.c;
    }
  }
  if (Ez) {
    Cells<R, V> d = ldv<R, V>(Bx + below);
    int64_t c = first;
    for (int j = j0; j < j1; ++j, c += g.nx) {
      const Cells<R, V> bx = ldv<R, V>(Bx + c);
      const W by = ldw<R, V, true, false>(By + c, lo, 0);
      Cells<R, V> ez = ldv<R, V>(Ez + c);
      const Cells<R, V> jz = Jz ? ldv<R, V>(Jz + c) : zerov<R, V>();
#pragma unroll
      for (int q = 0; q < V; ++q)
        ez.v[q] = update(ez.v[q], (by.at(q) - by.at(q - 1)) * f.idx - (bx.v[q] - d.v[q]) * f.idy, Jz, jz.v[q]);
      stv<R, V>(Ez + c, ez);
      d = bx;
    }
  }
}

// ---- 3D (all six components): threads over x and y, marching along z.
template <typename R, int V, bool TWICE>
__global__ void __launch_bounds__(128) k_faraday3(FdtdGrid g, R* Bx, R* By, R* Bz, const R* Ex, const R* Ey,
                                                  const R* Ez, FdtdCoef<R> f) {
  pass_begin();
  const int i0 = (blockIdx.x * blockDim.x + threadIdx.x) * V;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k0 = blockIdx.z * g.M;
  if (i0 >= g.nx || j >= g.ny) return;
  const int ro = i0 + V == g.nx ? -i0 : V;
  const int64_t up = j + 1 == g.ny ? -(int64_t)j * g.nx : g.nx;  // offset of row j + 1
  const int k1 = k0 + g.M < g.nz ? k0 + g.M : g.nz;
  int64_t c = (int64_t)k0 * g.plane + (int64_t)j * g.nx + i0;
  Cells<R, V> ex = ldv<R, V>(Ex + c), ey = ldv<R, V>(Ey + c);
  for (int k = k0; k < k1; ++k, c += g.plane) {
    const int64_t cn = k + 1 == g.nz ? c - (int64_t)k * g.plane : c + g.plane;  // plane k + 1
    const Cells<R, V> exn = ldv<R, V>(Ex + cn), eyn = ldv<R, V>(Ey + cn);
    const Cells<R, V> exu = ldv<R, V>(Ex + c + up), ezu = ldv<R, V>(Ez + c + up);
    const Wide<R, V> ez = ldw<R, V, false, true>(Ez + c, 0, ro);
    const R eyr = Ey[c + ro];
    Cells<R, V> bx = ldv<R, V>(Bx + c), by = ldv<R, V>(By + c), bz = ldv<R, V>(Bz + c);
#pragma unroll
    for (int q = 0; q < V; ++q) {
      const R y1 = q + 1 < V ? ey.v[q + 1 < V ? q + 1 : q] : eyr;
      bx.v[q] = half_step<R, TWICE>(bx.v[q], f.h, (ezu.v[q] - ez.at(q)) * f.idy - (eyn.v[q] - ey.v[q]) * f.idz);
      by.v[q] = half_step<R, TWICE>(by.v[q], f.h, (exn.v[q] - ex.v[q]) * f.idz - (ez.at(q + 1) - ez.at(q)) * f.idx);
      bz.v[q] = half_step<R, TWICE>(bz.v[q], f.h, (y1 - ey.v[q]) * f.idx - (exu.v[q] - ex.v[q]) * f.idy);
    }
    stv<R, V>(Bx + c, bx);
    stv<R, V>(By + c, by);
    stv<R, V>(Bz + c, bz);
    ex = exn;
    ey = eyn;
  }
}

template <typename R, int V>
__global__ void __launch_bounds__(128) k_ampere3(FdtdGrid g, R* Ex, R* Ey, R* Ez, const R* Bx, const R* By,
                                                 const R* Bz, const R* Jx, const R* Jy, const R* Jz, FdtdCoef<R> f) {
  pass_begin();
  const int i0 = (blockIdx.x * blockDim.x + threadIdx.x) * V;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k0 = blockIdx.z * g.M;
  if (i0 >= g.nx || j >= g.ny) return;
  const int lo = i0 == 0 ? g.nx - 1 : -1;
  const int64_t dn = j == 0 ? (int64_t)(g.ny - 1) * g.nx : -(int64_t)g.nx;  // offset of row j - 1
  const int k1 = k0 + g.M < g.nz ? k0 + g.M : g.nz;
  int64_t c = (int64_t)k0 * g.plane + (int64_t)j * g.nx + i0;
  const int64_t cp = k0 == 0 ? c + (int64_t)(g.nz - 1) * g.plane : c - g.plane;
  Cells<R, V> bxp = ldv<R, V>(Bx + cp), byp = ldv<R, V>(By + cp);
  auto update = [&](R e, R curl, const R* J, R j) {
    e = e + f.dt * (f.c2 * curl);
    return J ? e - f.dt_eps0 * j : e;
  };
  for (int k = k0; k < k1; ++k, c += g.plane) {
    const Cells<R, V> bx = ldv<R, V>(Bx + c), bxd = ldv<R, V>(Bx + c + dn), bzd = ldv<R, V>(Bz + c + dn);
    const Wide<R, V> by = ldw<R, V, true, false>(By + c, lo, 0), bz = ldw<R, V, true, false>(Bz + c, lo, 0);
    Cells<R, V> ex = ldv<R, V>(Ex + c), ey = ldv<R, V>(Ey + c), ez = ldv<R, V>(Ez + c);
    const Cells<R, V> jx = Jx ? ldv<R, V>(Jx + c) : zerov<R, V>(), jy = Jy ? ldv<R, V>(Jy + c) : zerov<R, V>(),
                      jz = Jz ? ldv<R, V>(Jz + c) : zerov<R, V>();
#pragma unroll
    for (int q = 0; q < V; ++q) {
      ex.v[q] = update(ex.v[q], (bz.at(q) - bzd.v[q]) * f.idy - (by.at(q) - byp.v[q]) * f.idz, Jx, jx.v[q]);
      ey.v[q] = update(ey.v[q], (bx.v[q] - bxp.v[q]) * f.idz - (bz.at(q) - bz.at(q - 1)) * f.idx, Jy, jy.v[q]);
      ez.v[q] = update(ez.v[q], (by.at(q) - by.at(q - 1)) * f.idx - (bx.v[q] - bxd.v[q]) * f.idy, Jz, jz.v[q]);
    }
    stv<R, V>(Ex + c, ex);
    stv<R, V>(Ey + c, ey);
    stv<R, V>(Ez + c, ez);
    bxp = bx;
    byp = by.c;
  }
}

template <typename R, int V>
static cudaError_t run_fdtd(int ndim, int scheme, int64_t nx, int64_t ny, int64_t nz, const FdtdCoef<R>& f,
                            R* const e[3], R* const b[3], const R* const j[3], int nsteps, cudaStream_t st) {
  FdtdGrid g{(int)nx, (int)ny, (int)nz, nx * ny, 1};
  const int tx = (int)((nx + V - 1) / V);
  const unsigned bx = tx >= 128 ? 128u : tx >= 64 ? 64u : 32u, by = 128u / bx;
  // two rows / planes per thread where that leaves each SM 512 threads: the next row's
  // values are loaded once; more rows make blocks too few for an even spread over the SMs
  // (CKC TE 2048^2, eight steps with 2 / 4 / 8 rows 156 / 159 / 193 us; Yee 200^3 291 / 301 / 331)
  const int64_t march = ndim == 3 ? nz : ny, across = (int64_t)tx * (ndim == 3 ? ny : 1);
  if (across * (march / 2) >= 152 * 512) g.M = 2;
  const unsigned gx = (unsigned)((tx + bx - 1) / bx);
  const dim3 block(bx, by);
  const int64_t span = (int64_t)by * (ndim == 3 ? 1 : g.M);
  const dim3 grid(gx, (unsigned)((ny + span - 1) / span), ndim == 3 ? (unsigned)((nz + g.M - 1) / g.M) : 1u);
  auto faraday = [&](bool twice) {
    if (ndim == 3) {
      if (twice) launch_pass(true, k_faraday3<R, V, true>, grid, block, 0, st, g, b[0], b[1], b[2], e[0], e[1], e[2], f);
      else launch_pass(true, k_faraday3<R, V, false>, grid, block, 0, st, g, b[0], b[1], b[2], e[0], e[1], e[2], f);
    } else if (scheme == 1) {
      if (twice) launch_pass(true, k_faraday2<R, V, true, true>, grid, block, 0, st, g, b[0], b[1], b[2], e[0], e[1], e[2], f);
      else launch_pass(true, k_faraday2<R, V, true, false>, grid, block, 0, st, g, b[0], b[1], b[2], e[0], e[1], e[2], f);
    } else {
      if (twice) launch_pass(true, k_faraday2<R, V, false, true>, grid, block, 0, st, g, b[0], b[1], b[2], e[0], e[1], e[2], f);
      else launch_pass(true, k_faraday2<R, V, false, false>, grid, block, 0, st, g, b[0], b[1], b[2], e[0], e[1], e[2], f);
    }
  };
  for (int s = 0; s < nsteps; ++s) {
    faraday(s > 0);
    if (ndim == 3)
      launch_pass(true, k_ampere3<R, V>, grid, block, 0, st, g, e[0], e[1], e[2], b[0], b[1], b[2], j[0], j[1], j[2], f);
    else
      launch_pass(true, k_ampere2<R, V>, grid, block, 0, st, g, e[0], e[1], e[2], b[0], b[1], b[2], j[0], j[1], j[2], f);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
  }
  faraday(false);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_fdtd(int ndim, int scheme, int64_t nx, int64_t ny, int64_t nz, const double* d,
                        double dt, double c, double eps0, void* const E[3], void* const B[3],
                        const void* const J[3], int nsteps, cudaStream_t st) {
  R* e[3] = {static_cast<R*>(E[0]), static_cast<R*>(E[1]), static_cast<R*>(E[2])};
  R* b[3] = {static_cast<R*>(B[0]), static_cast<R*>(B[1]), static_cast<R*>(B[2])};
  const R* j[3] = {static_cast<const R*>(J[0]), static_cast<const R*>(J[1]),
                   static_cast<const R*>(J[2])};
  FdtdCoef<R> f;
  f.h = R(0.5 * dt);
  f.dt = R(dt);
  f.c2 = R(c * c);
  f.dt_eps0 = R(dt / eps0);
  f.idx = R(1.0 / d[0]);
  f.idy = R(1.0 / d[1]);
  f.idz = R(ndim == 3 ? 1.0 / d[2] : 0.0);
  constexpr int V = 16 / sizeof(R);  // cells of 16 bytes (the arrays' base addresses are 16-byte aligned)
  return nx % V == 0 ? run_fdtd<R, V>(ndim, scheme, nx, ny, nz, f, e, b, j, nsteps, st)
                     : run_fdtd<R, 1>(ndim, scheme, nx, ny, nz, f, e, b, j, nsteps, st);
}

template cudaError_t launch_fdtd<float>(int, int, int64_t, int64_t, int64_t, const double*, double,
                                        double, double, void* const[3], void* const[3],
                                        const void* const[3], int, cudaStream_t);
template cudaError_t launch_fdtd<double>(int, int, int64_t, int64_t, int64_t, const double*, double,
                                         double, double, void* const[3], void* const[3],
                                         const void* const[3], int, cudaStream_t);

}  // namespace psatd
