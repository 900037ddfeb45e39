// farfield.cu -- the Fraunhofer far-field transform of a field snapshot, the
// diagnostic of the angularly resolved harmonic spectrum (Sec. II.B): for every
// requested wavevector k_j = (kx, ky),
//   U_j = sum over the window's cells of w(x, y) F(x, y) exp(-i (kx x + ky y)) dx dy,
// x = i dx, y = j dy, w an optional Hann apodisation (along x, or x and y).
//
// Rows first: S_j(y) = sum_x w_x F(x, y) exp(-i kx x) in the field's precision, then
// the sum over y in FP64.  A warp takes 4 wavevectors x 8 rows; its lanes take the
// cells x = lane, lane + 32, .. of the rows (each field value serves 4 wavevectors,
// each phase 8 rows), and a reduce-scatter over the lanes leaves every lane with one
// (wavevector, row) sum: the sum order of one warp per row.  The x phases (FP64, rounded
// once to the field's precision) are a table of the CTA's wavevectors in shared
// memory, kXs<R> cells at a time.  A CTA has 8 warps over KC = 4 nkw wavevectors and 8/nkw
// row parts, and a cluster splits the rows, then the columns, further where the wavevectors
// alone do not fill the GPU; every sum is taken in a fixed order, so the result does not depend on
// scheduling.
//
// FP64 runs at 2 operations per cycle and SM here, so the FP64 phases decide:
// one sincos per wavevector and row, on one lane of a warp, took most of 8.67 ms for
// 3848 wavevectors over 512 x 1024 cells.  For float fields the x phases come from
// ten sincos per wavevector (the binary powers of the cell step and the start) by
// products in FP64 (error 1e-13, against 6e-8 of the rounded phases), and the rows'
// phases enter by Horner's rule, U = U z + S, z = exp(-i ky 8 dy).  Double fields keep
// one sincos per phase, on all lanes.  That case: 8.67 ms -> 0.40 ms (20 TFLOP/s of the
// float sums; the operand loads and the table share the rest); double, 998 wavevectors
// over 874 x 734 cells, 6.04 -> 3.55 ms (the FP64 units' rate).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "farfield.h"

namespace psatd {

namespace {

template <typename R> struct FF;
template <> struct FF<float> {
  typedef float2 C2;
  static constexpr int kXs = 512;  // cells of the phase table
};
template <> struct FF<double> {
  typedef double2 C2;
  static constexpr int kXs = 256;
};
constexpr int kFfThreads = 256, kFfRows = 8, kFfKPerWarp = 4;
constexpr int kFfMaxWin = 4096;  // rows of a CTA with a table of apodisation weights

__device__ __forceinline__ double hann_w(int i, int n) {
  const double s = sinpi((i + 0.5) / (double)n);
  return s * s;
}
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 expi(double a) {  // exp(-i a)
  double s, c;
  sincos(a, &s, &c);
  return make_double2(c, -s);
}
// acc += f p for a real f
__device__ __forceinline__ void mac(float2& acc, float f, float2 p) { acc = __ffma2_rn(make_float2(f, f), p, acc); }
__device__ __forceinline__ void mac(double2& acc, double f, double2 p) {
  acc.x = fma(f, p.x, acc.x);
  acc.y = fma(f, p.y, acc.y);
}

}  // namespace

// A cluster's CTAs (blockIdx.y) are sx column ranges of each of gridDim.y / sx row ranges;
// a CTA's rows are 8 / nkw parts of whole 8-row tiles.
struct FarfieldSplit {
  int nkw;        // warps over the wavevectors (1, 2 or 4)
  int part_rows;  // rows per part, a multiple of 8
  int sx;
  int cols;       // columns per range, a multiple of 32
};

template <typename R>
__global__ void __launch_bounds__(kFfThreads, sizeof(R) == 4 ? 2 : 1) k_farfield(FarfieldArgs a, FarfieldSplit sp) {
  typedef typename FF<R>::C2 C2;
  constexpr int XS = FF<R>::kXs;
  extern __shared__ __align__(16) unsigned char ff_smem[];
  const int KC = kFfKPerWarp * sp.nkw, nrp = 8 / sp.nkw;
  C2* P = reinterpret_cast<C2*>(ff_smem);                                  // [KC][XS]
  double2* ang = reinterpret_cast<double2*>(ff_smem + (size_t)KC * XS * sizeof(C2));  // [KC][48]
  __shared__ double2 part[8][kFfKPerWarp];  // per warp and wavevector
  __shared__ __align__(16) double2 total[16];             // per wavevector of the CTA
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int kw = warp % sp.nkw, rp = warp / sp.nkw;
  const int k0 = blockIdx.x * KC;
  const int wx = (int)(a.x1 - a.x0), wy = (int)(a.y1 - a.y0);
  const int cta_rows = sp.part_rows * nrp;
  const int cta_row0 = (int)blockIdx.y / sp.sx * cta_rows;
  const int r_lo = cta_row0 + rp * sp.part_rows;  // this warp's rows
  const int c_lo = (int)blockIdx.y % sp.sx * sp.cols, c_hi = c_lo + sp.cols < wx ? c_lo + sp.cols : wx;
  const int r_hi = r_lo + sp.part_rows < wy ? r_lo + sp.part_rows : wy;
  double2* pw = ang + KC * 48;                                             // [KC][10]
  double* wxt = reinterpret_cast<double*>(pw + KC * 10);                   // x weights of the table's cells
  double* wtab = wxt + XS;                                                 // row weights
  const bool tabled = a.win_y && cta_rows <= kFfMaxWin;
  if (tabled)
    for (int i = tid; i < cta_rows; i += kFfThreads) wtab[i] = hann_w(cta_row0 + i, wy);
  // this lane's wavevector and row of a tile
  const int kl = kw * kFfKPerWarp + (lane >> 3), rl = lane & 7;
  const int kg = k0 + kl < a.nk ? k0 + kl : a.nk - 1;
  const double ky = a.k[2 * kg + 1];
  const double2 z = std::is_same<R, float>::value ? expi(ky * (8.0 * a.dy)) : make_double2(0.0, 0.0);
  const int tiles = r_lo < r_hi ? (r_hi - r_lo + 7) / 8 : 0;
  double2 usum = make_double2(0.0, 0.0);
  for (int xs = c_lo; xs < c_hi; xs += XS) {
    const int nx = c_hi - xs < XS ? c_hi - xs : XS;
    const int nstep = (nx + 31) / 32;
    __syncthreads();  // the previous table is read
    if (a.win_x)
      for (int i = tid; i < nx; i += kFfThreads) wxt[i] = hann_w(xs + i, wx);
    if constexpr (std::is_same<R, float>::value) {
      // pw[j] = exp(-i kx 2^j dx), j < 9, and the start of the table; ang: the cells 0..31
      // and the starts of the blocks of 32 as products of these
      for (int i = tid; i < KC * 10; i += kFfThreads) {
        const int kk = i / 10, e = i % 10;
        const double kx = a.k[2 * (k0 + kk < a.nk ? k0 + kk : a.nk - 1)];
        pw[i] = expi(kx * (e < 9 ? (double)(1 << e) : (double)(a.x0 + xs)) * a.dx);
      }
      __syncthreads();
      for (int i = tid; i < KC * 48; i += kFfThreads) {
        const int kk = i / 48, e = i % 48;
        double2 v = e < 32 ? make_double2(1.0, 0.0) : pw[kk * 10 + 9];
        const int bits = e < 32 ? e : e - 32, j0 = e < 32 ? 0 : 5;
        for (int j = 0; (bits >> j) != 0; ++j)
          if ((bits >> j) & 1) v = cmul(v, pw[kk * 10 + j0 + j]);
        ang[i] = v;
      }
    }
    __syncthreads();
    for (int kk = warp; kk < KC; kk += kFfThreads / 32) {
      const double kx = a.k[2 * (k0 + kk < a.nk ? k0 + kk : a.nk - 1)];
      for (int st = 0; st < nstep; ++st) {
        const int x = 32 * st + lane;
        C2 p;
        p.x = p.y = R(0);
        if (x < nx) {
          double2 e;
          if constexpr (std::is_same<R, float>::value) e = cmul(ang[kk * 48 + 32 + st], ang[kk * 48 + lane]);
          else e = expi(kx * (double)(a.x0 + xs + x) * a.dx);
          const double w = a.win_x ? wxt[x] : 1.0;
          p.x = (R)(w * e.x);
          p.y = (R)(w * e.y);
        }
        P[kk * XS + x] = p;
      }
    }
    __syncthreads();
    // accumulator q of a lane holds wavevector q ^ (lane >> 3) of the warp's four, so that the
    // reduce-scatter's first two steps keep and send the same accumulators in every lane
    const C2* Pl[kFfKPerWarp];
#pragma unroll
    for (int q = 0; q < kFfKPerWarp; ++q) Pl[q] = P + (kw * kFfKPerWarp + (q ^ (lane >> 3))) * XS + lane;
    const R* Fx = static_cast<const R*>(a.F) + a.x0 + xs + lane;
    double2 u = make_double2(0.0, 0.0);
    for (int tl = tiles - 1; tl >= 0; --tl) {  // descending: Horner's rule
      const int row0 = r_lo + 8 * tl;
      C2 acc[kFfKPerWarp * kFfRows];
#pragma unroll
      for (int i = 0; i < kFfKPerWarp * kFfRows; ++i) acc[i].x = acc[i].y = R(0);
      const int nr = r_hi - row0;  // valid rows of the tile: those r < nr
      const R* Fr[kFfRows];        // (rows past the last read the tile's first and count zero)
#pragma unroll
      for (int r = 0; r < kFfRows; ++r) Fr[r] = Fx + (a.y0 + row0 + (r < nr ? r : 0)) * a.nx;
      auto step = [&](int s, bool in) {
        R f[kFfRows];
#pragma unroll
        for (int r = 0; r < kFfRows; ++r) f[r] = in ? __ldg(Fr[r] + 32 * s) : R(0);
#pragma unroll
        for (int q = 0; q < kFfKPerWarp; ++q) {
          const C2 p = Pl[q][32 * s];
#pragma unroll
          for (int r = 0; r < kFfRows; ++r) mac(acc[q * kFfRows + r], f[r], p);
        }
      };
      const int full = nx / 32;
#pragma unroll 2
      for (int s = 0; s < full; ++s) step(s, true);
      if (full < nstep) step(full, 32 * full + lane < nx);
      // reduce-scatter: lane l ends with the sum of (wavevector l / 8, row l % 8)
#pragma unroll
      for (int o = 16; o >= 8; o >>= 1)
#pragma unroll
        for (int i = 0; i < o; ++i) {
          acc[i].x += __shfl_xor_sync(0xffffffffu, acc[i + o].x, o);
          acc[i].y += __shfl_xor_sync(0xffffffffu, acc[i + o].y, o);
        }
#pragma unroll
      for (int o = 4; o; o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < o; ++i) {
          const C2 keep = up ? acc[i + o] : acc[i], send = up ? acc[i] : acc[i + o];
          acc[i].x = keep.x + __shfl_xor_sync(0xffffffffu, send.x, o);
          acc[i].y = keep.y + __shfl_xor_sync(0xffffffffu, send.y, o);
        }
      }
      if (rl >= nr) acc[0].x = acc[0].y = R(0);
      double2 sv = make_double2((double)acc[0].x, (double)acc[0].y);
      const int row = row0 + rl;
      if (a.win_y) {
        const double w = row < wy ? (tabled ? wtab[row - cta_row0] : hann_w(row, wy)) : 0.0;
        sv.x *= w;
        sv.y *= w;
      }
      if constexpr (std::is_same<R, float>::value) {
        u = make_double2(fma(u.x, z.x, fma(-u.y, z.y, sv.x)), fma(u.x, z.y, fma(u.y, z.x, sv.y)));
      } else {
        const double2 e = expi(ky * (double)(a.y0 + row) * a.dy);
        u.x += sv.x * e.x - sv.y * e.y;
        u.y += sv.x * e.y + sv.y * e.x;
      }
    }
    if constexpr (std::is_same<R, float>::value) u = cmul(u, expi(ky * (double)(a.y0 + r_lo + rl) * a.dy));
    usum.x += u.x;
    usum.y += u.y;
  }
  // rows of a tile (8 lanes), row parts of the CTA, CTAs of the cluster
#pragma unroll
  for (int o = 4; o; o >>= 1) {
    usum.x += __shfl_xor_sync(0xffffffffu, usum.x, o);
    usum.y += __shfl_xor_sync(0xffffffffu, usum.y, o);
  }
  if (rl == 0) part[warp][lane >> 3] = usum;
  __syncthreads();
  if (tid < KC) {
    double2 s = make_double2(0.0, 0.0);
    for (int p = 0; p < nrp; ++p) {
      const double2 v = part[p * sp.nkw + tid / kFfKPerWarp][tid % kFfKPerWarp];
      s.x += v.x;
      s.y += v.y;
    }
    total[tid] = s;
  }
  // all CTAs' totals are written before the first reads them, and none leaves before
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (blockIdx.y == 0 && tid < KC && k0 + tid < a.nk) {
    double2 s = make_double2(0.0, 0.0);
    for (unsigned c = 0; c < gridDim.y; ++c) {
      double2 v;
      asm volatile(
          "{\n\t.reg .u32 p;\n\tmapa.shared::cluster.u32 p, %2, %3;\n\t"
          "ld.shared::cluster.v2.f64 {%0, %1}, [p];\n\t}"
          : "=d"(v.x), "=d"(v.y)
          : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(&total[tid]))), "r"(c)
          : "memory");
      s.x += v.x;
      s.y += v.y;
    }
    a.out[2 * (k0 + tid)] = s.x * a.dx * a.dy;
    a.out[2 * (k0 + tid) + 1] = s.y * a.dx * a.dy;
  }
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <typename R>
static cudaError_t launch_ff(const FarfieldArgs& a, cudaStream_t st) {
  const int wy = (int)(a.y1 - a.y0);
  FarfieldSplit sp;
  // 16 wavevectors per CTA once that gives every SM one, fewer (more row parts) below
  sp.nkw = a.nk >= 16 * 152 ? 4 : a.nk >= 8 * 152 ? 2 : 1;
  const int KC = kFfKPerWarp * sp.nkw, nrp = 8 / sp.nkw, gx = (a.nk + KC - 1) / KC;
  // CTAs of a cluster, up to two per SM in all: over the rows while every part keeps two
  // tiles, then over the columns while every range keeps two blocks of 32
  const int wx = (int)(a.x1 - a.x0), blocks = (wx + 31) / 32;
  int S = 1;
  while (S < 8 && (int64_t)gx * S < 2 * 152 && wy >= 2 * S * nrp * 16) S *= 2;
  sp.part_rows = ((wy + S * nrp - 1) / (S * nrp) + 7) / 8 * 8;
  const int cta_rows = sp.part_rows * nrp;
  sp.sx = 1;
  while (S * sp.sx < 8 && (int64_t)gx * S * sp.sx < 2 * 152 && blocks >= 4 * sp.sx) sp.sx *= 2;
  sp.cols = (blocks + sp.sx - 1) / sp.sx * 32;
  const size_t smem = (size_t)KC * FF<R>::kXs * sizeof(typename FF<R>::C2) + (size_t)KC * 58 * sizeof(double2) +
                      (size_t)FF<R>::kXs * 8 + (a.win_y && cta_rows <= kFfMaxWin ? (size_t)cta_rows * 8 : 0);
  cudaError_t e = cudaFuncSetAttribute(k_farfield<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)gx, (unsigned)(S * sp.sx));
  cfg.blockDim = dim3(kFfThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1;
  at[0].val.clusterDim.y = (unsigned)(S * sp.sx);
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_farfield<R>, a, sp);
}

cudaError_t launch_farfield(bool f32, const FarfieldArgs& a, cudaStream_t st) {
  return f32 ? launch_ff<float>(a, st) : launch_ff<double>(a, st);
}

}  // namespace psatd
