// pair_rows.cuh -- the FP32 transposing passes (no tensor cores): as k_fwd_T /
// k_inv_T (psatd_kernels.cuh), with two adjacent rows per thread in packed
// arithmetic (fft_line.cuh).
//
// A CTA takes TB = 1 << log_tb rows as TBp = max(TB/2, 1) row pairs of T threads
// (rows b0 + 2g, b0 + 2g + 1); TB = 1 runs one pair whose second row repeats the
// first and is not stored.  A pair's transposed elements (k, b), (k, b + 1) are 16
// contiguous bytes, moved by one access.  The R2C / C2R step takes the bins k and
// L - k together (they need the same two values and, up to conjugation, the same
// product), so every spectral value crosses shared memory once.
//
// Bound: the L1 / shared-memory data pipe and the latency between stages on small
// grids, HBM on large ones.  One row per thread -> pairs: 2048^2 TE forward 54.9 ->
// 43.4 us (75.1k -> 55.7k wavefronts per SM, 33.9 M -> 18.3 M instructions), inverse
// 41.3 -> 33.0 us; 256^3 with eleven components, x forward 319 -> 221 us, y forward
// 236 -> 216 us (6.1 TB/s of DRAM traffic), y inverse 157 -> 124 us.
#pragma once

#include "fft_line.cuh"
#include "psatd_kernels.cuh"

namespace psatd {

// Threads per CTA: half of the rows' threads of the one-row passes.  Registers: 128 (two
// CTAs of 256 threads per SM), 168 for 20 and 24 elements per thread.
template <int L>
struct RowPairThreads { static constexpr int value = RowThreads<float, L>::value / 2 > FFTPlan<L, RowEPT<L>::value>::kT
                                                         ? RowThreads<float, L>::value / 2
                                                         : FFTPlan<L, RowEPT<L>::value>::kT; };

// XOR mask of pair g's line in the transposed accesses (16-byte elements: 8 bank
// groups shared by the block's pairs); stays inside the line for L < 8.
__device__ __forceinline__ int pair_xor(int g, int log_tbp, int L) {
  return (log_tbp <= 3 ? g * (8 >> log_tbp) : g) & 7 & (L - 1);
}

__device__ __forceinline__ C2 mkpair(float2 r0, float2 r1) { return C2{F2{r0.x, r1.x}, F2{r0.y, r1.y}}; }
// adjacent rows (re, im, re, im) as stored
__device__ __forceinline__ C2 unpack_rows(float4 q) { return C2{F2{q.x, q.z}, F2{q.y, q.w}}; }
__device__ __forceinline__ float4 pack_rows(C2 c) { return make_float4(c.x.a, c.y.a, c.x.b, c.y.b); }

// One transposed element of the pair: 16 bytes, or 8 where the pair is one row.
__device__ __forceinline__ void put_rows(float2* p, C2 c, bool two) {
  if (two) *reinterpret_cast<float4*>(p) = pack_rows(c);
  else *p = make_float2(c.x.a, c.y.a);
}
__device__ __forceinline__ C2 get_rows(const float2* p, bool two) {
  if (two) return unpack_rows(*reinterpret_cast<const float4*>(p));
  const float2 v = *p;
  return mkpair(v, v);
}

template <int L, bool R2C, bool LOC = false>
__global__ void __launch_bounds__(RowPairThreads<L>::value, RowEPT<L>::value >= 20 ? 3 : 2)
k_fwd_P(LineIO io, const float4* __restrict__ tw, int64_t in_sa0, int64_t in_sb, int64_t out_sa0, int64_t out_sk,
        int log_tb, const int64_t* __restrict__ in_off) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pass_begin();
  constexpr int EPT = RowEPT<L>::value;
  typedef FFTPlan<L, EPT> P;
  constexpr int T = P::kT;
  constexpr int NK = R2C ? L + 1 : L;
  C2* smem = reinterpret_cast<C2*>(smem_raw);
  const int t = threadIdx.x, g = threadIdx.y;
  const bool two = log_tb > 0;
  const int log_tbp = two ? log_tb - 1 : 0;
  const int a0 = blockIdx.y, a1 = blockIdx.z;
  const int64_t b0 = (int64_t)blockIdx.x << log_tb;
  const int64_t b = b0 + 2 * g;  // the pair's rows b, b + 1
  const int64_t o0 = LOC ? 0 : in_off ? in_off[a0] : a0 * in_sa0;  // per-patch offsets of a batch
  if (io.in_ext) {  // checked mode: the rows read and the transposed block written
    int64_t in_end = o0 + (b + (two ? 1 : 0)) * in_sb + (R2C ? 2 * L : L);
    if constexpr (LOC)
      in_end = (int64_t)(max(LocalRow(io.loc, a0, (int)b).y, LocalRow(io.loc, a0, (int)b + (two ? 1 : 0)).y) + 1) * io.loc.nx;
    const int64_t out_end = a0 * out_sa0 + b0 + (1 << log_tb) + (int64_t)(NK - 1) * out_sk;
    if (cta_out_of_bounds(in_end > io.in_ext || out_end > io.out_ext || o0 < 0, io.chk_err)) return;
  }
  C2 v[EPT];
  if constexpr (LOC) {
    const LocalRow l0(io.loc, a0, (int)b), l1(io.loc, a0, (int)b + (two ? 1 : 0));
    const float* p = static_cast<const float*>(io.in[a1]);
    const float *r0 = p + (int64_t)l0.y * io.loc.nx, *r1 = p + (int64_t)l1.y * io.loc.nx;
#pragma unroll
    for (int m = 0; m < EPT; ++m)
      v[m] = mkpair(local_load(r0, io.loc, l0.x0, 2 * (t + T * m)), local_load(r1, io.loc, l0.x0, 2 * (t + T * m)));
  } else {
    const float2 *r0, *r1;
    if constexpr (R2C) {
      const float* p = static_cast<const float*>(io.in[a1]) + o0 + b * in_sb;
      r0 = reinterpret_cast<const float2*>(p);
      r1 = reinterpret_cast<const float2*>(p + (two ? in_sb : 0));
    } else {
      r0 = static_cast<const float2*>(io.in[a1]) + o0 + b * in_sb;
      r1 = r0 + (two ? in_sb : 0);
    }
#pragma unroll
    for (int m = 0; m < EPT; ++m) v[m] = mkpair(r0[t + T * m], r1[t + T * m]);
  }
  const int bar = 1 + g;
  C2* line = smem + g * L;
  line_fft_fwd<F2, L, EPT, false>(v, line, tw, t, line_gx<P>(g), bar);

  // this pair's spectrum to its line, then every thread takes whole (k, pair) elements
  if constexpr (P::kStages > 1) line_sync<T>(bar);  // the last exchange's reads are done
  const int xg = pair_xor(g, log_tbp, L);
#pragma unroll
  for (int m = 0; m < EPT; ++m) line[(t + T * m) ^ xg] = v[m];
  __syncthreads();
  const int tid = g * T + t;
  const int gg = tid & ((1 << log_tbp) - 1);
  const int k0 = tid >> log_tbp;  // in [0, T)
  const int xgg = pair_xor(gg, log_tbp, L);
  const C2* zr = smem + gg * L;
  float2* o = static_cast<float2*>(io.out[a1]) + a0 * out_sa0 + b0 + 2 * gg;
  if constexpr (R2C) {
    // X[k] = Fe + W Fo, X[L-k] = conj(Fe - W Fo), Fe = (Z[k] + Z*[L-k])/2,
    // Fo = (Z[k] - Z*[L-k])/(2i), W = W_2L^k; bins k = k0 + j T < L/2 with L - k, and
    // thread k0 = 0 also L/2
    const float4* wn = tw + P::kTwEntries;
    auto split = [&](C2 zk, C2 zm, float4 w, C2& fe, C2& wo) {
      fe = C2{0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y)};
      const C2 fo = C2{0.5f * (zk.y + zm.y), 0.5f * (zm.x - zk.x)};
      wo = twmul(fo, w);
    };
    constexpr int NP = EPT / 2;
    constexpr int GP = NP % 4 == 0 ? 4 : 2;
#pragma unroll
    for (int j0 = 0; j0 < NP; j0 += GP) {
      float4 w[GP];
#pragma unroll
      for (int j = 0; j < GP; ++j) w[j] = __ldg(&wn[k0 + (j0 + j) * T]);
#pragma unroll
      for (int j = 0; j < GP; ++j) {
        const int k = k0 + (j0 + j) * T;
        const C2 zk = zr[k ^ xgg];
        const C2 zm = zr[(k == 0 ? 0 : L - k) ^ xgg];
        C2 fe, wo;
        split(zk, zm, w[j], fe, wo);
        put_rows(o + (int64_t)k * out_sk, cadd(fe, wo), two);
        put_rows(o + (int64_t)(L - k) * out_sk, C2{fe.x - wo.x, wo.y - fe.y}, two);
      }
    }
    if (k0 == 0) {
      const C2 z = zr[(L / 2) ^ xgg];
      C2 fe, wo;
      split(z, z, __ldg(&wn[L / 2]), fe, wo);
      put_rows(o + (int64_t)(L / 2) * out_sk, cadd(fe, wo), two);
    }
  } else {
#pragma unroll
    for (int j = 0; j < EPT; ++j) {
      const int k = k0 + j * T;
      put_rows(o + (int64_t)k * out_sk, zr[k ^ xgg], two);
    }
  }
}

template <int L, bool C2R, bool LOC = false>
__global__ void __launch_bounds__(RowPairThreads<L>::value, RowEPT<L>::value >= 20 ? 3 : 2)
k_inv_P(LineIO io, const float4* __restrict__ tw, int64_t in_sa0, int64_t in_sk, int64_t out_sa0, int64_t out_sb,
        int log_tb, const int64_t* __restrict__ out_off) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pass_begin();
  constexpr int EPT = RowEPT<L>::value;
  typedef FFTPlan<L, EPT> P;
  constexpr int T = P::kT;
  constexpr int NK = C2R ? L + 1 : L;
  C2* smem = reinterpret_cast<C2*>(smem_raw);
  const int t = threadIdx.x, g = threadIdx.y;
  const bool two = log_tb > 0;
  const int log_tbp = two ? log_tb - 1 : 0;
  const int a0 = blockIdx.y, a1 = blockIdx.z;
  const int64_t b0 = (int64_t)blockIdx.x << log_tb;
  const int64_t b = b0 + 2 * g;
  const int64_t o0 = LOC ? 0 : out_off ? out_off[a0] : a0 * out_sa0;
  if (io.in_ext) {  // checked mode: the transposed block read and the rows written
    const int64_t in_end = a0 * in_sa0 + b0 + (1 << log_tb) + (int64_t)(NK - 1) * in_sk;
    int64_t out_end = o0 + (b + (two ? 1 : 0)) * out_sb + (C2R ? 2 * L : L);
    if constexpr (LOC) {
      const int64_t e0 = local_out(io.loc, a0, (int)b), e1 = local_out(io.loc, a0, (int)b + (two ? 1 : 0));
      out_end = e0 > e1 ? e0 : e1;
      out_end = out_end < 0 ? 0 : out_end + io.loc.ix;
    }
    if (cta_out_of_bounds(in_end > io.in_ext || out_end > io.out_ext || o0 < 0, io.chk_err)) return;
  }
  const int tid = g * T + t;
  const int gg = tid & ((1 << log_tbp) - 1);
  const int k0 = tid >> log_tbp;  // in [0, T)
  const int xgg = pair_xor(gg, log_tbp, L);
  C2* zr = smem + gg * L;
  const float2* ib = static_cast<const float2*>(io.in[a1]) + a0 * in_sa0 + b0 + 2 * gg;
  if constexpr (C2R) {
    // Z[k] = Fe + i Fo, Z[L-k] = Fe* + i Fo*, Fe = X[k] + X*[L-k], Fo = (X[k] - X*[L-k]) W_2L^-k:
    // bins k = k0 + j T < L/2 with L - k, and thread k0 = 0 also L/2
    const float4* wn = tw + P::kTwEntries;
    constexpr int NP = EPT / 2;
    constexpr int GP = NP % 4 == 0 ? 4 : 2;
#pragma unroll
    for (int j0 = 0; j0 < NP; j0 += GP) {
      C2 xk[GP], xm[GP];
      float4 w[GP];
#pragma unroll
      for (int j = 0; j < GP; ++j) {
        const int k = k0 + (j0 + j) * T;
        xk[j] = get_rows(ib + (int64_t)k * in_sk, two);
        xm[j] = get_rows(ib + (int64_t)(L - k) * in_sk, two);
        w[j] = __ldg(&wn[k]);
      }
#pragma unroll
      for (int j = 0; j < GP; ++j) {
        const int k = k0 + (j0 + j) * T;
        const C2 fe = C2{xk[j].x + xm[j].x, xk[j].y - xm[j].y};
        const C2 d = C2{xk[j].x - xm[j].x, xk[j].y + xm[j].y};
        const C2 fo = (k == 0) ? d : twmul_conj(d, w[j]);
        zr[k ^ xgg] = add_i(fe, fo);
        if (k > 0) zr[(L - k) ^ xgg] = C2{fe.x + fo.y, fo.x - fe.y};
      }
    }
    if (k0 == 0) {  // k = L/2: X[L/2] pairs with itself
      const C2 x = get_rows(ib + (int64_t)(L / 2) * in_sk, two);
      const C2 fe = C2{x.x + x.x, x.y - x.y};
      const C2 d = C2{x.x - x.x, x.y + x.y};
      zr[(L / 2) ^ xgg] = add_i(fe, twmul_conj(d, __ldg(&wn[L / 2])));
    }
  } else {
    C2 xv[EPT];
#pragma unroll
    for (int j = 0; j < EPT; ++j) xv[j] = get_rows(ib + (int64_t)(k0 + j * T) * in_sk, two);
#pragma unroll
    for (int j = 0; j < EPT; ++j) zr[(k0 + j * T) ^ xgg] = xv[j];
  }
  __syncthreads();
  const int bar = 1 + g;
  C2* line = smem + g * L;
  const int xg = pair_xor(g, log_tbp, L);
  C2 v[EPT];
#pragma unroll
  for (int m = 0; m < EPT; ++m) v[m] = line[(t + T * m) ^ xg];
  if constexpr (P::kStages > 1) line_sync<T>(bar);  // read by the whole line before the exchanges overwrite it
  line_fft_inv<F2, L, EPT, false>(v, line, tw, t, line_gx<P>(g), bar);
  if constexpr (LOC) {
    const int64_t e0 = local_out(io.loc, a0, (int)b), e1 = two ? local_out(io.loc, a0, (int)b + 1) : -1;
    float* p = static_cast<float*>(io.out[a1]) - io.loc.g;
    if (e0 >= 0) {
#pragma unroll
      for (int m = 0; m < EPT; ++m) local_store(p + e0, io.loc, 2 * (t + T * m), make_float2(v[m].x.a, v[m].y.a));
    }
    if (e1 >= 0) {
#pragma unroll
      for (int m = 0; m < EPT; ++m) local_store(p + e1, io.loc, 2 * (t + T * m), make_float2(v[m].x.b, v[m].y.b));
    }
    return;
  }
  float2 *r0, *r1;
  if constexpr (C2R) {
    float* p = static_cast<float*>(io.out[a1]) + o0 + b * out_sb;
    r0 = reinterpret_cast<float2*>(p);
    r1 = reinterpret_cast<float2*>(p + (two ? out_sb : 0));
  } else {
    r0 = static_cast<float2*>(io.out[a1]) + o0 + b * out_sb;
    r1 = r0 + (two ? out_sb : 0);
  }
#pragma unroll
  for (int m = 0; m < EPT; ++m) r0[t + T * m] = make_float2(v[m].x.a, v[m].y.a);
  if (two) {
#pragma unroll
    for (int m = 0; m < EPT; ++m) r1[t + T * m] = make_float2(v[m].x.b, v[m].y.b);
  }
}

}  // namespace psatd
