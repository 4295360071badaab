// Matrix-free element kernel of the SEM / SEM-NI operator (Algorithm 1's
// vectorized cell loop, Section 4) with sum factorization (Section 4.1):
//
//   y += sum_e  P_e^T (mass_coef M_e + K_e) P_e u          (P_e: gather through the map)
//
// per element, with n = p + 1 points per direction:
//   SEM-NI (LGL quadrature on the nodes):
//     g_d   = D along direction d of u_e                    3 sweeps
//     q     = G g,  m = mass_coef W u                       per quadrature point
//     y_e   = m + sum_d D^T along d of q_d                  3 sweeps
//   SEM (LG quadrature):
//     u_q   = Bi (x) Bi (x) Bi u_e                          3 sweeps to the Gauss points
//     g_d   = Dg along d of u_q  (collocation derivative on the Gauss points)
//     q, m  as above at the Gauss points
//     y_e   = Bi^T (x) Bi^T (x) Bi^T (m + sum_d Dg^T along d of q_d)
//
// GPU mapping: one CTA holds E elements in shared memory (three n^3 tiles per
// element).  A sweep along x or y gives each thread one 1-D line of n values
// (n^2 FMAs on registers, matrix entries read from the kernel-parameter bank);
// the z-sweep, the quadrature-point stage and the transposed z-sweep run on
// the (i, j) columns in registers.  The result is scatter-added with
// atomicAdd (RED) through the element-to-DOF map.
#pragma once

#include <algorithm>
#include <type_traits>

#include "sem_internal.cuh"

namespace sem {

constexpr int kApplyThreads = 256;

// Elements per CTA: E * n^2 close to the 256 threads of the CTA.
template <int P> struct ApplyCfg;
template <> struct ApplyCfg<1> { static constexpr int E = 64; };
template <> struct ApplyCfg<2> { static constexpr int E = 28; };
template <> struct ApplyCfg<3> { static constexpr int E = 16; };
template <> struct ApplyCfg<4> { static constexpr int E = 10; };
template <> struct ApplyCfg<5> { static constexpr int E = 7; };
template <> struct ApplyCfg<6> { static constexpr int E = 5; };

// Threads and elements of a CTA of the plain and the fused-inner-product apply.  Up
// to p = 4 a CTA of 128 threads is the faster one (more CTAs of an SM are in different
// phases between barriers): double-float, SEM-NI, 2 M nodes, 256 / 128 threads:
// p = 1 330 / 265, p = 2 144 / 129, p = 3 124 / 100, p = 4 88 / 85 us; FP64 p = 2
// 344 / 334, p = 4 292 / 291.  At p = 5, 6 128 threads hold 3 and 2 elements (84, 77 %
// of the lines): 97 and 102 us against 96 and 95.  The FP64 apply with the inner
// product keeps 256: sem_apply_dot_static's scratch holds one partial a CTA.
template <int P, typename T, bool DOT>
struct ApplyCta {
  static constexpr bool kNarrow = P <= 4 && !(std::is_same<T, double>::value && DOT);
  static constexpr int kThreads = kNarrow ? kApplyThreads / 2 : kApplyThreads;
  static constexpr int E = kNarrow ? ApplyCfg<P>::E / 2 : ApplyCfg<P>::E;
  static constexpr size_t smem = ((size_t)3 * E * (P + 1) * (P + 1) * (P + 1) * sizeof(T) + 15) / 16 * 16;
};

__device__ __forceinline__ double ldmetric(const double* p) { return __ldg(p); }
__device__ __forceinline__ float ldmetric(const float* p) { return __ldg(p); }
__device__ __forceinline__ float ldmetric(const __nv_bfloat16* p) {
  return __bfloat162float(__ldg(p));
}
__device__ __forceinline__ df ldmetric(const df_pair* p) {
  const float2 v = __ldg(reinterpret_cast<const float2*>(p));
  return df(v.x, v.y);
}

// Scatter-add of one element result; exact-match overloads so that no value is
// converted between precisions.
__device__ __forceinline__ void scatter_add(double* p, double v) { atomicAdd(p, v); }
__device__ __forceinline__ void scatter_add(float* p, float v) { atomicAdd(p, v); }
// the pair's halves widened by integer operations: one FP64 instruction per node
// instead of three (measured 0.2 % on the mixed step)
__device__ __forceinline__ void scatter_add(double* p, df v) { atomicAdd(p, df_to_double(v)); }
// Element-local store of one element result (deterministic mode).
__device__ __forceinline__ void store_loc(double* p, double v) { *p = v; }
__device__ __forceinline__ void store_loc(float* p, float v) { *p = v; }
__device__ __forceinline__ void store_loc(double* p, df v) { *p = (double)v; }

// The factor on an element result: none, out_scale, or a sign (no FP64 multiplication).
__device__ __forceinline__ df negated(df v) { return df(-v.h, -v.l); }
__device__ __forceinline__ double negated(double v) { return -v; }
__device__ __forceinline__ float negated(float v) { return -v; }
template <typename T, typename MT>
__device__ __forceinline__ T scale_result(const ApplyArgs<T, MT>& a, T v) {
  if (a.scale_out) v = a.scale_out == kNegateOut ? negated(v) : v * a.out_scale;
  return v;
}

// Base offset and stride of line l of an n^3 tile along direction DIR
// (0: x-line (j,k), l = j + n k; 1: y-line (i,k), l = i + n k; 2: z-line (i,j), l = i + n j).
template <int N, int DIR>
__device__ __forceinline__ void line_geom(int l, int& base, int& stride) {
  if (DIR == 0) { base = l * N; stride = 1; }
  else if (DIR == 1) { const int i = l % N, k = l / N; base = k * N * N + i; stride = N; }
  else { base = l; stride = N * N; }
}

// out = M in (ACC: out += M in) for M in even-odd form (EoMat), ANTI for
// s = -1.  With e_l = in_l + in_{n-1-l}, o_l = in_l - in_{n-1-l} (l < H):
//   se_q = sum_l a[q][l] e_l (+ a[q][H] in_H),  so_q = sum_l b[q][l] o_l,
//   out_q = se_q + so_q,  out_{n-1-q} = (ANTI ? so_q - se_q : se_q - so_q)   (q < H),
//   odd n: out_H = ANTI ? sum_l c[l] o_l : sum_l c[l] e_l + c[H] in_H.
// At n = 5 that is 12 multiply-adds and 8 additions instead of 25 multiply-adds.
template <int N, bool ANTI, bool ACC, typename T>
__device__ __forceinline__ void eo_line(const EoMat<N, T>& M, const T (&in)[N], T (&out)[N]) {
  if constexpr (N == 2 && ANTI) {
    // derivative of a linear function: both rows of D are (-d, d) (a = 0), and both
    // columns of D^T; D is only applied without ACC and D^T with it
    if constexpr (!ACC) {
      out[0] = out[1] = M.b[0][0] * (in[0] - in[1]);
    } else {
      const T y = M.a[0][0] * (in[0] + in[1]);
      out[0] = out[0] + y;
      out[1] = out[1] - y;
    }
    return;
  } else if constexpr (EoMat<N, T>::kDirect) {  // out_q (+)= sum_l m[q][l] in_l
#pragma unroll
    for (int q = 0; q < N; ++q) {
      T acc = ACC ? fma(M.m[q][0], in[0], out[q]) : M.m[q][0] * in[0];
#pragma unroll
      for (int l = 1; l < N; ++l) acc = fma(M.m[q][l], in[l], acc);
      out[q] = acc;
    }
    return;
  }
  constexpr int H = N / 2;
  constexpr bool ODD = (N & 1) != 0;
  T e[H], o[H];
#pragma unroll
  for (int l = 0; l < H; ++l) {
    e[l] = in[l] + in[N - 1 - l];
    o[l] = in[l] - in[N - 1 - l];
  }
#pragma unroll
  for (int q = 0; q < H; ++q) {
    T se = M.a[q][0] * e[0];
#pragma unroll
    for (int l = 1; l < H; ++l) se = fma(M.a[q][l], e[l], se);
    if (ODD) se = fma(M.a[q][H], in[H], se);
    T so = M.b[q][0] * o[0];
#pragma unroll
    for (int l = 1; l < H; ++l) so = fma(M.b[q][l], o[l], so);
    const T y0 = se + so;
    const T y1 = ANTI ? so - se : se - so;
    if (ACC) {
      out[q] = out[q] + y0;
      out[N - 1 - q] = out[N - 1 - q] + y1;
    } else {
      out[q] = y0;
      out[N - 1 - q] = y1;
    }
  }
  if (ODD) {
    T ym;
    if (ANTI) {
      ym = M.c[0] * o[0];
#pragma unroll
      for (int l = 1; l < H; ++l) ym = fma(M.c[l], o[l], ym);
    } else {
      ym = M.c[0] * e[0];
#pragma unroll
      for (int l = 1; l < H; ++l) ym = fma(M.c[l], e[l], ym);
      ym = fma(M.c[H], in[H], ym);
    }
    out[H] = ACC ? out[H] + ym : ym;
  }
}

// dst = M along DIR of src (ACC: dst += ...), for every line of ne element tiles
// (thread tid of a group of nth threads).  src may equal dst.
template <int N, int DIR, bool ANTI, bool ACC, typename T>
__device__ __forceinline__ void sweep(const EoMat<N, T>& M, const T* src, T* dst, int ne, int tid, int nth) {
  constexpr int N2 = N * N, N3 = N2 * N;
  for (int w = tid; w < ne * N2; w += nth) {
    const int s = w / N2, l = w - s * N2;
    int base, stride;
    line_geom<N, DIR>(l, base, stride);
    const T* ps = src + s * N3 + base;
    T* pd = dst + s * N3 + base;
    T in[N], out[N];
#pragma unroll
    for (int t = 0; t < N; ++t) in[t] = ps[t * stride];
    if (ACC) {
#pragma unroll
      for (int t = 0; t < N; ++t) out[t] = pd[t * stride];
    }
    eo_line<N, ANTI, ACC>(M, in, out);
#pragma unroll
    for (int t = 0; t < N; ++t) pd[t * stride] = out[t];
  }
}

// The same along a direction known at run time (one copy of the code for several
// directions).
template <int N, bool ANTI, bool ACC, typename T>
__device__ __forceinline__ void sweep_dir(const EoMat<N, T>& M, const T* src, T* dst, int dir, int ne, int tid, int nth) {
  constexpr int N2 = N * N, N3 = N2 * N;
  const int stride = dir == 0 ? 1 : dir == 1 ? N : N2;
  for (int w = tid; w < ne * N2; w += nth) {
    const int s = w / N2, l = w - s * N2;
    const int base = s * N3 + (dir == 0 ? l * N : dir == 1 ? (l / N) * N2 + l % N : l);
    T in[N], out[N];
#pragma unroll
    for (int t = 0; t < N; ++t) in[t] = src[base + t * stride];
    if (ACC) {
#pragma unroll
      for (int t = 0; t < N; ++t) out[t] = dst[base + t * stride];
    }
    eo_line<N, ANTI, ACC>(M, in, out);
#pragma unroll
    for (int t = 0; t < N; ++t) dst[base + t * stride] = out[t];
  }
}

// Block-wide sum of v (all threads must call); result valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) red[warp] = v;
  __syncthreads();
  v = 0.0;
  if (warp == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    v = (lane < nw) ? red[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  }
  return v;
}

// Writes this block's partial; the last block to arrive sums all partials in
// block order (deterministic) and returns true in its thread 0 with *total set.
__device__ __forceinline__ bool finish_reduction(double partial, double* partials,
                                                 unsigned int* ticket, double* total,
                                                 double* red) {
  __shared__ bool is_last;
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = partial;
    __threadfence();
    const unsigned int t = atomicAdd(ticket, 1u);
    is_last = (t == gridDim.x - 1);
  }
  __syncthreads();
  if (!is_last) return false;
  __threadfence();
  double v = 0.0;
  // fixed assignment of partials to threads, then a fixed-shape tree
  for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x)
    v += ((volatile double*)partials)[b];
  v = block_sum(v, red);
  if (threadIdx.x == 0) {
    *total = v;
    *ticket = 0u;
  }
  return threadIdx.x == 0;
}

// Shared-memory bytes of one CTA: three n^3 tiles per element.
template <int P, typename T>
__host__ __device__ constexpr size_t apply_tile_bytes() {
  return ((size_t)3 * ApplyCfg<P>::E * (P + 1) * (P + 1) * (P + 1) * sizeof(T) + 15) / 16 * 16;
}

// Warp-per-element mode (WARP): each warp of the CTA owns one element and
// synchronises with __syncwarp only, so the warps of an SM run their gather,
// sweep, metric and scatter phases independently.  Used for the FP32 mass operator up
// to p = 4, which is bound by memory latency rather than by arithmetic.
constexpr int kWarpsPerCta = kApplyThreads / 32;

// Elements per warp in warp mode: G n^2 lines close to 32 lanes (p <= 4).
template <int P> struct WarpCfg { static constexpr int G = 1; };
template <> struct WarpCfg<1> { static constexpr int G = 8; };
template <> struct WarpCfg<2> { static constexpr int G = 3; };
template <> struct WarpCfg<3> { static constexpr int G = 2; };

template <int P, typename T>
__host__ __device__ constexpr size_t apply_warp_tile_bytes() {
  return (size_t)3 * kWarpsPerCta * WarpCfg<P>::G * (P + 1) * (P + 1) * (P + 1) * sizeof(T);
}

// The element results (mass M_e + K_e) u_e (MASS_ONLY: mass M_e u_e) of ne element
// tiles, from the gathered values in sA into sA; sB, sC scratch of the same size.  The
// FP32 mass operator's metric is W alone, [element][padded n^3] (weight_lowp_count).  Tile
// s is element e0 + s, and those from e_end on have no metric (their values are zero).
template <int P, int QUAD, bool MASS_ONLY, bool ROLLED, bool WARP, typename T, typename MT>
__device__ __forceinline__ void element_results(const KTab<P + 1, T>& tab, const MT* metric, T mass, int e0, int e_end,
                                                int ne, T* sA, T* sB, T* sC, int tid, int nth) {
  constexpr int N = P + 1, N2 = N * N, N3 = N2 * N;
  using ML = MetricLayout<MT>;
  auto group_sync = [] {
    if (WARP) __syncwarp(); else __syncthreads();
  };
  if (QUAD == SEM_QUAD_LG) {  // values at the Gauss points
    if constexpr (ROLLED) {
#pragma unroll 1
      for (int d = 0; d < 3; ++d) {
        sweep_dir<N, false, false>(tab.Bi, sA, sA, d, ne, tid, nth);
        group_sync();
      }
    } else {
      sweep<N, 0, false, false>(tab.Bi, sA, sB, ne, tid, nth);
      group_sync();
      sweep<N, 1, false, false>(tab.Bi, sB, sC, ne, tid, nth);
      group_sync();
      sweep<N, 2, false, false>(tab.Bi, sC, sA, ne, tid, nth);
      group_sync();
    }
  }

  if (MASS_ONLY) {
    for (int idx = tid; idx < ne * N3; idx += nth) {
      const int s = idx / N3, loc = idx - s * N3, e = e0 + s;
      if (e < e_end) {
        const T W = ldmetric(metric + (std::is_same<T, float>::value ? (size_t)e * padded_n3(N) + loc
                                                                     : ML::offset(N, e, loc % N2, loc / N2, 6)));
        sA[idx] = (mass * W) * sA[idx];
      }
    }
    group_sync();
  } else {
    // reference gradient along x and y (into sB, sC)
    if constexpr (ROLLED) {
#pragma unroll 1
      for (int d = 0; d < 2; ++d) sweep_dir<N, true, false>(tab.D, sA, d == 0 ? sB : sC, d, ne, tid, nth);
    } else {
      sweep<N, 0, true, false>(tab.D, sA, sB, ne, tid, nth);
      sweep<N, 1, true, false>(tab.D, sA, sC, ne, tid, nth);
    }
    group_sync();
    // z-gradient, quadrature-point stage and transposed z-sweep on the columns
    for (int w = tid; w < ne * N2; w += nth) {
      const int s = w / N2, c = w - s * N2, e = e0 + s;
      if (e >= e_end) continue;
      T* pa = sA + s * N3 + c;
      T* pb = sB + s * N3 + c;
      T* pc = sC + s * N3 + c;
      T uz[N], g3[N], q3[N], m[N];
#pragma unroll
      for (int k = 0; k < N; ++k) uz[k] = pa[k * N2];
      eo_line<N, true, false>(tab.D, uz, g3);
      const MT* mp = metric + ML::offset(N, e, c, 0, 0);  // component-major, point by point
#pragma unroll
      for (int k = 0; k < N; ++k) {
        const T g1 = pb[k * N2], g2 = pc[k * N2];
        T gm[kMetricComps];
#pragma unroll
        for (int cc = 0; cc < kMetricComps; ++cc) gm[cc] = ldmetric(mp + k * N2 + cc * padded_n3(N));
        const T G00 = gm[0], G01 = gm[1], G02 = gm[2], G11 = gm[3], G12 = gm[4], G22 = gm[5], W = gm[6];
        pb[k * N2] = fma(G02, g3[k], fma(G01, g2, G00 * g1));
        pc[k * N2] = fma(G12, g3[k], fma(G11, g2, G01 * g1));
        q3[k] = fma(G22, g3[k], fma(G12, g2, G02 * g1));
        m[k] = (mass * W) * uz[k];
      }
      eo_line<N, true, true>(tab.Dt, q3, m);
#pragma unroll
      for (int k = 0; k < N; ++k) pa[k * N2] = m[k];
    }
    group_sync();
    if constexpr (ROLLED) {
#pragma unroll 1
      for (int d = 1; d >= 0; --d) {
        sweep_dir<N, true, true>(tab.Dt, d == 0 ? sB : sC, sA, d, ne, tid, nth);
        group_sync();
      }
    } else {
      sweep<N, 1, true, true>(tab.Dt, sC, sA, ne, tid, nth);
      group_sync();
      sweep<N, 0, true, true>(tab.Dt, sB, sA, ne, tid, nth);
      group_sync();
    }
  }

  if (QUAD == SEM_QUAD_LG) {  // back from the Gauss points to the nodes
    if constexpr (ROLLED) {
#pragma unroll 1
      for (int d = 0; d < 3; ++d) {
        sweep_dir<N, false, false>(tab.Bit, sA, sA, d, ne, tid, nth);
        group_sync();
      }
    } else {
      sweep<N, 0, false, false>(tab.Bit, sA, sB, ne, tid, nth);
      group_sync();
      sweep<N, 1, false, false>(tab.Bit, sB, sC, ne, tid, nth);
      group_sync();
      sweep<N, 2, false, false>(tab.Bit, sC, sA, ne, tid, nth);
      group_sync();
    }
  }
}

// The double-float kernel at p = 4 (the outer operator of the benchmark's mixed
// step) is bound by issue and memory latency: 10 CTAs per SM at 48 registers, without
// spills (8 measure the same in the plain apply, 1 % slower with the inner product; at
// p = 3, 5, 6, which take 90 to 124 registers, it would spill).
template <int P, int QUAD, typename T, typename MT, bool DOT, bool MASS_ONLY, bool WARP = false>
__global__ void __launch_bounds__(MASS_ONLY ? kApplyThreads : ApplyCta<P, T, DOT>::kThreads,
                                  (std::is_same<T, df>::value && !MASS_ONLY && P == 4)
                                      ? 5 * kApplyThreads / ApplyCta<P, T, DOT>::kThreads : 1)
    sem_apply_kernel(const ApplyArgs<T, MT> a, const __grid_constant__ KTab<P + 1, T> tab) {
  static_assert(!(WARP && DOT), "the fused inner product needs the CTA-wide mode");
  constexpr int N = P + 1, N3 = N * N * N;
  using ML = MetricLayout<MT>;
  constexpr int E = WARP ? WarpCfg<P>::G : MASS_ONLY ? ApplyCfg<P>::E : ApplyCta<P, T, DOT>::E;
  // One copy of the sweep code for the directions: double-float at p = 4 (85 -> 80 us,
  // SEM 120 -> 112) and FP64 at p = 1 (668 -> 644, SEM 1023 -> 975) gain by the shorter
  // code; at p = 6 the run-time strides cost more (95 -> 130 us).
  constexpr bool kRolled = (std::is_same<T, df>::value && P == 4) || (std::is_same<T, double>::value && P == 1 && !MASS_ONLY);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5;
  const int tid = WARP ? (threadIdx.x & 31) : threadIdx.x;
  const int nth = WARP ? 32 : blockDim.x;
  T* sA = reinterpret_cast<T*>(smem_raw) + (WARP ? warp * 3 * E * N3 : 0);
  T* sB = sA + E * N3;
  T* sC = sB + E * N3;
  __shared__ double red[32];
  auto group_sync = [] {
    if (WARP) __syncwarp(); else __syncthreads();
  };

  const int e0 = WARP ? (blockIdx.x * kWarpsPerCta + warp) * E : blockIdx.x * E;
  if (WARP && e0 >= a.nelem) return;  // no CTA-wide barrier follows in this mode
  // while the previous kernel drains: the group's map entries into L2
  prefetch_l2_lines(a.map + (size_t)e0 * N3, (size_t)min(E, a.nelem - e0) * N3 * sizeof(int), tid, nth);
  pdl_wait();
  if (a.done != nullptr && *a.done) return;

  if (std::is_same<T, df>::value && !MASS_ONLY) {
    // Bulk prefetch of the group's metric block (contiguous, 16-byte aligned, a
    // multiple of 16 bytes) into L2, in 16 KB pieces: the quadrature-point stage
    // reads it after the gather and two sweeps, and then hits L2.  Measured
    // faster for the memory-latency-bound double-float kernel only (the FP64
    // kernel is bound by the FP64 pipe).
    const int ne = min(E, a.nelem - e0);
    const unsigned bytes = (unsigned)(ML::offset(N, ne, 0, 0, 0) * sizeof(MT));
    const char* src = reinterpret_cast<const char*>(a.metric + ML::offset(N, e0, 0, 0, 0));
    for (unsigned off = (unsigned)tid * 16384u; off < bytes; off += (unsigned)nth * 16384u)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(src + off),
                   "r"(min(16384u, bytes - off))
                   : "memory");
  }

  // Gather and scatter loops.  The threads of a CTA are fixed (256 or 128 by
  // ApplyCta, 256 for the mass alone; a warp per element group in warp mode), so the
  // loops of the plain apply have compile-time trip counts: they unroll and keep the
  // loads of all their iterations in flight at once.  The apply with the fused
  // inner product keeps the rolled loops (both measured faster that way).
  constexpr int NTH = WARP ? 32 : MASS_ONLY ? kApplyThreads : ApplyCta<P, T, DOT>::kThreads;
  constexpr int IT = (E * N3 + NTH - 1) / NTH;

  // gather u_e = P_e u
  if constexpr (DOT) {
    // the double-float operator with the fused inner product gathers u as the
    // float pairs the CG kernel that formed u wrote (a.u2), converting nothing
    for (int idx = tid; idx < E * N3; idx += nth) {
      const int s = idx / N3, loc = idx - s * N3, e = e0 + s;
      if (e < a.nelem) {
        const int gi = (int)SEM_IDX(__ldg(a.map + (size_t)e * N3 + loc), a.ndofs, a.dbg, kDbgGather);
        if constexpr (std::is_same<T, df>::value) {
          const float2 v = __ldg(reinterpret_cast<const float2*>(a.u2) + gi);
          sA[idx] = df(v.x, v.y);
        } else {
          sA[idx] = T(a.u[gi]);
        }
      } else {
        sA[idx] = T(0);
      }
    }
  } else {
    const int nv = min(E, a.nelem - e0) * N3;  // nodal values of the group's elements
    const int* gmap = a.map + (size_t)e0 * N3;
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const int idx = tid + it * NTH;
      if (IT * NTH == E * N3 || idx < E * N3)
        sA[idx] = idx < nv ? T(a.u[SEM_IDX(__ldg(gmap + idx), a.ndofs, a.dbg, kDbgGather)]) : T(0);
    }
  }
  group_sync();

  element_results<P, QUAD, MASS_ONLY, kRolled, WARP>(tab, a.metric, a.mass_coef, e0, a.nelem, E, sA, sB, sC, tid, nth);

  pdl_trigger();
  // scatter-add y += P_e^T y_e, and with DOT the partial u_e . y_e
  double dot = 0.0;
  if constexpr (DOT) {
    if constexpr (std::is_same<T, df>::value) {
      // the partial u_e . y_e in double-float arithmetic from the float pairs of u
      // (in L1 since the gather)
      df dd(0);
      for (int idx = tid; idx < E * N3; idx += nth) {
        const int s = idx / N3, loc = idx - s * N3, e = e0 + s;
        if (e < a.nelem) {
          const int g = (int)SEM_IDX(__ldg(a.map + (size_t)e * N3 + loc), a.ndofs, a.dbg, kDbgScatter);
          T v = sA[idx];
          v = scale_result(a, v);
          if (a.yloc != nullptr) store_loc(a.yloc + (size_t)e * N3 + loc, v);
          else scatter_add(a.y + g, v);
          const float2 uu = __ldg(reinterpret_cast<const float2*>(a.u2) + g);
          dd = fma(df(uu.x, uu.y), v, dd);
        }
      }
      dot = (double)dd;
    } else {
      for (int idx = tid; idx < E * N3; idx += nth) {
        const int s = idx / N3, loc = idx - s * N3, e = e0 + s;
        if (e < a.nelem) {
          const int g = (int)SEM_IDX(__ldg(a.map + (size_t)e * N3 + loc), a.ndofs, a.dbg, kDbgScatter);
          T v = sA[idx];
          v = scale_result(a, v);
          if (a.yloc != nullptr) store_loc(a.yloc + (size_t)e * N3 + loc, v);
          else scatter_add(a.y + g, v);
          dot = fma((double)a.u[g], (double)v, dot);
        }
      }
    }
  } else {
    const int nv = min(E, a.nelem - e0) * N3;
    const int* gmap = a.map + (size_t)e0 * N3;
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const int idx = tid + it * NTH;
      if ((IT * NTH == E * N3 || idx < E * N3) && idx < nv) {
        T v = sA[idx];
        v = scale_result(a, v);
        if (a.yloc != nullptr) store_loc(a.yloc + (size_t)e0 * N3 + idx, v);
        else scatter_add(a.y + SEM_IDX(__ldg(gmap + idx), a.ndofs, a.dbg, kDbgScatter), v);
      }
    }
  }
  if (DOT) {  // this CTA's partial; the next kernel sums them
    const double bs = block_sum(dot, red);
    if (threadIdx.x == 0) a.dot_partials[blockIdx.x] = bs;
  }
}

// ---------------------------------------------------------------------------
// Plane kernel of the FP32 operator (stiffness and mass, every p).
//
// Each lane owns one (i, j) plane of n^2 nodes of one element in registers, a
// warp the n planes of each of the G = 32 / n elements of a "unit".  The x- and
// y-sweeps, the quadrature-point stage and their transposes are register
// arithmetic on the plane; only the two z-sweeps exchange data: every lane
// reads the n planes of its element from a shared tile by 16-byte loads (the
// lanes of one element read the same words) and accumulates them with its row
// of D (or of D^T), kept in registers.  At p = 4 a unit of 6 elements takes
// about 1,950 warp instructions, 325 an element.  The kernel with one 1-D line
// of one element per lane that this replaced took 551 and moved every sweep
// through shared memory (123 wavefronts an element, now 99).  Bound: the shared
// memory pipe (two z-sweeps read n planes a lane) and latency, at 12 warps an SM.
// Measured, apply with the clearing of y, SEM-NI, bf16 metric, 2 M nodes, before /
// after: p = 1..6 76 / 55, 41 / 31, 27 / 23, 27 / 21, 33 / 20, 31 / 25 us; 30 M
// nodes, p = 4: 307 / 231 us.  With 16 warps (128 registers) the p = 4 V-cycle on
// 2 M nodes took 387 us against 362 with 12 (168 registers).
//
// Each warp loops over units w, w + W, ... (W warps in the persistent grid)
// with the copies of the next unit in flight:
//   - its nodal values by 4-byte cp.async into the other of two tiles; the lanes
//     (s, i) of a copy read one x-row (j, k) of every element s of the unit, and
//     consecutive elements are neighbours in x, so a copy covers G n consecutive
//     words.  The nodes of an element follow from its first node and the strides of
//     the slab's lattice (the map is that lattice), so no per-node map entry is
//     read; the SEM_DEBUG build reads and checks every entry.  The first nodes are
//     an array of their own: read from the map they cost a 32-byte sector an
//     element, at p = 1 an eighth of the FP32 kernel's traffic (2.0 M DOFs,
//     FP32, SEM-NI: p = 1 84.7 -> 75.4 us, p = 2 44.2 -> 42.6; BF16 metric
//     55.4 -> 52.9 and 31.8 -> 28.8);
//   - its metric in chunks of rows by bulk copies (cp.async.bulk) into a ring of
//     kStages chunks, each issued as soon as the chunk before it in its place has
//     been read (a ring instead of the whole block, which at p = 6 and with the
//     float metric would leave room for 4 to 8 warps an SM).
// The result goes through the tile once more, so that the atomic adds have the
// row pattern of the gather.
template <int P, typename MT>
struct PlaneCfg {
  static constexpr int N = P + 1, N2 = N * N, N3 = N2 * N;
  static constexpr int G = 32 / N;            // elements of a unit
  static constexpr int NL = G * N;            // active lanes
  static constexpr int CH = (N2 + 3) / 4;     // 16-byte chunks of a plane
  // plane stride in words: an odd number of 16-byte chunks, so that the 16-byte
  // accesses of 8 consecutive lanes to their own planes have no bank conflict
  static constexpr int PS = 4 * (CH | 1);
  static constexpr int ES = N * PS;           // element stride of a tile
  static constexpr int TW = G * ES;           // words of a tile
  using ML = MetricLayout<MT>;
  static constexpr int NCH = ML::chunks(N), R = ML::rows(N);  // metric chunks of a unit, rows of a chunk
  static constexpr int kStages = NCH == 1 ? (sizeof(MT) == 2 ? 2 : 1) : (sizeof(MT) == 2 ? 3 : 2);
  static constexpr unsigned chunk_bytes = ML::chunk(N) * sizeof(MT);
  static constexpr size_t tile_offset = (size_t)kStages * chunk_bytes;
  static constexpr size_t bar_offset = tile_offset + 2 * (size_t)TW * sizeof(float);
  static constexpr size_t warp_bytes = bar_offset + 32;
  static constexpr int kWarps = 2;            // warps of a CTA
  static constexpr size_t cta_bytes = kWarps * warp_bytes;
  // warps an SM keeps resident (registers)
  static constexpr int kResident = P == 1 ? 24 : P == 2 ? 20 : P == 3 ? 16 : P <= 5 ? 12 : 8;
  static_assert(chunk_bytes % 16 == 0 && bar_offset % 16 == 0, "stages stay 16-byte aligned");
  static_assert(kStages <= 4, "four mbarriers of 8 bytes");
};

// Matrix rows of the z-sweeps, indexed by the lane's plane: D and D^T of the
// gradient, and for SEM the interpolation B and B^T.
template <int N>
struct ZTab {
  float D[N][N], Dt[N][N], B[N][N], Bt[N][N];
};

// The metric block of a unit reaches shared memory by one bulk copy (the TMA
// engine, cp.async.bulk) that lane 0 issues; 16-byte cp.async copies from every
// lane took four load instructions of the warp and about 11 more L1 tag-stage
// wavefronts per element, in a kernel bound by the L1 pipes and by issue.  The
// warp's stage has an mbarrier of count 1: lane 0 arrives with the expected byte
// count and the copy's completion ends the phase.
// Shared-memory addresses are passed as 32-bit shared-window offsets.
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void bulk_copy(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}
// Waits for the phase of the given parity to complete; false when it has not
// within kMbarTimeoutNs of the global timer (the copy takes microseconds: the
// bound only turns a copy that never completes into an error status).
#ifdef SEM_DEBUG
constexpr unsigned long long kMbarTimeoutNs = 20000000ull;  // 20 ms: a test of the timeout path ends quickly
#else
constexpr unsigned long long kMbarTimeoutNs = 1000000000ull;  // 1 s
#endif
__device__ __forceinline__ bool mbar_try(unsigned a, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(a), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t));
  return t;
}
// (the polling loop out of line: it keeps the hot loop's registers free)
static __device__ __noinline__ bool mbar_wait_timed(unsigned a, unsigned parity) {
  const unsigned long long t0 = global_ns();
  while (true) {
    for (int i = 0; i < 64; ++i)
      if (mbar_try(a, parity)) return true;
    if (global_ns() - t0 > kMbarTimeoutNs) return false;
  }
}
__device__ __forceinline__ bool mbar_wait(unsigned a, unsigned parity) {
  return mbar_try(a, parity) || mbar_wait_timed(a, parity);
}

// The warp's sequence of metric chunks: chunk `c` of unit `unit` next, into stage
// `stage`.  issue() copies it (lane 0) when it lies inside the mesh and steps on.
template <int P, typename MT>
struct PlaneFeed {
  using C = PlaneCfg<P, MT>;
  int unit, c, stage;
  __device__ __forceinline__ void issue(const ApplyArgs<float, MT>& a, int nunits, int tw, int lane, unsigned sM,
                                        unsigned bar) {
    if (unit < nunits) {
      if (lane == 0 && !(SEM_HOLD(a, unit) && c == 0))
        bulk_copy(sM + stage * C::chunk_bytes, a.metric + ((size_t)unit * C::NCH + c) * C::ML::chunk(C::N),
                  C::chunk_bytes, bar + 8 * stage);
      step(tw);
    }
  }
  __device__ __forceinline__ void step(int tw) {
    if (++c == C::NCH) {
      c = 0;
      unit += tw;
    }
    if (++stage == C::kStages) stage = 0;
  }
};

// First node of the lane's element of unit `unit` (0 past the mesh).
template <int P, typename MT>
__device__ __forceinline__ int plane_base(const ApplyArgs<float, MT>& a, int unit, int nunits, int s) {
  using C = PlaneCfg<P, MT>;
  const int e = unit * C::G + s;
  return (unit < nunits && e < a.nelem) ? __ldg(a.first + e) : 0;
}

// Node (i, j, k) of the element e whose first node is `base`.
template <int N, typename MT>
__device__ __forceinline__ int plane_node(const ApplyArgs<float, MT>& a, int e, int base, int i, int j, int k,
                                          unsigned kind) {
#ifdef SEM_DEBUG
  return e < a.nelem ? (int)SEM_IDX(__ldg(a.map + (size_t)e * N * N * N + i + N * (j + N * k)), a.ndofs, a.dbg, kind)
                     : 0;
#else
  (void)e;
  (void)kind;
  return base + i + j * a.row + k * a.plane;
#endif
}

// Copies the unit's nodal values into a tile: lane (s, i) the nodes (i, j, k) of
// element slot s for every (j, k), one 4-byte cp.async each.
template <int P, typename MT>
__device__ __forceinline__ void plane_gather(const ApplyArgs<float, MT>& a, int unit, int base, int s, int r, bool act,
                                             unsigned tile) {
  using C = PlaneCfg<P, MT>;
  constexpr int N = C::N;
  if (act) {
    const unsigned dst = tile + 4u * (unsigned)(s * C::ES + r);
#pragma unroll
    for (int k = 0; k < N; ++k)
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const float* src = a.u + plane_node<N>(a, unit * C::G + s, base, r, j, k, kDbgGather);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst + 4u * (k * C::PS + j * N)), "l"(src)
                     : "memory");
      }
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}

// out[m] (+)= sum_l z[l] x_l[m] over the n planes x_l of an element in a tile.
template <int N, int PS, bool ACC>
__device__ __forceinline__ void plane_zsweep(const float (&z)[N], const float* elem, float (&out)[N * N]) {
  constexpr int CH = (N * N + 3) / 4;
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    float4 v[N];
#pragma unroll
    for (int l = 0; l < N; ++l) v[l] = *reinterpret_cast<const float4*>(elem + l * PS + 4 * c);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int m = 4 * c + t;
      if (m < N * N) {
        auto at = [&](int l) { return t == 0 ? v[l].x : t == 1 ? v[l].y : t == 2 ? v[l].z : v[l].w; };
        float acc = ACC ? fmaf(z[0], at(0), out[m]) : z[0] * at(0);
#pragma unroll
        for (int l = 1; l < N; ++l) acc = fmaf(z[l], at(l), acc);
        out[m] = acc;
      }
    }
  }
}

// The lane's plane between registers and its place in a tile, by 16-byte accesses.
template <int N>
__device__ __forceinline__ void plane_load(const float* p, float (&v)[N * N]) {
#pragma unroll
  for (int c = 0; c < (N * N + 3) / 4; ++c) {
    const float4 q = reinterpret_cast<const float4*>(p)[c];
    v[4 * c] = q.x;
    if (4 * c + 1 < N * N) v[4 * c + 1] = q.y;
    if (4 * c + 2 < N * N) v[4 * c + 2] = q.z;
    if (4 * c + 3 < N * N) v[4 * c + 3] = q.w;
  }
}
template <int N>
__device__ __forceinline__ void plane_store(float* p, const float (&v)[N * N]) {
#pragma unroll
  for (int c = 0; c < (N * N + 3) / 4; ++c) {
    auto at = [&](int m) { return m < N * N ? v[m < N * N ? m : 0] : 0.f; };
    reinterpret_cast<float4*>(p)[c] = make_float4(at(4 * c), at(4 * c + 1), at(4 * c + 2), at(4 * c + 3));
  }
}

// v = M along x (DIR 0) or y (DIR 1) of the plane v, in place.
template <int N, int DIR, bool ANTI>
__device__ __forceinline__ void plane_sweep(const EoMat<N, float>& M, float (&v)[N * N]) {
#pragma unroll
  for (int t = 0; t < N; ++t) {
    float in[N], out[N];
#pragma unroll
    for (int l = 0; l < N; ++l) in[l] = DIR == 0 ? v[t * N + l] : v[l * N + t];
    eo_line<N, ANTI, false>(M, in, out);
#pragma unroll
    for (int l = 0; l < N; ++l) (DIR == 0 ? v[t * N + l] : v[l * N + t]) = out[l];
  }
}

// Metric values of row J of the rows at p: point i at g[7 i .. 7 i + 6], read by
// 8-byte (bf16) or 16-byte (float) loads of four values.
__device__ __forceinline__ void metric_quad(const __nv_bfloat16* p, float (&g)[4]) {
  const uint2 w = *reinterpret_cast<const uint2*>(p);
  g[0] = __uint_as_float(w.x << 16);
  g[1] = __uint_as_float(w.x & 0xffff0000u);
  g[2] = __uint_as_float(w.y << 16);
  g[3] = __uint_as_float(w.y & 0xffff0000u);
}
__device__ __forceinline__ void metric_quad(const float* p, float (&g)[4]) {
  const float4 w = *reinterpret_cast<const float4*>(p);
  g[0] = w.x;
  g[1] = w.y;
  g[2] = w.z;
  g[3] = w.w;
}
template <int N, int J, typename MT>
__device__ __forceinline__ void metric_row(const MT* p, float (&g)[kMetricComps * N]) {
  constexpr int v0 = kMetricComps * N * J, v1 = v0 + kMetricComps * N;
#pragma unroll
  for (int c = v0 / 4; c < (v1 + 3) / 4; ++c) {
    float q[4];
    metric_quad(p + 4 * c, q);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int v = 4 * c + t - v0;
      if (v >= 0 && v < kMetricComps * N) g[v] = q[t];
    }
  }
}

// Quadrature-point stage and x-sweeps of row J (row JC of the chunk whose values of
// this lane are at `metric`): on entry u the values, gy and gz the y- and
// z-derivatives of the plane; on exit row J of u holds m + D^T q1 along x, gy and gz
// hold q2 and q3.
template <int N, int JC, typename MT>
__device__ __forceinline__ void plane_row(const EoMat<N, float>& D, const EoMat<N, float>& Dt, const MT* metric,
                                          float mass, float* u, float* gy, float* gz) {
  float in[N], g1[N], q1[N], m[N], g[kMetricComps * N];
  metric_row<N, JC>(metric, g);
#pragma unroll
  for (int i = 0; i < N; ++i) in[i] = u[i];
  eo_line<N, true, false>(D, in, g1);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const float* G = g + kMetricComps * i;  // G00 G01 G02 G11 G12 G22 W
    const float x = g1[i], y = gy[i], z = gz[i];
    q1[i] = fmaf(G[2], z, fmaf(G[1], y, G[0] * x));
    gy[i] = fmaf(G[4], z, fmaf(G[3], y, G[1] * x));
    gz[i] = fmaf(G[5], z, fmaf(G[4], y, G[2] * x));
    m[i] = (mass * G[6]) * in[i];
  }
  eo_line<N, true, true>(Dt, q1, m);
#pragma unroll
  for (int i = 0; i < N; ++i) u[i] = m[i];
}
template <int N, int J, int JC, int R, typename MT>
__device__ __forceinline__ void plane_chunk(const EoMat<N, float>& D, const EoMat<N, float>& Dt, const MT* metric,
                                            float mass, float (&u)[N * N], float (&gy)[N * N], float (&gz)[N * N]) {
  if constexpr (JC < R) {
    plane_row<N, JC>(D, Dt, metric, mass, u + (J + JC) * N, gy + (J + JC) * N, gz + (J + JC) * N);
    plane_chunk<N, J, JC + 1, R>(D, Dt, metric, mass, u, gy, gz);
  }
}

// The lane's wait for the chunk in stage `use`; when it runs out: report it, let the
// warp's other copies land, false.
template <int P, typename MT>
__device__ __forceinline__ bool plane_wait(const ApplyArgs<float, MT>& a, unsigned bar, int use, unsigned phase,
                                           int behind, int lane) {
  using C = PlaneCfg<P, MT>;
  if (mbar_wait(bar + 8 * use, (phase >> use) & 1u)) return true;
  if (lane == 0 && a.fault != nullptr) atomicOr(a.fault, 1u);
  for (int t = 1; t < behind; ++t) {  // `behind` copies issued from this one on
    const int st = (use + t) % C::kStages;
    mbar_wait(bar + 8 * st, (phase >> st) & 1u);
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  return false;
}

// All chunks of a unit, from J = 0: wait, rows, release the stage to the next copy.
template <int P, int J, typename MT>
__device__ __forceinline__ bool plane_points(const ApplyArgs<float, MT>& a, const KTab<P + 1, float>& tab,
                                             PlaneFeed<P, MT>& feed, int& use, unsigned& phase, int& behind, int nunits,
                                             int tw, int lane, int lidx, unsigned char* wb, unsigned sM, unsigned bar,
                                             float (&u)[(P + 1) * (P + 1)], float (&gy)[(P + 1) * (P + 1)],
                                             float (&gz)[(P + 1) * (P + 1)]) {
  using C = PlaneCfg<P, MT>;
  if constexpr (J < C::N) {
    if (!plane_wait<P>(a, bar, use, phase, behind, lane)) return false;
    phase ^= 1u << use;
    const MT* m = reinterpret_cast<const MT*>(wb + use * C::chunk_bytes) + lidx * C::ML::stride(C::N);
    plane_chunk<C::N, J, 0, C::R>(tab.D, tab.Dt, m, a.mass_coef, u, gy, gz);
    __syncwarp();  // the chunk is read: its stage takes the next copy
    --behind;
    if (feed.unit < nunits) ++behind;
    feed.issue(a, nunits, tw, lane, sM, bar);
    if (++use == C::kStages) use = 0;
    return plane_points<P, J + C::R>(a, tab, feed, use, phase, behind, nunits, tw, lane, lidx, wb, sM, bar, u, gy, gz);
  }
  return true;
}

template <int P, int QUAD, typename MT>
__global__ void __launch_bounds__(32 * PlaneCfg<P, MT>::kWarps, PlaneCfg<P, MT>::kResident / PlaneCfg<P, MT>::kWarps)
    sem_apply_plane_kernel(const ApplyArgs<float, MT> a, const __grid_constant__ KTab<P + 1, float> tab,
                           const __grid_constant__ ZTab<P + 1> zt, int nunits) {
  using C = PlaneCfg<P, MT>;
  constexpr int N = C::N, N2 = C::N2, G = C::G;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int unit = blockIdx.x * C::kWarps + warp;
  if (unit >= nunits) return;  // no CTA-wide barrier in this kernel
  const int tw = gridDim.x * C::kWarps;
  unsigned char* wb = smem_raw + (size_t)warp * C::warp_bytes;
  float* tiles = reinterpret_cast<float*>(wb + C::tile_offset);
  const unsigned sm_s = smem_u32(wb), tile_s = smem_u32(tiles), bar_s = smem_u32(wb + C::bar_offset);
  // While the previous kernel drains, before pdl_wait: the first metric copies and
  // the first nodes (written by the set-up only, see pdl_trigger).
  if (lane == 0) {
    for (int t = 0; t < C::kStages; ++t) mbar_init(bar_s + 8 * t);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncwarp();
  PlaneFeed<P, MT> feed{unit, 0, 0};
  int behind = 0;  // copies issued and not yet waited for
#pragma unroll
  for (int t = 0; t < C::kStages; ++t) {
    if (feed.unit < nunits) ++behind;
    feed.issue(a, nunits, tw, lane, sm_s, bar_s);
  }
  // lane = slot s of the unit and r: plane k = r of the sweeps, node i = r of the
  // gather and scatter rows.  Idle lanes (32 - G n) run on the last slot's data
  // and neither copy nor store.
  const bool act = lane < C::NL;
  const int s = act ? lane / N : G - 1, r = act ? lane - s * N : 0;
  float dz[N], dtz[N];
#pragma unroll
  for (int l = 0; l < N; ++l) {
    dz[l] = zt.D[r][l];
    dtz[l] = zt.Dt[r][l];
  }
  int base = plane_base<P>(a, unit, nunits, s);
  int base_n = plane_base<P>(a, unit + tw, nunits, s);
  pdl_wait();
  const bool stop = a.done != nullptr && *a.done;
  plane_gather<P>(a, unit, base, s, r, act, tile_s);
  if (stop) {  // the CTA must not end under its own copies
    for (int t = 0; t < behind; ++t) mbar_wait(bar_s + 8 * t, 0);
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    return;
  }
  unsigned phase = 0;  // bit t: parity of stage t's next completion
  int use = 0;         // stage of the next chunk
  int b = 0;
  const int lidx = s * N + r;
  for (; unit < nunits; unit += tw) {
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncwarp();  // every lane's copies of this unit landed
    const int nxt = unit + tw;
    if (nxt >= nunits) pdl_trigger();  // the last unit
    if (nxt < nunits) plane_gather<P>(a, nxt, base_n, s, r, act, tile_s + 4u * (unsigned)((b ^ 1) * C::TW));
    const int base_nn = plane_base<P>(a, nxt + tw, nunits, s);
    float* elem = tiles + b * C::TW + s * C::ES;
    float* own = elem + r * C::PS;
    float u[N2], gy[N2], gz[N2];
    plane_load<N>(own, u);
    if (QUAD == SEM_QUAD_LG) {  // values at the Gauss points: x and y in the plane, then z
      plane_sweep<N, 0, false>(tab.Bi, u);
      plane_sweep<N, 1, false>(tab.Bi, u);
      if (act) plane_store<N>(own, u);
      __syncwarp();
      float bz[N];
#pragma unroll
      for (int l = 0; l < N; ++l) bz[l] = zt.B[r][l];
      plane_zsweep<N, C::PS, false>(bz, elem, u);
      __syncwarp();
      if (act) plane_store<N>(own, u);
      __syncwarp();
    }
    plane_zsweep<N, C::PS, false>(dz, elem, gz);
#pragma unroll
    for (int v = 0; v < N2; ++v) gy[v] = u[v];
    plane_sweep<N, 1, true>(tab.D, gy);
    if (!plane_points<P, 0>(a, tab, feed, use, phase, behind, nunits, tw, lane, lidx, wb, sm_s, bar_s, u, gy, gz)) return;
    __syncwarp();  // the planes of u are read
    if (act) plane_store<N>(own, gz);
#pragma unroll
    for (int i = 0; i < N; ++i) {  // u += D^T q2 along y
      float in[N], out[N];
#pragma unroll
      for (int j = 0; j < N; ++j) {
        in[j] = gy[j * N + i];
        out[j] = u[j * N + i];
      }
      eo_line<N, true, true>(tab.Dt, in, out);
#pragma unroll
      for (int j = 0; j < N; ++j) u[j * N + i] = out[j];
    }
    __syncwarp();
    plane_zsweep<N, C::PS, true>(dtz, elem, u);
    if (QUAD == SEM_QUAD_LG) {  // back from the Gauss points: z, then x and y in the plane
      __syncwarp();
      if (act) plane_store<N>(own, u);
      __syncwarp();
      float bz[N];
#pragma unroll
      for (int l = 0; l < N; ++l) bz[l] = zt.Bt[r][l];
      plane_zsweep<N, C::PS, false>(bz, elem, u);
      plane_sweep<N, 1, false>(tab.Bit, u);
      plane_sweep<N, 0, false>(tab.Bit, u);
    }
    __syncwarp();
    if (act) plane_store<N>(own, u);
    __syncwarp();
    // scatter-add y += P_e^T y_e, lane (s, i) along the rows of its element
    const int e = unit * G + s;
    if (act && e < a.nelem) {
      const float sc = a.scale_out ? a.out_scale : 1.f;
      const float* row = elem + r;
      if (a.yloc != nullptr) {  // deterministic mode: element-local results
#pragma unroll
        for (int v = 0; v < N2; ++v)
          a.yloc[(size_t)e * C::N3 + r + N * v] = row[(v / N) * C::PS + (v % N) * N] * sc;
      } else {
#pragma unroll
        for (int v = 0; v < N2; ++v)
          atomicAdd(a.y + plane_node<N>(a, e, base, r, v % N, v / N, kDbgScatter),
                    row[(v / N) * C::PS + (v % N) * N] * sc);
      }
    }
    __syncwarp();  // the next iteration's gather refills this tile
    base = base_n;
    base_n = base_nn;
    b ^= 1;
  }
}

// Persistent grid of the plane kernel: the CTAs resident on the device at once
// (set by prime_t, before any stream capture), at most one warp per unit.
template <int P, int QUAD, typename MT>
struct PlaneGrid {
  static inline int resident = 0;
};

template <int P, int QUAD, typename MT>
cudaError_t plane_prime() {
  using C = PlaneCfg<P, MT>;
  cudaError_t e = cudaFuncSetAttribute(sem_apply_plane_kernel<P, QUAD, MT>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::cta_bytes);
  int dev = 0, sms = 0, per_sm = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sem_apply_plane_kernel<P, QUAD, MT>, 32 * C::kWarps,
                                                      C::cta_bytes);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  PlaneGrid<P, QUAD, MT>::resident = sms * per_sm;
  return cudaSuccess;
}

template <int P, int QUAD, typename MT>
cudaError_t launch_apply_plane(const Level& L, const ApplyArgs<float, MT>& a, const KTab<P + 1, float>& tab,
                               cudaStream_t s) {
  using C = PlaneCfg<P, MT>;
  constexpr int N = P + 1;
  if (PlaneGrid<P, QUAD, MT>::resident < 1) return cudaErrorInitializationError;  // prime_apply_kernels was not called
  const int nunits = (L.nelem + C::G - 1) / C::G;
  if (nunits == 0) return cudaSuccess;
  const int grid = std::min(PlaneGrid<P, QUAD, MT>::resident, (nunits + C::kWarps - 1) / C::kWarps);
  ZTab<N> zt;
  for (int q = 0; q < N; ++q)
    for (int l = 0; l < N; ++l) {
      zt.D[q][l] = zt.Dt[l][q] = (float)(QUAD == SEM_QUAD_LG ? L.tab.Dg : L.tab.D)[q][l];
      zt.B[q][l] = zt.Bt[l][q] = (float)L.tab.Bi[q][l];
    }
  launch_k(sem_apply_plane_kernel<P, QUAD, MT>, grid, 32 * C::kWarps, C::cta_bytes, s, a, tab, zt, nunits);
  return cudaGetLastError();
}

// The FP32 operator on few elements (p >= 3): one 1-D line of an element per thread, E
// elements a CTA.  Below about a warp of the plane kernel an SM the apply takes as long
// as one warp takes for its unit, and a lane of that kernel works through a whole plane;
// here a thread works through one line a sweep, the column's metric waits in registers
// before pdl_wait, and the z-sweeps are registers only.  E fills the warps where that
// pays: one element a CTA took 5.9 instead of 5.1 us at p = 4 (2,808 elements, SEM-NI),
// 7.5 instead of 7.2 at p = 5; three a CTA at p = 6 lose by the wider barriers (88
// elements 3.5 us against 3.0).
// An apply, FP32 metric, plane kernel / this one, p = 3..6: 288 elements, SEM-NI
// 3.1 / 2.6, 3.9 / 2.8, 6.1 / 3.0, 7.1 / 3.4 us, SEM 3.5 / 2.9, 5.5 / 3.2, 8.0 / 3.5,
// 10.1 / 3.9; 1,250 elements 3.2 / 2.9, 4.0 / 3.4, 6.6 / 4.4, 8.0 / 5.9 and 3.6 / 3.3,
// 6.0 / 3.8, 8.8 / 5.0, 11.5 / 6.9; 2,808 elements 3.5 / 3.8, 4.6 / 5.1, 7.2 / 7.2,
// 9.0 / 10.2 and 4.0 / 4.5, 6.4 / 5.6, 9.4 / 8.5, 12.3 / 12.1; 5,760 elements
// 4.0 / 5.9, 6.1 / 8.0, 8.5 / 12.1 and 4.8 / 7.0, 7.8 / 9.3, 10.7 / 14.4 (p = 3..5).
// The line (kElements) lies where the two meet.  At p = 1 and 2 the plane kernel is as
// fast on any mesh.
template <int P, int QUAD>
struct FewCfg {
  static constexpr int N2 = (P + 1) * (P + 1), E = P == 3 ? 4 : P == 4 ? 5 : P == 5 ? 3 : 1;
  static constexpr int kThreads = (E * N2 + 31) / 32 * 32;
  static constexpr bool kSem = QUAD == SEM_QUAD_LG;
  static constexpr int kElements =
      P == 3 ? 1600 : P == 4 ? (kSem ? 3800 : 2200) : P == 5 ? (kSem ? 3400 : 2600) : kSem ? 2800 : 2200;
};

template <int P, int QUAD, typename MT>
__global__ void __launch_bounds__(FewCfg<P, QUAD>::kThreads)
    sem_apply_few_kernel(const ApplyArgs<float, MT> a, const __grid_constant__ KTab<P + 1, float> tab) {
  constexpr int N = P + 1, N2 = N * N, N3 = N2 * N, E = FewCfg<P, QUAD>::E;
  using ML = MetricLayout<MT>;
  __shared__ float sA[E * N3], sB[E * N3], sC[E * N3];
  const int slot = threadIdx.x / N2, c = threadIdx.x - slot * N2, e = blockIdx.x * E + slot;
  const bool act = slot < E && e < a.nelem;
  const int i = c % N, q = c / N;  // of the thread's column (i, j = q) and of its y-line (i, k = q)
  float* A = sA + (slot < E ? slot * N3 : 0);
  float* B = sB + (slot < E ? slot * N3 : 0);
  float* C = sC + (slot < E ? slot * N3 : 0);
  const int xl = N * c, yl = i + N2 * q;
  MT G[N][kMetricComps];
  int g0 = 0;
  if (act) {
    g0 = __ldg(a.first + e);
#pragma unroll
    for (int k = 0; k < N; ++k)
#pragma unroll
      for (int m = 0; m < kMetricComps; ++m) G[k][m] = __ldg(a.metric + ML::offset(N, e, c, k, m));
  }
  auto line = [](float* p, int stride, float (&v)[N]) {
#pragma unroll
    for (int t = 0; t < N; ++t) v[t] = p[t * stride];
  };
  auto put = [](float* p, int stride, const float (&v)[N]) {
#pragma unroll
    for (int t = 0; t < N; ++t) p[t * stride] = v[t];
  };
  auto result = [&](int ii, int jj, int kk, float v) {
    v = scale_result(a, v);
    if (a.yloc != nullptr) store_loc(a.yloc + (size_t)e * N3 + ii + N * jj + N2 * kk, v);
    else scatter_add(a.y + plane_node<N>(a, e, g0, ii, jj, kk, kDbgScatter), v);
  };
  pdl_wait();
  const bool stop = a.done != nullptr && *a.done;
  float z[N], w[N], v[N];
  if (act) {
#pragma unroll
    for (int k = 0; k < N; ++k) z[k] = a.u[plane_node<N>(a, e, g0, i, q, k, kDbgGather)];
  }
  if (stop) return;
  if (act) {
    if (QUAD == SEM_QUAD_LG) {
      eo_line<N, false, false>(tab.Bi, z, w);
      put(A + c, N2, w);
    } else {
      put(A + c, N2, z);
    }
  }
  __syncthreads();
  if (QUAD == SEM_QUAD_LG) {  // values at the Gauss points
    if (act) {
      line(A + xl, 1, v);
      eo_line<N, false, false>(tab.Bi, v, w);
      put(A + xl, 1, w);
    }
    __syncthreads();
  }
  if (act) {
    line(A + yl, N, v);
    if (QUAD == SEM_QUAD_LG) {
      eo_line<N, false, false>(tab.Bi, v, w);
      put(A + yl, N, w);
      eo_line<N, true, false>(tab.D, w, v);
      put(C + yl, N, v);
    } else {
      eo_line<N, true, false>(tab.D, v, w);
      put(C + yl, N, w);
    }
  }
  if (QUAD == SEM_QUAD_LG) __syncthreads();
  if (act) {
    line(A + xl, 1, v);
    eo_line<N, true, false>(tab.D, v, w);
    put(B + xl, 1, w);
    if (QUAD == SEM_QUAD_LG) line(A + c, N2, z);
  }
  __syncthreads();
  float m[N];
  if (act) {
    eo_line<N, true, false>(tab.D, z, v);
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const float g1 = B[c + k * N2], g2 = C[c + k * N2], g3 = v[k];
      float g[kMetricComps];
#pragma unroll
      for (int t = 0; t < kMetricComps; ++t) g[t] = (float)G[k][t];
      B[c + k * N2] = fmaf(g[2], g3, fmaf(g[1], g2, g[0] * g1));
      C[c + k * N2] = fmaf(g[4], g3, fmaf(g[3], g2, g[1] * g1));
      w[k] = fmaf(g[5], g3, fmaf(g[4], g2, g[2] * g1));
      m[k] = (a.mass_coef * g[6]) * z[k];
    }
    eo_line<N, true, true>(tab.Dt, w, m);
  }
  __syncthreads();
  if (act) {
    line(B + xl, 1, v);
    for (int t = 0; t < N; ++t) w[t] = 0.f;
    eo_line<N, true, true>(tab.Dt, v, w);
    put(B + xl, 1, w);
    line(C + yl, N, v);
    for (int t = 0; t < N; ++t) w[t] = 0.f;
    eo_line<N, true, true>(tab.Dt, v, w);
    put(C + yl, N, w);
  }
  __syncthreads();
  if (act) {
#pragma unroll
    for (int k = 0; k < N; ++k) m[k] += B[c + k * N2] + C[c + k * N2];
  }
  if (QUAD == SEM_QUAD_LG) {  // back to the nodes
    if (act) {
      eo_line<N, false, false>(tab.Bit, m, w);
      put(A + c, N2, w);
    }
    __syncthreads();
    if (act) {
      line(A + xl, 1, v);
      eo_line<N, false, false>(tab.Bit, v, w);
      put(A + xl, 1, w);
    }
    __syncthreads();
    if (act) {
      line(A + yl, N, v);
      eo_line<N, false, false>(tab.Bit, v, w);
    }
  }
  pdl_trigger();
  if (act) {
#pragma unroll
    for (int t = 0; t < N; ++t) {
      if (QUAD == SEM_QUAD_LG) result(i, t, q, w[t]);
      else result(i, q, t, m[t]);
    }
  }
}

template <int P, int QUAD, typename MT>
cudaError_t launch_apply_few(const Level& L, const ApplyArgs<float, MT>& a, const KTab<P + 1, float>& tab, cudaStream_t s) {
  using C = FewCfg<P, QUAD>;
  launch_k(sem_apply_few_kernel<P, QUAD, MT>, (L.nelem + C::E - 1) / C::E, C::kThreads, 0, s, a, tab);
  return cudaGetLastError();
}

// Even-odd form (EoMat) of the n x n matrix M (or of its transpose), from the
// host tables; the mirrored rows are implied by the symmetry of M.
template <int N, typename T>
void make_eo(EoMat<N, T>& E, const double (&M)[kMaxN][kMaxN], bool transpose) {
  constexpr int H = N / 2;
  auto m = [&](int q, int l) { return transpose ? M[l][q] : M[q][l]; };
  for (int q = 0; q < H; ++q) {
    for (int l = 0; l < H; ++l) {
      E.a[q][l] = (T)(0.5 * (m(q, l) + m(q, N - 1 - l)));
      E.b[q][l] = (T)(0.5 * (m(q, l) - m(q, N - 1 - l)));
    }
    E.a[q][H] = (T)((N & 1) ? m(q, H) : 0.0);
  }
  for (int l = 0; l <= H; ++l) E.c[l] = (T)((N & 1) ? m(H, l) : 0.0);
  if constexpr (EoMat<N, T>::kDirect)
    for (int q = 0; q < N; ++q)
      for (int l = 0; l < N; ++l) E.m[q][l] = (T)m(q, l);
}

// The apply kernels of one degree, quadrature and precision (atomic adds into
// y, or element-local results into a.yloc).
template <int P, int QUAD, typename T, typename MT>
cudaError_t launch_apply_kernels(const Level& L, const ApplyArgs<T, MT>& a, const KTab<P + 1, T>& tab,
                                 bool mass_only, bool dot, cudaStream_t s) {
  constexpr int E = ApplyCfg<P>::E;
  const int grid = (L.nelem + E - 1) / E;
  if (grid == 0) return cudaSuccess;
  constexpr size_t tiles = apply_tile_bytes<P, T>();
  if constexpr (std::is_same<T, float>::value) {
    if (dot) return cudaErrorInvalidValue;
    if constexpr (P >= 3) {
      // (the plane kernel where a metric copy is to be held back)
      if (!mass_only && L.nelem <= FewCfg<P, QUAD>::kElements && L.hold < 0) return launch_apply_few<P, QUAD, MT>(L, a, tab, s);
    }
    if (!mass_only) return launch_apply_plane<P, QUAD, MT>(L, a, tab, s);
    // mass only (Gauss quadrature; without it the mass is a diagonal), on the weights
    if (weight_lowp_count(L) == 0) return cudaErrorInvalidValue;
    ApplyArgs<T, MT> m = a;
    m.metric = a.metric + metric_lowp_count(L);
    // p <= 4: elements owned by warps (measured faster; at p = 5, 6 the n^2 = 36, 49
    // lines fill warps poorly and the CTA-wide mode is faster)
    if constexpr (P <= 4) {
      constexpr int per_cta = kWarpsPerCta * WarpCfg<P>::G;
      launch_k(sem_apply_kernel<P, QUAD, T, MT, false, true, true>, (L.nelem + per_cta - 1) / per_cta, kApplyThreads,
               apply_warp_tile_bytes<P, T>(), s, m, tab);
    } else {
      launch_k(sem_apply_kernel<P, QUAD, T, MT, false, true>, grid, kApplyThreads, tiles, s, m, tab);
    }
    return cudaGetLastError();
  } else {
  if (mass_only) {
    launch_k(sem_apply_kernel<P, QUAD, T, MT, false, true>, grid, kApplyThreads, tiles, s, a, tab);
  } else if (dot) {
    using C = ApplyCta<P, T, true>;
    const int dgrid = (L.nelem + C::E - 1) / C::E;
    launch_k(sem_apply_kernel<P, QUAD, T, MT, true, false>, dgrid, C::kThreads, C::smem, s, a, tab);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || (a.cg == nullptr && a.dot_out == nullptr)) return e;
    return launch_apply_dot_finish(a.dot_partials, dgrid, a.cg, a.dot_out, a.done, s);
  } else {
    using C = ApplyCta<P, T, false>;
    launch_k(sem_apply_kernel<P, QUAD, T, MT, false, false>, (L.nelem + C::E - 1) / C::E, C::kThreads, C::smem, s, a,
             tab);
  }
  return cudaGetLastError();
  }
}

// Launch helper shared by the precision-specific translation units.  With
// a.yloc set (deterministic mode) the kernels write element results and the
// node sums follow in a fixed order.
template <int P, int QUAD, typename T, typename MT>
cudaError_t launch_apply_t(const Level& L, const ApplyArgs<T, MT>& a, bool mass_only, bool dot,
                           cudaStream_t s) {
  constexpr int N = P + 1;
  KTab<N, T> tab;
  make_eo(tab.D, QUAD == SEM_QUAD_LG ? L.tab.Dg : L.tab.D, false);
  make_eo(tab.Dt, QUAD == SEM_QUAD_LG ? L.tab.Dg : L.tab.D, true);
  make_eo(tab.Bi, L.tab.Bi, false);
  make_eo(tab.Bit, L.tab.Bi, true);
  ApplyArgs<T, MT> b = a;
  b.ndofs = L.ndofs;
  b.row = P * L.nx + 1;
  b.first = L.first;
  b.plane = b.row * (P * L.ny + 1);
  b.dbg = L.dbg;
  b.fault = L.fault;
  b.hold = L.hold;
  const cudaError_t e = launch_apply_kernels<P, QUAD, T, MT>(L, b, tab, mass_only, dot, s);
  if (e != cudaSuccess || a.yloc == nullptr) return e;
  return launch_assemble(L, a.yloc, a.y, a.done, s);
}

// Dynamic shared-memory limits of the variants of one instantiation.
template <int P, int QUAD, typename T, typename MT>
cudaError_t prime_t() {
  constexpr int tiles = (int)apply_tile_bytes<P, T>();
  cudaError_t e = cudaFuncSetAttribute(sem_apply_kernel<P, QUAD, T, MT, false, true>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, tiles);
  if (e != cudaSuccess) return e;
  if constexpr (std::is_same<T, float>::value) {
    return plane_prime<P, QUAD, MT>();
  } else {
    if ((e = cudaFuncSetAttribute(sem_apply_kernel<P, QUAD, T, MT, false, false>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, tiles)) != cudaSuccess) return e;
    return cudaFuncSetAttribute(sem_apply_kernel<P, QUAD, T, MT, true, false>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, tiles);
  }
}

template <typename T, typename MT>
cudaError_t prime_all() {
  cudaError_t e;
#define SEM_PRIME(PP)                                                                   \
  if ((e = prime_t<PP, SEM_QUAD_LG, T, MT>()) != cudaSuccess) return e;                \
  if ((e = prime_t<PP, SEM_QUAD_LGL, T, MT>()) != cudaSuccess) return e;
  SEM_PRIME(1) SEM_PRIME(2) SEM_PRIME(3) SEM_PRIME(4) SEM_PRIME(5) SEM_PRIME(6)
#undef SEM_PRIME
  return cudaSuccess;
}

template <typename T, typename MT>
cudaError_t dispatch_apply(const Level& L, const ApplyArgs<T, MT>& a, bool mass_only, bool dot,
                           cudaStream_t s) {
#define SEM_CASE(PP)                                                                  \
  case PP:                                                                            \
    return L.quad == SEM_QUAD_LG ? launch_apply_t<PP, SEM_QUAD_LG, T, MT>(L, a, mass_only, dot, s) \
                                 : launch_apply_t<PP, SEM_QUAD_LGL, T, MT>(L, a, mass_only, dot, s);
  switch (L.p) {
    SEM_CASE(1)
    SEM_CASE(2)
    SEM_CASE(3)
    SEM_CASE(4)
    SEM_CASE(5)
    SEM_CASE(6)
    default:
      return cudaErrorInvalidValue;
  }
#undef SEM_CASE
}

}  // namespace sem
