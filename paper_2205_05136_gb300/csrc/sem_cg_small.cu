// Jacobi and plain CG of a small mesh in one kernel (FP64 operator).
//
// On a mesh of a few thousand nodes an iteration is four launches of kernels that each
// do a microsecond of work.  Here one cluster of 8 or 16 CTAs runs the whole solve: the
// nodes' x, r and 1 / diagonal stay in their threads' registers, p and A p go through
// global memory (L2) between the CTAs, the inner products through distributed shared
// memory, and the cluster's hardware barrier, three times an iteration, stands where the
// kernel boundaries were.  The latency of the FP64 sweeps between barriers bounds a
// solve of a thousand nodes, the 16 SMs' FP64 rate (2 operations a clock each) one of ten
// thousand, where the launch-per-step path, on all SMs, overtakes it (cg_small_fits).
// A time step, launches / one kernel, in us: p = 2 SEM-NI 1,125 nodes 131 / 82, 4,515
// nodes 201 / 128; p = 3 SEM 1,000 nodes 827 / 426, 6,517 nodes 651 / 430; p = 6 SEM
// 7,315 nodes 1,167 / 635.
//
// A launch runs at most kIterCap iterations and saves the iterate, so that a solve
// that does not converge returns to the host between launches as the other path does.
#include <algorithm>

#include "sem_apply_kernel.cuh"
#include "sem_context.cuh"

namespace sem {
namespace {

constexpr int kCtasMax = 16, kThreads = 256, kPer = 4;  // kPer nodes a thread at most
constexpr int kIterCap = 64;

struct SmallArgs {
  const int* map;
  const double* metric;
  int nelem, n;
  double mass;
  const double *b, *inv;  // inv: 1 / diagonal, or nullptr
  const double* ax0;      // A x of the initial iterate, or nullptr: applied here
  double *x, *r, *p, *Ap;
  CgScalars* sc;
  double rtol, atol;
  int maxit, resume;      // resume: continue from x, r, p and *sc
  int64_t ndofs;
  unsigned long long* dbg;
};

// The cluster's barrier: writes before it, to global and distributed shared memory, are
// visible to every thread of the cluster after it.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
  return r;
}
// *p of CTA `rank` (p: the same variable in this CTA's shared memory) = v
__device__ __forceinline__ void st_cluster(const double* p, unsigned rank, double v) {
  unsigned a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  asm volatile("st.shared::cluster.f64 [%0], %1;\n" ::"r"(a), "d"(v) : "memory");
}

// Sums of K values over the threads of the cluster's nc CTAs, the same in every thread:
// block sums, then every CTA's sums to every CTA, added in CTA order.  The barrier also
// orders the global writes before it.
template <int K>
__device__ __forceinline__ void cluster_sums(int nc, unsigned rank, double (&v)[K], double (*xch)[2],
                                             double (*red)[kThreads / 32]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) red[k][warp] = v[k];
  __syncthreads();
  if ((int)threadIdx.x < nc)
#pragma unroll
    for (int k = 0; k < K; ++k) {
      double t = 0.0;
#pragma unroll
      for (int w = 0; w < kThreads / 32; ++w) t += red[k][w];
      st_cluster(&xch[rank][k], threadIdx.x, t);
    }
  cluster_sync();
#pragma unroll
  for (int k = 0; k < K; ++k) {
    double t = 0.0;
    for (int c = 0; c < nc; ++c) t += xch[c][k];
    v[k] = t;
  }
}

template <int P, int QUAD>
__global__ void __launch_bounds__(kThreads)
    k_cg_small(const SmallArgs a, const __grid_constant__ KTab<P + 1, double> tab) {
  constexpr int N = P + 1, N3 = N * N * N, E = ApplyCfg<P>::E;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* sA = reinterpret_cast<double*>(smem_raw);
  double* sB = sA + E * N3;
  double* sC = sB + E * N3;
  __shared__ double red[2][kThreads / 32];
  __shared__ double xa[2][kCtasMax][2], xr[2][kCtasMax][2];  // two buffers: one is read while the other is written
  const int tid = threadIdx.x, rank = (int)cluster_rank(), gt = rank * kThreads + tid, nc = gridDim.x;
  const int per = (a.nelem + nc - 1) / nc, first = min(rank * per, a.nelem), last = min(first + per, a.nelem);

  // The nodes of the thread's gathered values of the CTA's first batch of elements, and
  // their values since the gather: an iteration then starts with one load and the inner
  // product takes none.
  constexpr int KEEP = 4;
  int node0[KEEP];
  const int ne0 = min(E, last - first);
#pragma unroll
  for (int k = 0; k < KEEP; ++k) {
    const int i = tid + k * kThreads;
    node0[k] = i < ne0 * N3 ? (int)SEM_IDX(__ldg(a.map + (size_t)first * N3 + i), a.ndofs, a.dbg, kDbgGather) : 0;
  }
  // y += A u over the CTA's elements; the thread's share of u . A u
  auto apply = [&](const double* u, double* y) {
    double dot = 0.0;
    for (int e0 = first; e0 < last; e0 += E) {
      const int ne = min(E, last - e0);
      const int* gmap = a.map + (size_t)e0 * N3;
      auto at = [&](int i, unsigned kind) { return SEM_IDX(__ldg(gmap + i), a.ndofs, a.dbg, kind); };
      const bool kept = e0 == first;
      double u0[KEEP];
      if (kept) {
#pragma unroll
        for (int k = 0; k < KEEP; ++k) {
          const int i = tid + k * kThreads;
          u0[k] = i < ne * N3 ? __ldcg(u + node0[k]) : 0.0;
        }
#pragma unroll
        for (int k = 0; k < KEEP; ++k) {
          const int i = tid + k * kThreads;
          if (i < ne * N3) sA[i] = u0[k];
        }
      }
      for (int i = tid + (kept ? KEEP * kThreads : 0); i < ne * N3; i += kThreads)
        sA[i] = __ldcg(u + at(i, kDbgGather));
      __syncthreads();
      element_results<P, QUAD, false, false, false>(tab, a.metric, a.mass, e0, last, ne, sA, sB, sC, tid, kThreads);
      if (kept) {
#pragma unroll
        for (int k = 0; k < KEEP; ++k) {
          const int i = tid + k * kThreads;
          if (i < ne * N3) {
            const double v = sA[i];
            atomicAdd(y + node0[k], v);
            dot = fma(u0[k], v, dot);
          }
        }
      }
      for (int i = tid + (kept ? KEEP * kThreads : 0); i < ne * N3; i += kThreads) {
        const int64_t g = at(i, kDbgScatter);
        const double v = sA[i];
        atomicAdd(y + g, v);
        dot = fma(__ldcg(u + g), v, dot);
      }
      if (e0 + E < last) __syncthreads();
    }
    return dot;
  };

  pdl_wait();
  cluster_sync();  // every CTA runs before another writes to its shared memory
  double x[kPer], r[kPer], inv[kPer], p[kPer];
  double rz, tol2;
  int iters = 0, done = 0, status = 0;
  double rr;
  const auto node = [&](int k) { return gt + k * nc * kThreads; };
  if (a.resume) {
    rz = a.sc->rz;
    rr = a.sc->rr;
    tol2 = a.sc->tol2;
    iters = a.sc->iters;
#pragma unroll
    for (int k = 0; k < kPer; ++k)
      if (node(k) < a.n) {
        x[k] = a.x[node(k)];
        r[k] = a.r[node(k)];
        p[k] = a.p[node(k)];
        inv[k] = a.inv ? a.inv[node(k)] : 1.0;
      }
    cluster_sync();  // every CTA has read *sc
  } else {
#pragma unroll
    for (int k = 0; k < kPer; ++k)
      if (node(k) < a.n) a.Ap[node(k)] = 0.0;
    if (a.ax0 == nullptr) {
      cluster_sync();
      apply(a.x, a.Ap);
      cluster_sync();
    }
    double v[2] = {0.0, 0.0}, bb[1] = {0.0};
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int i = node(k);
      if (i < a.n) {
        const double bi = a.b[i];
        x[k] = a.x[i];
        inv[k] = a.inv ? a.inv[i] : 1.0;
        r[k] = bi - (a.ax0 ? a.ax0[i] : __ldcg(a.Ap + i));
        p[k] = inv[k] * r[k];
        a.p[i] = p[k];
        a.Ap[i] = 0.0;
        v[0] = fma(r[k], p[k], v[0]);
        v[1] = fma(r[k], r[k], v[1]);
        bb[0] = fma(bi, bi, bb[0]);
      }
    }
    cluster_sums<2>(nc, rank, v, xr[1], red);
    __syncthreads();
    cluster_sums<1>(nc, rank, bb, xa[1], red);
    rz = v[0];
    rr = v[1];
    tol2 = fmax(a.rtol * a.rtol * bb[0], a.atol * a.atol);
    const bool finite = isfinite(v[0]) && isfinite(v[1]) && isfinite(bb[0]);
    if (!finite) status = SEM_ERR_NONFINITE;
    done = (!finite || rr <= tol2) ? 1 : 0;
    if (gt == 0) a.sc->bb = bb[0];
  }
  // p and a zero A p are visible to the cluster here
  const int stop = min(a.maxit, iters + kIterCap);
  for (int it = 0; !done && iters < stop; ++it) {
    double d[1] = {apply(a.p, a.Ap)};
    cluster_sums<1>(nc, rank, d, xa[it & 1], red);
    const double alpha = rz / d[0];
    double v[2] = {0.0, 0.0}, z[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int i = node(k);
      if (i < a.n) {
        x[k] = fma(alpha, p[k], x[k]);
        r[k] = fma(-alpha, __ldcg(a.Ap + i), r[k]);
        z[k] = inv[k] * r[k];
        a.Ap[i] = 0.0;
        v[0] = fma(r[k], z[k], v[0]);
        v[1] = fma(r[k], r[k], v[1]);
      }
    }
    cluster_sums<2>(nc, rank, v, xr[it & 1], red);
    const double beta = v[0] / rz;
    rz = v[0];
    rr = v[1];
    iters += 1;
    if (!(isfinite(v[0]) && isfinite(v[1]) && isfinite(alpha))) {
      status = SEM_ERR_NONFINITE;
      done = 1;
    } else if (rr <= tol2) {
      done = 1;
    }
#pragma unroll
    for (int k = 0; k < kPer; ++k)
      if (node(k) < a.n) {
        p[k] = fma(beta, p[k], z[k]);
        a.p[node(k)] = p[k];
      }
    cluster_sync();  // p complete, A p zero
  }
#pragma unroll
  for (int k = 0; k < kPer; ++k)
    if (node(k) < a.n) {
      a.x[node(k)] = x[k];
      a.r[node(k)] = r[k];
    }
  if (gt == 0) {
    a.sc->rz = rz;
    a.sc->rr = rr;
    a.sc->tol2 = tol2;
    a.sc->iters = iters;
    a.sc->done = done;
    a.sc->status = status;
  }
  cluster_sync();  // no CTA ends while another may write to its shared memory
}

// CTAs of the cluster: 8 up to 1,500 nodes (cheaper barriers and sums), above and at
// p = 1 (most elements a node) 16.  A Jacobi step, 8 / 16, SEM-NI and SEM, us: p = 1 532
// nodes 79 / 81 and 486 / 519, 1,350 94 / 93 and 705 / 576, 2,304 146 / 119 and 1,050 /
// 746; p = 2 1,035 nodes 81 / 93 and 408 / 442, 1,485 96 / 106 and 430 / 437, 1,595 104 /
// 104 and 440 / 426, 3,367 132 / 116 and 609 / 451; p = 3 1,120 nodes 103 / 114 and 354 /
// 388, 2,821 117 / 117 and 475 / 444.  From p = 4 on (fewer, longer elements) 8 would stay
// the faster to about 2,500 nodes (p = 4 2,145 nodes 131 / 143 and 480 / 513, p = 6 2,275
// 156 / 168 and 539 / 570; even at 3,400 to 4,000); the line does not follow that.
int small_ctas(const Level& L) { return L.p >= 2 && L.ndofs <= 1500 ? 8 : kCtasMax; }

template <int P>
constexpr size_t small_smem() {
  return (size_t)3 * ApplyCfg<P>::E * (P + 1) * (P + 1) * (P + 1) * sizeof(double);
}

// Grid, block, shared memory and cluster of nc CTAs (at[0]).
template <int P>
void small_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at, int nc) {
  static_assert(small_smem<P>() <= 46 * 1024, "within the default limit beside the static arrays");
  cfg.gridDim = dim3((unsigned)nc);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = small_smem<P>();
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)nc;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
}

// Whether the device can hold the cluster (a partition of a GPU may have no 16 SMs in one
// GPC); also allows the kernel the cluster size beyond the portable 8.
template <int P, int QUAD>
bool small_placeable(int nc) {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[1];
  small_config<P>(cfg, at, nc);
  int clusters = 0;
  const bool ok = cudaFuncSetAttribute(k_cg_small<P, QUAD>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                  cudaOccupancyMaxActiveClusters(&clusters, k_cg_small<P, QUAD>, &cfg) == cudaSuccess;
  if (!ok) cudaGetLastError();  // the launches of cg_solve take the mesh instead
  return ok && clusters > 0;
}

template <int P, int QUAD>
cudaError_t launch_small(const Level& L, const SmallArgs& a, cudaStream_t s) {
  constexpr int N = P + 1;
  KTab<N, double> tab;
  make_eo(tab.D, QUAD == SEM_QUAD_LG ? L.tab.Dg : L.tab.D, false);
  make_eo(tab.Dt, QUAD == SEM_QUAD_LG ? L.tab.Dg : L.tab.D, true);
  make_eo(tab.Bi, L.tab.Bi, false);
  make_eo(tab.Bit, L.tab.Bi, true);
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[2];
  small_config<P>(cfg, at, small_ctas(L));
  cfg.stream = s;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.numAttrs = pdl_enabled() ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, k_cg_small<P, QUAD>, a, tab);
}

}  // namespace

// Whether the one-kernel solve takes a mesh on the current device: up to where it
// measured even with the launches of cg_solve (us a time step, launches / one kernel):
//   SEM-NI  p = 1 175 / 146 at 3,920 nodes, 174 / 185 at 5,760; p = 2 216 / 181 at 7,497,
//           209 / 211 at 9,063; p = 3 246 / 232 at 9,880, 257 / 274 at 13,420; p = 4 313 /
//           243 at 11,529, 342 / 342 at 14,625; p = 5 376 / 296 at 12,936, 406 / 337 at
//           15,246; p = 6 441 / 338 at 13,975
//   SEM     p = 1 799 / 764 at 2,730, 808 / 939 at 3,920; p = 2 696 / 633 at 5,355, 679 /
//           687 at 7,497; p = 3 744 / 517 at 6,517, 723 / 752 at 9,880; p = 4 849 / 674 at
//           11,529, 827 / 871 at 14,625; p = 5 962 / 749 at 12,936, 967 / 814 at 15,246;
//           p = 6 1,074 / 824 at 13,975
// (p = 5 and 6: the nodes that the cluster's threads hold are the limit).
bool cg_small_fits(const Level& L, int max_ctas) {
  static constexpr int64_t kNodes[2][kMaxP + 1] = {
      {0, 2500, 6000, 9000, 12000, 14000, 14000},    // SEM
      {0, 4500, 8000, 10000, 12000, 14000, 14000}};  // SEM-NI
  static_assert(14000 <= kCtasMax * kThreads * kPer, "every node has a place");
  if (L.p < 1 || L.p > kMaxP || L.ndofs > kNodes[L.quad == SEM_QUAD_LGL ? 1 : 0][L.p]) return false;
  const int nc = small_ctas(L);
  if (nc > max_ctas) return false;
#define SEM_CASE(PP) \
  case PP:           \
    return L.quad == SEM_QUAD_LG ? small_placeable<PP, SEM_QUAD_LG>(nc) : small_placeable<PP, SEM_QUAD_LGL>(nc);
  switch (L.p) {
    SEM_CASE(1)
    SEM_CASE(2)
    SEM_CASE(3)
    SEM_CASE(4)
    SEM_CASE(5)
    SEM_CASE(6)
  }
#undef SEM_CASE
  return false;
}

cudaError_t launch_cg_small(const Level& L, double alpha, const double* b, const double* inv, const double* ax0, double* x,
                            double* r, double* p, double* Ap, CgScalars* sc, double rtol, double atol, int maxit,
                            bool resume, cudaStream_t s) {
  SmallArgs a{};
  a.map = L.map; a.metric = L.metric; a.nelem = L.nelem; a.n = (int)L.ndofs; a.mass = alpha;
  a.b = b; a.inv = inv; a.ax0 = ax0; a.x = x; a.r = r; a.p = p; a.Ap = Ap; a.sc = sc;
  a.rtol = rtol; a.atol = atol; a.maxit = maxit; a.resume = resume; a.ndofs = L.ndofs; a.dbg = L.dbg;
#define SEM_CASE(PP)                                                      \
  case PP:                                                                \
    return L.quad == SEM_QUAD_LG ? launch_small<PP, SEM_QUAD_LG>(L, a, s) \
                                 : launch_small<PP, SEM_QUAD_LGL>(L, a, s);
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
