// Geometric multigrid preconditioner (Section 4.3) and the flexible PCG it drives.
//
// Levels: the fine Q_p level, then p-coarsened levels on the same mesh
// (p -> max(1, p/2) -> ... -> 1), then 2:1 h-coarsened Q_1 levels (each
// direction's n elements -> ceil(n/2) elements built from every other vertex)
// until a level has at most `min_coarse_dofs` nodes.  Every level
// rediscretises alpha M + K with its own metric; a coarse element takes the
// tissue of its first fine child.
//
// Transfers (matrix-vector products, Section 4.3):
//   p-levels: nodal interpolation Q_pc -> Q_pf, the tensor product of 1-D
//     prolongations on the lattice (sem_transfer.cu); restriction is its
//     transpose;
//   h-levels: per fine vertex, the coarse trilinear function evaluated at the
//     reference coordinates -1, 0, +1 of the coarse element (a trailing odd
//     element spans one fine element: -1, +1); restriction by the transpose.
// Smoother: Chebyshev semi-iteration with point-Jacobi on [0.08, 1.2] x the
//   largest eigenvalue of D^{-1} A, estimated by 10 preconditioned CG
//   (Lanczos) steps from a fixed start vector; degree `degree` before and after
//   the coarse correction, degree `coarse_degree` on the coarsest level.
// Precision: the V-cycle runs in FP32 with an FP32 or bf16 metric, or in FP64;
//   the outer CG, its inner products and residual stay in FP64.  A V-cycle in
//   FP32 is not exactly symmetric, so the outer iteration is the flexible
//   (Polak-Ribiere) PCG: beta = r_{k+1} . (z_{k+1} - z_k) / (r_k . z_k).
#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "sem_apply_kernel.cuh"
#include "sem_context.cuh"
#include "sem_dfmath.cuh"

namespace sem {

// p-transfers on the slab lattice (sem_transfer.cu).
template <typename T>
cudaError_t p_transfer(bool prolong, const Level& F, const Level& C, const double (*P)[kMaxN], const T* src, T* dst,
                       T* dst_d, const int* done, cudaStream_t s);

struct GmgLevel {
  Level* L = nullptr;
  bool owned = false;
  int to_next = 0;  // 0: p-transfer to the next level, 1: h-transfer
  double *sl = nullptr, *st = nullptr, *th = nullptr;
  bool owns_tissue = false;
  // residual (right-hand side at first), iterate, correction, 1 / diagonal
  void *r = nullptr, *x = nullptr, *d = nullptr, *invd = nullptr;
  double* dinv64 = nullptr;
  double lam = 0.0;
};

constexpr int kLanczosSteps = 10;
struct LanczosScalars {
  double rz, a, b;  // r . z; step length and conjugation coefficient of the current step
  double alpha[kLanczosSteps], beta[kLanczosSteps];
  int m, stop;      // steps recorded
};

struct Gmg {
  std::vector<GmgLevel> lv;
  double alpha = -1.0;
  bool stale = false;  // the tissue changed: metrics, diagonals and estimates are renewed on the next use
  int precision = SEM_PREC_FP32;
  int degree = 3, coarse_degree = 10;
  double* z = nullptr;                                 // outer PCG preconditioned residual
  // CUDA graphs of the PCG set-up and of one PCG iteration (V-cycle included),
  // keyed by the solution pointer and alpha; captured on a private stream.
  struct Graphs {
    bool used = false;
    const double* x = nullptr;
    const double* b = nullptr;
    double alpha = 0.0;
    double rtol = 0.0, atol = 0.0;
    // one executable graph and its kernel count, captured when it is first launched
    struct Exec {
      cudaGraphExec_t exec = nullptr;
      int64_t kernels = 0;
    };
    Exec init[3];     // the set-up: A x applied, carried (ws.Ax), carried where ws.same reads nonzero
    Exec iter[2];     // an iteration; [1] with event nodes around two applies
    int last_iters = 0;  // iterations the previous solve with these graphs took
    // the set-up (variant v) and its first `n` iterations as one graph: one launch
    // where n + 1 were.  Captured once two solves in a row took n iterations.
    struct Combo : Exec {
      int n = 0, seen = 0;
    } combo[3];
    void drop() {
      for (Exec& e : init) if (e.exec) cudaGraphExecDestroy(e.exec);
      for (Exec& e : iter) if (e.exec) cudaGraphExecDestroy(e.exec);
      for (Combo& c : combo) if (c.exec) cudaGraphExecDestroy(c.exec);
      *this = Graphs();
    }
  };
  Graphs graphs[16];
  int next_graph = 0;
  cudaStream_t capture = nullptr;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;           // recorded around the outer operator apply
  cudaEvent_t ev2 = nullptr, ev3 = nullptr;           // around the fine-level smoother apply
  double *lr = nullptr, *lz = nullptr, *lp = nullptr, *lAp = nullptr;  // Lanczos
  LanczosScalars* lanczos = nullptr;            // device scalars, one record per level
  double* partials = nullptr;
  unsigned int* tickets = nullptr;
  int partial_len = 0;
};

namespace {

constexpr int kThreads = 256;

int grid1d(int64_t n) {
  const int64_t g = (n + kThreads - 1) / kThreads;
  return (int)std::max<int64_t>(1, std::min<int64_t>(g, 152 * 8));
}

// Grid of a kernel that moves K entries per thread and iteration (16-byte
// chunks): one thread per chunk up to 8 CTAs per SM.  On a small level a grid
// sized by entries would launch 4x the CTAs, most of them without work.
template <typename T>
int grid_chunks(int64_t n) {
  constexpr int K = 16 / (int)sizeof(T);
  const int64_t g = (n / K + kThreads - 1) / kThreads;
  return (int)std::max<int64_t>(1, std::min<int64_t>(g, 152 * 8));
}

#define GRID_LOOP(i, n)                                                          \
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (n); \
       i += (int64_t)gridDim.x * blockDim.x)

// Whether the solve has ended.  The kernels read the flag beside their data and act on
// it before they store: tested first, its load put one more memory latency in front of
// every kernel.  One PCG iteration, before / now: 3,255 nodes 63.5 / 60.3 us, 2.06 M
// nodes 430 / 422 us.  The kernels of the outer PCG and the FP64 and double-float
// applies test it first: held across the loads it costs them registers (the mixed step
// on 2.06 M nodes, 10 steps, 18.8 ms so and 20.0 ms with the flag read late there too).
__device__ __forceinline__ bool skip(const int* done) { return done != nullptr && *done; }

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// ---------------------------------------------------------------- vectors
// Streaming vector kernels: consecutive entries are handled in 16-byte groups
// (4 floats or 2 doubles) by vector loads and stores, which keeps enough bytes
// in flight per thread to stream at HBM speed; the remaining n % K entries go
// one by one.  Level and workspace vectors come from cudaMalloc (256-byte
// aligned); kernels that also touch a caller's vector take a VEC flag that the
// host sets from the pointers' alignment.
template <typename T, int K>
struct alignas(K * sizeof(T)) Pk {
  T e[K];
};
template <typename T>
__host__ __device__ constexpr int k16() { return 16 / (int)sizeof(T); }

// Grid-stride loops over 16-byte chunks and over the scalar tail.  They stay
// rolled: with grids of 8 CTAs per SM a thread runs only a few iterations, and
// an unrolled body would only raise the register count (to 56-72 registers a
// thread, which halves the resident CTAs) without ever running.
#define GRID_CHUNKS(c, nc)                                                         \
  _Pragma("unroll 1")                                                              \
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < (nc);     \
       c += (int64_t)gridDim.x * blockDim.x)
#define GRID_TAIL(i, start, n)                                                     \
  _Pragma("unroll 1")                                                              \
  for (int64_t i = (start) + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (n); \
       i += (int64_t)gridDim.x * blockDim.x)

template <typename T>
__global__ void k_zero(int64_t n, T* x, const int* done) {
  pdl_wait();
  if (skip(done)) return;
  constexpr int K = k16<T>();
  const int64_t nc = n / K;
  GRID_CHUNKS(c, nc) reinterpret_cast<Pk<T, K>*>(x)[c] = Pk<T, K>{};
  GRID_TAIL(i, nc * K, n) x[i] = T(0);
  pdl_trigger();
}

template <typename T>
__global__ void k_level_inv_diag(int64_t n, double alpha, const double* m, const double* k,
                                 T* inv, double* inv64) {
  pdl_wait();
  GRID_LOOP(i, n) {
    const double v = 1.0 / fma(alpha, m[i], k[i]);
    inv[i] = (T)v;
    inv64[i] = v;
  }
  pdl_trigger();
}

// Chebyshev smoothing in residual form.  A level keeps the residual r of its
// current iterate in place of the right-hand side (the apply subtracts A d from it),
// so no vector t = A x is written, cleared and read back, and the restriction takes
// r as it is.  x takes its corrections two at a time, so a pair of steps moves 10
// vectors where b, t, x, d moved 16, the first two of a zero start 8 instead of 13, the
// last one 5 (its d is not stored).  Fine-level vectors of a V-cycle of degree 6 on
// 2.06 M nodes: 462 MB; 545 with x updated in every step, 768 with b and t.  The
// V-cycle there (bf16 metric): 310 us, 317 with x updated in every step.
//
// First step from zero: d = D^{-1} r / theta (x = d follows with the next step, or
// here with with_x).
template <typename T>
__global__ void k_cheb_zero_start(int64_t n, const T* __restrict__ r, const T* __restrict__ invd,
                                  T* __restrict__ x, T* __restrict__ d, T inv_theta, int with_x, const int* done) {
  pdl_wait();
  const bool stop = skip(done);
  constexpr int K = k16<T>();
  using V = Pk<T, K>;
  const int64_t nc = n / K;
  GRID_CHUNKS(c, nc) {
    const V rr = reinterpret_cast<const V*>(r)[c], ii = reinterpret_cast<const V*>(invd)[c];
    if (stop) return;
    V dd;
#pragma unroll
    for (int k = 0; k < K; ++k) dd.e[k] = ii.e[k] * rr.e[k] * inv_theta;
    reinterpret_cast<V*>(d)[c] = dd;
    if (with_x) reinterpret_cast<V*>(x)[c] = dd;
  }
  GRID_TAIL(i, nc * K, n) {
    const T di = invd[i] * r[i] * inv_theta;
    if (stop) return;
    d[i] = di;
    if (with_x) x[i] = di;
  }
  pdl_trigger();
}

// Chebyshev step from the residual r: d = c1 d + c2 D^{-1} r (kChebFirst: d = c2
// D^{-1} r).  A step reads the d before it in any case, so x takes two corrections
// every second step: it is left alone with kChebDefer, gains old d + d with kChebPair,
// becomes old d + d with kChebStartX (the second step of a zero start) and gains d with
// none of these.  kChebLast: d is not needed any more and not stored.
constexpr int kChebFirst = 1, kChebStartX = 2, kChebLast = 4, kChebDefer = 8, kChebPair = 16;
template <typename T>
__global__ void k_cheb_step(int64_t n, const T* __restrict__ r, const T* __restrict__ invd,
                            T* __restrict__ x, T* __restrict__ d, T c1, T c2, int mode, const int* done) {
  pdl_wait();
  const bool stop = skip(done);
  const bool first = (mode & kChebFirst) != 0, startx = (mode & kChebStartX) != 0, last = (mode & kChebLast) != 0;
  const bool defer = (mode & kChebDefer) != 0, pair = (mode & (kChebPair | kChebStartX)) != 0;
  constexpr int K = k16<T>();
  using V = Pk<T, K>;
  const int64_t nc = n / K;
  GRID_CHUNKS(c, nc) {
    const V rr = reinterpret_cast<const V*>(r)[c], ii = reinterpret_cast<const V*>(invd)[c];
    const V od = first ? V{} : reinterpret_cast<const V*>(d)[c];
    V xx = startx || defer ? V{} : reinterpret_cast<const V*>(x)[c];
    if (stop) return;
    V dd;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      dd.e[k] = first ? c2 * ii.e[k] * rr.e[k] : fma(c1, od.e[k], c2 * ii.e[k] * rr.e[k]);
      xx.e[k] += pair ? od.e[k] + dd.e[k] : dd.e[k];
    }
    if (!last) reinterpret_cast<V*>(d)[c] = dd;
    if (!defer) reinterpret_cast<V*>(x)[c] = xx;
  }
  GRID_TAIL(i, nc * K, n) {
    const T od = first ? T(0) : d[i];
    const T di = first ? c2 * invd[i] * r[i] : fma(c1, od, c2 * invd[i] * r[i]);
    const T xi = startx || defer ? T(0) : x[i];
    if (stop) return;
    if (!last) d[i] = di;
    if (!defer) x[i] = xi + (pair ? od + di : di);
  }
  pdl_trigger();
}

// ---- all Chebyshev steps of a small coarsest level in one CTA
//
// Steps of a level of a few hundred nodes cost two launches each, about 1 us a launch
// whatever the level's size.  One CTA of kCoarseThreads threads runs all of them with
// everything on chip: the metric (in its storage type, word by word across the
// elements so that the lanes' reads do not conflict), d and the element results in
// shared memory, r, x, 1 / diagonal and the elements' node numbers in registers.  A
// step is two phases between barriers: every thread evaluates its elements (Q_1 in
// registers); every thread sums the results of its nodes' elements in a fixed order
// (the deterministic mode needs no variant) and updates.  The metric is copied before
// the wait for the previous kernel.  The launcher takes it for a Q_1 level in FP32 of
// at most kCoarseNodes nodes whose metric fits.  One PCG iteration, before / now,
// with coarsest levels of 608, 108, 30 and 990 nodes: 113 / 102, 145 / 125, 103 / 81,
// 437 / 430 us (degree 10, with the one-launch restriction below).  (With the metric read from L1 at every step, lane by lane, a step of the
// 608-node level took as long as its two launches.)
constexpr int kCoarseThreads = 512, kCoarseNodes = 1024, kCoarsePer = kCoarseNodes / kCoarseThreads;
constexpr int kCoarseDegree = 200;
constexpr size_t kCoarseSmem = 227 * 1024;

struct ChebCoef {
  float c1[kCoarseDegree], c2[kCoarseDegree];
};

// Shared-memory words of an element's metric: 56 values of the storage type.
template <typename MT> __host__ __device__ constexpr int coarse_words() { return 56 * (int)sizeof(MT) / 4; }
__device__ __forceinline__ void coarse_point(const unsigned* w, int nep, int pt, float (&G)[kMetricComps],
                                             const __nv_bfloat16*) {
#pragma unroll
  for (int c = 0; c < kMetricComps; ++c) {
    const int v = kMetricComps * pt + c;
    const unsigned u = w[(v >> 1) * nep];
    G[c] = __uint_as_float((v & 1) ? u & 0xffff0000u : u << 16);
  }
}
__device__ __forceinline__ void coarse_point(const unsigned* w, int nep, int pt, float (&G)[kMetricComps], const float*) {
#pragma unroll
  for (int c = 0; c < kMetricComps; ++c) G[c] = __uint_as_float(w[(kMetricComps * pt + c) * nep]);
}

// Element results y = (mass M + K) u of one Q_1 element, in place; w: its first
// metric word, nep words between its words.
template <int QUAD, typename MT>
__device__ __forceinline__ void q1_element(const KTab<2, float>& tab, const unsigned* w, int nep, float mass,
                                           float (&u)[8]) {
  // f(node, node) for the four lines of a direction; nodes a = i + 2 j + 4 k
  auto lines = [](int dir, auto f) {
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const int base = dir == 0 ? 2 * l : dir == 1 ? (l & 1) + 4 * (l >> 1) : l;
      f(base, base + (1 << dir));
    }
  };
  auto interpolate = [&](const EoMat<2, float>& M) {
#pragma unroll
    for (int dir = 0; dir < 3; ++dir)
      lines(dir, [&](int p, int q) {
        const float in[2] = {u[p], u[q]};
        float out[2];
        eo_line<2, false, false>(M, in, out);
        u[p] = out[0];
        u[q] = out[1];
      });
  };
  if (QUAD == SEM_QUAD_LG) interpolate(tab.Bi);
  float g[3][8];
#pragma unroll
  for (int dir = 0; dir < 3; ++dir)
    lines(dir, [&](int p, int q) {
      const float in[2] = {u[p], u[q]};
      float out[2];
      eo_line<2, true, false>(tab.D, in, out);
      g[dir][p] = out[0];
      g[dir][q] = out[1];
    });
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    float G[kMetricComps];
    coarse_point(w, nep, a, G, static_cast<const MT*>(nullptr));
    const float x = g[0][a], y = g[1][a], z = g[2][a];
    g[0][a] = fmaf(G[2], z, fmaf(G[1], y, G[0] * x));
    g[1][a] = fmaf(G[4], z, fmaf(G[3], y, G[1] * x));
    g[2][a] = fmaf(G[5], z, fmaf(G[4], y, G[2] * x));
    u[a] = (mass * G[6]) * u[a];
  }
#pragma unroll
  for (int dir = 2; dir >= 0; --dir)
    lines(dir, [&](int p, int q) {
      const float in[2] = {g[dir][p], g[dir][q]};
      float out[2] = {u[p], u[q]};
      eo_line<2, true, true>(tab.Dt, in, out);
      u[p] = out[0];
      u[q] = out[1];
    });
  if (QUAD == SEM_QUAD_LG) interpolate(tab.Bit);
}

template <int QUAD, typename MT>
__global__ void __launch_bounds__(kCoarseThreads, 1)
    k_cheb_coarse(int nx, int ny, int nz, const int* __restrict__ map, const MT* __restrict__ metric, float mass,
                  const __grid_constant__ KTab<2, float> tab, const __grid_constant__ ChebCoef cf, int degree,
                  const float* __restrict__ rhs, const float* __restrict__ invd, float* __restrict__ x_out,
                  int64_t ndofs, unsigned long long* dbg, const int* done) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int W = coarse_words<MT>();
  static_assert(MetricLayout<MT>::unit(2) * 2 * MetricLayout<MT>::stride(2) == MetricLayout<MT>::chunk(2) &&
                    2 * MetricLayout<MT>::stride(2) == 56, "the elements' 56 values follow one another at n = 2");
  const int n = (nx + 1) * (ny + 1) * (nz + 1), ne = nx * ny * nz, nep = ne | 1;
  float* sd = reinterpret_cast<float*>(smem_raw);  // d on the nodes
  float* sy = sd + n;                              // element results [8][nep]
  unsigned* sm = reinterpret_cast<unsigned*>(sy + 8 * nep);  // metric [W][nep]
  const unsigned* gm = reinterpret_cast<const unsigned*>(metric);
#pragma unroll 8
  for (int t = threadIdx.x; t < ne * W; t += kCoarseThreads) sm[(t % W) * nep + t / W] = __ldg(gm + t);
  unsigned short node[kCoarsePer][8];
#pragma unroll
  for (int q = 0; q < kCoarsePer; ++q) {
    const int e = threadIdx.x + q * kCoarseThreads;
#pragma unroll
    for (int a = 0; a < 8; ++a)
      node[q][a] = e < ne ? (unsigned short)SEM_IDX(__ldg(map + 8 * e + a), ndofs, dbg, kDbgGather) : 0;
  }
  pdl_wait();
  const bool stop = skip(done);
  float r[kCoarsePer], x[kCoarsePer], inv[kCoarsePer];
  const float c0 = cf.c2[0];  // 1 / theta
#pragma unroll
  for (int t = 0; t < kCoarsePer; ++t) {
    const int i = threadIdx.x + t * kCoarseThreads;
    if (i < n) {
      r[t] = rhs[i];
      inv[t] = invd[i];
      x[t] = inv[t] * r[t] * c0;
      sd[i] = x[t];
    }
  }
  if (stop) return;
  __syncthreads();
#pragma unroll 1
  for (int s = 1; s < degree; ++s) {
#pragma unroll
    for (int q = 0; q < kCoarsePer; ++q) {
      const int e = threadIdx.x + q * kCoarseThreads;
      if (e < ne) {
        float u[8];
#pragma unroll
        for (int a = 0; a < 8; ++a) u[a] = sd[node[q][a]];
        q1_element<QUAD, MT>(tab, sm + e, nep, mass, u);
#pragma unroll
        for (int a = 0; a < 8; ++a) sy[a * nep + e] = u[a];
      }
    }
    __syncthreads();
    const float c1 = cf.c1[s], c2 = cf.c2[s];
#pragma unroll
    for (int t = 0; t < kCoarsePer; ++t) {
      const int i = threadIdx.x + t * kCoarseThreads;
      if (i < n) {
        const int I = i % (nx + 1), J = i / (nx + 1) % (ny + 1), K = i / ((nx + 1) * (ny + 1));
        float y = 0.f;
#pragma unroll
        for (int a = 7; a >= 0; --a) {  // the node is local node a of the element below it by a's bits
          const int ex = I - (a & 1), ey = J - (a >> 1 & 1), ez = K - (a >> 2);
          if (ex >= 0 && ex < nx && ey >= 0 && ey < ny && ez >= 0 && ez < nz)
            y += sy[a * nep + ex + nx * (ey + ny * ez)];
        }
        r[t] -= y;
        const float d = fmaf(c1, sd[i], c2 * inv[t] * r[t]);
        sd[i] = d;
        x[t] += d;
      }
    }
    __syncthreads();
  }
  pdl_trigger();
#pragma unroll
  for (int t = 0; t < kCoarsePer; ++t) {
    const int i = threadIdx.x + t * kCoarseThreads;
    if (i < n) x_out[i] = x[t];
  }
}

template <typename MT>
size_t coarse_smem(const Level& L) {
  const size_t nep = (size_t)L.nelem | 1;
  return 4 * ((size_t)L.ndofs + 8 * nep + coarse_words<MT>() * nep);
}
cudaError_t prime_coarse() {
  auto set = [](auto kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCoarseSmem);
  };
  cudaError_t e = set(k_cheb_coarse<SEM_QUAD_LG, float>);
  if (e == cudaSuccess) e = set(k_cheb_coarse<SEM_QUAD_LGL, float>);
  if (e == cudaSuccess) e = set(k_cheb_coarse<SEM_QUAD_LG, __nv_bfloat16>);
  if (e == cudaSuccess) e = set(k_cheb_coarse<SEM_QUAD_LGL, __nv_bfloat16>);
  return e;
}

// ---------------------------------------------------------------- transfers
struct PTab {
  int nf, nc;
  double P[kMaxN][kMaxN];  // P[i][a] = l^c_a(x^f_i)
};

// Coarse vertex k (and k+1) and weights of fine vertex I along one direction.
__device__ __forceinline__ void hweights(int I, int nf, int nc, int& k, double& w0, double& w1) {
  k = min(I / 2, nc - 1);
  const int t = I - 2 * k;
  if (2 * k + 2 <= nf) {  // coarse element made of two fine elements
    w0 = t == 0 ? 1.0 : (t == 1 ? 0.5 : 0.0);
  } else {                // trailing single fine element
    w0 = t == 0 ? 1.0 : 0.0;
  }
  w1 = 1.0 - w0;
}

template <typename T>
__global__ void k_prolong_h(int nfx, int nfy, int nfz, int ncx, int ncy, int ncz,
                            const T* __restrict__ xc, T* __restrict__ xf, T* __restrict__ df,
                            const int* done) {
  pdl_wait();
  const bool stop = skip(done);
  // node numbers are 32-bit (checked by sem_create): 32-bit divisions
  const unsigned NX = nfx + 1, NY = nfy + 1, n = NX * NY * (nfz + 1);
  const int64_t CX = ncx + 1, CY = ncy + 1;
  for (unsigned g = blockIdx.x * blockDim.x + threadIdx.x; g < n; g += gridDim.x * blockDim.x) {
    const int I = (int)(g % NX), J = (int)(g / NX % NY), K = (int)(g / NX / NY);
    int kx, ky, kz;
    double wx[2], wy[2], wz[2];
    hweights(I, nfx, ncx, kx, wx[0], wx[1]);
    hweights(J, nfy, ncy, ky, wy[0], wy[1]);
    hweights(K, nfz, ncz, kz, wz[0], wz[1]);
    const T x = xf[g];
    T v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {  // all loads in flight
      const int a = q & 1, b = q >> 1 & 1, c = q >> 2;
      v[q] = (wx[a] != 0.0 && wy[b] != 0.0 && wz[c] != 0.0) ? xc[(kx + a) + CX * ((ky + b) + CY * (kz + c))] : T(0);
    }
    T s = T(0);
#pragma unroll
    for (int q = 0; q < 8; ++q) s = fma((T)wx[q & 1] * (T)wy[q >> 1 & 1] * (T)wz[q >> 2], v[q], s);  // exact weights
    if (stop) return;
    xf[g] = x + s;
    df[g] = s;
  }
  pdl_trigger();
}

// Restriction gathered per coarse node: the fine nodes within 1 of 2 C in each
// direction (also at a trailing single element), in a fixed order, weighted by the
// trilinear prolongation's weight of that coarse node.  Every coarse node is written
// once: nothing is cleared before and the result is the same in every run.
template <typename T>
__global__ void k_restrict_h(int nfx, int nfy, int nfz, int ncx, int ncy, int ncz,
                             const T* __restrict__ rf, T* __restrict__ rc, const int* done) {
  pdl_wait();
  const bool stop = skip(done);
  const int64_t NX = nfx + 1, NY = nfy + 1;
  const unsigned CX = ncx + 1, CY = ncy + 1, nc = CX * CY * (ncz + 1);
  for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x) {
    const int CI = (int)(c % CX), CJ = (int)(c / CX % CY), CK = (int)(c / CX / CY);
    // weights of the fine nodes 2 C - 1, 2 C, 2 C + 1: 1/2 beside C, 1 on it; a trailing
    // single element has its only inner neighbour at the mesh's end, weight 1
    auto weights = [](int C, int nf, T (&w)[3]) {
      const bool odd_end = 2 * C > nf;  // C is the closing node of an odd nf: fine node nf is 2 C - 1
      w[0] = C == 0 ? T(0) : (odd_end ? T(1) : T(0.5));
      w[1] = odd_end ? T(0) : T(1);
      w[2] = 2 * C + 2 <= nf ? T(0.5) : T(0);
    };
    T wx[3], wy[3], wz[3], v[27];
    weights(CI, nfx, wx);
    weights(CJ, nfy, wy);
    weights(CK, nfz, wz);
    const int64_t base = (2 * CI - 1) + NX * ((2 * CJ - 1) + NY * (int64_t)(2 * CK - 1));
#pragma unroll
    for (int a = 0; a < 27; ++a) {  // all loads in flight
      const int i = a % 3, j = a / 3 % 3, k = a / 9;
      v[a] = (wx[i] != T(0) && wy[j] != T(0) && wz[k] != T(0)) ? rf[base + i + NX * (j + NY * (int64_t)k)] : T(0);
    }
    T acc = T(0);
#pragma unroll
    for (int a = 0; a < 27; ++a) acc = fma(wx[a % 3] * wy[a / 3 % 3] * wz[a / 9], v[a], acc);
    if (stop) return;
    rc[c] = acc;
  }
  pdl_trigger();
}

__global__ void k_coarse_tissue(int ncx, int ncy, int ncz, int nfx, int nfy, const double* sl,
                                const double* st, const double* th, double* csl, double* cst,
                                double* cth) {
  pdl_wait();
  const int64_t n = (int64_t)ncx * ncy * ncz;
  GRID_LOOP(e, n) {
    const int kx = (int)(e % ncx), ky = (int)((e / ncx) % ncy), kz = (int)(e / ((int64_t)ncx * ncy));
    const int64_t f = 2 * kx + (int64_t)nfx * (2 * ky + (int64_t)nfy * 2 * kz);
    csl[e] = sl[f];
    cst[e] = st[f];
    cth[e] = th[f];
  }
  pdl_trigger();
}

// ---------------------------------------------------------------- reductions
// Lanczos estimate of one level: ten Jacobi-PCG steps with their scalars on the
// device, read by the host once for all levels.  The kernels return at once when a
// step found a scalar that is not positive (the estimate then has fewer steps).

// r = start vector, z = D^{-1} r, p = z, Ap = 0; r . z.
__global__ void k_lanczos_start(int64_t n, const double* __restrict__ dinv, double* __restrict__ r,
                                double* __restrict__ p, double* __restrict__ Ap, LanczosScalars* sc, double* partials,
                                unsigned int* ticket) {
  pdl_wait();
  __shared__ double red[32];
  double v = 0.0;
  GRID_LOOP(i, n) {
    const unsigned long long h = ((unsigned long long)i * 2654435761ull) & 0xffffffffull;
    const double ri = (double)h / 4294967296.0 - 0.5, zi = dinv[i] * ri;
    r[i] = ri;
    p[i] = zi;
    Ap[i] = 0.0;
    v = fma(ri, zi, v);
  }
  pdl_trigger();
  v = block_sum(v, red);
  double total;
  if (finish_reduction(v, partials, ticket, &total, red)) {
    sc->rz = total;
    sc->m = 0;
    sc->stop = 0;
  }
}

// p . Ap and the step length.
__global__ void k_lanczos_dot(int64_t n, const double* __restrict__ p, const double* __restrict__ Ap,
                              LanczosScalars* sc, double* partials, unsigned int* ticket) {
  pdl_wait();
  if (sc->stop) return;
  __shared__ double red[32];
  double v = 0.0;
  GRID_LOOP(i, n) v = fma(p[i], Ap[i], v);
  pdl_trigger();
  v = block_sum(v, red);
  double total;
  if (finish_reduction(v, partials, ticket, &total, red)) {
    if (total > 0.0 && sc->rz > 0.0) sc->a = sc->rz / total;
    else sc->stop = 1;
  }
}

// r -= a Ap, z = D^{-1} r; r . z, the conjugation coefficient, the step's record.
__global__ void k_lanczos_update(int64_t n, const double* __restrict__ Ap, double* __restrict__ r,
                                 const double* __restrict__ dinv, double* __restrict__ z, LanczosScalars* sc,
                                 double* partials, unsigned int* ticket) {
  pdl_wait();
  if (sc->stop) return;
  const double a = sc->a;
  __shared__ double red[32];
  double v = 0.0;
  GRID_LOOP(i, n) {
    const double ri = fma(-a, Ap[i], r[i]), zi = dinv[i] * ri;
    r[i] = ri;
    z[i] = zi;
    v = fma(ri, zi, v);
  }
  pdl_trigger();
  v = block_sum(v, red);
  double total;
  if (finish_reduction(v, partials, ticket, &total, red)) {
    const int m = sc->m;
    sc->alpha[m] = a;
    sc->b = sc->beta[m] = total / sc->rz;
    sc->rz = total;
    sc->m = m + 1;
    if (!(total > 0.0)) sc->stop = 1;
  }
}

__global__ void k_lanczos_p(int64_t n, const double* __restrict__ z, double* __restrict__ p, double* __restrict__ Ap,
                            const LanczosScalars* sc) {
  pdl_wait();
  if (sc->stop) return;
  const double b = sc->b;
  GRID_LOOP(i, n) {
    p[i] = fma(b, p[i], z[i]);
    Ap[i] = 0.0;
  }
  pdl_trigger();
}

// ---------------------------------------------------------------- outer flexible PCG
template <int K>
__device__ __forceinline__ bool grid_sums_k(double (&v)[K], double* partials, int stride,
                                            unsigned int* ticket, double (&tot)[K]) {
  __shared__ double red[K][32];
  __shared__ bool is_last;
  double bs[K];
#pragma unroll
  for (int k = 0; k < K; ++k) bs[k] = block_sum(v[k], red[k]);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) partials[k * stride + blockIdx.x] = bs[k];
    __threadfence();
    const unsigned int t = atomicAdd(ticket, 1u);
    is_last = (t == gridDim.x - 1);
  }
  __syncthreads();
  if (!is_last) return false;
  __threadfence();
#pragma unroll
  for (int k = 0; k < K; ++k) {
    double s = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x)
      s += ((volatile double*)partials)[k * stride + b];
    tot[k] = block_sum(s, red[k]);
    __syncthreads();
  }
  if (threadIdx.x == 0) *ticket = 0u;
  return threadIdx.x == 0;
}

// r = b - Ap, Ap = 0, b0 = (T) r; r.r, b.b; stopping threshold.  VEC: b is
// 16-byte aligned (pairs of entries by 16-byte accesses).
template <typename T, bool VEC>
__global__ void k_fpcg_init(int64_t n, const double* __restrict__ b, double* Ap_main, double* Ap_alt,
                            const int* use_main, double* __restrict__ r, T* __restrict__ b0, CgScalars* cg,
                            double* partials, int stride, unsigned int* ticket, double rtol,
                            double atol) {
  pdl_wait();
  // A x: Ap_main, or Ap_alt where the flag use_main reads zero
  double* __restrict__ Ap = (use_main == nullptr || *use_main != 0) ? Ap_main : Ap_alt;
  double v[2] = {0.0, 0.0};
  const int64_t nc = VEC ? n / 2 : 0;
  GRID_CHUNKS(c, nc) {
    const Pk<double, 2> bb = reinterpret_cast<const Pk<double, 2>*>(b)[c];
    const Pk<double, 2> aa = reinterpret_cast<const Pk<double, 2>*>(Ap)[c];
    Pk<double, 2> rr;
    Pk<T, 2> rb;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      rr.e[k] = bb.e[k] - aa.e[k];
      rb.e[k] = (T)rr.e[k];
      v[0] = fma(rr.e[k], rr.e[k], v[0]);
      v[1] = fma(bb.e[k], bb.e[k], v[1]);
    }
    reinterpret_cast<Pk<double, 2>*>(r)[c] = rr;
    reinterpret_cast<Pk<double, 2>*>(Ap)[c] = Pk<double, 2>{};
    reinterpret_cast<Pk<T, 2>*>(b0)[c] = rb;
  }
  GRID_TAIL(i, nc * 2, n) {
    const double bi = b[i];
    const double ri = bi - Ap[i];
    r[i] = ri;
    Ap[i] = 0.0;
    b0[i] = (T)ri;
    v[0] = fma(ri, ri, v[0]);
    v[1] = fma(bi, bi, v[1]);
  }
  pdl_trigger();
  double tot[2];
  if (grid_sums_k<2>(v, partials, stride, ticket, tot)) {
    cg->rr = tot[0];
    cg->bb = tot[1];
    cg->tol2 = fmax(rtol * rtol * tot[1], atol * atol);
    cg->iters = 0;
    cg->status = 0;
    const bool finite = isfinite(tot[0]) && isfinite(tot[1]);
    if (!finite) cg->status = SEM_ERR_NONFINITE;
    cg->done = (!finite || tot[0] <= cg->tol2) ? 1 : 0;
  }
}

// z_new = (double) x0; first iteration (no iteration finished yet): p = z_new,
// rz = r.z_new; else beta = (r.z_new - r.z_old) / rz, rz = r.z_new (z holds
// z_old on entry).  Pairs of entries by 16-byte (8-byte for float x0) accesses.
// With p2 set, p is also written there as float pairs.
template <typename T>
__global__ void k_fpcg_z(int64_t n, const T* __restrict__ x0, double* __restrict__ z,
                         const double* __restrict__ r, double* __restrict__ p, df_pair* __restrict__ p2,
                         CgScalars* cg, double* partials, int stride, unsigned int* ticket) {
  pdl_wait();
  if (cg->done) return;
  const bool first = cg->iters == 0;
  double v[2] = {0.0, 0.0};
  using D2 = Pk<double, 2>;
  const int64_t nc = n / 2;
  GRID_CHUNKS(c, nc) {
    const Pk<T, 2> xx = reinterpret_cast<const Pk<T, 2>*>(x0)[c];
    const D2 rr = reinterpret_cast<const D2*>(r)[c];
    const D2 zo = first ? D2{} : reinterpret_cast<const D2*>(z)[c];
    D2 zn;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      zn.e[k] = (double)xx.e[k];
      if (!first) v[1] = fma(rr.e[k], zo.e[k], v[1]);
      v[0] = fma(rr.e[k], zn.e[k], v[0]);
    }
    if (first) {
      reinterpret_cast<D2*>(p)[c] = zn;
      if (p2 != nullptr) {
        const df_pair a0 = split_pair(zn.e[0]), a1 = split_pair(zn.e[1]);
        reinterpret_cast<float4*>(p2)[c] = make_float4(a0.h, a0.l, a1.h, a1.l);
      }
    }
    reinterpret_cast<D2*>(z)[c] = zn;
  }
  GRID_TAIL(i, nc * 2, n) {
    const double zi = (double)x0[i];
    const double ri = r[i];
    if (first) {
      p[i] = zi;
      if (p2 != nullptr) p2[i] = split_pair(zi);
    } else {
      v[1] = fma(ri, z[i], v[1]);
    }
    z[i] = zi;
    v[0] = fma(ri, zi, v[0]);
  }
  pdl_trigger();
  double tot[2];
  if (grid_sums_k<2>(v, partials, stride, ticket, tot)) {
    if (first) {
      cg->beta = 0.0;
    } else {
      cg->beta = (tot[0] - tot[1]) / cg->rz;
    }
    cg->rz = tot[0];
    if (!isfinite(tot[0]) || !isfinite(tot[1])) {
      cg->status = SEM_ERR_NONFINITE;
      cg->done = 1;
    }
  }
}

__global__ void k_fpcg_p(int64_t n, const double* __restrict__ z, double* __restrict__ p,
                         df_pair* __restrict__ p2, const CgScalars* cg) {
  pdl_wait();
  if (cg->done || cg->iters == 0) return;  // first iteration: k_fpcg_z set p = z
  const double beta = cg->beta;
  using D2 = Pk<double, 2>;
  const int64_t nc = n / 2;
  GRID_CHUNKS(c, nc) {
    const D2 zz = reinterpret_cast<const D2*>(z)[c];
    D2 pp = reinterpret_cast<const D2*>(p)[c];
#pragma unroll
    for (int k = 0; k < 2; ++k) pp.e[k] = fma(beta, pp.e[k], zz.e[k]);
    reinterpret_cast<D2*>(p)[c] = pp;
    if (p2 != nullptr) {
      const df_pair a0 = split_pair(pp.e[0]), a1 = split_pair(pp.e[1]);
      reinterpret_cast<float4*>(p2)[c] = make_float4(a0.h, a0.l, a1.h, a1.l);
    }
  }
  GRID_TAIL(i, nc * 2, n) {
    const double pi = fma(beta, p[i], z[i]);
    p[i] = pi;
    if (p2 != nullptr) p2[i] = split_pair(pi);
  }
  pdl_trigger();
}

// x += alpha p, r -= alpha Ap, Ap = 0, b0 = (T) r; r.r; convergence.  VEC: x is
// 16-byte aligned.
template <typename T, bool VEC>
__global__ void k_fpcg_xr(int64_t n, double* __restrict__ x, const double* __restrict__ p,
                          double* __restrict__ Ap, double* __restrict__ r, T* __restrict__ b0,
                          CgScalars* cg, double* partials, int stride, unsigned int* ticket) {
  pdl_wait();
  if (cg->done) return;
  const double alpha = cg->alpha;
  double v[1] = {0.0};
  using D2 = Pk<double, 2>;
  const int64_t nc = VEC ? n / 2 : 0;
  GRID_CHUNKS(c, nc) {
    D2 xx = reinterpret_cast<const D2*>(x)[c];
    const D2 pp = reinterpret_cast<const D2*>(p)[c];
    const D2 aa = reinterpret_cast<const D2*>(Ap)[c];
    D2 rr = reinterpret_cast<const D2*>(r)[c];
    Pk<T, 2> rb;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      xx.e[k] = fma(alpha, pp.e[k], xx.e[k]);
      rr.e[k] = fma(-alpha, aa.e[k], rr.e[k]);
      rb.e[k] = (T)rr.e[k];
      v[0] = fma(rr.e[k], rr.e[k], v[0]);
    }
    reinterpret_cast<D2*>(x)[c] = xx;
    reinterpret_cast<D2*>(r)[c] = rr;
    reinterpret_cast<D2*>(Ap)[c] = D2{};
    reinterpret_cast<Pk<T, 2>*>(b0)[c] = rb;
  }
  GRID_TAIL(i, nc * 2, n) {
    x[i] = fma(alpha, p[i], x[i]);
    const double ri = fma(-alpha, Ap[i], r[i]);
    r[i] = ri;
    Ap[i] = 0.0;
    b0[i] = (T)ri;
    v[0] = fma(ri, ri, v[0]);
  }
  pdl_trigger();
  double tot[1];
  if (grid_sums_k<1>(v, partials, stride, ticket, tot)) {
    cg->rr = tot[0];
    cg->iters += 1;
    if (!isfinite(tot[0]) || !isfinite(alpha)) {
      cg->status = SEM_ERR_NONFINITE;
      cg->done = 1;
    } else if (tot[0] <= cg->tol2) {
      cg->done = 1;
    }
  }
}

// ---- the same flexible PCG with the double-float operator: r and p are kept
// as float pairs, z as the V-cycle's own values (type T), and their updates and
// inner products run in double-float arithmetic on the FP32 pipe; only x, the
// caller's FP64 solution, is updated by FP64 instructions (one DFMA and one
// addition per entry).  GB300 issues two FP64 operations per clock per SM, which
// bound the FP64 forms of these kernels (FP64 pipe 76 % busy).

// double-float value of a T (exact for float)
__device__ __forceinline__ df df_of(float v) { return df(v, 0.f); }
__device__ __forceinline__ df df_of(double v) { return dfd(v); }
// T-rounded high part for the V-cycle's right-hand side
template <typename T> __device__ __forceinline__ T t_of(df v);
template <> __device__ __forceinline__ float t_of<float>(df v) { return v.h; }
template <> __device__ __forceinline__ double t_of<double>(df v) { return df_to_double(v); }

// Block sum of double-float values: the warps add in double-float (FP32
// shuffles), each warp's sum becomes a double once, and warp 0 adds those.
__device__ __forceinline__ double block_sum_df(df v, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float h = __shfl_down_sync(0xffffffffu, v.h, o), l = __shfl_down_sync(0xffffffffu, v.l, o);
    v = v + df(h, l);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) red[warp] = (double)v.h + (double)v.l;
  __syncthreads();
  double d = 0.0;
  if (warp == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    d = (lane < nw) ? red[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d += __shfl_down_sync(0xffffffffu, d, o);
  }
  return d;
}

// grid_sums_k with double-float per-thread values.
template <int K>
__device__ __forceinline__ bool grid_sums_df(df (&v)[K], double* partials, int stride, unsigned int* ticket,
                                             double (&tot)[K]) {
  __shared__ double red[K][32];
  __shared__ bool is_last;
  double bs[K];
#pragma unroll
  for (int k = 0; k < K; ++k) bs[k] = block_sum_df(v[k], red[k]);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) partials[k * stride + blockIdx.x] = bs[k];
    __threadfence();
    const unsigned int t = atomicAdd(ticket, 1u);
    is_last = (t == gridDim.x - 1);
  }
  __syncthreads();
  if (!is_last) return false;
  __threadfence();
#pragma unroll
  for (int k = 0; k < K; ++k) {
    double s = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x)
      s += ((volatile double*)partials)[k * stride + b];
    tot[k] = block_sum(s, red[k]);
    __syncthreads();
  }
  if (threadIdx.x == 0) *ticket = 0u;
  return threadIdx.x == 0;
}

// The double-float PCG kernels move two entries per thread and iteration
// (16-byte accesses to FP64 and float-pair vectors) and the odd last entry
// alone.  Workspace and level vectors come from cudaMalloc; VEC is false when a
// caller's FP64 vector is not 16-byte aligned (then every entry goes the scalar
// way).  8 CTAs of 256 threads per SM stay resident (32 registers); 6 for
// k_dfpcg_xr (40 registers: at 32 it spills), whose grid is sized to match.
template <typename T> using C2 = Pk<T, 2>;
constexpr int kXrCtasPerSm = 6;

// one entry of the set-up: r = b - A x (pairs), b0 = r rounded to T
template <typename T>
__device__ __forceinline__ void init_entry(double bi, df ax, df_pair& r2, T& b0, df (&v)[2]) {
  const df bd = dfd(bi);
  const df r = dfnorm(bd - ax);
  r2 = df_pair{r.h, r.l};
  b0 = t_of<T>(r);
  v[0] = fma(r, r, v[0]);
  v[1] = fma(bd, bd, v[1]);
}

// r = b - A x, b0 = r; r.r, b.b; stopping threshold.  A x is the FP64 result of
// an apply in Ap (zeroed here), or the carried float pairs in ax2_in (Ap is then
// already zero).
template <typename T, bool VEC>
__global__ void __launch_bounds__(kThreads, 8)
    k_dfpcg_init(int64_t n, const double* __restrict__ b, double* __restrict__ Ap,
                 const df_pair* __restrict__ ax2_in, const int* ax2_ok, df_pair* __restrict__ r2,
                 T* __restrict__ b0, CgScalars* cg, double* partials, int stride, unsigned int* ticket,
                 double rtol, double atol) {
  pdl_wait();
  // the carried pairs, unless the flag ax2_ok reads zero (then A x is in Ap)
  const df_pair* __restrict__ ax2 = (ax2_ok == nullptr || *ax2_ok != 0) ? ax2_in : nullptr;
  df v[2] = {df(0.f, 0.f), df(0.f, 0.f)};
  const int64_t nc = VEC ? n / 2 : 0;
  GRID_CHUNKS(c, nc) {
    const C2<double> bb = reinterpret_cast<const C2<double>*>(b)[c];
    C2<df_pair> ax, rr;
    C2<double> aa;
    if (ax2 != nullptr) {
      ax = reinterpret_cast<const C2<df_pair>*>(ax2)[c];
    } else {
      aa = reinterpret_cast<const C2<double>*>(Ap)[c];
      reinterpret_cast<C2<double>*>(Ap)[c] = C2<double>{};
    }
    C2<T> rb;
#pragma unroll
    for (int k = 0; k < 2; ++k)
      init_entry(bb.e[k], ax2 != nullptr ? df(ax.e[k].h, ax.e[k].l) : dfd(aa.e[k]), rr.e[k], rb.e[k], v);
    reinterpret_cast<C2<df_pair>*>(r2)[c] = rr;
    reinterpret_cast<C2<T>*>(b0)[c] = rb;
  }
  GRID_TAIL(i, nc * 2, n) {
    df ax;
    if (ax2 != nullptr) {
      ax = df(ax2[i].h, ax2[i].l);
    } else {
      ax = dfd(Ap[i]);
      Ap[i] = 0.0;
    }
    init_entry(b[i], ax, r2[i], b0[i], v);
  }
  pdl_trigger();
  double tot[2];
  if (grid_sums_df<2>(v, partials, stride, ticket, tot)) {
    cg->rr = tot[0];
    cg->bb = tot[1];
    cg->tol2 = fmax(rtol * rtol * tot[1], atol * atol);
    cg->iters = 0;
    cg->status = 0;
    const bool finite = isfinite(tot[0]) && isfinite(tot[1]);
    if (!finite) cg->status = SEM_ERR_NONFINITE;
    cg->done = (!finite || tot[0] <= cg->tol2) ? 1 : 0;
  }
}

// z_new = the V-cycle's result (kept in zs, which holds z_old on entry); first
// iteration: p = z_new, rz = r.z_new; else beta = (r.z_new - r.z_old) / rz, rz = r.z_new.
template <typename T>
__device__ __forceinline__ void z_entry(T z, T& zs, df_pair rp, df_pair& p2, bool first, df (&v)[2]) {
  const df r(rp.h, rp.l), zd = df_of(z);
  v[0] = fma(r, zd, v[0]);
  if (first) p2 = df_pair{zd.h, zd.l};
  else v[1] = fma(r, df_of(zs), v[1]);
  zs = z;
}

template <typename T>
__global__ void __launch_bounds__(kThreads, 8)
    k_dfpcg_z(int64_t n, const T* __restrict__ x0, T* __restrict__ zs, const df_pair* __restrict__ r2,
              df_pair* __restrict__ p2, CgScalars* cg, double* partials, int stride, unsigned int* ticket) {
  pdl_wait();
  if (cg->done) return;
  const bool first = cg->iters == 0;
  df v[2] = {df(0.f, 0.f), df(0.f, 0.f)};
  const int64_t nc = n / 2;
  GRID_CHUNKS(c, nc) {
    const C2<T> z = reinterpret_cast<const C2<T>*>(x0)[c];
    C2<T> zz = reinterpret_cast<const C2<T>*>(zs)[c];
    const C2<df_pair> rr = reinterpret_cast<const C2<df_pair>*>(r2)[c];
    C2<df_pair> pp;
#pragma unroll
    for (int k = 0; k < 2; ++k) z_entry(z.e[k], zz.e[k], rr.e[k], pp.e[k], first, v);
    reinterpret_cast<C2<T>*>(zs)[c] = zz;
    if (first) reinterpret_cast<C2<df_pair>*>(p2)[c] = pp;
  }
  GRID_TAIL(i, nc * 2, n) {
    df_pair pp;
    z_entry(x0[i], zs[i], r2[i], pp, first, v);
    if (first) p2[i] = pp;
  }
  pdl_trigger();
  double tot[2];
  if (grid_sums_df<2>(v, partials, stride, ticket, tot)) {
    cg->beta = first ? 0.0 : (tot[0] - tot[1]) / cg->rz;
    cg->rz = tot[0];
    if (!isfinite(tot[0]) || !isfinite(tot[1])) {
      cg->status = SEM_ERR_NONFINITE;
      cg->done = 1;
    }
  }
}

// p = z + beta p (float pairs)
template <typename T>
__device__ __forceinline__ df_pair p_entry(df beta, df_pair pp, T z) {
  const df pn = dfnorm(fma(beta, df(pp.h, pp.l), df_of(z)));
  return df_pair{pn.h, pn.l};
}

template <typename T>
__global__ void __launch_bounds__(kThreads, 8)
    k_dfpcg_p(int64_t n, const T* __restrict__ zs, df_pair* __restrict__ p2, const CgScalars* cg) {
  pdl_wait();
  if (cg->done || cg->iters == 0) return;  // first iteration: k_dfpcg_z set p = z
  const df beta = dfd(cg->beta);
  const int64_t nc = n / 2;
  GRID_CHUNKS(c, nc) {
    const C2<T> zz = reinterpret_cast<const C2<T>*>(zs)[c];
    C2<df_pair> pp = reinterpret_cast<const C2<df_pair>*>(p2)[c];
#pragma unroll
    for (int k = 0; k < 2; ++k) pp.e[k] = p_entry(beta, pp.e[k], zz.e[k]);
    reinterpret_cast<C2<df_pair>*>(p2)[c] = pp;
  }
  GRID_TAIL(i, nc * 2, n) p2[i] = p_entry(beta, p2[i], zs[i]);
  pdl_trigger();
}

// x += alpha p (FP64), r -= alpha Ap, Ap = 0, b0 = r; r.r; convergence.
template <typename T>
__device__ __forceinline__ T xr_entry(double alpha, df nalpha, df_pair pp, double& x, double& ap, df_pair& r2,
                                      df (&v)[1]) {
  x = fma(alpha, df_to_double(df(pp.h, pp.l)), x);
  const df r = dfnorm(fma(nalpha, dfd(ap), df(r2.h, r2.l)));
  r2 = df_pair{r.h, r.l};
  ap = 0.0;
  v[0] = fma(r, r, v[0]);
  return t_of<T>(r);
}

template <typename T, bool VEC>
__global__ void __launch_bounds__(kThreads, kXrCtasPerSm)
    k_dfpcg_xr(int64_t n, double* __restrict__ x, const df_pair* __restrict__ p2, double* __restrict__ Ap,
               df_pair* __restrict__ r2, T* __restrict__ b0, CgScalars* cg, double* partials, int stride,
               unsigned int* ticket) {
  pdl_wait();
  if (cg->done) return;
  const double alpha = cg->alpha;
  const df nalpha = dfneg(dfd(alpha));
  df v[1] = {df(0.f, 0.f)};
  const int64_t nc = VEC ? n / 2 : 0;
  GRID_CHUNKS(c, nc) {
    const C2<df_pair> pp = reinterpret_cast<const C2<df_pair>*>(p2)[c];
    C2<double> xx = reinterpret_cast<const C2<double>*>(x)[c];
    C2<double> aa = reinterpret_cast<const C2<double>*>(Ap)[c];
    C2<df_pair> rr = reinterpret_cast<const C2<df_pair>*>(r2)[c];
    C2<T> rb;
#pragma unroll
    for (int k = 0; k < 2; ++k) rb.e[k] = xr_entry<T>(alpha, nalpha, pp.e[k], xx.e[k], aa.e[k], rr.e[k], v);
    reinterpret_cast<C2<double>*>(x)[c] = xx;
    reinterpret_cast<C2<df_pair>*>(r2)[c] = rr;
    reinterpret_cast<C2<double>*>(Ap)[c] = aa;
    reinterpret_cast<C2<T>*>(b0)[c] = rb;
  }
  GRID_TAIL(i, nc * 2, n) {
    b0[i] = xr_entry<T>(alpha, nalpha, p2[i], x[i], Ap[i], r2[i], v);
  }
  pdl_trigger();
  double tot[1];
  if (grid_sums_df<1>(v, partials, stride, ticket, tot)) {
    cg->rr = tot[0];
    cg->iters += 1;
    if (!isfinite(tot[0]) || !isfinite(alpha)) {
      cg->status = SEM_ERR_NONFINITE;
      cg->done = 1;
    } else if (tot[0] <= cg->tol2) {
      cg->done = 1;
    }
  }
}

template <typename T>
__global__ void k_to_level0(int64_t n, const double* __restrict__ r, T* __restrict__ b0) {
  pdl_wait();
  GRID_LOOP(i, n) b0[i] = (T)r[i];
  pdl_trigger();
}

template <typename T>
__global__ void k_from_level0(int64_t n, const T* __restrict__ x0, double* __restrict__ z) {
  pdl_wait();
  GRID_LOOP(i, n) z[i] = (double)x0[i];
  pdl_trigger();
}

// ---------------------------------------------------------------- host helpers
#define GMG_CK(call)                                          \
  do {                                                        \
    cudaError_t e_ = (call);                                  \
    if (e_ != cudaSuccess) return cuda_fail(ctx, e_, #call);  \
  } while (0)

size_t elem_size(int precision) { return precision == SEM_PREC_FP64 ? sizeof(double) : sizeof(float); }

// Largest eigenvalue of the symmetric tridiagonal matrix (diag a, off-diagonal e) by bisection.
double tridiag_max_eig(const std::vector<double>& a, const std::vector<double>& e) {
  const int m = (int)a.size();
  double lo = 1e300, hi = -1e300;
  for (int i = 0; i < m; ++i) {
    const double r = (i > 0 ? std::fabs(e[i - 1]) : 0.0) + (i + 1 < m ? std::fabs(e[i]) : 0.0);
    lo = std::min(lo, a[i] - r);
    hi = std::max(hi, a[i] + r);
  }
  auto count_below = [&](double x) {
    int c = 0;
    double d = 1.0;
    for (int i = 0; i < m; ++i) {
      d = a[i] - x - (i > 0 ? e[i - 1] * e[i - 1] / d : 0.0);
      if (d == 0.0) d = -1e-300;
      if (d < 0.0) ++c;
    }
    return c;
  };
  for (int it = 0; it < 200; ++it) {
    const double mid = 0.5 * (lo + hi);
    if (mid <= lo || mid >= hi) break;
    if (count_below(mid) >= m) hi = mid; else lo = mid;
  }
  return 0.5 * (lo + hi);
}

// r -= (alpha M + K) d on one level in the V-cycle's precision.
int level_apply(sem_ctx* ctx, const Level& L, int precision, double alpha, const void* d, void* r,
                const int* done, cudaStream_t s) {
  cudaError_t e;
  // deterministic mode: element-local results and fixed-order node sums (scalar kernels)
  void* loc = ctx->deterministic ? ctx->det_scratch : nullptr;
  if (precision == SEM_PREC_FP64) {
    ApplyArgs64 a{};
    a.map = L.map; a.metric = L.metric; a.u = (const double*)d; a.y = (double*)r;
    a.nelem = L.nelem; a.mass_coef = alpha; a.out_scale = -1.0; a.scale_out = kNegateOut; a.done = done;
    a.yloc = (double*)loc;
    e = launch_apply_fp64(L, a, false, s);
  } else if (precision == SEM_PREC_FP32_BF16 || precision == SEM_PREC_BF16_TC) {
    ApplyArgs<float, __nv_bfloat16> a{};
    a.map = L.map; a.metric = L.metric16; a.u = (const float*)d; a.y = (float*)r;
    a.nelem = L.nelem; a.mass_coef = (float)alpha; a.out_scale = -1.f; a.scale_out = kNegateOut; a.done = done;
    a.yloc = (float*)loc;
    e = (precision == SEM_PREC_BF16_TC && tc_supported(L) && loc == nullptr) ? launch_apply_tc(L, a, s)
                                                                             : launch_apply_bf16(L, a, false, s);
  } else {
    ApplyArgs<float, float> a{};
    a.map = L.map; a.metric = L.metric32; a.u = (const float*)d; a.y = (float*)r;
    a.nelem = L.nelem; a.mass_coef = (float)alpha; a.out_scale = -1.f; a.scale_out = kNegateOut; a.done = done;
    a.yloc = (float*)loc;
    e = launch_apply_fp32(L, a, false, s);
  }
  if (e != cudaSuccess) return cuda_fail(ctx, e, "level apply");
  ctx->launches += 1;
  return SEM_OK;
}

PTab make_ptab(const Level& fine, const Level& coarse) {
  PTab t{};
  t.nf = fine.n;
  t.nc = coarse.n;
  // l^c_a(x^f_i) by the barycentric formula on the coarse LGL nodes
  const double* xc = coarse.tab.xg;
  const double* xf = fine.tab.xg;
  double lam[kMaxN];
  for (int a = 0; a < t.nc; ++a) {
    double prod = 1.0;
    for (int b = 0; b < t.nc; ++b) if (b != a) prod *= (xc[a] - xc[b]);
    lam[a] = 1.0 / prod;
  }
  for (int i = 0; i < t.nf; ++i) {
    int hit = -1;
    for (int a = 0; a < t.nc; ++a) if (std::fabs(xf[i] - xc[a]) < 1e-15) hit = a;
    if (hit >= 0) {
      for (int a = 0; a < t.nc; ++a) t.P[i][a] = (a == hit) ? 1.0 : 0.0;
      continue;
    }
    double den = 0.0;
    for (int a = 0; a < t.nc; ++a) den += lam[a] / (xf[i] - xc[a]);
    for (int a = 0; a < t.nc; ++a) t.P[i][a] = (lam[a] / (xf[i] - xc[a])) / den;
  }
  return t;
}

// Restrict r_l into r_{l+1}.
template <typename T>
int restrict_to(sem_ctx* ctx, Gmg& g, int l, const int* done, cudaStream_t s) {
  GmgLevel& F = g.lv[l];
  GmgLevel& C = g.lv[l + 1];
  if (F.to_next == 0) {
    const PTab tab = make_ptab(*F.L, *C.L);
    GMG_CK(p_transfer<T>(false, *F.L, *C.L, tab.P, (const T*)F.r, (T*)C.r, nullptr, done, s));
    ctx->launches += 1;
    return SEM_OK;
  }
  launch_k(k_restrict_h<T>, grid1d(C.L->ndofs), kThreads, 0, s, F.L->nx, F.L->ny, F.L->nz, C.L->nx, C.L->ny, C.L->nz,
           (const T*)F.r, (T*)C.r, done);
  GMG_CK(cudaGetLastError());
  ctx->launches += 1;
  return SEM_OK;
}

// d_l = P x_{l+1}, x_l += d_l.
template <typename T>
int prolong_from(sem_ctx* ctx, Gmg& g, int l, const int* done, cudaStream_t s) {
  GmgLevel& F = g.lv[l];
  GmgLevel& C = g.lv[l + 1];
  if (F.to_next == 0) {
    const PTab tab = make_ptab(*F.L, *C.L);
    GMG_CK(p_transfer<T>(true, *F.L, *C.L, tab.P, (const T*)C.x, (T*)F.x, (T*)F.d, done, s));
    ctx->launches += 1;
    return SEM_OK;
  } else {
    launch_k(k_prolong_h<T>, grid1d(F.L->ndofs), kThreads, 0, s,
        F.L->nx, F.L->ny, F.L->nz, C.L->nx, C.L->ny, C.L->nz, (const T*)C.x, (T*)F.x, (T*)F.d,
        done);
  }
  GMG_CK(cudaGetLastError());
  ctx->launches += 1;
  return SEM_OK;
}

// `degree` Chebyshev steps on level l: from a zero start with r the right-hand side,
// or from the current x with r the residual before its last correction d.  On exit r
// is the residual before the last correction, which is in d when keep_d.
template <typename T>
int chebyshev(sem_ctx* ctx, Gmg& g, int l, int degree, bool zero_start, bool keep_d, const int* done,
              cudaStream_t s) {
  GmgLevel& V = g.lv[l];
  const Level& L = *V.L;
  const int64_t n = L.ndofs;
  const double lo = 0.08 * V.lam, hi = 1.2 * V.lam;
  const double theta = 0.5 * (hi + lo), delta = 0.5 * (hi - lo), sigma = theta / delta;
  double rho_old = 1.0 / sigma;
  T* r = (T*)V.r; T* x = (T*)V.x; T* d = (T*)V.d; const T* invd = (const T*)V.invd;
  int k0 = 0;
  bool owed = false;  // the correction in d is not in x yet
  if (zero_start) {
    owed = degree > 1;
    launch_k(k_cheb_zero_start<T>, grid_chunks<T>(n), kThreads, 0, s, n, r, invd, x, d, (T)(1.0 / theta),
             degree == 1 ? 1 : 0, done);
    GMG_CK(cudaGetLastError());
    ctx->launches += 1;
    k0 = 1;
  }
  for (int k = k0; k < degree; ++k) {
    int rc = level_apply(ctx, L, g.precision, g.alpha, d, r, done, s);
    if (rc != SEM_OK) return rc;
    const bool end = k == degree - 1;
    int mode = end && !keep_d ? kChebLast : 0;
    if (owed) mode |= zero_start && k == 1 ? kChebStartX : kChebPair;
    else if (!end) mode |= kChebDefer;
    owed = !owed && !end;
    double c1 = 0.0, c2 = 1.0 / theta;
    if (k == 0) {
      mode |= kChebFirst;
    } else {
      const double rho = 1.0 / (2.0 * sigma - rho_old);
      c1 = rho * rho_old;
      c2 = 2.0 * rho / delta;
      rho_old = rho;
    }
    launch_k(k_cheb_step<T>, grid_chunks<T>(n), kThreads, 0, s, n, r, invd, x, d, (T)c1, (T)c2, mode, done);
    GMG_CK(cudaGetLastError());
    ctx->launches += 1;
  }
  return SEM_OK;
}

// Whether k_cheb_coarse takes the coarsest level.
bool coarse_in_one_cta(const Gmg& g) {
  const Level& L = *g.lv.back().L;
  if (g.precision == SEM_PREC_FP64 || L.p != 1 || L.ndofs > kCoarseNodes || g.coarse_degree > kCoarseDegree) return false;
  return (g.precision == SEM_PREC_FP32 ? coarse_smem<float>(L) : coarse_smem<__nv_bfloat16>(L)) <= kCoarseSmem;
}

template <int QUAD, typename MT>
cudaError_t launch_coarse(const GmgLevel& V, const MT* metric, double alpha, int degree, const int* done, cudaStream_t s) {
  const Level& L = *V.L;
  const double lo = 0.08 * V.lam, hi = 1.2 * V.lam;
  const double theta = 0.5 * (hi + lo), delta = 0.5 * (hi - lo), sigma = theta / delta;
  ChebCoef cf;
  double rho_old = 1.0 / sigma;
  cf.c1[0] = 0.f;
  cf.c2[0] = (float)(1.0 / theta);
  for (int k = 1; k < degree; ++k) {
    const double rho = 1.0 / (2.0 * sigma - rho_old);
    cf.c1[k] = (float)(rho * rho_old);
    cf.c2[k] = (float)(2.0 * rho / delta);
    rho_old = rho;
  }
  KTab<2, float> tab;
  make_eo(tab.D, QUAD == SEM_QUAD_LG ? L.tab.Dg : L.tab.D, false);
  make_eo(tab.Dt, QUAD == SEM_QUAD_LG ? L.tab.Dg : L.tab.D, true);
  make_eo(tab.Bi, L.tab.Bi, false);
  make_eo(tab.Bit, L.tab.Bi, true);
  return launch_k(k_cheb_coarse<QUAD, MT>, 1, kCoarseThreads, coarse_smem<MT>(L), s, L.nx, L.ny, L.nz, L.map, metric,
                  (float)alpha, tab, cf, degree, (const float*)V.r, (const float*)V.invd, (float*)V.x, L.ndofs, L.dbg,
                  done);
}

int chebyshev_coarse(sem_ctx* ctx, Gmg& g, const int* done, cudaStream_t s) {
  const GmgLevel& V = g.lv.back();
  const bool lg = V.L->quad == SEM_QUAD_LG;
  if (g.precision == SEM_PREC_FP32)
    GMG_CK((lg ? launch_coarse<SEM_QUAD_LG, float> : launch_coarse<SEM_QUAD_LGL, float>)(V, V.L->metric32, g.alpha,
                                                                                        g.coarse_degree, done, s));
  else
    GMG_CK((lg ? launch_coarse<SEM_QUAD_LG, __nv_bfloat16> : launch_coarse<SEM_QUAD_LGL, __nv_bfloat16>)(
        V, V.L->metric16, g.alpha, g.coarse_degree, done, s));
  ctx->launches += 1;
  return SEM_OK;
}

template <typename T>
int vcycle_level(sem_ctx* ctx, Gmg& g, int l, const int* done, cudaStream_t s, bool record) {
  const int last = (int)g.lv.size() - 1;
  int rc;
  if (l == last)
    return coarse_in_one_cta(g) ? chebyshev_coarse(ctx, g, done, s)
                                : chebyshev<T>(ctx, g, l, g.coarse_degree, true, false, done, s);
  if ((rc = chebyshev<T>(ctx, g, l, g.degree, true, true, done, s)) != SEM_OK) return rc;
  GmgLevel& V = g.lv[l];
  // r -= A d: the residual of x, then r_{l+1} = R r
  // the fine-level residual apply is bracketed by event nodes when `record`
  if (record && l == 0) GMG_CK(cudaEventRecordWithFlags(g.ev2, s, cudaEventRecordExternal));
  if ((rc = level_apply(ctx, *V.L, g.precision, g.alpha, V.d, V.r, done, s)) != SEM_OK) return rc;
  if (record && l == 0) GMG_CK(cudaEventRecordWithFlags(g.ev3, s, cudaEventRecordExternal));
  if ((rc = restrict_to<T>(ctx, g, l, done, s)) != SEM_OK) return rc;
  if ((rc = vcycle_level<T>(ctx, g, l + 1, done, s, false)) != SEM_OK) return rc;
  if ((rc = prolong_from<T>(ctx, g, l, done, s)) != SEM_OK) return rc;
  return chebyshev<T>(ctx, g, l, g.degree, false, false, done, s);
}

int vcycle(sem_ctx* ctx, Gmg& g, const int* done, cudaStream_t s, bool record = false) {
  if (g.precision == SEM_PREC_FP64) return vcycle_level<double>(ctx, g, 0, done, s, record);
  return vcycle_level<float>(ctx, g, 0, done, s, record);
}

// Enqueues 10 Jacobi-PCG steps on level V from the fixed start vector (scalars to sc).
int launch_lanczos(sem_ctx* ctx, Gmg& g, GmgLevel& V, double alpha, LanczosScalars* sc, cudaStream_t s) {
  const Level& L = *V.L;
  const int64_t n = L.ndofs;
  const int gr = grid1d(n);
  launch_k(k_lanczos_start, gr, kThreads, 0, s, n, V.dinv64, g.lr, g.lp, g.lAp, sc, g.partials, g.tickets);
  const int iters = (int)std::min<int64_t>(kLanczosSteps, n);
  for (int it = 0; it < iters; ++it) {
    ApplyArgs64 a{};
    a.map = L.map; a.metric = L.metric; a.u = g.lp; a.y = g.lAp; a.nelem = L.nelem;
    a.mass_coef = alpha; a.out_scale = 1.0; a.scale_out = 0; a.done = &sc->stop;
    a.yloc = ctx->deterministic ? ctx->det_scratch : nullptr;
    GMG_CK(launch_apply_fp64(L, a, false, s));
    launch_k(k_lanczos_dot, gr, kThreads, 0, s, n, g.lp, g.lAp, sc, g.partials, g.tickets);
    launch_k(k_lanczos_update, gr, kThreads, 0, s, n, g.lAp, g.lr, V.dinv64, g.lz, sc, g.partials, g.tickets);
    if (it + 1 < iters) launch_k(k_lanczos_p, gr, kThreads, 0, s, n, g.lz, g.lp, g.lAp, sc);
  }
  GMG_CK(cudaGetLastError());
  return SEM_OK;
}

// Largest eigenvalue of the Lanczos tridiagonal of the recorded steps (0: none).
double lanczos_lambda(const LanczosScalars& sc) {
  const int m = sc.m;
  if (m == 0) return 0.0;
  std::vector<double> d(m), e(std::max(0, m - 1));
  for (int j = 0; j < m; ++j) {
    d[j] = 1.0 / sc.alpha[j] + (j > 0 ? sc.beta[j - 1] / sc.alpha[j - 1] : 0.0);
    if (j + 1 < m) e[j] = std::sqrt(sc.beta[j]) / sc.alpha[j];
  }
  return tridiag_max_eig(d, e);
}

// Diagonals and eigenvalue estimates of every level for alpha.  All levels' estimates
// are enqueued before the one host read (each step read two scalars back before: 1.8 ms
// for the three levels of a 70,000-node hierarchy, now 0.64).  That read is also the full
// dependency between the levels' metric conversions and the first applies (pdl_wait).
int set_alpha(sem_ctx* ctx, Gmg& g, double alpha, cudaStream_t s) {
  if (g.alpha == alpha) return SEM_OK;
  const size_t nl = g.lv.size();
  g.alpha = -1.0;
  for (size_t l = 0; l < nl; ++l) {
    GmgLevel& V = g.lv[l];
    const Level& L = *V.L;
    if (g.precision == SEM_PREC_FP64)
      launch_k(k_level_inv_diag<double>, grid1d(L.ndofs), kThreads, 0, s, L.ndofs, alpha, L.mdiag, L.kdiag,
                                                                   (double*)V.invd, V.dinv64);
    else
      launch_k(k_level_inv_diag<float>, grid1d(L.ndofs), kThreads, 0, s, L.ndofs, alpha, L.mdiag, L.kdiag,
                                                                  (float*)V.invd, V.dinv64);
    GMG_CK(cudaGetLastError());
    int rc = launch_lanczos(ctx, g, V, alpha, g.lanczos + l, s);
    if (rc != SEM_OK) return rc;
  }
  std::vector<LanczosScalars> sc(nl);
  GMG_CK(cudaMemcpyAsync(sc.data(), g.lanczos, sizeof(LanczosScalars) * nl, cudaMemcpyDeviceToHost, s));
  GMG_CK(cudaStreamSynchronize(s));
  for (size_t l = 0; l < nl; ++l) {
    g.lv[l].lam = lanczos_lambda(sc[l]);
    if (sc[l].m == 0) return fail(ctx, SEM_ERR_NONFINITE, "eigenvalue estimate failed on a multigrid level");
  }
  g.alpha = alpha;
  return SEM_OK;
}

void free_gmg_struct(Gmg* g) {
  if (!g) return;
  for (GmgLevel& V : g->lv) {
    if (V.owned && V.L) {
      level_free(*V.L);
      delete V.L;
    }
    if (V.owns_tissue) {
      cudaFree(V.sl); cudaFree(V.st); cudaFree(V.th);
    }
    cudaFree(V.r); cudaFree(V.x); cudaFree(V.d); cudaFree(V.invd);
    cudaFree(V.dinv64);
  }
  cudaFree(g->z);
  for (auto& gr : g->graphs) gr.drop();
  if (g->capture) cudaStreamDestroy(g->capture);
  if (g->ev0) cudaEventDestroy(g->ev0);
  if (g->ev1) cudaEventDestroy(g->ev1);
  if (g->ev2) cudaEventDestroy(g->ev2);
  if (g->ev3) cudaEventDestroy(g->ev3);
  cudaFree(g->lr); cudaFree(g->lz); cudaFree(g->lp); cudaFree(g->lAp);
  cudaFree(g->lanczos); cudaFree(g->partials); cudaFree(g->tickets);
  delete g;
}

// The low-precision metrics of every level that the V-cycle reads.
int level_metrics(sem_ctx* ctx, Gmg& g, cudaStream_t s) {
  for (GmgLevel& V : g.lv) {
    Level& L = *V.L;
    if (g.precision == SEM_PREC_FP32 && !L.metric32_valid) {
      if (!L.metric32) GMG_CK(cudaMalloc(&L.metric32, sizeof(float) * metric_lowp_values(L)));
      GMG_CK(setup_metric_lowp(L, false, s));
    }
    const bool tc = g.precision == SEM_PREC_BF16_TC && tc_supported(L) && !ctx->deterministic;
    if ((g.precision == SEM_PREC_FP32_BF16 || (g.precision == SEM_PREC_BF16_TC && !tc)) &&
        !L.metric16_valid) {
      if (!L.metric16) GMG_CK(cudaMalloc(&L.metric16, sizeof(__nv_bfloat16) * metric_lowp_values(L)));
      GMG_CK(setup_metric_lowp(L, true, s));
    }
    if (tc && !L.metric_tc_valid) GMG_CK(setup_metric_tc(L, s));
  }
  return SEM_OK;
}

// New tissue on a standing hierarchy: the coarse levels' tissue, metrics and diagonals
// (the fine level's are sem_set_tissue's), the estimates (alpha = -1) and the graphs,
// whose launches hold the smoother's coefficients.
int refresh(sem_ctx* ctx, Gmg& g, cudaStream_t s) {
  for (auto& gr : g.graphs) gr.drop();
  g.alpha = -1.0;
  for (size_t l = 1; l < g.lv.size(); ++l) {
    GmgLevel &F = g.lv[l - 1], &V = g.lv[l];
    Level& L = *V.L;
    if (V.owns_tissue) {
      launch_k(k_coarse_tissue, grid1d(L.nelem), kThreads, 0, s, L.nx, L.ny, L.nz, F.L->nx, F.L->ny, F.sl, F.st, F.th,
               V.sl, V.st, V.th);
      GMG_CK(cudaGetLastError());
    }
    GMG_CK(setup_geometry(L, V.sl, V.st, V.th, ctx->d_flag, s));
    GMG_CK(setup_diagonals(L, s));
  }
  const int rc = level_metrics(ctx, g, s);
  if (rc == SEM_OK) g.stale = false;
  return rc;
}

int build(sem_ctx* ctx, cudaStream_t s) {
  if (ctx->gmg) return ctx->gmg->stale ? refresh(ctx, *ctx->gmg, s) : SEM_OK;
  GMG_CK(prime_coarse());
  Gmg* g = new Gmg();
  g->precision = ctx->gmg_precision;
  g->degree = ctx->gmg_degree;
  g->coarse_degree = ctx->gmg_coarse_degree;
  struct Guard {
    Gmg*& g;
    ~Guard() { if (g) free_gmg_struct(g); }
  } guard{g};
  GmgLevel top;
  top.L = &ctx->L;
  top.sl = ctx->sigma_l; top.st = ctx->sigma_t; top.th = ctx->theta;
  g->lv.push_back(top);
  std::vector<double> verts = ctx->vertices;
  int nx = ctx->L.nx, ny = ctx->L.ny, nz = ctx->L.nz, p = ctx->L.p;
  const int quad = ctx->L.quad;
  GMG_CK(cudaMemsetAsync(ctx->d_flag, 0, sizeof(int), s));
  // p-coarsening on the fine mesh, then h-coarsening, while the level is larger
  // than min_coarse_dofs (a p-level may be the coarsest)
  while (p > 1 && g->lv.back().L->ndofs > ctx->gmg_min_coarse_dofs) {
    const int pc = std::max(1, p / 2);
    GmgLevel V;
    V.L = new Level();
    V.owned = true;
    V.sl = ctx->sigma_l; V.st = ctx->sigma_t; V.th = ctx->theta;
    g->lv.back().to_next = 0;
    g->lv.push_back(V);
    GMG_CK(level_create(*g->lv.back().L, nx, ny, nz, verts.data(), pc, quad, false, s));
    g->lv.back().L->dbg = ctx->L.dbg;
    g->lv.back().L->fault = ctx->L.fault;
    GMG_CK(setup_geometry(*g->lv.back().L, V.sl, V.st, V.th, ctx->d_flag, s));
    GMG_CK(setup_diagonals(*g->lv.back().L, s));
    p = pc;
  }
  while (g->lv.back().L->ndofs > ctx->gmg_min_coarse_dofs && std::max(nx, std::max(ny, nz)) > 1) {
    const int cx = (nx + 1) / 2, cy = (ny + 1) / 2, cz = (nz + 1) / 2;
    std::vector<double> cv((size_t)(cx + 1) * (cy + 1) * (cz + 1) * 3);
    for (int K = 0; K <= cz; ++K)
      for (int J = 0; J <= cy; ++J)
        for (int I = 0; I <= cx; ++I) {
          const size_t f = (size_t)std::min(2 * I, nx) +
                           (size_t)(nx + 1) * (std::min(2 * J, ny) + (size_t)(ny + 1) * std::min(2 * K, nz));
          const size_t c = (size_t)I + (size_t)(cx + 1) * (J + (size_t)(cy + 1) * K);
          for (int d = 0; d < 3; ++d) cv[c * 3 + d] = verts[f * 3 + d];
        }
    GmgLevel& F = g->lv.back();
    GmgLevel V;
    V.L = new Level();
    V.owned = true;
    V.owns_tissue = true;
    const size_t ne = (size_t)cx * cy * cz;
    GMG_CK(cudaMalloc(&V.sl, sizeof(double) * ne));
    GMG_CK(cudaMalloc(&V.st, sizeof(double) * ne));
    GMG_CK(cudaMalloc(&V.th, sizeof(double) * ne));
    launch_k(k_coarse_tissue, grid1d((int64_t)ne), kThreads, 0, s, cx, cy, cz, nx, ny, F.sl, F.st, F.th,
                                                              V.sl, V.st, V.th);
    GMG_CK(cudaGetLastError());
    F.to_next = 1;
    g->lv.push_back(V);
    GMG_CK(level_create(*g->lv.back().L, cx, cy, cz, cv.data(), 1, quad, false, s));
    g->lv.back().L->dbg = ctx->L.dbg;
    g->lv.back().L->fault = ctx->L.fault;
    GMG_CK(setup_geometry(*g->lv.back().L, V.sl, V.st, V.th, ctx->d_flag, s));
    GMG_CK(setup_diagonals(*g->lv.back().L, s));
    verts.swap(cv);
    nx = cx; ny = cy; nz = cz;
  }
  int bad = 0;
  GMG_CK(cudaMemcpyAsync(&bad, ctx->d_flag, sizeof(int), cudaMemcpyDeviceToHost, s));
  GMG_CK(cudaStreamSynchronize(s));
  if (bad) return fail(ctx, SEM_ERR_BAD_MESH, "a coarsened multigrid level has an inverted element");
  if (const int rc = level_metrics(ctx, *g, s); rc != SEM_OK) return rc;
  const size_t es = elem_size(g->precision);
  int64_t nmax = 0;
  for (GmgLevel& V : g->lv) {
    Level& L = *V.L;
    nmax = std::max(nmax, L.ndofs);
    void** vecs[] = {&V.r, &V.x, &V.d, &V.invd};
    for (void** v : vecs) GMG_CK(cudaMalloc(v, es * L.ndofs));
    GMG_CK(cudaMalloc(&V.dinv64, sizeof(double) * L.ndofs));
  }
  const int64_t nf = ctx->L.ndofs;
  GMG_CK(cudaMalloc(&g->z, sizeof(double) * nf));
  GMG_CK(cudaStreamCreateWithFlags(&g->capture, cudaStreamNonBlocking));
  GMG_CK(cudaEventCreate(&g->ev0));
  GMG_CK(cudaEventCreate(&g->ev1));
  GMG_CK(cudaEventCreate(&g->ev2));
  GMG_CK(cudaEventCreate(&g->ev3));
  double** lv4[] = {&g->lr, &g->lz, &g->lp, &g->lAp};
  for (double** v : lv4) GMG_CK(cudaMalloc(v, sizeof(double) * nmax));
  GMG_CK(cudaMalloc(&g->lanczos, sizeof(LanczosScalars) * g->lv.size()));
  g->partial_len = 2048;
  GMG_CK(cudaMalloc(&g->partials, sizeof(double) * 4 * g->partial_len));
  GMG_CK(cudaMalloc(&g->tickets, sizeof(unsigned int) * 4));
  GMG_CK(cudaMemsetAsync(g->tickets, 0, sizeof(unsigned int) * 4, s));
  GMG_CK(cudaStreamSynchronize(s));
  ctx->gmg = g;
  g = nullptr;  // ownership moved to the context
  return SEM_OK;
}

// Kernel nodes of an instantiated graph's source graph.
int64_t count_kernels(cudaGraph_t graph) {
  size_t n = 0;
  if (cudaGraphGetNodes(graph, nullptr, &n) != cudaSuccess) return 0;
  std::vector<cudaGraphNode_t> nodes(n);
  if (cudaGraphGetNodes(graph, nodes.data(), &n) != cudaSuccess) return 0;
  int64_t k = 0;
  for (auto nd : nodes) {
    cudaGraphNodeType t;
    if (cudaGraphNodeGetType(nd, &t) == cudaSuccess && t == cudaGraphNodeTypeKernel) ++k;
  }
  return k;
}

// The PCG launch sequences, issued on stream s (a capture stream when graphs are built).
// Set-up: r = b - A x, stopping threshold, convergence test.  One iteration:
// z = V(r), beta, p = z + beta p, A p with alpha = r.z / p.Ap, x and r updated,
// convergence test.  The iteration ends with the test, so the host launches no
// V-cycle after convergence.
// carried: A x is read from ws.Ax (the last time step's b - r) instead of
// applied; ws.Ap is then already zero (every PCG iteration leaves it zero).
// checked (with carried): a device flag; the zeroing of ws.Ap and the apply run
// only where it reads zero (they return at once otherwise), and the residual
// kernel reads ws.Ax or ws.Ap accordingly.
template <typename T>
int pcg_init_seq(sem_ctx* ctx, Gmg& g, double alpha, const double* b, const double* x, double rtol,
                 double atol, bool carried, const int* checked, cudaStream_t s) {
  Workspace& w = ctx->ws;
  Level& L = ctx->L;
  const int64_t n = L.ndofs;
  const int gr = grid1d(n);
  T* b0 = (T*)g.lv[0].r;
  const int stride = g.partial_len;
  if (!carried || checked != nullptr) {
    launch_k(k_zero<double>, gr, kThreads, 0, s, n, w.Ap, checked);
    ApplyArgs64 a{};
    a.map = L.map; a.metric = L.metric; a.u = x; a.y = w.Ap; a.nelem = L.nelem;
    a.mass_coef = alpha; a.out_scale = 1.0; a.scale_out = 0; a.done = checked;
    a.yloc = ctx->deterministic ? ctx->det_scratch : nullptr;
    GMG_CK(launch_operator(ctx, a, s));
  }
  if (ctx->op_precision == SEM_PREC_DF64) {  // r kept as float pairs in ws.r, carried A x as pairs in ws.Ax
    auto kern = aligned16(b) ? k_dfpcg_init<T, true> : k_dfpcg_init<T, false>;
    launch_k(kern, gr, kThreads, 0, s, n, b, w.Ap, carried ? reinterpret_cast<const df_pair*>(w.Ax) : nullptr,
             checked, reinterpret_cast<df_pair*>(w.r), b0, w.cg, g.partials, stride, g.tickets, rtol, atol);
  } else {
    auto kern = aligned16(b) ? k_fpcg_init<T, true> : k_fpcg_init<T, false>;
    launch_k(kern, gr, kThreads, 0, s, n, b, carried ? w.Ax : w.Ap, w.Ap, checked, w.r, b0, w.cg, g.partials,
             stride, g.tickets, rtol, atol);
  }
  GMG_CK(cudaGetLastError());
  return SEM_OK;
}

// timed: external event nodes around the fine-level residual apply of the V-cycle
// (ev2, ev3) and the outer operator apply (ev0, ev1).  Each event node costs a few
// microseconds of the step (it breaks the programmatic dependent launch around it),
// so only the sampled iterations use the timed graph.
template <typename T>
int pcg_iter_seq(sem_ctx* ctx, Gmg& g, double alpha, double* x, bool timed, cudaStream_t s) {
  Workspace& w = ctx->ws;
  Level& L = ctx->L;
  const int64_t n = L.ndofs;
  const int gr = grid1d(n);
  const int stride = g.partial_len;
  const int* done = &w.cg->done;
  int rc = vcycle(ctx, g, done, s, timed);
  if (rc != SEM_OK) return rc;
  // the double-float operator gathers p as the float pairs the p kernels write
  const bool dfop = ctx->op_precision == SEM_PREC_DF64;
  df_pair* p2 = dfop ? w.p2 : nullptr;
  df_pair* r2 = reinterpret_cast<df_pair*>(w.r);
  if (dfop) {
    launch_k(k_dfpcg_z<T>, gr, kThreads, 0, s, n, (const T*)g.lv[0].x, reinterpret_cast<T*>(g.z), r2, p2, w.cg,
             g.partials, stride, g.tickets + 1);
    launch_k(k_dfpcg_p<T>, gr, kThreads, 0, s, n, reinterpret_cast<const T*>(g.z), p2, w.cg);
  } else {
    launch_k(k_fpcg_z<T>, gr, kThreads, 0, s, n, (const T*)g.lv[0].x, g.z, w.r, w.p, p2, w.cg, g.partials,
             stride, g.tickets + 1);
    launch_k(k_fpcg_p, gr, kThreads, 0, s, n, g.z, w.p, p2, w.cg);
  }
  GMG_CK(cudaGetLastError());
  ApplyArgs64 ap{};
  ap.map = L.map; ap.metric = L.metric; ap.u = w.p; ap.y = w.Ap; ap.nelem = L.nelem;
  ap.mass_coef = alpha; ap.out_scale = 1.0; ap.scale_out = 0; ap.done = done;
  ap.dot_partials = w.apply_partials; ap.cg = w.cg; ap.u2 = p2;
  ap.yloc = ctx->deterministic ? ctx->det_scratch : nullptr;
  // external records become event nodes of the captured graph (timing of the outer apply)
  if (timed) GMG_CK(cudaEventRecordWithFlags(g.ev0, s, cudaEventRecordExternal));
  GMG_CK(launch_operator(ctx, ap, s));
  if (timed) GMG_CK(cudaEventRecordWithFlags(g.ev1, s, cudaEventRecordExternal));
  if (dfop)
    launch_k(aligned16(x) ? k_dfpcg_xr<T, true> : k_dfpcg_xr<T, false>, std::min(gr, 152 * kXrCtasPerSm),
             kThreads, 0, s, n, x, p2, w.Ap, r2, (T*)g.lv[0].r, w.cg, g.partials, stride, g.tickets + 2);
  else if (aligned16(x))
    launch_k(k_fpcg_xr<T, true>, gr, kThreads, 0, s, n, x, w.p, w.Ap, w.r, (T*)g.lv[0].r, w.cg, g.partials,
                                             stride, g.tickets + 2);
  else
    launch_k(k_fpcg_xr<T, false>, gr, kThreads, 0, s, n, x, w.p, w.Ap, w.r, (T*)g.lv[0].r, w.cg, g.partials,
                                              stride, g.tickets + 2);
  GMG_CK(cudaGetLastError());
  return SEM_OK;
}

// The graphs of one solution pointer, right-hand side, alpha and tolerances (all baked
// into the captured launches); sixteen are cached.
Gmg::Graphs& get_graphs(Gmg& g, double alpha, const double* b, double* x, double rtol, double atol) {
  for (auto& gr : g.graphs)
    if (gr.used && gr.x == x && gr.b == b && gr.alpha == alpha && gr.rtol == rtol && gr.atol == atol) return gr;
  Gmg::Graphs& gr = g.graphs[g.next_graph];
  g.next_graph = (g.next_graph + 1) % 16;
  gr.drop();
  gr.used = true;
  gr.x = x;
  gr.b = b;
  gr.alpha = alpha;
  gr.rtol = rtol;
  gr.atol = atol;
  return gr;
}

// Captures what seq issues on the private stream into e.
template <typename F>
int capture(sem_ctx* ctx, Gmg& g, Gmg::Graphs::Exec& e, F seq) {
  cudaStream_t cs = g.capture;
  const int64_t l0 = ctx->launches;
  GMG_CK(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
  const int rc = seq(cs);
  cudaGraph_t graph = nullptr;
  const cudaError_t ec = cudaStreamEndCapture(cs, &graph);
  ctx->launches = l0;  // capture launched nothing; replays are counted
  if (rc != SEM_OK) {
    if (graph) cudaGraphDestroy(graph);
    return rc;
  }
  if (ec != cudaSuccess) return cuda_fail(ctx, ec, "cudaStreamEndCapture");
  cudaGraphExec_t exec = nullptr;
  const cudaError_t ei = cudaGraphInstantiate(&exec, graph, 0);
  const int64_t nk = count_kernels(graph);
  cudaGraphDestroy(graph);
  if (ei != cudaSuccess) return cuda_fail(ctx, ei, "cudaGraphInstantiate");
  e.exec = exec;
  e.kernels = nk;
  return SEM_OK;
}

template <typename T>
int pcg_t(sem_ctx* ctx, Gmg& g, double alpha, const double* b, double* x, double rtol,
          double atol, int maxit, int* iters, double* final_res, sem_stats* stats, bool carried,
          bool checked, cudaStream_t s) {
  Workspace& w = ctx->ws;
  Gmg::Graphs& gr = get_graphs(g, alpha, b, x, rtol, atol);
  Timing& tm = ctx->timing;
  bool done_h = false;
  int launched = 0;
  // with timing on, the first iteration of one solve in kTimingEvery is the timed one
  bool sample = tm.enabled && (tm.solves++ % kTimingEvery) == 0;
  const int variant = !carried ? 0 : (checked ? 2 : 1);
  auto seq_init = [&](cudaStream_t cs) {
    return pcg_init_seq<T>(ctx, g, alpha, b, x, rtol, atol, variant >= 1, variant == 2 ? w.same : nullptr, cs);
  };
  auto launch = [&](Gmg::Graphs::Exec& e, auto seq) -> int {
    if (e.exec == nullptr) {
      const int rc = capture(ctx, g, e, seq);
      if (rc != SEM_OK) return rc;
    }
    GMG_CK(cudaGraphLaunch(e.exec, s));
    ctx->launches += e.kernels;
    return SEM_OK;
  };
  auto launch_iter = [&]() -> int {
    const bool timed = sample && launched == 0;
    return launch(gr.iter[timed ? 1 : 0], [&](cudaStream_t cs) { return pcg_iter_seq<T>(ctx, g, alpha, x, timed, cs); });
  };
  // Successive solves (time steps) take about the same number of iterations: the
  // set-up and the previous count go out before the scalars are read, as one graph
  // once the count has repeated, so that a solve that needs no more costs one launch
  // and one host round trip.  An iteration launched after convergence runs kernels
  // that return at once.
  const int ahead = std::min(maxit, std::max(0, gr.last_iters));
  Gmg::Graphs::Combo& c = gr.combo[variant];
  if (c.n != ahead) {
    if (c.exec) cudaGraphExecDestroy(c.exec);
    c = Gmg::Graphs::Combo();
    c.n = ahead;
  }
  int rc;
  if (ahead > 0 && !sample && (c.exec != nullptr || c.seen++ > 0)) {
    rc = launch(c, [&](cudaStream_t cs) {
      int r = seq_init(cs);
      for (int i = 0; i < ahead && r == SEM_OK; ++i) r = pcg_iter_seq<T>(ctx, g, alpha, x, false, cs);
      return r;
    });
    if (rc != SEM_OK) return rc;
    launched = ahead;
  } else {
    if ((rc = launch(gr.init[variant], seq_init)) != SEM_OK) return rc;
    for (; launched < ahead; ++launched)
      if ((rc = launch_iter()) != SEM_OK) return rc;
  }
  while (true) {
    GMG_CK(cudaMemcpyAsync(w.cg_host, w.cg, sizeof(CgScalars), cudaMemcpyDeviceToHost, s));
    GMG_CK(cudaMemcpyAsync(w.fault_host, ctx->L.fault, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
    GMG_CK(cudaStreamSynchronize(s));
    if (*w.fault_host != 0u) {  // an apply kernel gave up waiting for its metric copy
      *w.fault_host = 0u;
      GMG_CK(cudaMemsetAsync(ctx->L.fault, 0, sizeof(unsigned), s));
      GMG_CK(cudaStreamSynchronize(s));
      return fail(ctx, SEM_ERR_TIMEOUT, "an apply kernel's wait for its metric copy timed out");
    }
    if (sample && launched > 0 && w.cg_host->iters >= 1) {  // the timed first iteration ran
      sample = false;
      float ms = 0.f;
      if (cudaEventElapsedTime(&ms, g.ev0, g.ev1) == cudaSuccess) {
        tm.ms += ms;
        tm.count += 1;
      } else {
        cudaGetLastError();  // timing unavailable for these event nodes: not an error
      }
      if (cudaEventElapsedTime(&ms, g.ev2, g.ev3) == cudaSuccess) {
        tm.smoother_ms += ms;
        tm.smoother_count += 1;
      } else {
        cudaGetLastError();
      }
    }
    if (w.cg_host->done) { done_h = true; break; }
    if (launched >= maxit) break;
    if ((rc = launch_iter()) != SEM_OK) return rc;
    ++launched;
  }
  const CgScalars& h = *w.cg_host;
  gr.last_iters = h.iters;
  if (iters) *iters = h.iters;
  if (final_res) *final_res = std::sqrt(h.rr);
  if (stats) {
    stats->cg_iters += h.iters;
    stats->last_residual = std::sqrt(h.rr);
  }
  if (h.status == SEM_ERR_NONFINITE)
    return fail(ctx, SEM_ERR_NONFINITE, "non-finite value in a CG inner product");
  if (!done_h)
    return fail(ctx, SEM_ERR_NOT_CONVERGED,
                "multigrid PCG did not converge in " + std::to_string(maxit) + " iterations");
  return SEM_OK;
}

}  // namespace

void gmg_tissue_changed(sem_ctx* ctx) {
  if (ctx->gmg) ctx->gmg->stale = true;
}

void gmg_free(sem_ctx* ctx) {
  if (ctx->gmg) {
    free_gmg_struct(ctx->gmg);
    ctx->gmg = nullptr;
  }
}

int gmg_pcg(sem_ctx* ctx, double alpha, const double* b, double* x, double rtol, double atol,
            int maxit, int* iters, double* final_res, sem_stats* stats, cudaStream_t s, double* ax0,
            const int* ax0_ok) {
  int rc = ensure_workspace(ctx);
  if (rc != SEM_OK) return rc;
  // the carried A x and its check flag are always the workspace's (captured into the set-up graphs)
  if (ax0 != nullptr && ax0 != ctx->ws.Ax) return fail(ctx, SEM_ERR_ARG, "carried A x must be the workspace's");
  if (ax0_ok != nullptr && ax0_ok != ctx->ws.same) return fail(ctx, SEM_ERR_ARG, "carry check must be the workspace's");
  if (rc != SEM_OK) return rc;
  if ((rc = build(ctx, s)) != SEM_OK) return rc;
  GMG_CK(prepare_operator(ctx, s));
  Gmg& g = *ctx->gmg;
  if ((rc = set_alpha(ctx, g, alpha, s)) != SEM_OK) return rc;
  if (g.precision == SEM_PREC_FP64)
    return pcg_t<double>(ctx, g, alpha, b, x, rtol, atol, maxit, iters, final_res, stats, ax0 != nullptr,
                         ax0_ok != nullptr, s);
  return pcg_t<float>(ctx, g, alpha, b, x, rtol, atol, maxit, iters, final_res, stats, ax0 != nullptr,
                      ax0_ok != nullptr, s);
}

int gmg_vcycle(sem_ctx* ctx, double alpha, const double* r, double* z, cudaStream_t s) {
  int rc = build(ctx, s);
  if (rc != SEM_OK) return rc;
  Gmg& g = *ctx->gmg;
  if ((rc = set_alpha(ctx, g, alpha, s)) != SEM_OK) return rc;
  const int64_t n = ctx->L.ndofs;
  if (g.precision == SEM_PREC_FP64)
    launch_k(k_to_level0<double>, grid1d(n), kThreads, 0, s, n, r, (double*)g.lv[0].r);
  else
    launch_k(k_to_level0<float>, grid1d(n), kThreads, 0, s, n, r, (float*)g.lv[0].r);
  GMG_CK(cudaGetLastError());
  if ((rc = vcycle(ctx, g, nullptr, s)) != SEM_OK) return rc;
  if (g.precision == SEM_PREC_FP64)
    launch_k(k_from_level0<double>, grid1d(n), kThreads, 0, s, n, (const double*)g.lv[0].x, z);
  else
    launch_k(k_from_level0<float>, grid1d(n), kThreads, 0, s, n, (const float*)g.lv[0].x, z);
  GMG_CK(cudaGetLastError());
  return SEM_OK;
}

int gmg_info(sem_ctx* ctx, double alpha, int max_levels, int* nlevels, int* p, int* dims,
             int64_t* ndofs, double* lambda_max, cudaStream_t s) {
  int rc = build(ctx, s);
  if (rc != SEM_OK) return rc;
  Gmg& g = *ctx->gmg;
  if ((rc = set_alpha(ctx, g, alpha, s)) != SEM_OK) return rc;
  const int nl = (int)g.lv.size();
  if (nlevels) *nlevels = nl;
  for (int l = 0; l < std::min(nl, max_levels); ++l) {
    const Level& L = *g.lv[l].L;
    if (p) p[l] = L.p;
    if (dims) { dims[3 * l] = L.nx; dims[3 * l + 1] = L.ny; dims[3 * l + 2] = L.nz; }
    if (ndofs) ndofs[l] = L.ndofs;
    if (lambda_max) lambda_max[l] = g.lv[l].lam;
  }
  return SEM_OK;
}

}  // namespace sem
