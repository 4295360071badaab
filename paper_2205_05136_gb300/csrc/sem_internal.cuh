// Internal declarations of libsem (not part of the C ABI).
//
// Layout of the data in HBM (one context = one slab, one device):
//   map      int32  [nelem][n^3]   local node a = i + n j + n^2 k -> global node
//   metric   double [nelem][7][n3p] per quadrature point: G00 G01 G02 G11 G12 G22 W,
//            n3p = n^3 rounded up to a multiple of 8 (16-byte aligned blocks),
//            G = w |det J| J^{-1} D J^{-T}, W = w |det J|  (element-blocked SoA)
//   metric32 float, metric16 bf16  copies in the order the plane kernel consumes:
//            [unit][chunk of rows][element of the unit][plane k][RS] (MetricLayout)
//   mdiag    double [ndofs]  diagonal of the assembled mass matrix
//   kdiag    double [ndofs]  diagonal of the assembled stiffness matrix
//   xyz      double [3][ndofs] node coordinates
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <string>
#include <type_traits>
#include <utility>

#include "sem.h"
#include "sem_df64.cuh"

namespace sem {

// Index checks of the SEM_DEBUG build.  dbg_index returns a node index read
// from an element-to-DOF map (or computed from the lattice) when it lies in
// [0, n); otherwise it records the first offender in *word as
// (kind << 56) | (32-bit index) and returns 0, so no access leaves the vector.
// The host reads and clears the word after the call (debug_check) and returns
// SEM_ERR_ARG with the index.  In the normal build SEM_IDX is the index itself.
constexpr unsigned kDbgGather = 1, kDbgScatter = 2, kDbgLine = 3;
#if defined(SEM_DEBUG) && defined(__CUDACC__)
__device__ __forceinline__ int64_t dbg_index(int64_t g, int64_t n, unsigned long long* word, unsigned kind) {
  if (g >= 0 && g < n) return g;
  if (word != nullptr)
    atomicCAS(word, 0ull, ((unsigned long long)kind << 56) | (unsigned long long)(uint32_t)g);
  return 0;
}
#define SEM_IDX(g, n, word, kind) dbg_index((g), (n), (word), (kind))
// a copy the SEM_DEBUG build leaves out on request (sem_debug_hold_copy), so that
// the wait for it runs out and the timeout path runs
#define SEM_HOLD(a, unit) ((unit) == (a).hold)
// the same for a CTA's arrival at a grid barrier (sem_debug_hold_update)
#define SEM_HOLD_CTA(hold) ((int)blockIdx.x == (hold))
#else
#define SEM_IDX(g, n, word, kind) (g)
#define SEM_HOLD(a, unit) false
#define SEM_HOLD_CTA(hold) ((void)(hold), false)
#endif

// Programmatic dependent launch (PDL).  A kernel launched by launch_k may be
// scheduled before the kernel ahead of it in the stream has completed, and then
// runs its blocks up to pdl_wait(), which returns when the previous grid has
// completed and its writes are visible (griddepcontrol.wait).  Every kernel
// launched by launch_k waits in every block before it touches memory that another
// kernel writes, so that grids still complete in stream order and each kernel sees
// all earlier results.  In a kernel launched without the attribute both
// instructions return at once.  Inside a CUDA graph the attribute becomes a
// programmatic edge between the two kernel nodes.
// pdl_trigger() (griddepcontrol.launch_dependents) lets the next kernel's blocks be
// scheduled once every block has called it or ended.  It stands at the end of a
// kernel's main loop (before the reduction's tail or the last scatter), not at its
// start: blocks launched early take the SMs that come free first, up to their full
// occupancy, and leave the others without any; launched when all SMs are about to
// come free they spread evenly, and the launch latency is hidden all the same.
// Measured with the plane kernel: V-cycle on 2.06 M nodes 404 us with triggers at
// the start, 362 us at the end (476 us without the attribute).
// Before pdl_wait() a kernel may read the map, the elements' first nodes and the
// metric copies, which only the set-up writes, because a full dependency always lies
// between them.  That the set-up kernels do not trigger is not enough: their blocks
// have then ended before a kernel launched by launch_k starts, but their writes are
// promised to it by its wait only.  The full dependency is a memset or a host
// synchronisation: apply_fp32 clears y between the conversion and the apply, and the
// multigrid set-up, first or after a tissue update, ends in set_alpha's synchronisation.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
// L2 prefetch of the 128-byte lines of [p, p + bytes), line `first` and every
// `step`-th after it by this thread.
__device__ __forceinline__ void prefetch_l2_lines(const void* p, size_t bytes, int first, int step) {
  const uintptr_t a0 = reinterpret_cast<uintptr_t>(p) & ~(uintptr_t)127;
  const uintptr_t end = reinterpret_cast<uintptr_t>(p) + bytes;
  for (uintptr_t a = a0 + (uintptr_t)first * 128u; a < end; a += (uintptr_t)step * 128u)
    asm volatile("prefetch.global.L2 [%0];\n" ::"l"(a));
}
#endif
bool pdl_enabled();  // false when the environment sets SEM_NO_PDL (read once)
template <typename... P, typename... A>
cudaError_t launch_k(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                     A&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl_enabled() ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

// Storage type of the vectors an operator kernel reads and writes: the df64
// operator works on FP64 vectors.
template <typename T> struct VecOf { using type = T; };
template <> struct VecOf<df> { using type = double; };

constexpr int kMaxP = 6;
constexpr int kMaxN = kMaxP + 1;
constexpr int kMetricComps = 7;

// Quadrature points per element rounded up to a multiple of 8: every element's
// metric block and each of its 7 components then start on a 16-byte boundary
// in every storage precision (bf16, float, double, float pairs).
__host__ __device__ constexpr int padded_n3(int n) { return ((n * n * n + 7) / 8) * 8; }

// 1-D tables of one degree p and one quadrature kind (host side, double).
struct Tables1D {
  int p = 0, n = 0, quad = 0;
  double xg[kMaxN] = {}, wg[kMaxN] = {};  // LGL nodes / weights
  double xq[kMaxN] = {}, wq[kMaxN] = {};  // quadrature nodes / weights
  double D[kMaxN][kMaxN] = {};   // D[q][l] = l_l'(xg_q)  (GLL collocation derivative)
  double Bi[kMaxN][kMaxN] = {};  // Bi[q][l] = l_l(xq_q)   (GLL basis at quadrature points)
  double Dg[kMaxN][kMaxN] = {};  // Dg[q][m] = g_m'(xq_q)  (collocation derivative on the quadrature points)
};

// Builds the tables of degree p (1..kMaxP) for quad SEM_QUAD_LG / SEM_QUAD_LGL.
void build_tables(int p, int quad, Tables1D* t);

// Even-odd form of an n x n matrix M with M[n-1-q][n-1-l] = s M[q][l]: s = -1
// for a derivative matrix on points symmetric about 0 (and its transpose),
// s = +1 for interpolation between two symmetric point sets.  With H = n / 2,
// for q, l < H:
//   a[q][l] = (M[q][l] + M[q][n-1-l]) / 2,   b[q][l] = (M[q][l] - M[q][n-1-l]) / 2,
// and for odd n the middle column a[q][H] = M[q][H] and the middle row
// c[l] = M[H][l] (l <= H).  A product y = M x then takes about half the
// multiplications (see eo_line).  For n = 2 and 4 the split saves no
// multiplication, so the matrix itself (m) is kept and multiplied directly; but in
// double-float, where a multiply-add takes 13 instructions and an addition 8, the
// split is shorter at n = 4 (132 instead of 172 instructions a line).
template <int N, typename T>
struct EoMat {
  static constexpr int H = N / 2;
  static constexpr bool kDirect = (N == 2 || (N == 4 && !std::is_same<T, df>::value));
  static constexpr int NM = kDirect ? N : 1;
  T a[H][H + 1];
  T b[H][H];
  T c[H + 1];
  T m[NM][NM];
};

// Tables in the kernel's arithmetic type, passed to kernels by value (kernel
// parameter space): accesses with compile-time indices become constant-bank
// operands of the FMA instructions.
template <int N, typename T>
struct KTab {
  EoMat<N, T> D, Dt;    // derivative matrix of the gradient (D for SEM-NI, Dg for SEM), its transpose
  EoMat<N, T> Bi, Bit;  // interpolation GLL -> quadrature points (SEM only), its transpose
};

// Deterministic grid reductions: every block writes a partial, the last block
// to finish (atomic ticket) sums the partials in block order.
// Partials of the vector kernels: kVecBlocksMax per reduction slot.
constexpr int kVecBlocksMax = 2048;
constexpr int kReduceSlots = 4;

// Device scalars of one CG solve.
struct CgScalars {
  double rz;      // r . z of the current iterate
  double rr;      // r . r
  double bb;      // b . b
  double pAp;     // p . A p
  double alpha;   // step length
  double beta;    // conjugation coefficient
  double tol2;    // squared stopping threshold on ||r||
  int done;       // 1 when converged or failed
  int iters;      // iterations taken
  int status;     // 0 ok, SEM_ERR_NONFINITE
  int pad;
};

struct Level {
  int p = 0, quad = 0, n = 0;
  int nx = 0, ny = 0, nz = 0;
  int nelem = 0;
  int64_t ndofs = 0;
  Tables1D tab;
  int* map = nullptr;
  int* first = nullptr;      // [nelem] first node of each element (map[e][0])
  double* evert = nullptr;   // [nelem][8][3] element vertices
  double* metric = nullptr;  // [nelem][7][n^3]
  float* metric32 = nullptr;
  __nv_bfloat16* metric16 = nullptr;
  df_pair* metric2 = nullptr;  // FP64 metric split into FP32 pairs (df64 operator)
  uint32_t* metric_tc = nullptr;  // bf16 metric in the tensor-core kernel's order (sem_apply_tc.cu)
  uint32_t* tc_frag = nullptr;    // constant MMA fragments of the tensor-core kernel
  bool metric32_valid = false, metric16_valid = false, metric2_valid = false, metric_tc_valid = false;
  bool weight32_valid = false, weight16_valid = false;  // the weights behind them (geometry only: written once)
  unsigned long long* dbg = nullptr;  // SEM_DEBUG build: the context's index-error word
  unsigned* fault = nullptr;  // the context's wait-timeout word (nonzero: a kernel gave up a wait)
  int hold = -1;  // SEM_DEBUG build: element group whose metric copy the plane kernel skips
  double* mdiag = nullptr;
  double* kdiag = nullptr;
  double* xyz = nullptr;
};

// Number of metric values of a level (7 components x padded points per element).
inline size_t metric_count(const Level& L) {
  return (size_t)L.nelem * kMetricComps * padded_n3(L.n);
}

// Offset of component `comp` of the quadrature point on column c = i + n j at
// level k of element e.
//   double, float pairs: element-blocked, component-major [7][padded n^3], point
//   c + n^2 k;
//   float, bf16: the order in which the plane kernel consumes it.  A unit of
//   G = 32 / n consecutive elements has n / R chunks of R rows j; a chunk holds, for
//   each element of the unit and each plane k, the 7 n R values of its points, point
//   by point, in RS values.  A chunk is one contiguous copy, and RS is an odd number
//   of the loads of four values that read it (8 bytes bf16, 16 bytes float), so that
//   the loads of neighbouring lanes, each of its own plane, fall on different banks.
//   R = n at n <= 3 (one chunk), 1 above: the kernel keeps a short ring of chunks in
//   shared memory instead of the unit's whole metric.  The last unit is padded.
template <typename MT>
struct MetricLayout {
  __host__ __device__ static constexpr int block(int n) { return kMetricComps * padded_n3(n); }
  __host__ __device__ static constexpr size_t offset(int n, int64_t e, int c, int k, int comp) {
    return (size_t)e * block(n) + comp * padded_n3(n) + c + k * n * n;
  }
};
struct PlaneMetricLayout {
  __host__ __device__ static constexpr int unit(int n) { return 32 / n; }                // G
  __host__ __device__ static constexpr int rows(int n) { return n <= 3 ? n : 1; }        // R
  __host__ __device__ static constexpr int chunks(int n) { return n / rows(n); }
  __host__ __device__ static constexpr int stride(int n) {                               // RS
    return 4 * (((kMetricComps * n * rows(n) + 3) / 4) | 1);
  }
  __host__ __device__ static constexpr int chunk(int n) { return unit(n) * n * stride(n); }
  __host__ __device__ static constexpr size_t offset(int n, int64_t e, int c, int k, int comp) {
    const int64_t u = e / unit(n);
    const int s = (int)(e - u * unit(n)), i = c % n, j = c / n;
    return (size_t)(u * chunks(n) + j / rows(n)) * chunk(n) + (s * n + k) * stride(n) +
           kMetricComps * (i + n * (j % rows(n))) + comp;
  }
};
template <> struct MetricLayout<float> : PlaneMetricLayout {};
template <> struct MetricLayout<__nv_bfloat16> : PlaneMetricLayout {};

// Number of values of the float or bf16 metric of a level (whole units).
inline size_t metric_lowp_count(const Level& L) {
  using ML = PlaneMetricLayout;
  const size_t units = ((size_t)L.nelem + ML::unit(L.n) - 1) / ML::unit(L.n);
  return units * ML::chunks(L.n) * ML::chunk(L.n);
}
// Behind them, on a SEM fine level, the weights W alone, [nelem][n3p]: the FP32 mass
// operator reads nothing else, and taken from the seven values of each point they cost
// it the whole metric.  An apply on 2 M nodes, p = 1..6: FP32 99 58 40 38 35 34 us so, 92
// 49 31 25 25 25 from the FP64 metric, 83 41 29 23 23 25 from here; bf16 90 53 35 29 30 30
// and 76 40 29 23 23 24.  The other levels only apply alpha M + K.
inline size_t weight_lowp_count(const Level& L) {
  return L.quad == SEM_QUAD_LG && L.xyz != nullptr ? (size_t)L.nelem * padded_n3(L.n) : 0;
}
inline size_t metric_lowp_values(const Level& L) { return metric_lowp_count(L) + weight_lowp_count(L); }

constexpr int kScaleOut = 1, kNegateOut = 2;  // ApplyArgs::scale_out

// Arguments of the element kernel y += A_e u_e (scatter-add into y).
template <typename T, typename MT>
struct ApplyArgs {
  const int* map;
  const MT* metric;
  const typename VecOf<T>::type* u;
  typename VecOf<T>::type* y;
  int nelem;
  T mass_coef;        // coefficient of the mass term inside the element kernel
  T out_scale;        // factor applied to the element result before the scatter
  int scale_out;      // 0: out_scale is 1; kScaleOut; kNegateOut: it is -1
  const int* done;    // optional: skip all work when *done != 0
  // optional fused u . (A u) (CG's p . A p): every CTA writes its partial sum
  // to dot_partials (one double per CTA of the launch, dot_blocks of them) and a
  // one-CTA kernel launched after the apply adds them up
  double* dot_partials;
  CgScalars* cg;      // when set, the sum goes to pAp, and alpha = rz / pAp
  double* dot_out;    // otherwise the sum goes here; with neither the caller sums
  // optional (double-float operator with the fused inner product): u split into
  // float pairs by the kernel that formed u; the gather then reads the pairs and
  // converts nothing
  const df_pair* u2;
  // optional (deterministic mode): element results go to yloc[e][n^3] instead of
  // atomic adds, and a node kernel then adds each node's contributions to y in a
  // fixed order
  typename VecOf<T>::type* yloc;
  // set by the launcher: the vectors' length and strides, the elements' first
  // nodes, the SEM_DEBUG index-error word and the wait-timeout word
  int64_t ndofs;
  int row, plane;  // lattice strides: nodes of an x-row and of an (x, y) plane
  const int* first;  // Level::first
  unsigned long long* dbg;
  unsigned* fault;
  int hold;  // SEM_DEBUG build: Level::hold
};
using ApplyArgs64 = ApplyArgs<double, double>;

// Kernel launchers (sem_apply_fp64.cu, sem_apply_fp32.cu).
cudaError_t launch_apply_fp64(const Level& L, const ApplyArgs64& a, bool mass_only, cudaStream_t s);
cudaError_t launch_apply_fp32(const Level& L, const ApplyArgs<float, float>& a, bool mass_only,
                              cudaStream_t s);
cudaError_t launch_apply_bf16(const Level& L, const ApplyArgs<float, __nv_bfloat16>& a,
                              bool mass_only, cudaStream_t s);
cudaError_t launch_apply_df64(const Level& L, const ApplyArgs<df, df_pair>& a, bool mass_only,
                              cudaStream_t s);
int apply_grid_blocks(const Level& L);
// Partials the FP64 (or, df64 set, the double-float) apply with the inner product writes.
int dot_blocks(const Level& L, bool df64);
// y[g] += the element contributions yloc[e][n^3] of node g, elements in a fixed
// order (ez, ey, ex ascending): the deterministic assembly of the apply kernels'
// element results.
cudaError_t launch_assemble(const Level& L, const double* yloc, double* y, const int* done, cudaStream_t s);
cudaError_t launch_assemble(const Level& L, const float* yloc, float* y, const int* done, cudaStream_t s);
// Sum, in a fixed order, of the n per-CTA partials of a fused inner product:
// to cg (pAp and alpha = rz / pAp) when set, else to *out; nothing when *done.
cudaError_t launch_apply_dot_finish(const double* partials, int n, CgScalars* cg, double* out,
                                    const int* done, cudaStream_t s);
// Raises the dynamic shared-memory limit of the kernels that stage the metric in
// shared memory; call once per device before any stream capture.
cudaError_t prime_apply_kernels();

// Tensor-core FP32 operator with the bf16 metric (sem_apply_tc.cu): SEM-NI, p = 2..4.
bool tc_supported(const Level& L);
size_t tc_metric_words(const Level& L);
// Builds the level's metric_tc (from the FP64 metric) and constant fragments.
cudaError_t setup_metric_tc(Level& L, cudaStream_t s);
// y += (mass_coef M + K) u with a.u, a.y float vectors (a.map, a.metric unused).
cudaError_t launch_apply_tc(const Level& L, const ApplyArgs<float, __nv_bfloat16>& a, cudaStream_t s);
cudaError_t prime_apply_tc();

// Level construction (sem_setup.cu): structured numbering of an nx x ny x nz
// slab with host vertices, device allocation of map, element vertices, metric,
// diagonals (and node coordinates when `coords`).  Metric and diagonals are
// filled by setup_geometry / setup_diagonals.
cudaError_t level_create(Level& L, int nx, int ny, int nz, const double* vertices, int p, int quad,
                         bool coords, cudaStream_t s);
void level_free(Level& L);

// Setup kernels (sem_setup.cu).
cudaError_t setup_geometry(Level& L, const double* sigma_l, const double* sigma_t,
                           const double* theta, int* d_bad, cudaStream_t s);
cudaError_t setup_diagonals(Level& L, cudaStream_t s);
cudaError_t setup_metric_lowp(Level& L, bool bf16, cudaStream_t s);
cudaError_t setup_metric_df(Level& L, cudaStream_t s);
cudaError_t setup_node_coords(Level& L, cudaStream_t s);
cudaError_t setup_region_mask(const Level& L, int region, const double* prm, double* mask,
                              cudaStream_t s);

// CG of a small mesh in one kernel (sem_cg_small.cu): the solve of cg_solve with the FP64
// operator, inv = 1 / diagonal or nullptr.  At most 64 iterations a launch; resume
// continues from x, r, p and *sc.  p and Ap are scratch.  cg_small_fits: whether it takes
// the mesh and the current device can place its cluster (of at most max_ctas CTAs); it
// must have returned true before launch_cg_small.
bool cg_small_fits(const Level& L, int max_ctas);
cudaError_t launch_cg_small(const Level& L, double alpha, const double* b, const double* inv, const double* ax0, double* x,
                            double* r, double* p, double* Ap, CgScalars* sc, double rtol, double atol, int maxit,
                            bool resume, cudaStream_t s);

// Vector kernels (sem_solver.cu).
int vec_blocks(int64_t n);
cudaError_t vec_axpby_diag(int64_t n, double a, const double* x, double b, const double* y,
                           double* out, cudaStream_t s);  // out = a x + b y
cudaError_t vec_inv_diag(int64_t n, double alpha, const double* mdiag, const double* kdiag,
                         double* inv, cudaStream_t s);     // inv = 1/(alpha m + k)
cudaError_t vec_scale_mul(int64_t n, double a, const double* d, const double* x, double* y,
                          cudaStream_t s);                 // y = a d x

}  // namespace sem
