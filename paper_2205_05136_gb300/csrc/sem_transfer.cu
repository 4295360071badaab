// p-multigrid transfers between Q_pf and Q_pc on the same slab mesh
// (Section 4.3: transfers are matrix-vector products).
//
// On the structured slab lattice the global prolongation is the tensor product
// P = Pz Py Px of 1-D global prolongations: along x, fine node I of element
// e = min(I / pf, nx - 1) takes sum_a P[I - pf e][a] x_c[pc e + a], with
// P[i][a] = l^c_a(x^f_i) the 1-D interpolation matrix.  A node on an element
// boundary gets the same value from either element, because the interpolation
// is exact at the shared end points (rows 0 and pf of P are unit rows).  So
//   prolongation  d_f = P x_c, x_f += d_f: three 1-D passes, coarse lattice ->
//                 (NXc, NYc, NZf) -> (NXc, NYf, NZf) -> fine lattice;
//   restriction   r_c = P^T r_f: three 1-D passes the other way,
//                 coarse node A summing P1[I][A] over the fine nodes I of the
//                 elements that hold it, each fine node once.
// Both run as one kernel: a CTA takes a brick of elements and contracts along one
// axis after the other, and writes the nodes that it owns (those of its elements
// without the upper faces, which belong to the next brick; the mesh's last nodes with
// its last brick).  A restriction reads one element more on the lower sides.  The
// lanes of a warp are neighbours in x, so global rows are read and written whole; the
// z-contraction runs on registers with all its loads in flight, the y- and
// x-contractions on shared memory, every coefficient a constant-bank operand.  Values
// outside the mesh read as zero, which makes the edges of the mesh no special case.
// Every node is written by one thread and summed in a fixed order, so the result is
// the same in every run (the deterministic mode needs no variant).  Latency bounds
// it: one global read, two short passes between barriers.  Restriction and
// prolongation as three kernels each, through two scratch lattices in global memory,
// took the V-cycle on 2.06 M nodes 331 us, these 326; one kernel with the whole brick in
// shared memory and one node a thread in every pass 343 (index arithmetic).
#include <algorithm>

#include "sem_apply_kernel.cuh"
#include "sem_context.cuh"

namespace sem {
namespace {

template <int NF, int NC, typename T>
struct PMat {
  T P[NF][NC];
};

// Elements of a brick: in x as many as 32 lanes hold fine nodes of a restriction,
// PF (X + 1) <= 32; a warp for each of its PF (Y + 1) fine rows.
template <int PF> struct Brick;
template <> struct Brick<2> { static constexpr int X = 15, Y = 4, Z = 8; };
template <> struct Brick<3> { static constexpr int X = 9, Y = 3, Z = 4; };
template <> struct Brick<4> { static constexpr int X = 7, Y = 2, Z = 4; };
template <> struct Brick<5> { static constexpr int X = 5, Y = 1, Z = 2; };
template <> struct Brick<6> { static constexpr int X = 4, Y = 1, Z = 2; };

template <int NF, int NC>
struct BrickCfg {
  static constexpr int PF = NF - 1, PC = NC - 1;
  using B = Brick<PF>;
  // fine nodes read by a restriction (from PF (e0 - 1) + 1 on), coarse nodes and fine
  // nodes of the brick, closing ones included
  static constexpr int RX = PF * (B::X + 1), RY = PF * (B::Y + 1), RZ = PF * (B::Z + 1);
  static constexpr int CX = PC * B::X + 1, CY = PC * B::Y + 1, CZ = PC * B::Z + 1;
  static constexpr int FX = PF * B::X + 1, FY = PF * B::Y + 1, FZ = PF * B::Z + 1;
  static constexpr int kWarps = RY, kThreads = 32 * kWarps;
  static_assert(RX <= 32 && FX <= 32 && FY <= kWarps, "a row of the brick is one warp");
};

// Position of a brick: its first element along each axis, the elements inside the
// mesh, and the owned coarse and fine nodes (the closing one with the last brick).
template <int NF, int NC>
struct BrickPos {
  using C = BrickCfg<NF, NC>;
  int ex, ey, ez, lx, ly, lz, cx, cy, cz, fx, fy, fz;
  __device__ __forceinline__ BrickPos(int nx, int ny, int nz) {
    using B = typename C::B;
    const int bx = (nx + B::X - 1) / B::X, by = (ny + B::Y - 1) / B::Y, i = blockIdx.x;
    ex = (i % bx) * B::X;
    ey = (i / bx % by) * B::Y;
    ez = (i / bx / by) * B::Z;
    lx = min(B::X, nx - ex);
    ly = min(B::Y, ny - ey);
    lz = min(B::Z, nz - ez);
    const int tx = ex + lx == nx, ty = ey + ly == ny, tz = ez + lz == nz;
    cx = C::PC * lx + tx;
    cy = C::PC * ly + ty;
    cz = C::PC * lz + tz;
    fx = C::PF * lx + tx;
    fy = C::PF * ly + ty;
    fz = C::PF * lz + tz;
  }
};

// The coarse nodes of E elements and the closing one from their fine nodes f, f[0]
// the first node inside the element before: out(c, value) for c = 0 .. PC E.
template <int NF, int NC, int E, typename T, typename F>
__device__ __forceinline__ void restrict_line(const PMat<NF, NC, T>& pm, const T (&f)[(NF - 1) * (E + 1)], F out) {
  constexpr int PF = NF - 1, PC = NC - 1;
#pragma unroll
  for (int e = 0; e <= E; ++e) {
    const int v = PF * (e + 1) - 1;  // the vertex between the elements e - 1 and e
    T acc = f[v];
#pragma unroll
    for (int i = 1; i < PF; ++i) acc = fma(pm.P[i][PC], f[v - PF + i], acc);
    if (e < E) {
#pragma unroll
      for (int i = 1; i < PF; ++i) acc = fma(pm.P[i][0], f[v + i], acc);
    }
    out(PC * e, acc);
    if (e < E) {
#pragma unroll
      for (int a = 1; a < PC; ++a) {
        T s = pm.P[1][a] * f[v + 1];
#pragma unroll
        for (int i = 2; i < PF; ++i) s = fma(pm.P[i][a], f[v + i], s);
        out(PC * e + a, s);
      }
    }
  }
}

// The fine nodes of E elements and the closing one from their coarse nodes:
// out(i, value) for i = 0 .. PF E.
template <int NF, int NC, int E, typename T, typename F>
__device__ __forceinline__ void prolong_line(const PMat<NF, NC, T>& pm, const T (&c)[(NC - 1) * E + 1], F out) {
  constexpr int PF = NF - 1, PC = NC - 1;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    out(PF * e, c[PC * e]);
#pragma unroll
    for (int i = 1; i < PF; ++i) {
      T acc = pm.P[i][0] * c[PC * e];
#pragma unroll
      for (int a = 1; a < NC; ++a) acc = fma(pm.P[i][a], c[PC * e + a], acc);
      out(PF * e + i, acc);
    }
  }
  out(PF * E, c[PC * E]);
}

template <int NF, int NC, typename T>
__global__ void __launch_bounds__(BrickCfg<NF, NC>::kThreads)
    k_restrict_p(int nx, int ny, int nz, const T* __restrict__ in, T* __restrict__ out,
                 const __grid_constant__ PMat<NF, NC, T> pm, const int* done) {
  using C = BrickCfg<NF, NC>;
  using B = typename C::B;
  constexpr int PF = C::PF, PC = C::PC;
  __shared__ T s1[C::CZ][C::RY][32];
  __shared__ T s2[C::CZ][C::CY][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const BrickPos<NF, NC> q(nx, ny, nz);
  const int xf = PF * nx + 1, yf = PF * ny + 1, zf = PF * nz + 1;
  pdl_wait();
  const bool stop = done != nullptr && *done;  // acted on before the first store (sem_gmg.cu, skip)
  {  // z: the lane's column (x, y) of the fine nodes
    const int x = PF * (q.ex - 1) + 1 + lane, y = PF * (q.ey - 1) + 1 + warp, z0 = PF * (q.ez - 1) + 1;
    const bool col = lane < C::RX && x >= 0 && x < xf && y >= 0 && y < yf;
    const T* p = in + x + (int64_t)xf * (y + (int64_t)yf * z0);
    T f[C::RZ];
#pragma unroll
    for (int k = 0; k < C::RZ; ++k) f[k] = (col && z0 + k >= 0 && z0 + k < zf) ? p[(int64_t)xf * yf * k] : T(0);
    if (stop) return;
    restrict_line<NF, NC, B::Z>(pm, f, [&](int c, T v) { s1[c][warp][lane] = v; });
  }
  __syncthreads();
  pdl_trigger();
  for (int t = threadIdx.x; t < C::CZ * 32; t += C::kThreads) {  // y: one (z, x) a thread
    T f[C::RY];
#pragma unroll
    for (int j = 0; j < C::RY; ++j) f[j] = s1[t >> 5][j][t & 31];
    restrict_line<NF, NC, B::Y>(pm, f, [&](int c, T v) { s2[t >> 5][c][t & 31] = v; });
  }
  __syncthreads();
  const int xc = PC * nx + 1, yc = PC * ny + 1;
  constexpr int EX = B::X + 1;  // x: one element (or the closing node) of one row a thread
  for (int t = threadIdx.x; t < C::CZ * C::CY * EX; t += C::kThreads) {
    const int e = t % EX, y = t / EX % C::CY, z = t / (EX * C::CY);
    if (y >= q.cy || z >= q.cz || PC * e >= q.cx) continue;
    T f[2 * PF];
#pragma unroll
    for (int i = 0; i < 2 * PF; ++i) f[i] = (e < B::X || i < PF) ? s2[z][y][PF * e + i] : T(0);
    T* o = out + PC * (q.ex + e) + (int64_t)xc * (PC * q.ey + y + (int64_t)yc * (PC * q.ez + z));
    restrict_line<NF, NC, 1>(pm, f, [&](int c, T v) {
      if (c < PC && PC * e + c < q.cx) o[c] = v;
    });
  }
}

template <int NF, int NC, typename T>
__global__ void __launch_bounds__(BrickCfg<NF, NC>::kThreads)
    k_prolong_p(int nx, int ny, int nz, const T* __restrict__ in, T* __restrict__ out, T* __restrict__ out_d,
                const __grid_constant__ PMat<NF, NC, T> pm, const int* done) {
  using C = BrickCfg<NF, NC>;
  using B = typename C::B;
  constexpr int PF = C::PF, PC = C::PC;
  __shared__ T s1[C::CZ][C::CY][32];
  __shared__ T s2[C::CZ][C::FY][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const BrickPos<NF, NC> q(nx, ny, nz);
  const int xc = PC * nx + 1, yc = PC * ny + 1;
  pdl_wait();
  const bool stop = done != nullptr && *done;  // acted on before the first store (sem_gmg.cu, skip)
  // the fine column (x, y) of the lane, read while the coarse nodes are
  const int xf = PF * nx + 1, yf = PF * ny + 1;
  const int64_t o = PF * q.ex + lane + (int64_t)xf * (PF * q.ey + warp + (int64_t)yf * (PF * q.ez)),
                zs = (int64_t)xf * yf;
  const bool col = warp < q.fy && lane < q.fx;
  T x[C::FZ];
#pragma unroll
  for (int i = 0; i < C::FZ; ++i) x[i] = col && i < q.fz ? out[o + zs * i] : T(0);
  for (int t = threadIdx.x; t < C::CZ * C::CY * B::X; t += C::kThreads) {  // x: one element of one row a thread
    const int e = t % B::X, y = t / B::X % C::CY, z = t / (B::X * C::CY);
    if (e >= q.lx) continue;
    const bool inside = y <= PC * q.ly && z <= PC * q.lz;
    const T* p = in + PC * (q.ex + e) + (int64_t)xc * (PC * q.ey + y + (int64_t)yc * (PC * q.ez + z));
    T c[NC];
#pragma unroll
    for (int a = 0; a < NC; ++a) c[a] = inside ? p[a] : T(0);
    prolong_line<NF, NC, 1>(pm, c, [&](int i, T v) {
      if (i < PF || e == q.lx - 1) s1[z][y][PF * e + i] = v;
    });
  }
  if (stop) return;
  __syncthreads();
  for (int t = threadIdx.x; t < C::CZ * 32; t += C::kThreads) {  // y: one (z, x) a thread
    T c[C::CY];
#pragma unroll
    for (int j = 0; j < C::CY; ++j) c[j] = s1[t >> 5][j][t & 31];
    prolong_line<NF, NC, B::Y>(pm, c, [&](int i, T v) { s2[t >> 5][i][t & 31] = v; });
  }
  __syncthreads();
  if (col) {  // z
    T c[C::CZ];
#pragma unroll
    for (int k = 0; k < C::CZ; ++k) c[k] = s2[k][warp][lane];
    prolong_line<NF, NC, B::Z>(pm, c, [&](int i, T v) {
      if (i < q.fz) {
        out_d[o + zs * i] = v;
        out[o + zs * i] = x[i] + v;
      }
    });
  }
  pdl_trigger();
}

template <int NF, int NC, typename T>
cudaError_t launch_transfer(bool prolong, const Level& F, const double (*P)[kMaxN], const T* src, T* dst, T* dst_d,
                            const int* done, cudaStream_t s) {
  using C = BrickCfg<NF, NC>;
  using B = typename C::B;
  PMat<NF, NC, T> pm;
  for (int i = 0; i < NF; ++i)
    for (int a = 0; a < NC; ++a) pm.P[i][a] = (T)P[i][a];
  const int nx = F.nx, ny = F.ny, nz = F.nz;
  const int64_t bricks = (int64_t)((nx + B::X - 1) / B::X) * ((ny + B::Y - 1) / B::Y) * ((nz + B::Z - 1) / B::Z);
  if (prolong)
    return launch_k(k_prolong_p<NF, NC, T>, (unsigned)bricks, C::kThreads, 0, s, nx, ny, nz, src, dst, dst_d, pm, done);
  return launch_k(k_restrict_p<NF, NC, T>, (unsigned)bricks, C::kThreads, 0, s, nx, ny, nz, src, dst, pm, done);
}

}  // namespace

// prolong: dst_d (fine d) = P src (coarse x), dst (fine x) += dst_d.
// restrict: dst (coarse r) = P^T src (fine r).
template <typename T>
cudaError_t p_transfer(bool prolong, const Level& F, const Level& C, const double (*P)[kMaxN], const T* src, T* dst,
                       T* dst_d, const int* done, cudaStream_t s) {
  const int nf = F.n, nc = C.n;
#define SEM_PAIR(A, B) \
  if (nf == A && nc == B) return launch_transfer<A, B, T>(prolong, F, P, src, dst, dst_d, done, s);
  SEM_PAIR(7, 4)
  SEM_PAIR(6, 3)
  SEM_PAIR(5, 3)
  SEM_PAIR(4, 2)
  SEM_PAIR(3, 2)
#undef SEM_PAIR
  return cudaErrorInvalidValue;
}

template cudaError_t p_transfer<float>(bool, const Level&, const Level&, const double (*)[kMaxN], const float*, float*,
                                       float*, const int*, cudaStream_t);
template cudaError_t p_transfer<double>(bool, const Level&, const Level&, const double (*)[kMaxN], const double*,
                                        double*, double*, const int*, cudaStream_t);

}  // namespace sem
