// Setup kernels: node coordinates, quadrature-point metric terms with the
// fibre conductivity tensor, assembled diagonals, stimulus masks and the
// low-precision metric copies.
//
// Metric (Section 4: "the Jacobian of the transformation ... is cached";
// Section 4.2: D evaluated at every quadrature point, Eq. diffusiontensor):
//   J[d][c] = dx_d / dxi_c at each quadrature point, the derivative of the
//   element's trilinear map,
//   D_e = sigma_t I + (sigma_l - sigma_t) f f^T,  f = (cos theta, sin theta, 0),
//   G   = w |det J| J^{-1} D_e J^{-T}  (6 entries),  W = w |det J|.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "sem_internal.cuh"

namespace sem {
namespace {

struct SetupTab {
  int n;
  double xg[kMaxN];          // LGL nodes
  double xq[kMaxN];          // quadrature nodes
  double wq[kMaxN];          // quadrature weights
  double Bq[kMaxN][kMaxN];   // GLL basis at the quadrature points (identity for SEM-NI)
  double Dq[kMaxN][kMaxN];   // derivative of the GLL basis at the quadrature points
};

SetupTab make_setup_tab(const Tables1D& t) {
  SetupTab s{};
  s.n = t.n;
  for (int i = 0; i < t.n; ++i) { s.xg[i] = t.xg[i]; s.xq[i] = t.xq[i]; s.wq[i] = t.wq[i]; }
  for (int q = 0; q < t.n; ++q)
    for (int l = 0; l < t.n; ++l) {
      s.Bq[q][l] = t.Bi[q][l];
      double d = 0.0;
      if (t.quad == SEM_QUAD_LGL) {
        d = t.D[q][l];
      } else {
        for (int m = 0; m < t.n; ++m) d += t.Dg[q][m] * t.Bi[m][l];
      }
      s.Dq[q][l] = d;
    }
  return s;
}

__device__ __forceinline__ double trilinear(const double (*V)[3], int d, double x, double y,
                                            double z) {
  double acc = 0.0;
#pragma unroll
  for (int v = 0; v < 8; ++v) {
    const double sx = (v & 1) ? 1.0 : -1.0, sy = (v & 2) ? 1.0 : -1.0, sz = (v & 4) ? 1.0 : -1.0;
    const double N = 0.125 * (1.0 + sx * x) * (1.0 + sy * y) * (1.0 + sz * z);
    acc += N * V[v][d];
  }
  return acc;
}

constexpr int kSetupThreads = 256;
// Elements of a CTA of the metric and diagonal kernels: about four points a thread.
__host__ __device__ constexpr int setup_elems(int n3) { return n3 < 1024 ? 1024 / n3 : 1; }

// Metric of E elements per CTA, one quadrature point a thread and turn.  The trilinear
// map x_d = c0 + c1 xi + c2 eta + c3 xi eta + c4 zeta + c5 xi zeta + c6 eta zeta +
// c7 xi eta zeta is kept by its coefficients, so a column of J takes three
// multiply-adds an entry; with A = adj J = det J J^{-1} (rows the cross products of
// J's columns), G = w / det A D_e A^T takes one division.  About 100 FP64 operations a
// point, which bound the kernel (2 a clock and SM); differentiating the nodal
// coordinates and dividing nine entries took about 400 (2.0 ms on 15,410 elements at
// p = 5, now 0.60 ms).
template <int N>
__global__ void __launch_bounds__(kSetupThreads)
    k_metric(int nelem, const double* __restrict__ evert, const double* __restrict__ sigma_l,
             const double* __restrict__ sigma_t, const double* __restrict__ theta,
             const __grid_constant__ SetupTab tab, double* __restrict__ metric, int* bad) {
  constexpr int N2 = N * N, N3 = N2 * N, E = setup_elems(N3), N3P = padded_n3(N);
  __shared__ double coef[E][3][8];
  __shared__ double tens[E][4];  // sigma_t, sigma_l - sigma_t, cos theta, sin theta
  __shared__ double xq[N], wq[N];
  const int e0 = blockIdx.x * E, ne = min(E, nelem - e0);
  if (threadIdx.x < N) {
    xq[threadIdx.x] = tab.xq[threadIdx.x];
    wq[threadIdx.x] = tab.wq[threadIdx.x];
  }
  for (int t = threadIdx.x; t < ne * 3; t += kSetupThreads) {
    const int el = t / 3, d = t - 3 * el;
    const double* v = evert + (size_t)(e0 + el) * 24 + d;
    double x[8];
    for (int i = 0; i < 8; ++i) x[i] = v[3 * i];
    // sums and differences over the corners' bits (1: xi, 2: eta, 4: zeta)
    for (int bit = 1; bit < 8; bit <<= 1)
      for (int i = 0; i < 8; ++i)
        if (!(i & bit)) {
          const double lo = x[i], hi = x[i | bit];
          x[i] = 0.5 * (hi + lo);
          x[i | bit] = 0.5 * (hi - lo);
        }
    for (int i = 0; i < 8; ++i) coef[el][d][i] = x[i];
  }
  for (int el = threadIdx.x; el < ne; el += kSetupThreads) {
    const double st = sigma_t[e0 + el], th = theta[e0 + el];
    tens[el][0] = st;
    tens[el][1] = sigma_l[e0 + el] - st;
    tens[el][2] = cos(th);
    tens[el][3] = sin(th);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < ne * N3; t += kSetupThreads) {
    const int el = t / N3, a = t - el * N3, qx = a % N, qy = a / N % N, qz = a / N2;
    const double x = xq[qx], y = xq[qy], z = xq[qz];
    double J[3][3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double* c = coef[el][d];  // index bits: 1 xi, 2 eta, 4 zeta
      J[d][0] = fma(z, fma(y, c[7], c[5]), fma(y, c[3], c[1]));
      J[d][1] = fma(z, fma(x, c[7], c[6]), fma(x, c[3], c[2]));
      J[d][2] = fma(y, fma(x, c[7], c[6]), fma(x, c[5], c[4]));
    }
    double A[3][3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int p = (r + 1) % 3, q = (r + 2) % 3;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const int u = (d + 1) % 3, v = (d + 2) % 3;
        A[r][d] = fma(J[u][p], J[v][q], -(J[v][p] * J[u][q]));
      }
    }
    const double det = fma(J[2][0], A[0][2], fma(J[1][0], A[0][1], J[0][0] * A[0][0]));
    if (!(det > 0.0)) atomicExch(bad, 1);
    const double w = wq[qx] * wq[qy] * wq[qz], s = w / det;
    const double st = s * tens[el][0], sd = s * tens[el][1], f0 = tens[el][2], f1 = tens[el][3];
    double af[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) af[r] = fma(A[r][1], f1, A[r][0] * f0);
    double* out = metric + (size_t)(e0 + el) * kMetricComps * N3P + a;
    auto g = [&](int r, int c) {
      const double aa = fma(A[r][2], A[c][2], fma(A[r][1], A[c][1], A[r][0] * A[c][0]));
      return fma(sd * af[r], af[c], st * aa);
    };
    out[0 * N3P] = g(0, 0);
    out[1 * N3P] = g(0, 1);
    out[2 * N3P] = g(0, 2);
    out[3 * N3P] = g(1, 1);
    out[4 * N3P] = g(1, 2);
    out[5 * N3P] = g(2, 2);
    out[6 * N3P] = w * det;
  }
}

// Node coordinates; each global node is written by exactly one element (the
// highest-index element that holds it).
__global__ void k_nodes(int nelem, int nx, int ny, int nz, const double* __restrict__ evert,
                        const int* __restrict__ map, const __grid_constant__ SetupTab tab,
                        int64_t ndofs, double* __restrict__ xyz) {
  const int e = blockIdx.x;
  if (e >= nelem) return;
  const int n = tab.n, p = n - 1, n3 = n * n * n;
  const int ex = e % nx, ey = (e / nx) % ny, ez = e / (nx * ny);
  __shared__ double V[8][3];
  if (threadIdx.x < 24) V[threadIdx.x / 3][threadIdx.x % 3] = evert[(size_t)e * 24 + threadIdx.x];
  __syncthreads();
  for (int a = threadIdx.x; a < n3; a += blockDim.x) {
    const int i = a % n, j = (a / n) % n, k = a / (n * n);
    const bool own = (i < p || ex == nx - 1) && (j < p || ey == ny - 1) && (k < p || ez == nz - 1);
    if (!own) continue;
    const int g = map[(size_t)e * n3 + a];
    for (int d = 0; d < 3; ++d) xyz[d * ndofs + g] = trilinear(V, d, tab.xg[i], tab.xg[j], tab.xg[k]);
  }
}

// Assembled diagonals of M and K: per element and local node a,
//   M_aa = sum_q W_q phi_a(q)^2,  K_aa = sum_q grad phi_a(q) . G_q grad phi_a(q)
// (reference gradients; G already holds J^{-1} D J^{-T} w |det J|).  With the 1-D
// tables' products bb = B^2, bd = B D, dd = D^2 every term is separable:
//   K_aa: G00 (dd bb bb) + G11 (bb dd bb) + G22 (bb bb dd)
//         + 2 G01 (bd bd bb) + 2 G02 (bd bb bd) + 2 G12 (bb bd bd),
//   M_aa: W (bb bb bb)                                       (factors along x y z).
// SEM-NI (k_diagonals_ni): B is the identity, so a node sums three lines of points and
// its own point.  SEM (k_diagonals): three sweeps over 7, 7 and 4 fields.  The direct
// sum over all points of every node took n^6 terms an element: 31.9 ms on 15,410
// elements at p = 5, now 0.15 ms (SEM-NI) and 0.67 ms (SEM).
template <int N>
__global__ void __launch_bounds__(kSetupThreads)
    k_diagonals_ni(int nelem, const int* __restrict__ map, const double* __restrict__ metric,
                   const __grid_constant__ SetupTab tab, double* __restrict__ mdiag, double* __restrict__ kdiag) {
  constexpr int N2 = N * N, N3 = N2 * N, E = setup_elems(N3), N3P = padded_n3(N);
  __shared__ double dd[N][N], dq[N];  // D[q][a]^2, D[a][a]
  const int e0 = blockIdx.x * E, ne = min(E, nelem - e0);
  if (threadIdx.x < N2) {
    const int q = threadIdx.x / N, a = threadIdx.x % N;
    dd[q][a] = tab.Dq[q][a] * tab.Dq[q][a];
    if (q == a) dq[a] = tab.Dq[a][a];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < ne * N3; t += kSetupThreads) {
    const int el = t / N3, a = t - el * N3, i = a % N, j = a / N % N, k = a / N2;
    const double* me = metric + (size_t)(e0 + el) * kMetricComps * N3P;
    const double *mx = me + (a - i), *my = me + 3 * N3P + (a - j * N), *mz = me + 5 * N3P + (a - k * N2);
    double s = 2.0 * (me[1 * N3P + a] * dq[i] * dq[j] + me[2 * N3P + a] * dq[i] * dq[k] + me[4 * N3P + a] * dq[j] * dq[k]);
#pragma unroll
    for (int q = 0; q < N; ++q)
      s = fma(mz[q * N2], dd[q][k], fma(my[q * N], dd[q][j], fma(mx[q], dd[q][i], s)));
    const int g = map[(size_t)(e0 + el) * N3 + a];
    atomicAdd(mdiag + g, me[6 * N3P + a]);
    atomicAdd(kdiag + g, s);
  }
}

template <int N>
__global__ void __launch_bounds__(kSetupThreads)
    k_diagonals(int nelem, const int* __restrict__ map, const double* __restrict__ metric,
                const __grid_constant__ SetupTab tab, double* __restrict__ mdiag, double* __restrict__ kdiag) {
  constexpr int N2 = N * N, N3 = N2 * N, N3P = padded_n3(N), E = N3 < 256 ? 256 / N3 : 1;
  // [0..2]: bb, bd, dd; fields after the x-sweep (7) and after the y-sweep (4)
  __shared__ double T[3][N][N];
  __shared__ double X[7][E * N3];
  __shared__ double Y[4][E * N3];
  const int e0 = blockIdx.x * E, ne = min(E, nelem - e0);
  if (threadIdx.x < N2) {
    const int q = threadIdx.x / N, a = threadIdx.x % N;
    const double B = tab.Bq[q][a], D = tab.Dq[q][a];
    T[0][q][a] = B * B;
    T[1][q][a] = B * D;
    T[2][q][a] = D * D;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < ne * N3; t += kSetupThreads) {
    const int el = t / N3, a = t - el * N3, i = a % N;
    const double* me = metric + (size_t)(e0 + el) * kMetricComps * N3P + (a - i);
    double s[7] = {0, 0, 0, 0, 0, 0, 0};  // G00 dd, G01 bd, G02 bd, G11 bb, G12 bb, G22 bb, W bb
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const double bb = T[0][q][i], bd = T[1][q][i], dd = T[2][q][i];
      s[0] = fma(me[q], dd, s[0]);
      s[1] = fma(me[N3P + q], bd, s[1]);
      s[2] = fma(me[2 * N3P + q], bd, s[2]);
#pragma unroll
      for (int c = 3; c < 7; ++c) s[c] = fma(me[c * N3P + q], bb, s[c]);
    }
    for (int c = 0; c < 7; ++c) X[c][t] = s[c];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < ne * N3; t += kSetupThreads) {
    const int j = t / N % N, b = t - j * N;
    double v0 = 0, v1 = 0, v2 = 0, v3 = 0;  // with bb, bd, dd along z, and the mass
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const double bb = T[0][q][j], bd = T[1][q][j], dd = T[2][q][j];
      const int p = b + q * N;
      v0 = fma(X[0][p], bb, fma(X[3][p], dd, fma(2.0 * X[1][p], bd, v0)));
      v1 = fma(X[2][p], bb, fma(X[4][p], bd, v1));
      v2 = fma(X[5][p], bb, v2);
      v3 = fma(X[6][p], bb, v3);
    }
    Y[0][t] = v0;
    Y[1][t] = 2.0 * v1;
    Y[2][t] = v2;
    Y[3][t] = v3;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < ne * N3; t += kSetupThreads) {
    const int k = t / N2 % N, b = t - k * N2;
    double ks = 0, ms = 0;
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const int p = b + q * N2;
      ks = fma(Y[0][p], T[0][q][k], fma(Y[1][p], T[1][q][k], fma(Y[2][p], T[2][q][k], ks)));
      ms = fma(Y[3][p], T[0][q][k], ms);
    }
    const int g = map[(size_t)e0 * N3 + t];
    atomicAdd(mdiag + g, ms);
    atomicAdd(kdiag + g, ks);
  }
}

__global__ void k_region_mask(int64_t ndofs, const double* __restrict__ xyz, int region,
                              double a0, double a1, double a2, double a3, double a4, double a5,
                              double* __restrict__ mask) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ndofs;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double x = xyz[i], y = xyz[ndofs + i], z = xyz[2 * ndofs + i];
    bool in;
    if (region == SEM_REGION_BOX) {
      in = x >= a0 && y >= a1 && z >= a2 && x <= a3 && y <= a4 && z <= a5;
    } else {
      const double dx = x - a0, dy = y - a1, dz = z - a2;
      in = dx * dx + dy * dy + dz * dz <= a3 * a3;
    }
    mask[i] = in ? 1.0 : 0.0;
  }
}

template <typename OT>
__device__ __forceinline__ OT metric_round(double v);
template <>
__device__ __forceinline__ float metric_round<float>(double v) { return __double2float_rn(v); }
template <>
__device__ __forceinline__ __nv_bfloat16 metric_round<__nv_bfloat16>(double v) {
  return __float2bfloat16_rn(__double2float_rn(v));
}

// FP64 component-major metric -> the plane kernel's low-precision order (MetricLayout);
// zero in the padding.  A CTA rounds the values of E elements into shared memory as it
// reads them (coalesced: an element is one contiguous block) and writes them in the
// target's order, four values a thread and store; every index is split by constants.
// DRAM bounds it.  A thread per target value, with 64-bit divisions by run-time sizes
// and 8-byte loads seven components apart, took 2.46 ms on 462,024 elements at p = 4 for
// bf16 and 2.36 for FP32; now 0.69 and 0.88 (6.2 TB/s both).  weight: where W alone goes
// too (weight_lowp_count), or nullptr.
template <int N, typename OT>
__global__ void __launch_bounds__(kSetupThreads)
    k_convert_planes(int nelem, int padded, const double* __restrict__ in, OT* __restrict__ out,
                     OT* __restrict__ weight) {
  using ML = MetricLayout<OT>;
  constexpr int N2 = N * N, N3P = padded_n3(N), E = setup_elems(N2 * N), block = kMetricComps * N3P;
  constexpr int R = ML::rows(N), chunks = ML::chunks(N), RS = ML::stride(N), G = ML::unit(N);
  constexpr int vectors = chunks * N * (RS / 4);  // an element's stores of four values
  struct alignas(4 * sizeof(OT)) Four { OT v[4]; };
  __shared__ OT m[E * block];
  const int e0 = blockIdx.x * E, ne = min(E, nelem - e0), nout = min(E, padded - e0);
#pragma unroll 8
  for (int t = threadIdx.x; t < ne * block; t += kSetupThreads) m[t] = metric_round<OT>(__ldcs(in + (size_t)e0 * block + t));
  __syncthreads();
  if (weight != nullptr)
    for (int t = threadIdx.x; t < ne * N3P; t += kSetupThreads)
      weight[(size_t)e0 * N3P + t] = m[t / N3P * block + 6 * N3P + t % N3P];
  for (int t = threadIdx.x; t < nout * vectors; t += kSetupThreads) {
    const int el = t / vectors, q = t - el * vectors, v0 = 4 * (q % (RS / 4)), k = q / (RS / 4) % N,
              chunk = q / (RS / 4) / N, e = e0 + el, unit = e / G, slot = e - unit * G;
    Four w;
    for (int i = 0; i < 4; ++i) {
      const int point = (v0 + i) / kMetricComps, comp = (v0 + i) - kMetricComps * point;
      w.v[i] = el < ne && point < R * N ? m[el * block + comp * N3P + chunk * R * N + point + N2 * k] : metric_round<OT>(0.0);
    }
    *(Four*)(out + (size_t)(unit * (int64_t)chunks + chunk) * ML::chunk(N) + (slot * N + k) * RS + v0) = w;
  }
}

__global__ void k_split_pairs(int64_t n, const double* __restrict__ in, df_pair* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double x = in[i];
    const float h = __double2float_rn(x);
    out[i].h = h;
    out[i].l = __double2float_rn(x - (double)h);
  }
}

int setup_threads(int n3) { return n3 <= 64 ? 64 : (n3 <= 128 ? 128 : 256); }

}  // namespace

cudaError_t level_create(Level& L, int nx, int ny, int nz, const double* vertices, int p, int quad,
                         bool coords, cudaStream_t s) {
  L.p = p; L.quad = quad; L.n = p + 1;
  L.nx = nx; L.ny = ny; L.nz = nz;
  L.nelem = nx * ny * nz;
  const int64_t NX = (int64_t)p * nx + 1, NY = (int64_t)p * ny + 1, NZ = (int64_t)p * nz + 1;
  L.ndofs = NX * NY * NZ;
  build_tables(p, quad, &L.tab);
  const int n = L.n, n3 = n * n * n;
  std::vector<int> map((size_t)L.nelem * n3);
  std::vector<int> first((size_t)L.nelem);
  std::vector<double> ev((size_t)L.nelem * 24);
  for (int ez = 0; ez < nz; ++ez)
    for (int ey = 0; ey < ny; ++ey)
      for (int ex = 0; ex < nx; ++ex) {
        const size_t e = (size_t)ex + (size_t)nx * (ey + (size_t)ny * ez);
        for (int k = 0; k < n; ++k)
          for (int j = 0; j < n; ++j)
            for (int i = 0; i < n; ++i) {
              const int64_t g = (ex * (int64_t)p + i) + NX * ((ey * (int64_t)p + j) + NY * (ez * (int64_t)p + k));
              map[e * n3 + i + n * (j + n * k)] = (int)g;
            }
        first[e] = map[e * n3];
        for (int c = 0; c < 2; ++c)
          for (int b = 0; b < 2; ++b)
            for (int a = 0; a < 2; ++a) {
              const size_t v = (size_t)(ex + a) + (size_t)(nx + 1) * ((ey + b) + (size_t)(ny + 1) * (ez + c));
              for (int d = 0; d < 3; ++d) ev[e * 24 + (a + 2 * b + 4 * c) * 3 + d] = vertices[v * 3 + d];
            }
      }
  const size_t nm = metric_count(L);
  cudaError_t e;
  if ((e = cudaMalloc(&L.map, sizeof(int) * map.size())) != cudaSuccess) return e;
  if ((e = cudaMalloc(&L.first, sizeof(int) * first.size())) != cudaSuccess) return e;
  if ((e = cudaMalloc(&L.evert, sizeof(double) * ev.size())) != cudaSuccess) return e;
  if ((e = cudaMalloc(&L.metric, sizeof(double) * nm)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(L.metric, 0, sizeof(double) * nm, s)) != cudaSuccess) return e;  // padding
  if ((e = cudaMalloc(&L.mdiag, sizeof(double) * L.ndofs)) != cudaSuccess) return e;
  if ((e = cudaMalloc(&L.kdiag, sizeof(double) * L.ndofs)) != cudaSuccess) return e;
  if (coords && (e = cudaMalloc(&L.xyz, sizeof(double) * 3 * L.ndofs)) != cudaSuccess) return e;
  if ((e = cudaMemcpyAsync(L.map, map.data(), sizeof(int) * map.size(), cudaMemcpyHostToDevice, s)) != cudaSuccess) return e;
  if ((e = cudaMemcpyAsync(L.first, first.data(), sizeof(int) * first.size(), cudaMemcpyHostToDevice, s)) != cudaSuccess) return e;
  if ((e = cudaMemcpyAsync(L.evert, ev.data(), sizeof(double) * ev.size(), cudaMemcpyHostToDevice, s)) != cudaSuccess) return e;
  // the host vectors must outlive the copies
  return cudaStreamSynchronize(s);
}

void level_free(Level& L) {
  cudaFree(L.map);
  cudaFree(L.first);
  cudaFree(L.evert);
  cudaFree(L.metric);
  cudaFree(L.metric32);
  cudaFree(L.metric16);
  cudaFree(L.metric2);
  cudaFree(L.metric_tc);
  cudaFree(L.tc_frag);
  cudaFree(L.mdiag);
  cudaFree(L.kdiag);
  cudaFree(L.xyz);
  L = Level();
}

// The instantiation of one degree: f(std::integral_constant<int, n>).
template <typename F>
cudaError_t for_points(int n, F f) {
  switch (n) {
    case 2: f(std::integral_constant<int, 2>()); break;
    case 3: f(std::integral_constant<int, 3>()); break;
    case 4: f(std::integral_constant<int, 4>()); break;
    case 5: f(std::integral_constant<int, 5>()); break;
    case 6: f(std::integral_constant<int, 6>()); break;
    case 7: f(std::integral_constant<int, 7>()); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t setup_geometry(Level& L, const double* sigma_l, const double* sigma_t,
                           const double* theta, int* d_bad, cudaStream_t s) {
  const SetupTab tab = make_setup_tab(L.tab);
  L.metric32_valid = false;
  L.metric16_valid = false;
  L.metric2_valid = false;
  L.metric_tc_valid = false;
  return for_points(L.n, [&](auto n) {
    constexpr int N = decltype(n)::value, E = setup_elems(N * N * N);
    k_metric<N><<<(L.nelem + E - 1) / E, kSetupThreads, 0, s>>>(L.nelem, L.evert, sigma_l, sigma_t, theta, tab, L.metric,
                                                                d_bad);
  });
}

cudaError_t setup_node_coords(Level& L, cudaStream_t s) {
  const SetupTab tab = make_setup_tab(L.tab);
  const int n3 = L.n * L.n * L.n;
  k_nodes<<<L.nelem, setup_threads(n3), 0, s>>>(L.nelem, L.nx, L.ny, L.nz, L.evert, L.map, tab,
                                                L.ndofs, L.xyz);
  return cudaGetLastError();
}

cudaError_t setup_diagonals(Level& L, cudaStream_t s) {
  const SetupTab tab = make_setup_tab(L.tab);
  cudaError_t err = cudaMemsetAsync(L.mdiag, 0, sizeof(double) * L.ndofs, s);
  if (err != cudaSuccess) return err;
  err = cudaMemsetAsync(L.kdiag, 0, sizeof(double) * L.ndofs, s);
  if (err != cudaSuccess) return err;
  return for_points(L.n, [&](auto n) {
    constexpr int N = decltype(n)::value, N3 = N * N * N;
    if (L.quad == SEM_QUAD_LGL) {
      constexpr int E = setup_elems(N3);
      k_diagonals_ni<N><<<(L.nelem + E - 1) / E, kSetupThreads, 0, s>>>(L.nelem, L.map, L.metric, tab, L.mdiag, L.kdiag);
    } else {
      constexpr int E = N3 < 256 ? 256 / N3 : 1;
      k_diagonals<N><<<(L.nelem + E - 1) / E, kSetupThreads, 0, s>>>(L.nelem, L.map, L.metric, tab, L.mdiag, L.kdiag);
    }
  });
}

cudaError_t setup_metric_lowp(Level& L, bool bf16, cudaStream_t s) {
  const int G = PlaneMetricLayout::unit(L.n), padded = (L.nelem + G - 1) / G * G;
  (bf16 ? L.metric16_valid : L.metric32_valid) = true;
  bool& written = bf16 ? L.weight16_valid : L.weight32_valid;
  const bool weights = weight_lowp_count(L) > 0 && !written;
  const size_t at = metric_lowp_count(L);
  written = written || weights;
  return for_points(L.n, [&](auto n) {
    constexpr int N = decltype(n)::value, E = setup_elems(N * N * N);
    const int ctas = (padded + E - 1) / E;
    if (bf16)
      k_convert_planes<N><<<ctas, kSetupThreads, 0, s>>>(L.nelem, padded, L.metric, L.metric16,
                                                 weights ? L.metric16 + at : nullptr);
    else
      k_convert_planes<N><<<ctas, kSetupThreads, 0, s>>>(L.nelem, padded, L.metric, L.metric32,
                                                 weights ? L.metric32 + at : nullptr);
  });
}

cudaError_t setup_metric_df(Level& L, cudaStream_t s) {
  const int64_t count = (int64_t)metric_count(L);
  const int threads = 256;
  const int blocks = (int)std::min<int64_t>((count + threads - 1) / threads, 152 * 16);
  k_split_pairs<<<blocks, threads, 0, s>>>(count, L.metric, L.metric2);
  L.metric2_valid = true;
  return cudaGetLastError();
}

cudaError_t setup_region_mask(const Level& L, int region, const double* prm, double* mask,
                              cudaStream_t s) {
  double a[6] = {0, 0, 0, 0, 0, 0};
  const int cnt = region == SEM_REGION_BOX ? 6 : 4;
  for (int i = 0; i < cnt; ++i) a[i] = prm[i];
  const int threads = 256;
  const int blocks = (int)std::min<int64_t>((L.ndofs + threads - 1) / threads, 152 * 8);
  k_region_mask<<<blocks, threads, 0, s>>>(L.ndofs, L.xyz, region, a[0], a[1], a[2], a[3], a[4],
                                           a[5], mask);
  return cudaGetLastError();
}

}  // namespace sem
