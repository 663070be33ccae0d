// Pressure coupling of the FP64 Stokes operator K = [[A, B^T], [B, 0]],
// B = -P^T B_f with B_f the P1-P1 divergence on the velocity grid.
//
// B_f does not depend on the viscosity, and on a Kuhn grid its rows are one
// stencil: with D_o f = f(v + o) - f(v - o),
//   (B_f u)(v) = (h^2 / 12) sum_c [3 D_c + D_cd + D_ce + D_cde - D_d - D_e - D_de] u_c,
// d and e the other two axes (D_cd: offset e_c + e_d, and so on), and
// (-B_f^T q)_c at an interior vertex is the same combination of q.  The
// velocity is zero on the boundary and counts as zero outside it, so the
// stencil holds at every vertex.  P^T B_f at a pressure vertex K is again one
// stencil around 2K, over sums of two Kuhn offsets and odd in the offset: 26
// differences with a non-zero weight a component.
//
// Per tetrahedron, with the coupling recomputed for every element, this took
// some 190 FP64 operations a vertex (665 us at 128^3 cubes, 0.60 of the
// operator's time); here they are 22 for the gradient and 20 for the
// divergence, and the divergence is formed where the pressure lives, without
// a fine-grid vector and its restriction: 119 + 94 us, the operator at 64^3
// pressure cubes 1105 -> 650 us (FP64 pipe-bound, as the viscous part).
#include <utility>

#include "agca_internal.cuh"

namespace agca {

namespace {

// integer weights of (12 / h^2) times the x part of B_f by offset in [-1, 1]^3
constexpr int bweight(int x, int y, int z) {
  const int ax = x < 0 ? -x : x, ay = y < 0 ? -y : y, az = z < 0 ? -z : z;
  if (ax > 1 || ay > 1 || az > 1) return 0;
  const int s = x + y + z;
  if (s != ax + ay + az && s != -(ax + ay + az)) return 0;  // entries of both signs: no Kuhn offset
  if (s == 0) return 0;
  const int sg = s > 0 ? 1 : -1;
  return ax ? (ay + az == 0 ? 3 * sg : sg) : -sg;
}
// 2 * (P^T B_f): twice the weight at 2K plus those at the 14 midpoints around it
constexpr int pbweight(int x, int y, int z) {
  int w = 2 * bweight(x, y, z);
  for (int d = 1; d < 8; ++d) {
    const int dx = d & 1, dy = (d >> 1) & 1, dz = d >> 2;
    w += bweight(x - dx, y - dy, z - dz) + bweight(x + dx, y + dy, z + dz);
  }
  return w;
}
// the offsets with positive position in (z, y, x) order and a non-zero weight
struct HalfStencil {
  signed char x[62], y[62], z[62], w[62];
  int n;
};
constexpr HalfStencil make_half() {
  HalfStencil h{};
  for (int z = 0; z <= 2; ++z)
    for (int y = -2; y <= 2; ++y)
      for (int x = -2; x <= 2; ++x) {
        if (z == 0 && (y < 0 || (y == 0 && x <= 0))) continue;
        const int w = pbweight(x, y, z);
        if (w == 0) continue;
        h.x[h.n] = (signed char)x;
        h.y[h.n] = (signed char)y;
        h.z[h.n] = (signed char)z;
        h.w[h.n] = (signed char)w;
        ++h.n;
      }
  return h;
}
constexpr HalfStencil kHalf = make_half();
static_assert(kHalf.n == 26, "differences a component of the divergence");

// sum_q w_q (at(o_q) - at(-o_q)), in the order of q
template <typename F, int... Q>
__device__ __forceinline__ double half_sum(F at, std::integer_sequence<int, Q...>) {
  double acc = 0.0;
  (
      [&] {
        constexpr int x = kHalf.x[Q], y = kHalf.y[Q], z = kHalf.z[Q], w = kHalf.w[Q];
        acc = fma((double)w, at(x, y, z) - at(-x, -y, -z), acc);
      }(),
      ...);
  return acc;
}

// y = scale * (a - B_f^T q) at vertex v of a grid with n cubes per axis (a, scale
// may be nullptr: 0 and 1), 0 on the boundary
__device__ __forceinline__ void gradient_point(const int n, const double* __restrict__ q, const double* a,
                                               const double* __restrict__ scale, double* y, const int v) {
  const int nv = n + 1, V = nv * nv * nv;
  const int vk = v / (nv * nv), vr = v - vk * nv * nv, vj = vr / nv, vi = vr - vj * nv;
  if (vi == 0 || vj == 0 || vk == 0 || vi == n || vj == n || vk == n) {
#pragma unroll
    for (int c = 0; c < 3; ++c) y[v + c * V] = 0.0;
    return;
  }
  double y0[3] = {0.0, 0.0, 0.0};
  if (a) {
#pragma unroll
    for (int c = 0; c < 3; ++c) y0[c] = a[v + c * V];
  }
  const int sy = nv, sz = nv * nv;
  auto D = [&](int o) { return __ldg(q + v + o) - __ldg(q + v - o); };
  const double dx = D(1), dy = D(sy), dz = D(sz), dxy = D(1 + sy), dxz = D(1 + sz), dyz = D(sy + sz),
               dxyz = D(1 + sy + sz);
  // component c: base + 4 D_c - 2 D_de
  const double base = ((dxy + dxz) + (dyz + dxyz)) - ((dx + dy) + dz);
  const double w = 1.0 / (12.0 * (double)n * n);
  y0[0] = fma(w, fma(4.0, dx, fma(-2.0, dyz, base)), y0[0]);
  y0[1] = fma(w, fma(4.0, dy, fma(-2.0, dxz, base)), y0[1]);
  y0[2] = fma(w, fma(4.0, dz, fma(-2.0, dxy, base)), y0[2]);
#pragma unroll
  for (int c = 0; c < 3; ++c) y[v + c * V] = scale ? __ldg(scale + v + c * V) * y0[c] : y0[c];
}

// y = B u on pressure vertices 32 b .. 32 b + 31 (np cubes per axis): warp c adds
// component c's part, which is one formula in axes (c, d, e), and warp 0 sums
__device__ __forceinline__ void divergence_block(const int np, const double* __restrict__ u, double* __restrict__ y,
                                                 const int b, double (&part)[3][32]) {
  const int n = 2 * np, nv = n + 1, nvp = np + 1, V = nv * nv * nv, Vp = nvp * nvp * nvp;
  const int c = threadIdx.x >> 5, lane = threadIdx.x & 31, v = b * 32 + lane;
  const bool exists = v < Vp;
  const int K = exists ? v / (nvp * nvp) : 0, r = exists ? v - K * nvp * nvp : 0, J = r / nvp, I = r - J * nvp;
  // axes: component c first, then the other two (the stencil is symmetric in them)
  const int st[3] = {1, nv, nv * nv}, ps[3] = {2 * I, 2 * J, 2 * K};
  const int sa = c == 0 ? st[0] : (c == 1 ? st[1] : st[2]), sb = c == 0 ? st[1] : st[0], sc = c == 2 ? st[1] : st[2];
  const int pa = c == 0 ? ps[0] : (c == 1 ? ps[1] : ps[2]), pb = c == 0 ? ps[1] : ps[0], pc = c == 2 ? ps[1] : ps[2];
  const int f = 2 * I + nv * (2 * J + nv * 2 * K);
  const double* uc = u + c * V;
  double acc = 0.0;
  if (exists) {
    const bool deep = pa > 2 && pb > 2 && pc > 2 && pa < n - 2 && pb < n - 2 && pc < n - 2;
    auto at = [&](int x, int y2, int z) -> double {  // zero on and outside the boundary
      const int i = pa + x, j = pb + y2, k = pc + z;
      if (!deep && (i <= 0 || j <= 0 || k <= 0 || i >= n || j >= n || k >= n)) return 0.0;
      return __ldg(uc + f + x * sa + y2 * sb + z * sc);
    };
    acc = half_sum(at, std::make_integer_sequence<int, kHalf.n>{});
  }
  part[c][lane] = acc;
  __syncthreads();
  if (c == 0 && exists) y[v] = -(((part[0][lane] + part[1][lane]) + part[2][lane]) * (1.0 / (24.0 * (double)n * n)));
}

__global__ void __launch_bounds__(128) gradient_kernel(const int n, const double* __restrict__ q,
                                                       const double* a, const double* __restrict__ scale, double* y) {
  grid_dep_entry();
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < (n + 1) * (n + 1) * (n + 1)) gradient_point(n, q, a, scale, y, v);
}
__global__ void __launch_bounds__(96) divergence_kernel(const int np, const double* __restrict__ u,
                                                        double* __restrict__ y) {
  grid_dep_entry();
  __shared__ double part[3][32];
  divergence_block(np, u, y, blockIdx.x, part);
}

// many problems: grid (blocks of the largest, problems)
__global__ void __launch_bounds__(128) gradient_batch_kernel(const XferTask* __restrict__ tasks) {
  grid_dep_entry();
  const XferTask tk = tasks[blockIdx.y];
  if (tk.sc && tk.sc[MS_DONE] != 0.0) return;
  const int v = blockIdx.x * blockDim.x + threadIdx.x, nv = tk.nf + 1;
  if (v < nv * nv * nv) gradient_point(tk.nf, static_cast<const double*>(tk.src), static_cast<double*>(tk.dst), nullptr,
                                      static_cast<double*>(tk.dst), v);
}
__global__ void __launch_bounds__(96) divergence_batch_kernel(const XferTask* __restrict__ tasks) {
  grid_dep_entry();
  __shared__ double part[3][32];
  const XferTask tk = tasks[blockIdx.y];
  if (tk.sc && tk.sc[MS_DONE] != 0.0) return;
  const int nvp = tk.nf / 2 + 1;
  if ((int)blockIdx.x * 32 >= nvp * nvp * nvp) return;
  divergence_block(tk.nf / 2, static_cast<const double*>(tk.src), static_cast<double*>(tk.dst), blockIdx.x, part);
}

}  // namespace

cudaError_t launch_gradient(int n, const double* q, const double* a, const double* scale, double* y, cudaStream_t s) {
  return launch_k(gradient_kernel, dim3((unsigned)((nverts(n) + 127) / 128)), dim3(128), 0, s, n, q, a, scale, y);
}
cudaError_t launch_divergence(int np, const double* u, double* y, cudaStream_t s) {
  return launch_k(divergence_kernel, dim3((unsigned)((nverts(np) + 31) / 32)), dim3(96), 0, s, np, u, y);
}
cudaError_t launch_gradient_batch(const XferTask* tasks, int ntasks, int64_t max_count, cudaStream_t s) {
  return launch_k(gradient_batch_kernel, dim3((unsigned)((max_count + 127) / 128), (unsigned)ntasks), dim3(128), 0, s,
                  tasks);
}
cudaError_t launch_divergence_batch(const XferTask* tasks, int ntasks, int64_t max_count, cudaStream_t s) {
  return launch_k(divergence_batch_kernel, dim3((unsigned)((max_count + 31) / 32), (unsigned)ntasks), dim3(96), 0, s,
                  tasks);
}

}  // namespace agca
