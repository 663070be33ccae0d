// Per-point device arithmetic shared by the single-problem kernels and the
// batched kernels, so that both compute each value with the same operations
// in the same order (a batched cycle is bit-for-bit equal to the cycle of one
// problem).
#pragma once

#include "agca_internal.cuh"

namespace agca {

__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// ------------------------------------------------------------ element action
// For a tetrahedron with nodal values x_a (a = 0..3) the scaled displacement
// gradient is Gx = sum_a x_a (x) G_a; along the Kuhn path its column p_k is the
// edge difference x_{k+1} - x_k.  With S = Gx + Gx^T, the element
// contribution to local vertex a is y_a = eta (h/6) S G_a, i.e. with the edge
// "fluxes" F_k = eta (h/6) S[:, p_k]:
//   y_0 = -F_0, y_1 = F_0 - F_1, y_2 = F_1 - F_2, y_3 = F_2.
// This equals A_e x_e for the element matrix of Eq. 3.5 and needs only
// differences of nodal values.  Xl / Xh: the cube's corner values on its
// lower / upper z-plane (index qx + 2 qy), c[t]: eta_t h / 6 per type; the
// contributions are added to Y[corner qx + 2 qy + 4 qz][component].
template <typename T, int NC>
__device__ __forceinline__ void cube_dca(const T (&Xl)[4][NC], const T (&Xh)[4][NC], const T (&c)[6], T (&Y)[8][NC]) {
#pragma unroll
  for (int t = 0; t < 6; ++t) {
    T G[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int qa = tet_corner(t, k), qb = tet_corner(t, k + 1), m = perm(t, k);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const T xb = (qb & 4) ? Xh[qb & 3][i] : Xl[qb & 3][i];
        const T xa = (qa & 4) ? Xh[qa & 3][i] : Xl[qa & 3][i];
        G[i][m] = xb - xa;
      }
    }
    const T ct = c[t], nct = -c[t], c2 = c[t] + c[t], nc2 = -c2;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int qa = tet_corner(t, k), qb = tet_corner(t, k + 1), m = perm(t, k);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        if (i == m) {
          Y[qb][i] = fma(c2, G[m][m], Y[qb][i]);
          Y[qa][i] = fma(nc2, G[m][m], Y[qa][i]);
        } else {
          const T sv = G[i][m] + G[m][i];
          Y[qb][i] = fma(ct, sv, Y[qb][i]);
          Y[qa][i] = fma(nct, sv, Y[qa][i]);
        }
      }
    }
  }
}

// Velocity block plus the divergence pieces on the finest grid: with the
// fine-grid pressure q = P p (component 3 of the tile) the element adds
// -(h^2/6) qbar_T G_a to the velocity row of vertex a (that is -B_f^T q with
// B_f the P1-P1 divergence, |T| g = (h^2/6) G) and (h^2/24) tr(Gx) to the
// scalar row of each vertex ((|T|/4) div u).  c[t] = eta_t h/6, hq = h^2/6.
template <typename T>
__device__ __forceinline__ void cube_stokes(const T (&Xl)[4][4], const T (&Xh)[4][4], const T (&c)[6], const T hq,
                                            T (&Y)[8][4]) {
#pragma unroll
  for (int t = 0; t < 6; ++t) {
    T G[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int qa = tet_corner(t, k), qb = tet_corner(t, k + 1), m = perm(t, k);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const T xb = (qb & 4) ? Xh[qb & 3][i] : Xl[qb & 3][i];
        const T xa = (qa & 4) ? Xh[qa & 3][i] : Xl[qa & 3][i];
        G[i][m] = xb - xa;
      }
    }
    T qsum = T(0);
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int q = tet_corner(t, a);
      qsum += (q & 4) ? Xh[q & 3][3] : Xl[q & 3][3];
    }
    const T pq = T(0.25) * hq * qsum;  // (h^2/6) qbar
    const T ct = c[t], nct = -c[t], c2 = c[t] + c[t];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int qa = tet_corner(t, k), qb = tet_corner(t, k + 1), m = perm(t, k);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        if (i == m) {
          const T dm = fma(c2, G[m][m], -pq);
          Y[qb][i] += dm;
          Y[qa][i] -= dm;
        } else {
          const T sv = G[i][m] + G[m][i];
          Y[qb][i] = fma(ct, sv, Y[qb][i]);
          Y[qa][i] = fma(nct, sv, Y[qa][i]);
        }
      }
    }
    const T dv = T(0.25) * hq * (G[0][0] + G[1][1] + G[2][2]);  // (|T|/4) div u
#pragma unroll
    for (int a = 0; a < 4; ++a) Y[tet_corner(t, a)][3] += dv;
  }
}

// ------------------------------------------------------------------ transfers
// Linear interpolation between Kuhn grids and its transpose (Sec. 2.1).  Every
// fine vertex is either 2i (a coarse vertex) or the midpoint 2i + d of the
// coarse Kuhn edge (i, i + d), d in {0,1}^3 \ {0} (Kuhn edges join corners
// whose difference has entries of one sign), hence
//   (P e)(2i) = e(i),  (P e)(2i + d) = (e(i) + e(i + d)) / 2,
//   (P^T r)(i) = r(2i) + 1/2 sum_d [ r(2i + d) + r(2i - d) ].
// The weights are known a priori and never stored.

// One warp's piece w of the vertices of a grid with nv vertices per axis: 32
// consecutive ones of a row (whose position is warp-uniform: the per-vertex
// divisions of a flat index would cost more than the arithmetic)
struct RowPiece {
  int i, j, k;  // this lane's vertex; i < nv must hold for it to exist
};
__device__ __forceinline__ int row_pieces(const int nv) { return nv * nv * ((nv + 31) / 32); }
__device__ __forceinline__ RowPiece row_piece(const int nv, const int w, const int lane) {
  const int per = (nv + 31) / 32, row = w / per, k = row / nv;
  return RowPiece{32 * (w - row * per) + lane, row - k * nv, k};
}

// scale * P^T r at coarse vertex (I, J, K) for one component of a fine grid with
// nf cubes per axis; 0 on the coarse boundary when mask is set; with fi.x1, the
// first Chebyshev iterate beside it.  The sum runs over d = 1 .. 7, +d before -d,
// and a neighbour outside the grid contributes nothing.
template <typename T>
__device__ __forceinline__ void restrict_point(const int nf, const bool mask, const T scale, const T* __restrict__ rf,
                                               T* __restrict__ rc, const FirstIterate<T>& fi, const int I, const int J,
                                               const int K) {
  const int nc = nf / 2, nvc = nc + 1, nvf = nf + 1;
  const bool edge = I == 0 || J == 0 || K == 0 || I == nc || J == nc || K == nc;
  const int c0 = I + nvc * (J + nvc * K);
  const T* r = rf + 2 * I + nvf * (2 * J + nvf * 2 * K);
  T v = T(0);
  if (!edge) {
    T acc = T(0);
#pragma unroll
    for (int d = 1; d < 8; ++d) {
      const int o = (d & 1) + nvf * (((d >> 1) & 1) + nvf * ((d >> 2) & 1));
      acc += __ldg(r + o);
      acc += __ldg(r - o);
    }
    v = scale * (__ldg(r) + T(0.5) * acc);
  } else if (!mask) {
    T acc = T(0);
#pragma unroll
    for (int d = 1; d < 8; ++d) {
      const int dx = d & 1, dy = (d >> 1) & 1, dz = (d >> 2) & 1, o = dx + nvf * (dy + nvf * dz);
      if (2 * I + dx <= nf && 2 * J + dy <= nf && 2 * K + dz <= nf) acc += __ldg(r + o);
      if (2 * I >= dx && 2 * J >= dy && 2 * K >= dz) acc += __ldg(r - o);
    }
    v = scale * (__ldg(r) + T(0.5) * acc);
  }
  rc[c0] = v;
  if (fi.x1) fi.x1[c0] = fi.s2 * __ldg(fi.invD + c0) * v;
}

// P e at fine vertex (i, j, k) (added to xf when ADD) for NC components; 0 on the
// fine boundary when mask is set.  Explicit roundings: x + (P e) rounds the same
// in every kernel that adds it.
template <typename T, int NC, bool ADD>
__device__ __forceinline__ void prolong_point(const int nf, const bool mask, const T* __restrict__ ec,
                                              T* __restrict__ xf, const RowPiece& p) {
  const int nvf = nf + 1, nvc = nf / 2 + 1, Vc = nvc * nvc * nvc, Vf = nvf * nvf * nvf;
  const int i = p.i, j = p.j, k = p.k;
  if (i >= nvf) return;
  const bool zero = mask && (i == 0 || j == 0 || k == 0 || i == nf || j == nf || k == nf);
  if (ADD && zero) return;
  const int dx = i & 1, dy = j & 1, dz = k & 1;
  const int e0 = (i >> 1) + nvc * ((j >> 1) + nvc * (k >> 1)), e1 = e0 + dx + nvc * (dy + nvc * dz);
  T* x = xf + i + nvf * (j + nvf * k);
  T a[NC], b[NC], o[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    a[c] = zero ? T(0) : __ldg(ec + c * Vc + e0);
    b[c] = zero ? T(0) : __ldg(ec + c * Vc + e1);
    if (ADD) o[c] = x[c * Vf];
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const T v = (dx | dy | dz) ? mul_rn(T(0.5), add_rn(a[c], b[c])) : a[c];
    x[c * Vf] = ADD ? add_rn(o[c], v) : v;
  }
}

// ------------------------------------------------------------- coarsest solve
// z = A_1^-1 r on the interior DoFs of the coarsest grid (n cubes) with the
// explicit inverse ainv (m x m, m = 3 (n-1)^3, symmetric bit for bit): block
// b of nb forms the rows b * 8 .. b * 8 + 7, one warp each, from a copy of r
// in shared memory (sm: m doubles); r, z are full-grid vectors.  A row's sum is
// formed by one warp in a fixed order, so the result depends on no grid shape.
// One block doing both triangular products of L^-T L^-1 took 16 us at m = 81 and
// 200 us for twelve problems of up to m = 648; the rows of the inverse are
// independent, need half the passes and spread over the SMs.
constexpr int kCoarseWarps = 8;
template <typename T>
__device__ __forceinline__ void coarse_solve_rows(const int n, const double* __restrict__ ainv, const T* r, T* z,
                                                  double* sm, const int b, const int nb) {
  const int nv = n + 1, ni = n - 1, V = nv * nv * nv;
  const int nI = ni * ni * ni, m = 3 * nI;
  auto grid_index = [&](int q) {
    const int c = q / nI, iv = q - c * nI;
    const int t = iv / ni, i = iv - t * ni, k = t / ni, j = t - k * ni;
    return c * V + (1 + i) + nv * ((1 + j) + nv * (1 + k));
  };
  const int lane = threadIdx.x & 31, q = b * kCoarseWarps + (threadIdx.x >> 5);
  for (int p = threadIdx.x; p < m; p += blockDim.x) sm[p] = (double)__ldg(r + grid_index(p));
  // Dirichlet entries of z
  for (int id = b * blockDim.x + threadIdx.x; id < 3 * V; id += nb * blockDim.x) {
    const int v = id % V, t = v / nv, i = v - t * nv, k = t / nv, j = t - k * nv;
    if (i == 0 || j == 0 || k == 0 || i == n || j == n || k == n) z[id] = T(0);
  }
  __syncthreads();
  if (q >= m) return;
  const double* row = ainv + (int64_t)q * m;
  double s = 0.0;
#pragma unroll 4
  for (int p = lane; p < m; p += 32) s = fma(row[p], sm[p], s);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  if (lane == 0) z[grid_index(q)] = (T)s;
}

// ------------------------------------------------------------ MINRES scalars
// The recurrence of one MINRES iteration on the device scalars sc (MinresSlot), by
// one thread: the single solve's reduction and the batched one both end with it.
__device__ inline void minres_scalars(double* sc) {
  if (sc[MS_DONE] != 0.0) {
    sc[MS_UPD_SKIP] = 1.0;  // iterations past convergence change nothing
    return;
  }
  const double g = sc[MS_GAMMA];
  const double delta = sc[MS_DOT_KZZ] / (g * g);
  const double gn2 = sc[MS_DOT_ZV];
  const double gn = gn2 > 0.0 ? sqrt(gn2) : 0.0;
  const double c = sc[MS_C], co = sc[MS_C_OLD], s = sc[MS_S], so = sc[MS_S_OLD];
  const double a0 = c * delta - co * s * g;
  const double a1 = sqrt(a0 * a0 + gn * gn);
  const double a2 = s * delta + co * c * g;
  const double a3 = so * g;
  const double eta = sc[MS_ETA];
  if (!(a1 > 0.0) || !isfinite(a1)) {  // exact convergence or breakdown
    sc[MS_DONE] = 2.0;
    sc[MS_UPD_SKIP] = 1.0;
    return;
  }
  const double cn = a0 / a1, sn = gn / a1;
  sc[MS_A1] = a1;
  sc[MS_A2] = a2;
  sc[MS_A3] = a3;
  sc[MS_XCOEF] = cn * eta;
  sc[MS_INV_GAMMA_PREV] = 1.0 / g;
  sc[MS_UPD_SKIP] = 0.0;
  sc[MS_ETA] = -sn * eta;
  sc[MS_C_OLD] = c;
  sc[MS_C] = cn;
  sc[MS_S_OLD] = s;
  sc[MS_S] = sn;
  sc[MS_GAMMA_OLD] = g;
  sc[MS_GAMMA] = gn;
  sc[MS_ITERS] += 1.0;
  if (fabs(sc[MS_ETA]) <= sc[MS_TOL_ABS] || !(gn > 0.0)) sc[MS_DONE] = 1.0;
}

}  // namespace agca
