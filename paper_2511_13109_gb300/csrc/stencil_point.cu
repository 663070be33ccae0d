// Operator application on the small levels (Eq. 2.9), eight lanes per vertex,
// fused with the smoother and residual epilogues.
//
// A tile marching z-planes over a level of up to 33^3 vertices, which does not
// fill the chip, is bound by the length of its dependency chain: a copy wait
// and two block barriers per plane (12 to 16 us a launch in FP32, 26 to 60 us
// in FP64, whatever the level's size).  Here nothing is staged and nothing
// waits on a barrier.  What bounds this kernel is load latency, except in FP64
// from about 17^3 vertices on: every flux is formed at both its ends and the
// sums by shuffles add in all lanes, some 35 FP64 warp instructions per four
// vertices, four times the tiles' arithmetic a vertex, so that at 33^3 vertices
// the FP64 pipe takes 24 to 26 us a launch (39 for the step from zero, which
// forms its input on the fly) where FP32 takes 7 (9.5).  The operator at a vertex is the difference of the
// fluxes along its six axis edges (edge form, see stencil_edge.cu), and lane
// 2 m + s of a vertex's eight computes one of them: the edge of axis m that
// ends (s = 0) or starts (s = 1) at the vertex.  All six follow one formula:
// with c < k the other two axes and S the edge's start vertex,
//   F[m] = 2 H d[m],   F[c] = H d[c] + sum of four differences along c of
//   component m, at S + e_m, S - e_c, S + e_m + e_k and S - e_c - e_k,
// so a lane's 12 vector values and 6 coefficients (or 9 record values) are
// independent loads, and three shuffles add the fluxes as
//   ((F_x- - F_x+) + (F_y- - F_y+)) + (F_z- - F_z+),
// the order of the tile kernels of stencil_edge.cu: in FP64 with coefficient
// records both give the same bits.  The stored-Galerkin stencils of touched
// vertices are spread over the lanes too, two of the 15 offsets each.
//
// Measured (whole V-cycles, tile kernels -> this kernel on the levels up to 32
// cubes per axis): 8-sphere field at 32^3 pressure cubes, mixed 195 -> 138 us;
// at 16^3, FP64 357 -> 182 us; at 4^3, FP64 70 -> 27 us.  The limit is where
// the tiles begin to win: with all levels up to 64 cubes here, a finest level
// of 40 cubes made the mixed cycle slower (76 -> 86 us) and the FP64 one too
// (243 -> 285 us), one of 36 cubes changed the FP64 cycle by 1 % (205 -> 208).
#include "agca_internal.cuh"
#include "device_ops.cuh"

namespace agca {

namespace {

constexpr int PT = 128;  // threads per block: 16 vertices, so that small levels still spread over the SMs

// coefficient sources of a level
enum PointCoef { PC_PLAIN = 0, PC_MASK = 1, PC_RECORD = 2 };  // op.coef, op.coef with flagged elements zero, op.hedge

// Stored-Galerkin part of a coarse operator at vertex (vi, vj, vk) with stencil
// index sv (Remark 5), by the eight lanes e of the vertex (lanes without a
// stencil pass sv < 0): g = sum_o S[o] x(v + o) over the 15 Kuhn offsets,
// offsets e and e + 8 in lane e, added by shuffles so that every lane holds g.
// Dirichlet neighbours contribute nothing.  All lanes of the warp call it.
template <typename T, typename XF>
__device__ __forceinline__ void gather_lanes(const LevelOp<T>& op, const int sv, const int vi, const int vj,
                                             const int vk, const int e, XF xat, T (&g)[3]) {
  const int n = op.n, nv = n + 1;
  if (sv >= 0) {
    const T* St = op.sten + (int64_t)sv * 135;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int o = e + 8 * r;
      // offset pair (o - 1) / 2 of x, y, z, xy, xz, yz, xyz; odd o: +, even o: -
      const int p = o > 0 ? (o - 1) >> 1 : 0, sg = o == 0 ? 0 : ((o & 1) ? 1 : -1);
      const int bits = (int)((0x7653421u >> (4 * p)) & 7u);
      const int i = vi + sg * (bits & 1), j = vj + sg * ((bits >> 1) & 1), k = vk + sg * (bits >> 2);
      if (o < 15 && i > 0 && j > 0 && k > 0 && i < n && j < n && k < n) {
        const int wv = i + nv * (j + nv * k);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const T xv = xat(d, wv, true);
#pragma unroll
          for (int q = 0; q < 3; ++q) g[q] = fma(__ldg(St + o * 9 + q * 3 + d), xv, g[q]);
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
#pragma unroll
    for (int off = 1; off < 8; off <<= 1) g[q] += __shfl_xor_sync(0xffffffffu, g[q], off);
  }
  if (sv >= 0 && op.sscale) {
    const T s = op.sscale[sv];
#pragma unroll
    for (int q = 0; q < 3; ++q) g[q] *= s;
  }
}

template <typename T, int MODE, int COEF>
__device__ __forceinline__ void stencil_point(const LevelOp<T>& op, const StencilArgs<T>& a, const int64_t id) {
  const int n = op.n, nv = n + 1, V = nv * nv * nv;
  const int e = (int)(id & 7);
  const int64_t v64 = id >> 3;
  const bool exists = v64 < V;
  const int v = exists ? (int)v64 : 0;
  const int vk = v / (nv * nv), vr = v - vk * nv * nv, vj = vr / nv, vi = vr - vj * nv;
  const bool inner = exists && vi > 0 && vj > 0 && vk > 0 && vi < n && vj < n && vk < n;
  constexpr bool PRE = MODE == ST_CHEB_PRE;

  // epilogue inputs of component e, read early
  const bool out_lane = exists && e < 3;
  const int vo = (e < 3 ? e : 0) * V + v;
  T eb = T(0), ed = T(0), ep = T(0), xo = T(0);
  if (out_lane && inner) {
    if (MODE != ST_APPLY && MODE != ST_POWER) eb = __ldg(a.b + vo);
    if (MODE == ST_CHEB_FIRST || MODE == ST_CHEB_STEP || PRE || MODE == ST_POWER) ed = __ldg(a.invD + vo);
    if (MODE == ST_CHEB_STEP) ep = a.xprev[vo];
    if (MODE == ST_CHEB_FIRST || MODE == ST_CHEB_STEP) xo = __ldg(a.x + vo);
  }

  // operator input, component d at vertex w (PRE: the first Chebyshev iterate)
  auto xat = [&](int d, int w, bool in) -> T {
    if (!in) return T(0);  // Dirichlet
    if (PRE) return a.s2 * __ldg(a.invD + d * V + w) * __ldg(a.b + d * V + w);
    return __ldg(a.x + d * V + w);
  };

  T F[3] = {T(0), T(0), T(0)};  // flux by component, negative where the edge starts at v
  const int m = e >> 1;
  if (inner && m < 3) {
    const int c = m == 0 ? 1 : 0, k = m == 2 ? 1 : 2;
    const int back = (e & 1) ? 0 : 1;
    auto str = [&](int ax, int s1, int s2) { return ax == 0 ? 1 : (ax == 1 ? s1 : s2); };
    const int sm = str(m, nv, nv * nv), sc = str(c, nv, nv * nv), sk = str(k, nv, nv * nv);
    auto pos = [&](int ax) { return ax == 0 ? vi : (ax == 1 ? vj : vk); };
    const int pm = pos(m) - back, pc = pos(c), pk = pos(k);
    const int S = v - back * sm;
    // v is interior: along c and k the offsets -1, 0, 1 stay on the grid, along m 0 and 1
    const bool m0 = pm > 0, m1 = pm + 1 < n;
    const bool cl = pc > 1, ch = pc + 1 < n, kl = pk > 1, kh = pk + 1 < n;
    T d[3];  // differences along the edge: components m, c, k
    const T xm0 = xat(m, S, m0), xm1 = xat(m, S + sm, m1);
    d[0] = xm1 - xm0;
    d[1] = xat(c, S + sm, m1) - xat(c, S, m0);
    d[2] = xat(k, S + sm, m1) - xat(k, S, m0);
    // component m on the squares S + e_m + {0, e_c, e_k, e_c + e_k} and S - {0, e_c, e_k, e_c + e_k}
    const T pc1 = xat(m, S + sm + sc, m1 && ch), pk1 = xat(m, S + sm + sk, m1 && kh);
    const T pck = xat(m, S + sm + sc + sk, m1 && ch && kh);
    const T nc1 = xat(m, S - sc, m0 && cl), nk1 = xat(m, S - sk, m0 && kl);
    const T nck = xat(m, S - sc - sk, m0 && cl && kl);
    T h, w[8];
    if constexpr (COEF == PC_RECORD) {
      const T* rec = op.hedge + S;
      h = __ldg(rec + (int64_t)m * V);
#pragma unroll
      for (int q = 0; q < 8; ++q) w[q] = __ldg(rec + (int64_t)(3 + 8 * m + q) * V);
    } else {
      // the six tetrahedra around the edge, named by their path order
      const int im = 1 * (m == 0 ? pm : vi), jm = m == 1 ? pm : vj, km = m == 2 ? pm : vk;
      const int C = im + n * (jm + n * km);
      const int tc = str(c, n, n * n), tk = str(k, n, n * n);
      auto cf = [&](int cube, int t) -> T {
        const T q = __ldg(op.coef + 6 * cube + t);
        if constexpr (COEF == PC_MASK) return __ldg(op.fidx + 6 * cube + t) >= 0 ? T(0) : q;
        return q;
      };
      const T mck = cf(C, 2 * m), mkc = cf(C, 2 * m + 1);
      const T cmk = cf(C - tc, 2 * c + (m > k)), kmc = cf(C - tk, 2 * k + (m > c));
      const T ckm = cf(C - tc - tk, 2 * c + (k > m)), kcm = cf(C - tc - tk, 2 * k + (c > m));
      h = ((mck + mkc) + (cmk + kmc)) + (ckm + kcm);
      w[0] = mck + kmc, w[1] = cmk + kcm, w[2] = mkc, w[3] = ckm;
      w[4] = mkc + cmk, w[5] = kmc + ckm, w[6] = mck, w[7] = kcm;
    }
    const T fm = T(2) * (h * d[0]);
    T fc = fma(pc1 - xm1, w[0], h * d[1]);
    fc = fma(xm0 - nc1, w[1], fc);
    fc = fma(pck - pk1, w[2], fc);
    fc = fma(nk1 - nck, w[3], fc);
    T fk = fma(pk1 - xm1, w[4], h * d[2]);
    fk = fma(xm0 - nk1, w[5], fk);
    fk = fma(pck - pc1, w[6], fk);
    fk = fma(nc1 - nck, w[7], fk);
    F[0] = m == 0 ? fm : fc;
    F[1] = m == 1 ? fm : (m == 0 ? fc : fk);
    F[2] = m == 2 ? fm : fk;
    if (!back) {
#pragma unroll
      for (int q = 0; q < 3; ++q) F[q] = -F[q];
    }
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
#pragma unroll
    for (int off = 1; off < 8; off <<= 1) F[q] += __shfl_xor_sync(0xffffffffu, F[q], off);
  }

  // stored-Galerkin part of a touched vertex
  T g[3] = {T(0), T(0), T(0)};
  if (op.sten) {
    const int sv = inner ? op.sidx[v] : -1;
    if (__any_sync(0xffffffffu, sv >= 0)) gather_lanes<T>(op, sv, vi, vj, vk, e, xat, g);
  }
  if (!out_lane) return;
  const T sum = e == 0 ? F[0] : (e == 1 ? F[1] : F[2]);
  const T gs = e == 0 ? g[0] : (e == 1 ? g[1] : g[2]);
  T o = T(0);
  if (inner) {
    if (MODE == ST_APPLY || MODE == ST_POWER) {
      o = op.sten ? fma(op.h6, sum, gs) : op.h6 * sum;
      if (MODE == ST_POWER) o = ed * o;
    } else {
      const T r = op.sten ? eb - fma(op.h6, sum, gs) : fma(-op.h6, sum, eb);  // b - A x
      if (MODE == ST_RESID) o = r;
      if (MODE == ST_CHEB_FIRST) o = fma(a.s0, ed * r, xo);
      if (MODE == ST_CHEB_STEP) o = fma(a.s1, ed * r, fma(a.s0, xo - ep, xo));
      if (PRE) {
        const T x1 = a.s2 * ed * eb;
        o = fma(a.s1, ed * r, fma(a.s0, x1, x1));
      }
    }
  }
  if (a.out64)
    a.out64[vo] = (double)o;  // the mixed cycle's result, widened
  else
    a.out[vo] = o;
}

// The stored-Galerkin part alone, for the tile kernels: op.ye[3 s + c] for the
// vertex with stencil index s (its room is the 12 values per flagged element,
// and an element has four vertices).  Inside a tile one thread would walk its
// vertex's 135 stencil values alone while the block waits: that made the coarse
// levels of a twelve-problem batch eight times slower per vertex.
template <typename T>
__device__ __forceinline__ void gather_point(const LevelOp<T>& op, const T* __restrict__ x, const int64_t id) {
  const int nv = op.n + 1, V = nv * nv * nv;
  const int e = (int)(id & 7);
  const int64_t s64 = id >> 3;
  const bool exists = s64 < op.n_sv;
  const int v = exists ? __ldg(op.slist + s64) : 0;
  const int vk = v / (nv * nv), vr = v - vk * nv * nv, vj = vr / nv, vi = vr - vj * nv;
  T g[3] = {T(0), T(0), T(0)};
  gather_lanes<T>(op, exists ? (int)s64 : -1, vi, vj, vk, e,
                  [&](int d, int w, bool) -> T { return __ldg(x + d * V + w); }, g);
  if (exists && e < 3) op.ye[3 * s64 + e] = e == 0 ? g[0] : (e == 1 ? g[1] : g[2]);
}

template <typename T>
__global__ void __launch_bounds__(PT) gather_kernel(const LevelOp<T> op, const T* __restrict__ x) {
  grid_dep_entry();
  gather_point<T>(op, x, blockIdx.x * (int64_t)PT + threadIdx.x);
}

template <typename T>
__global__ void __launch_bounds__(PT) gather_batch_kernel(const StencilTask<T, T>* __restrict__ tasks) {
  grid_dep_entry();
  const StencilTask<T, T>& tk = tasks[blockIdx.y];
  if (tk.sc && tk.sc[MS_DONE] != 0.0) return;  // converged problem
  if (blockIdx.x * (int64_t)(PT / 8) >= tk.op.n_sv) return;
  gather_point<T>(tk.op, tk.a.x, blockIdx.x * (int64_t)PT + threadIdx.x);
}

template <typename T, int MODE, int COEF>
__global__ void __launch_bounds__(PT) stencil_point_kernel(const LevelOp<T> op, const StencilArgs<T> a) {
  grid_dep_entry();
  stencil_point<T, MODE, COEF>(op, a, blockIdx.x * (int64_t)PT + threadIdx.x);
}

// many problems: grid (blocks of the largest, problems)
template <typename T, int MODE, int COEF>
__global__ void __launch_bounds__(PT) stencil_point_batch_kernel(const StencilTask<T, T>* __restrict__ tasks) {
  grid_dep_entry();
  const StencilTask<T, T>& tk = tasks[blockIdx.y];
  if (tk.sc && tk.sc[MS_DONE] != 0.0) return;  // converged problem
  const int64_t nv = tk.op.n + 1;
  if (blockIdx.x * (int64_t)(PT / 8) >= nv * nv * nv) return;
  stencil_point<T, MODE, COEF>(tk.op, tk.a, blockIdx.x * (int64_t)PT + threadIdx.x);
}

unsigned point_blocks(int n) { return (unsigned)((nverts(n) * 8 + PT - 1) / PT); }

}  // namespace

template <typename T>
cudaError_t launch_stencil_point(int mode, const LevelOp<T>& op, const StencilArgs<T>& a, cudaStream_t s) {
  const dim3 grid(point_blocks(op.n)), block(PT);
#define AGCA_PLAUNCH(M)                                                                             \
  do {                                                                                              \
    if constexpr (sizeof(T) == 8) {                                                                 \
      if (op.hedge)                                                                                 \
        KL(launch_k(stencil_point_kernel<T, M, PC_RECORD>, grid, block, 0, s, op, a));              \
      else if (op.fidx)                                                                             \
        KL(launch_k(stencil_point_kernel<T, M, PC_MASK>, grid, block, 0, s, op, a));                \
      else                                                                                          \
        KL(launch_k(stencil_point_kernel<T, M, PC_PLAIN>, grid, block, 0, s, op, a));               \
    } else {                                                                                        \
      KL(launch_k(stencil_point_kernel<T, M, PC_PLAIN>, grid, block, 0, s, op, a));                 \
    }                                                                                               \
  } while (0)
  switch (mode) {
    case ST_APPLY: AGCA_PLAUNCH(ST_APPLY); break;
    case ST_RESID: AGCA_PLAUNCH(ST_RESID); break;
    case ST_CHEB_FIRST: AGCA_PLAUNCH(ST_CHEB_FIRST); break;
    case ST_CHEB_STEP: AGCA_PLAUNCH(ST_CHEB_STEP); break;
    case ST_CHEB_PRE: AGCA_PLAUNCH(ST_CHEB_PRE); break;
    case ST_POWER:
      if constexpr (sizeof(T) == 8) {
        AGCA_PLAUNCH(ST_POWER);
        break;
      }
      [[fallthrough]];
    default: return cudaErrorInvalidValue;
  }
#undef AGCA_PLAUNCH
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_stencil_point_batch(int mode, const StencilTask<T, T>* tasks, int ntasks, int max_n,
                                       cudaStream_t s) {
  if (ntasks <= 0) return cudaSuccess;
  constexpr int COEF = sizeof(T) == 8 ? PC_RECORD : PC_PLAIN;  // batched FP64 steps belong to FP64 contexts
  const dim3 grid(point_blocks(max_n), (unsigned)ntasks), block(PT);
  switch (mode) {
    case ST_APPLY: KL(launch_k(stencil_point_batch_kernel<T, ST_APPLY, COEF>, grid, block, 0, s, tasks)); break;
    case ST_RESID: KL(launch_k(stencil_point_batch_kernel<T, ST_RESID, COEF>, grid, block, 0, s, tasks)); break;
    case ST_CHEB_FIRST:
      KL(launch_k(stencil_point_batch_kernel<T, ST_CHEB_FIRST, COEF>, grid, block, 0, s, tasks));
      break;
    case ST_CHEB_STEP: KL(launch_k(stencil_point_batch_kernel<T, ST_CHEB_STEP, COEF>, grid, block, 0, s, tasks)); break;
    case ST_CHEB_PRE: KL(launch_k(stencil_point_batch_kernel<T, ST_CHEB_PRE, COEF>, grid, block, 0, s, tasks)); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_gather(const LevelOp<T>& op, const T* x, cudaStream_t s) {
  if (!op.sten || op.n_sv <= 0) return cudaSuccess;
  return launch_k(gather_kernel<T>, dim3((unsigned)((op.n_sv * 8 + PT - 1) / PT)), dim3(PT), 0, s, op, x);
}

template <typename T>
cudaError_t launch_gather_batch(const StencilTask<T, T>* tasks, int ntasks, int64_t max_sv, cudaStream_t s) {
  if (ntasks <= 0 || max_sv <= 0) return cudaSuccess;
  return launch_k(gather_batch_kernel<T>, dim3((unsigned)((max_sv * 8 + PT - 1) / PT), (unsigned)ntasks), dim3(PT), 0,
                  s, tasks);
}

template cudaError_t launch_gather<float>(const LevelOp<float>&, const float*, cudaStream_t);
template cudaError_t launch_gather<double>(const LevelOp<double>&, const double*, cudaStream_t);
template cudaError_t launch_gather_batch<float>(const StencilTask<float, float>*, int, int64_t, cudaStream_t);
template cudaError_t launch_gather_batch<double>(const StencilTask<double, double>*, int, int64_t, cudaStream_t);
template cudaError_t launch_stencil_point<float>(int, const LevelOp<float>&, const StencilArgs<float>&, cudaStream_t);
template cudaError_t launch_stencil_point<double>(int, const LevelOp<double>&, const StencilArgs<double>&,
                                                  cudaStream_t);
template cudaError_t launch_stencil_point_batch<float>(int, const StencilTask<float, float>*, int, int, cudaStream_t);
template cudaError_t launch_stencil_point_batch<double>(int, const StencilTask<double, double>*, int, int,
                                                        cudaStream_t);

}  // namespace agca
