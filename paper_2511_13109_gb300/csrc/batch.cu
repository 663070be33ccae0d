// Batched element-wise kernels: many independent problems per launch.
// Grid (chunks, problems): block row y serves problem y, blocks past the end
// of a smaller problem exit at once.  A problem whose MINRES has converged
// (sc[MS_DONE] != 0) is skipped.  Used by the batched solve of
// agca_batch_solve (the stencil launches live in the stencil files).
#include <math.h>

#include <algorithm>

#include "agca_internal.cuh"
#include "device_ops.cuh"

namespace agca {

namespace {

constexpr int kBT = 256;
constexpr int kDotBlocks = 64;  // per problem: fixed, so the reductions are deterministic

__device__ __forceinline__ bool skip(const double* sc) { return sc && sc[MS_DONE] != 0.0; }

// FP32 right-hand sides (XK_D2F) or the FP64 ones in place (XK_X1, WRITE false), with the first Chebyshev iterate
template <typename TO, bool WRITE>
__global__ void rhs_batch_kernel(const XferTask* __restrict__ tasks) {
  grid_dep_entry();
  const XferTask tk = tasks[blockIdx.y];
  if (skip(tk.sc)) return;
  const double* in = static_cast<const double*>(tk.src);
  TO* out = static_cast<TO*>(tk.dst);
  TO* x1 = static_cast<TO*>(tk.x1);
  const TO* invD = static_cast<const TO*>(tk.invD);
  const TO s2 = (TO)tk.s2;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < tk.count; i += (int64_t)gridDim.x * blockDim.x) {
    const TO v = (TO)in[i];
    if (WRITE) out[i] = v;
    if (x1) x1[i] = s2 * __ldg(invD + i) * v;
  }
}

// coarsest solves, grid (row blocks of the largest, problems)
template <typename T>
__global__ void __launch_bounds__(32 * kCoarseWarps) coarse_solve_batch_kernel(const XferTask* __restrict__ tasks) {
  grid_dep_entry();
  extern __shared__ double sm[];
  const XferTask tk = tasks[blockIdx.y];
  if (skip(tk.sc)) return;
  const int ni = tk.nf - 1, nb = (3 * ni * ni * ni + kCoarseWarps - 1) / kCoarseWarps;
  if ((int)blockIdx.x >= nb) return;
  coarse_solve_rows<T>(tk.nf, tk.m1, static_cast<const T*>(tk.src), static_cast<T*>(tk.dst), sm, blockIdx.x, nb);
}

// ------------------------------------------------------------------ Krylov
template <int OP>
__global__ void __launch_bounds__(kBT) reduce_batch_kernel(const KTask* __restrict__ tasks, double* partials) {
  grid_dep_entry();
  const KTask tk = tasks[blockIdx.y];
  double acc = 0.0;
  if (!skip(tk.sc)) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < tk.n; i += (int64_t)gridDim.x * blockDim.x)
      acc = (OP == KB_DOT) ? fma(tk.a[i], tk.b[i], acc) : acc + tk.a[i];
  }
  __shared__ double red[kBT / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
  if (lane == 0) red[warp] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < kBT / 32; ++w) v += red[w];
    partials[blockIdx.y * kDotBlocks + blockIdx.x] = v;
  }
}

__global__ void reduce_batch_final_kernel(const KTask* __restrict__ tasks, const double* partials) {
  grid_dep_entry();
  const KTask tk = tasks[blockIdx.x];
  if (skip(tk.sc)) return;
  __shared__ double red[kDotBlocks];
  red[threadIdx.x] = partials[blockIdx.x * kDotBlocks + threadIdx.x];
  __syncthreads();
  for (int s = kDotBlocks / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) tk.sc[tk.slot] = tk.scale * red[0];
}

__global__ void vec_batch_kernel(const KTask* __restrict__ tasks, int op) {
  grid_dep_entry();
  const KTask tk = tasks[blockIdx.y];
  if (op == KB_UPDATE ? tk.sc[MS_UPD_SKIP] != 0.0 : skip(tk.sc)) return;
  const double* sc = tk.sc;
  const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, st = (int64_t)gridDim.x * blockDim.x;
  if (op == KB_LANCZOS) {  // c <- a/g - (delta/g) b - (g/g_old) c   (a = Kz, b = v, c = v_old)
    const double g = sc[MS_GAMMA], go = sc[MS_GAMMA_OLD];
    const double ig = 1.0 / g;
    const double delta = sc[MS_DOT_KZZ] * ig * ig;
    const double al = delta * ig, be = g / go;
    for (int64_t i = i0; i < tk.n; i += st) tk.c[i] = tk.a[i] * ig - al * tk.b[i] - be * tk.c[i];
  } else if (op == KB_UPDATE) {  // c <- (a/g_prev - a3 c - a2 b)/a1 ; d += xcoef c   (a = z, b = w, c = w_old, d = x)
    const double ig = sc[MS_INV_GAMMA_PREV], a1 = sc[MS_A1], a2 = sc[MS_A2], a3 = sc[MS_A3], xc = sc[MS_XCOEF];
    const double ia1 = 1.0 / a1;
    for (int64_t i = i0; i < tk.n; i += st) {
      const double wn = (tk.a[i] * ig - a3 * tk.c[i] - a2 * tk.b[i]) * ia1;
      tk.c[i] = wn;
      tk.d[i] = fma(xc, wn, tk.d[i]);
    }
  } else if (op == KB_PDIV) {  // c <- (a - sc[slot]) * b
    const double m = sc[tk.slot];
    for (int64_t i = i0; i < tk.n; i += st) tk.c[i] = (tk.a[i] - m) * tk.b[i];
  } else if (op == KB_SUBS) {  // c <- a - sc[slot]
    const double m = sc[tk.slot];
    for (int64_t i = i0; i < tk.n; i += st) tk.c[i] = tk.a[i] - m;
  }
}

// MINRES scalar recurrence, one thread per problem
__global__ void scalars_batch_kernel(const KTask* __restrict__ tasks, int ntasks) {
  grid_dep_entry();
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= ntasks) return;
  double* sc = tasks[p].sc;
  minres_scalars(sc);
  if (tasks[p].c) tasks[p].c[0] = sc[MS_DONE];  // contiguous copy of the done flags for the host
}

inline unsigned chunks(int64_t n, int bs) { return (unsigned)((n + bs - 1) / bs); }

}  // namespace

template <typename T>
cudaError_t launch_xfer_batch(int kind, int ncomp, const XferTask* tasks, int ntasks, int64_t max_count, int max_m,
                              cudaStream_t s) {
  if (ntasks <= 0) return cudaSuccess;
  const dim3 g(chunks(max_count, kBT), (unsigned)ntasks);
  const dim3 gc(std::min<unsigned>(g.x, 1216u), (unsigned)ntasks);
  switch (kind) {
    case XK_RESTRICT:
    case XK_PROLONG_ADD:
    case XK_PROLONG: return launch_transfer_batch<T>(kind, ncomp, tasks, ntasks, max_m, s);
    case XK_D2F:
      KL(launch_k(rhs_batch_kernel<float, true>, gc, dim3(kBT), 0, s, tasks));
      break;
    case XK_GRADIENT: return launch_gradient_batch(tasks, ntasks, max_count, s);
    case XK_DIVERGENCE: return launch_divergence_batch(tasks, ntasks, max_count, s);
    case XK_X1:
      KL(launch_k(rhs_batch_kernel<double, false>, gc, dim3(kBT), 0, s, tasks));
      break;
    case XK_COARSE:
      KL(launch_k(coarse_solve_batch_kernel<T>, dim3(chunks(max_m, kCoarseWarps), (unsigned)ntasks),
                  dim3(32 * kCoarseWarps), (size_t)max_m * sizeof(double), s, tasks));
      break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}
template cudaError_t launch_xfer_batch<float>(int, int, const XferTask*, int, int64_t, int, cudaStream_t);
template cudaError_t launch_xfer_batch<double>(int, int, const XferTask*, int, int64_t, int, cudaStream_t);

cudaError_t launch_krylov_batch(int op, const KTask* tasks, int ntasks, int64_t max_n, double* partials,
                                cudaStream_t s) {
  if (ntasks <= 0) return cudaSuccess;
  switch (op) {
    case KB_DOT:
      KL(launch_k(reduce_batch_kernel<KB_DOT>, dim3(kDotBlocks, ntasks), dim3(kBT), 0, s, tasks, partials));
      KL(launch_k(reduce_batch_final_kernel, dim3(ntasks), dim3(kDotBlocks), 0, s, tasks, partials));
      break;
    case KB_SUM:
      KL(launch_k(reduce_batch_kernel<KB_SUM>, dim3(kDotBlocks, ntasks), dim3(kBT), 0, s, tasks, partials));
      KL(launch_k(reduce_batch_final_kernel, dim3(ntasks), dim3(kDotBlocks), 0, s, tasks, partials));
      break;
    case KB_SCALARS: KL(launch_k(scalars_batch_kernel, dim3(chunks(ntasks, 32)), dim3(32), 0, s,
                        tasks, ntasks)); break;
    default: {
      dim3 g(std::min<unsigned>(chunks(max_n, kBT), 1216u), (unsigned)ntasks);
      KL(launch_k(vec_batch_kernel, dim3(g), dim3(kBT), 0, s, tasks, op));
    }
  }
  return cudaGetLastError();
}

}  // namespace agca
