// Interpolation between Kuhn grids and its transpose (Sec. 2.1); the per-point
// formulas are restrict_point / prolong_point in device_ops.cuh.
//
// Prolongation: one thread per fine vertex, all components at once, a warp on 32
// vertices of one row.  With flat vertex indices (two integer divisions each) and
// a loop over the components the finest FP32 level at 128^3 pressure cubes took
// 131 us, now 92; floor 64.  (One warp per row, looping over it, left too little
// in flight: 134 us.)
//
// Restriction: one thread per coarse vertex and component, flat indices.  In FP64
// it is bound by the FP64 pipe (16 operations a value: 164 us at 256^3 cubes; 18
// with the first iterate), so lanes must not idle: rows of 32 vertices waste a fifth of them at 129 vertices
// a row.  Measured alone, 256^3 / 128^3 / 64^3 cubes: FP64 196 / 30 / 9 us (rows of
// 32 with all components per thread 216 / 34 / 12, flat with a loop over the
// components 198 / 32 / 12), FP32 53 / 12 / 6 us (54 / 14 / 9, 78 / 18 / 11); with
// the first iterate FP64 221 / 35 / 10, FP32 60 / 14 / 6 us.
#include <stdlib.h>

#include "agca_internal.cuh"
#include "device_ops.cuh"

namespace agca {

namespace {

constexpr int kRowWarps = 8;
constexpr int kRestrictThreads = 256;

// grid (blocks of the vertices, components)
template <typename T>
__device__ __forceinline__ void restrict_thread(const int nf, const bool mask, const T scale, const T* rf, T* rc,
                                                FirstIterate<T> fi, const int c) {
  const int nvf = nf + 1, nv = nf / 2 + 1, V = nv * nv * nv, id = blockIdx.x * kRestrictThreads + threadIdx.x;
  if (id >= V) return;
  const int t = id / nv, K = t / nv;
  if (fi.x1) {
    fi.x1 += c * V;
    fi.invD += c * V;
  }
  restrict_point<T>(nf, mask, scale, rf + c * (nvf * nvf * nvf), rc + c * V, fi, id - t * nv, t - K * nv, K);
}

template <typename T>
__global__ void __launch_bounds__(kRestrictThreads)
    restrict_kernel(int nf, bool mask, T scale, const T* __restrict__ rf, T* __restrict__ rc, const FirstIterate<T> fi) {
  grid_dep_entry();
  restrict_thread<T>(nf, mask, scale, rf, rc, fi, blockIdx.y);
}

template <typename T, int NC, bool ADD>
__global__ void __launch_bounds__(32 * kRowWarps)
    prolong_kernel(int nf, bool mask, const T* __restrict__ ec, T* __restrict__ xf) {
  grid_dep_entry();
  const int w = blockIdx.x * kRowWarps + (threadIdx.x >> 5), nv = nf + 1;
  if (w < row_pieces(nv)) prolong_point<T, NC, ADD>(nf, mask, ec, xf, row_piece(nv, w, threadIdx.x & 31));
}

// many problems: grid (blocks of the largest, problems, components of a restriction)
template <typename T>
__global__ void __launch_bounds__(kRestrictThreads) restrict_batch_kernel(const XferTask* __restrict__ tasks) {
  grid_dep_entry();
  const XferTask tk = tasks[blockIdx.y];
  if (tk.sc && tk.sc[MS_DONE] != 0.0) return;
  FirstIterate<T> fi;
  fi.invD = static_cast<const T*>(tk.invD);
  fi.x1 = static_cast<T*>(tk.x1);
  fi.s2 = (T)tk.s2;
  restrict_thread<T>(tk.nf, tk.mask, (T)tk.scale, static_cast<const T*>(tk.src), static_cast<T*>(tk.dst), fi,
                     blockIdx.z);
}

template <typename T, int NC, bool ADD>
__global__ void __launch_bounds__(32 * kRowWarps) prolong_batch_kernel(const XferTask* __restrict__ tasks) {
  grid_dep_entry();
  const XferTask tk = tasks[blockIdx.y];
  if (tk.sc && tk.sc[MS_DONE] != 0.0) return;
  const int w = blockIdx.x * kRowWarps + (threadIdx.x >> 5), nv = tk.nf + 1;
  if (w < row_pieces(nv))
    prolong_point<T, NC, ADD>(tk.nf, tk.mask, static_cast<const T*>(tk.src), static_cast<T*>(tk.dst),
                              row_piece(nv, w, threadIdx.x & 31));
}

unsigned row_blocks(int n) {
  const int64_t nv = n + 1;
  return (unsigned)((nv * nv * ((nv + 31) / 32) + kRowWarps - 1) / kRowWarps);
}

unsigned vertex_blocks(int n) { return (unsigned)((nverts(n) + kRestrictThreads - 1) / kRestrictThreads); }

}  // namespace

bool pdl_enabled(cudaStream_t s) {
  static const bool on = [] {
    const char* v = getenv("AGCA_PDL");
    return !(v && v[0] == '0');
  }();
  return on && s != nullptr && s != cudaStreamLegacy;
}

// ncomp: 3 (velocity) or 1 (pressure)
template <typename T>
cudaError_t launch_restrict(int nf, int ncomp, bool mask, T scale, const T* rf, T* rc, cudaStream_t s,
                            const FirstIterate<T>& fi) {
  if (ncomp != 3 && ncomp != 1) return cudaErrorInvalidValue;
  return launch_k(restrict_kernel<T>, dim3(vertex_blocks(nf / 2), (unsigned)ncomp), dim3(kRestrictThreads), 0, s, nf, mask,
                  scale, rf, rc, fi);
}

template <typename T>
cudaError_t launch_prolong(int nf, int ncomp, bool mask, bool add, const T* ec, T* xf, cudaStream_t s) {
  const dim3 g(row_blocks(nf)), t(32 * kRowWarps);
  if (ncomp == 3 && add) return launch_k(prolong_kernel<T, 3, true>, g, t, 0, s, nf, mask, ec, xf);
  if (ncomp == 1 && !add) return launch_k(prolong_kernel<T, 1, false>, g, t, 0, s, nf, mask, ec, xf);
  return cudaErrorInvalidValue;
}

// velocity restriction and correction, pressure interpolation; the pressure's restriction (ncomp 1) in FP64 only
template <typename T>
cudaError_t launch_transfer_batch(int kind, int ncomp, const XferTask* tasks, int ntasks, int max_n, cudaStream_t s) {
  const dim3 g(row_blocks(max_n), (unsigned)ntasks), t(32 * kRowWarps);
  switch (kind) {
    case XK_RESTRICT:
      return launch_k(restrict_batch_kernel<T>, dim3(vertex_blocks(max_n), (unsigned)ntasks, (unsigned)ncomp),
                      dim3(kRestrictThreads), 0, s, tasks);
    case XK_PROLONG_ADD: return launch_k(prolong_batch_kernel<T, 3, true>, g, t, 0, s, tasks);
    case XK_PROLONG: return launch_k(prolong_batch_kernel<T, 1, false>, g, t, 0, s, tasks);
    default: return cudaErrorInvalidValue;
  }
}

template cudaError_t launch_restrict<float>(int, int, bool, float, const float*, float*, cudaStream_t,
                                            const FirstIterate<float>&);
template cudaError_t launch_restrict<double>(int, int, bool, double, const double*, double*, cudaStream_t,
                                             const FirstIterate<double>&);
template cudaError_t launch_prolong<float>(int, int, bool, bool, const float*, float*, cudaStream_t);
template cudaError_t launch_prolong<double>(int, int, bool, bool, const double*, double*, cudaStream_t);
template cudaError_t launch_transfer_batch<float>(int, int, const XferTask*, int, int, cudaStream_t);
template cudaError_t launch_transfer_batch<double>(int, int, const XferTask*, int, int, cudaStream_t);

}  // namespace agca
