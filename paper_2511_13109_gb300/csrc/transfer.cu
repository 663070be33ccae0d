// Interpolation between Kuhn grids and its transpose (Sec. 2.1): one thread per
// written vertex, all components at once, a warp on 32 vertices of one row.  The
// per-point formulas are restrict_point / prolong_point in device_ops.cuh.  With
// flat vertex indices (two integer divisions each) and a loop over the components
// the finest FP32 level at 128^3 pressure cubes took 131 us (prolongation) and
// 87 us (restriction with the first iterate); now 92 and 54 us, floors 64 and 41.
// (One warp per row, looping over it, left too little in flight: 134 and 106 us.)
#include <stdlib.h>

#include "agca_internal.cuh"
#include "device_ops.cuh"

namespace agca {

namespace {

constexpr int kRowWarps = 8;

template <typename T, int NC>
__global__ void __launch_bounds__(32 * kRowWarps)
    restrict_kernel(int nf, bool mask, T scale, const T* __restrict__ rf, T* __restrict__ rc, const FirstIterate<T> fi) {
  grid_dep_entry();
  const int w = blockIdx.x * kRowWarps + (threadIdx.x >> 5), nv = nf / 2 + 1;
  if (w < row_pieces(nv)) restrict_point<T, NC>(nf, mask, scale, rf, rc, fi, row_piece(nv, w, threadIdx.x & 31));
}

template <typename T, int NC, bool ADD>
__global__ void __launch_bounds__(32 * kRowWarps)
    prolong_kernel(int nf, bool mask, const T* __restrict__ ec, T* __restrict__ xf) {
  grid_dep_entry();
  const int w = blockIdx.x * kRowWarps + (threadIdx.x >> 5), nv = nf + 1;
  if (w < row_pieces(nv)) prolong_point<T, NC, ADD>(nf, mask, ec, xf, row_piece(nv, w, threadIdx.x & 31));
}

// many problems: grid (blocks of the largest, problems)
template <typename T, int NC>
__global__ void __launch_bounds__(32 * kRowWarps) restrict_batch_kernel(const XferTask* __restrict__ tasks) {
  grid_dep_entry();
  const XferTask tk = tasks[blockIdx.y];
  if (tk.sc && tk.sc[MS_DONE] != 0.0) return;
  const int w = blockIdx.x * kRowWarps + (threadIdx.x >> 5), nv = tk.nf / 2 + 1;
  if (w >= row_pieces(nv)) return;
  FirstIterate<T> fi;
  fi.invD = static_cast<const T*>(tk.invD);
  fi.x1 = static_cast<T*>(tk.x1);
  fi.s2 = (T)tk.s2;
  restrict_point<T, NC>(tk.nf, tk.mask, (T)tk.scale, static_cast<const T*>(tk.src), static_cast<T*>(tk.dst), fi,
                        row_piece(nv, w, threadIdx.x & 31));
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
  const dim3 g(row_blocks(nf / 2)), t(32 * kRowWarps);
  if (ncomp == 3) return launch_k(restrict_kernel<T, 3>, g, t, 0, s, nf, mask, scale, rf, rc, fi);
  if (ncomp == 1) return launch_k(restrict_kernel<T, 1>, g, t, 0, s, nf, mask, scale, rf, rc, fi);
  return cudaErrorInvalidValue;
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
      if (ncomp == 3) return launch_k(restrict_batch_kernel<T, 3>, g, t, 0, s, tasks);
      return launch_k(restrict_batch_kernel<T, 1>, g, t, 0, s, tasks);
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
