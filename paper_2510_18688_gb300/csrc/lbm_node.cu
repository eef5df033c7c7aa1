// lbm_node.cu -- the two-kernel node step (lbm_node.cuh) of two-dimensional
// double-precision and tangent contexts, single grids and batches (sm_103a).
#include "lbm_launch.h"

namespace lbmn {

// The bound that sets the registers a thread, not a block's size (blocks have
// 32 to 128 threads, warps_per_block): 128 registers in double, so that sixteen
// warps fit an SM, which saturate its FP64 pipe; all 255 for a tangent.
constexpr int NTN = 256;
template <typename R>
constexpr int min_blocks() {
  return std::is_same<R, double>::value ? 2 : 1;
}

template <typename R, int LATC>
__global__ void __launch_bounds__(NTN, min_blocks<R>())
    node_local_kernel(const __grid_constant__ NodeArgs<R, 2> a) {
  lbmk::after_previous();
  node_local_linear<R, 2, LATC, int>(a, blockIdx.x * blockDim.x + threadIdx.x);
}

template <typename R, int LATC, bool DIAG>
__global__ void __launch_bounds__(NTN, min_blocks<R>())
    node_collide_kernel(const __grid_constant__ NodeArgs<R, 2> a) {
  lbmk::after_previous();
  node_collide_linear<R, 2, LATC, false, DIAG, int>(a, nullptr, blockIdx.x * blockDim.x + threadIdx.x);
}

template <typename R, int LATC, bool DIAG>
__global__ void __launch_bounds__(NTN, min_blocks<R>())
    node_read_kernel(const __grid_constant__ NodeArgs<R, 2> a,
                     const __grid_constant__ ReadOut ro) {
  lbmk::after_previous();
  node_collide_linear<R, 2, LATC, true, DIAG, int>(a, &ro, blockIdx.x * blockDim.x + threadIdx.x);
}

// Warps per block: four where that still gives each of GB300's 152 SMs several blocks; a
// grid of a few thousand nodes is spread warp by warp, so that no SM gets
// more than its share of the FP64 work.
static int warps_per_block(int nwarps) {
  return nwarps >= 4 * 4 * 152 ? 4 : (nwarps >= 2 * 2 * 152 ? 2 : 1);
}

template <typename R, int LATC>
static void launch_lat(const NodeArgs<R, 2>& a, const ReadOut* ro, bool diag, int wpb,
                       cudaStream_t s) {
  const int nt = 32 * wpb, nb = (a.nwarps + wpb - 1) / wpb;
  lbmk::launch_dep(node_local_kernel<R, LATC>, nb, nt, 0, s, a);
  if (ro) {
    if (diag) lbmk::launch_dep(node_read_kernel<R, LATC, true>, nb, nt, 0, s, a, *ro);
    else lbmk::launch_dep(node_read_kernel<R, LATC, false>, nb, nt, 0, s, a, *ro);
  } else {
    if (diag) lbmk::launch_dep(node_collide_kernel<R, LATC, true>, nb, nt, 0, s, a);
    else lbmk::launch_dep(node_collide_kernel<R, LATC, false>, nb, nt, 0, s, a);
  }
}

template <typename R>
cudaError_t launch_node(const NodeArgs<R, 2>& a, const ReadOut* ro, bool diag,
                        cudaStream_t s) {
  const int wpb = warps_per_block(a.nwarps);
  // the all-lattices case is specialised at compile time
  if (a.g.lattices == (LAT_FLOW | LAT_PHASE | LAT_HEAT)) launch_lat<R, 7>(a, ro, diag, wpb, s);
  else launch_lat<R, 0>(a, ro, diag, wpb, s);
  return cudaGetLastError();
}
template cudaError_t launch_node<double>(const NodeArgs<double, 2>&, const ReadOut*, bool, cudaStream_t);
template cudaError_t launch_node<Dual>(const NodeArgs<Dual, 2>&, const ReadOut*, bool, cudaStream_t);

cudaError_t launch_node_local(const NodeArgs<double, 2>& a, cudaStream_t s) {
  const int wpb = warps_per_block(a.nwarps), nt = 32 * wpb, nb = (a.nwarps + wpb - 1) / wpb;
  if (a.g.lattices == (LAT_FLOW | LAT_PHASE | LAT_HEAT)) lbmk::launch_dep(node_local_kernel<double, 7>, nb, nt, 0, s, a);
  else lbmk::launch_dep(node_local_kernel<double, 0>, nb, nt, 0, s, a);
  return cudaGetLastError();
}

// Batches: block t takes block t of the concatenated block lists of the
// grids (its grid by bisection); a node's arithmetic and its warp's partial
// sums are those of the single-grid kernels.
template <bool COLLIDE, int LATC, bool DIAG>
__global__ void __launch_bounds__(NTN, 2)
    node_batch_kernel(const __grid_constant__ NodeBatch B) {
  const int t = blockIdx.x;
  int lo = 0, hi = B.ngrids;  // base[lo] <= t < base[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (B.base[mid] <= t) lo = mid;
    else hi = mid;
  }
  const int id = (t - B.base[lo]) * blockDim.x + threadIdx.x;
  lbmk::after_previous();
  if (COLLIDE) node_collide_linear<double, 2, LATC, false, DIAG, int>(B.args[lo], nullptr, id);
  else node_local_linear<double, 2, LATC, int>(B.args[lo], id);
}

template <int LATC>
static void launch_batch_lat(const NodeBatch& b, bool diag, cudaStream_t s) {
  const int nt = NODE_BATCH_THREADS, nb = b.base[b.ngrids];
  lbmk::launch_dep(node_batch_kernel<false, LATC, false>, nb, nt, 0, s, b);
  if (diag) lbmk::launch_dep(node_batch_kernel<true, LATC, true>, nb, nt, 0, s, b);
  else lbmk::launch_dep(node_batch_kernel<true, LATC, false>, nb, nt, 0, s, b);
}

cudaError_t launch_node_batch(const NodeBatch& b, bool diag, bool all, cudaStream_t s) {
  if (all) launch_batch_lat<7>(b, diag, s);
  else launch_batch_lat<0>(b, diag, s);
  return cudaGetLastError();
}

}  // namespace lbmn
