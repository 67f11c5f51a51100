// noalloc.cu -- exact Poisson solves on single 8^3 boxes that allocate no
// memory.
//
// Some callers cannot call cudaMalloc: code that runs while another
// component owns every byte of device memory (a caching allocator or a
// memory pool it must not bypass), code that runs inside a region where
// allocation is forbidden or would synchronise the device, and embedders
// that only hand over their own input and output buffers.  For them
// sm_box_solve_noalloc solves the 7-point Poisson problem of many single
// boxes with the same eigenbasis method as the level-0 solve of the
// multigrid cycle.  It keeps nothing on the device: the four 1-D eigenbases
// (one per pair of end conditions) are 2.3 KB of launch parameters.
#include <cooperative_groups.h>
#include <math.h>
#include <mutex>

#include "sm_internal.cuh"

using namespace sm;
namespace cg = cooperative_groups;

namespace {

// Orthonormal eigenvectors (component i of vector m at 8 i + m) and
// h^2-scaled eigenvalues of the 1-D cell-centred 3-point operator on 8
// cells, by end conditions lo + 2 hi (0 Neumann, 1 Dirichlet): cosine (NN),
// sine (DD) and quarter-wave sine (DN, ND) families.
struct Bases {
  double v[4][64], lam[4][8];
  Bases() {
    const double pi = 3.14159265358979323846;
    for (int ty = 0; ty < 4; ++ty) {
      const bool lo = ty & 1, hi = ty & 2;
      for (int m = 0; m < NC; ++m) {
        const double th = !lo && !hi ? m : (lo && hi ? m + 1 : m + 0.5);
        double w[NC], nrm = 0.0;
        for (int i = 0; i < NC; ++i) {
          const double x = lo || !hi ? (i + 0.5) / NC : (NC - i - 0.5) / NC;
          w[i] = !lo && !hi ? cos(pi * th * x) : sin(pi * th * x);
          nrm += w[i] * w[i];
        }
        for (int i = 0; i < NC; ++i) v[ty][8 * i + m] = w[i] / sqrt(nrm);
        const double sn = sin(pi * th / (2.0 * NC));
        lam[ty][m] = -4.0 * sn * sn;
      }
    }
  }
};

// One problem per cluster of C blocks of 512 / C threads, a cell each.  The
// solve is FP64-pipe work (six 8-term transforms a cell, 2 instructions per
// clock and SM), so a call of few problems spreads each over several SMs:
// block r holds z-planes of the box (wall terms, x and y forward), then the
// slab of y modes r (z forward from the planes in the blocks' shared memory,
// eigenvalue scaling, z and x backward), then its z-planes again (y backward,
// store).
template <int C>
__global__ void __launch_bounds__(CELLS / C) k_box_solve(const double *__restrict__ f, double *__restrict__ phi,
                                                         const int32_t *__restrict__ bc_type,
                                                         const double *__restrict__ bc_val, double h2, double inv_h2,
                                                         const __grid_constant__ Bases B) {
  constexpr int T = CELLS / C, S = NC / C;  // threads, planes a block
  __shared__ double pa[T], pb[T], pc[T], V[3][64], lam[3][8], wall[6];
  cg::cluster_group cl = cg::this_cluster();
  const int p = blockIdx.x / C, r = blockIdx.x % C, t = threadIdx.x;
  const int i = t & 7, j = (t >> 3) & 7, s = t >> 6;
  const int32_t *bt = bc_type + 6 * p;
  auto kind = [&](int a) { return (bt[2 * a] != 0) | (bt[2 * a + 1] != 0) << 1; };
  double x = f[(size_t)p * CELLS + 64 * S * r + t];
  if (t < 6) wall[t] = bt[t] ? 2.0 * bc_val[6 * p + t] * inv_h2 : 0.0;  // 2g / h^2
  for (int n = t; n < 216; n += T) {
    if (n < 192) V[n >> 6][n & 63] = B.v[kind(n >> 6)][n & 63];
    else lam[(n - 192) >> 3][n & 7] = B.lam[kind((n - 192) >> 3)][n & 7];
  }
  __syncthreads();
  const int z = S * r + s;
  if (i == 0) x -= wall[0];
  if (i == NC - 1) x -= wall[1];
  if (j == 0) x -= wall[2];
  if (j == NC - 1) x -= wall[3];
  if (z == 0) x -= wall[4];
  if (z == NC - 1) x -= wall[5];
  pa[t] = x;
  __syncthreads();
  double acc = 0.0;
#pragma unroll
  for (int m = 0; m < NC; ++m) acc = fma(V[0][m * 8 + i], pa[m + 8 * j + 64 * s], acc);
  pb[t] = acc;
  __syncthreads();
  acc = 0.0;
#pragma unroll
  for (int m = 0; m < NC; ++m) acc = fma(V[1][m * 8 + j], pb[i + 8 * m + 64 * s], acc);
  __syncthreads();
  pa[t] = acc;  // read by the other blocks after the cluster barrier
  auto all = [&] {
    if constexpr (C == 1) __syncthreads();
    else cl.sync();
  };
  auto of = [&](double *q, int rank) {
    if constexpr (C == 1) return q;
    else return cl.map_shared_rank(q, rank);
  };
  all();
  {  // thread: x mode i, z (mode) j, y mode S r + s
    acc = 0.0;
#pragma unroll
    for (int m = 0; m < NC; ++m)
      acc = fma(V[2][m * 8 + j], of(pa, m / S)[i + 8 * (S * r + s) + 64 * (m % S)], acc);
    // a problem without a Dirichlet face has a zero eigenvalue (the constant
    // mode); that mode is set to zero
    const double ev = lam[0][i] + lam[1][S * r + s] + lam[2][j];
    pb[t] = ev != 0.0 ? quotient(acc * h2, ev) : 0.0;
    __syncthreads();
    acc = 0.0;
#pragma unroll
    for (int m = 0; m < NC; ++m) acc = fma(V[2][j * 8 + m], pb[i + 8 * m + 64 * s], acc);
    pc[t] = acc;
    __syncthreads();
    acc = 0.0;
#pragma unroll
    for (int m = 0; m < NC; ++m) acc = fma(V[0][i * 8 + m], pc[m + 8 * j + 64 * s], acc);
    pb[t] = acc;  // read by the other blocks after the cluster barrier
  }
  all();
  acc = 0.0;
#pragma unroll
  for (int m = 0; m < NC; ++m) acc = fma(V[1][j * 8 + m], of(pb, m / S)[i + 8 * z + 64 * (m % S)], acc);
  phi[(size_t)p * CELLS + 64 * S * r + t] = acc;
  if constexpr (C > 1) cl.sync();  // no block leaves while its shared memory is read
}

// The first call on a device loads the kernels, all of them whatever its
// problem count: CUDA would load each when it is first launched (10 us for a
// kernel, 110 for the module), inside a stream capture or where nothing may
// be loaded or allocated.  So that call has to be made outside a capture.
constexpr int MAX_DEVICES = 64;
std::mutex g_ready_mtx;
bool g_ready[MAX_DEVICES];

int device_ready(cudaStream_t stream) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return SM_ECUDA;
  }
  if (dev < 0 || dev >= MAX_DEVICES) return SM_EINVAL;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(stream, &cs) != cudaSuccess) {
    cudaGetLastError();
    return SM_ECUDA;
  }
  std::lock_guard<std::mutex> lock(g_ready_mtx);
  if (g_ready[dev]) return SM_OK;
  if (cs != cudaStreamCaptureStatusNone) return SM_ECUDA;
  cudaFuncAttributes a;  // asking for them loads the kernel
  if (cudaFuncGetAttributes(&a, k_box_solve<1>) != cudaSuccess ||
      cudaFuncGetAttributes(&a, k_box_solve<2>) != cudaSuccess ||
      cudaFuncGetAttributes(&a, k_box_solve<4>) != cudaSuccess ||
      cudaFuncGetAttributes(&a, k_box_solve<8>) != cudaSuccess) {
    cudaGetLastError();
    return SM_ECUDA;
  }
  g_ready[dev] = true;
  return SM_OK;
}

template <int C>
cudaError_t launch(int n, const double *f, double *phi, const int32_t *bc_type, const double *bc_val, double h2,
                   const Bases &B, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n * C);
  cfg.blockDim = dim3(CELLS / C);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_box_solve<C>, f, phi, bc_type, bc_val, h2, 1.0 / h2, B);
}

}  // namespace

extern "C" int sm_box_solve_noalloc(double length, int n_problems, const int32_t *bc_type, const double *bc_val,
                                    const double *f, double *phi, void *stream) {
  if (n_problems > SM_NOALLOC_MAX_PROBLEMS) return SM_ENOMEM;
  if (n_problems < 0 || !(length > 0.0)) return SM_EINVAL;
  if (n_problems > 0 && (!bc_type || !bc_val || !f || !phi)) return SM_EINVAL;
  if (const int st = device_ready((cudaStream_t)stream)) return st;
  if (n_problems == 0) return SM_OK;
  static const Bases bases;
  const double h = length / NC, h2 = h * h;
  const cudaStream_t st = (cudaStream_t)stream;
  // as many blocks per problem as still put every block on an SM of its own
  // (152): a block more on an SM's FP64 pipe costs what the split saves
  const cudaError_t e = n_problems <= 19   ? launch<8>(n_problems, f, phi, bc_type, bc_val, h2, bases, st)
                        : n_problems <= 38 ? launch<4>(n_problems, f, phi, bc_type, bc_val, h2, bases, st)
                        : n_problems <= 76 ? launch<2>(n_problems, f, phi, bc_type, bc_val, h2, bases, st)
                                           : launch<1>(n_problems, f, phi, bc_type, bc_val, h2, bases, st);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return SM_ECUDA;
  }
  return SM_OK;
}
