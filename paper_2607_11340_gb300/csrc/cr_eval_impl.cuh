// Kernels of the kinematics and cost entry points (cr_fk, cr_fk_jac, cr_cost_grad,
// cr_reduce_rows). One thread per state; states are structure-of-arrays [q][B] so that the
// per-component loads and stores of a warp are coalesced.
#pragma once

#include <cooperative_groups.h>

#include <atomic>

#include "cr_host.h"

namespace crk {

template <typename T, int N, int MODEL = CR_MODEL_TENDON>
__global__ void __launch_bounds__(128) k_fk(RobotK<T> rb, const T* __restrict__ u, int64_t B,
                                             T* __restrict__ Tout, T* __restrict__ bb) {
  int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  T uu[3 * N];
#pragma unroll
  for (int q = 0; q < 3 * N; ++q) uu[q] = u[q * B + b];
  Chain<T, N> ch;
  chain_forward<T, N, MODEL>(rb, uu, ch);
#pragma unroll
  for (int a = 0; a < 9; ++a) Tout[a * B + b] = ch.R[a];
#pragma unroll
  for (int a = 0; a < 3; ++a) Tout[(9 + a) * B + b] = ch.p[a];
  if (bb) {
    const T inb = T(1) / T(rb.nb);
#pragma unroll
    for (int i = 0; i < N; ++i)
      for (int k = 1; k <= rb.nb; ++k) {
        T q[3], w[3], s, c;
        backbone_point(ch.Rb[i], ch.pb[i], ch.ax[i], ch.ay[i], ch.x[i], ch.L[i], T(k) * inb, q, w, s, c);
        int64_t row = (int64_t)(i * rb.nb + (k - 1)) * 3;
        bb[(row + 0) * B + b] = w[0];
        bb[(row + 1) * B + b] = w[1];
        bb[(row + 2) * B + b] = w[2];
      }
  }
}

template <typename T, int N, int MODEL = CR_MODEL_TENDON>
__global__ void __launch_bounds__(128) k_fk_jac(RobotK<T> rb, const T* __restrict__ u, int64_t B,
                                                 T* __restrict__ J) {
  constexpr int D = 3 * N;
  int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  T uu[D];
#pragma unroll
  for (int q = 0; q < D; ++q) uu[q] = u[q * B + b];
  Chain<T, N> ch;
  chain_forward<T, N, MODEL>(rb, uu, ch);
  T Jp[3][D], Jw[3][D];
  tip_jacobian<T, N, MODEL>(rb, ch, Jp, Jw);
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int q = 0; q < D; ++q) {
      J[((int64_t)a * D + q) * B + b] = Jp[a][q];
      J[((int64_t)(3 + a) * D + q) * B + b] = Jw[a][q];
    }
}

// MODE 0: cost only; 1: cost + dF/du; 2: cost + dF/du + dF/d(L, r_c)
template <typename T, int N, bool OBST, int MODE, int MODEL = CR_MODEL_TENDON>
__global__ void __launch_bounds__(128) k_cost_grad(RobotK<T> rb, WeightsK<T> w, int kind,
                                                    const double* __restrict__ targets, int64_t P,
                                                    int S, const double* __restrict__ spheres, int no,
                                                    const double* __restrict__ prims, int np,
                                                    const T* __restrict__ u, int64_t B, T* cost,
                                                    T* coll, T* gu, T* gp, const T* __restrict__ upstream) {
  constexpr int D = 3 * N;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ObsK<T> ob(nullptr);
  const Sphere4<float>* f32 = nullptr;
  if (OBST) {
    ob = stage_obstacles(spheres, no, prims, np, rb, w.delta, smem_raw);
    __syncthreads();
    if constexpr (sizeof(T) == 8) {  // the FP32 copy of the table for the broad phase
      Sphere4<float>* f = reinterpret_cast<Sphere4<float>*>(smem_raw + ((obstacles_smem<T>(no, np) + 15) & ~(size_t)15));
      bool fits = true;
      for (int j = threadIdx.x; j < no + np; j += blockDim.x) {
        f[j] = Sphere4<float>{float(ob.s[j].x), float(ob.s[j].y), float(ob.s[j].z), float(ob.s[j].reach)};
        fits = fits && cull_entry_fits(f[j].reach);
      }
      f32 = __syncthreads_and(fits) ? f : nullptr;
    }
  }
  int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  T uu[D];
#pragma unroll
  for (int q = 0; q < D; ++q) uu[q] = u[q * B + b];
  TargetK<T> tg = load_target<T>(targets, P, b / S, kind);
  T g[D], gL[N], grc[N], cl;
  T F = eval_ik<T, N, OBST, (MODE >= 1), (MODE >= 2), true, MODEL, true>(rb, w, kind, tg, ob, no + np, uu, g, gL, grc,
                                                                          &cl, f32);
  if (cost) cost[b] = F;
  if (coll) coll[b] = cl;
  const T up = upstream ? upstream[b] : T(1);  // vector-Jacobian product weight
  if (MODE >= 1) {
#pragma unroll
    for (int q = 0; q < D; ++q) gu[q * B + b] = up * g[q];
  }
  if (MODE >= 2) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      gp[(int64_t)i * B + b] = up * gL[i];
      gp[(int64_t)(N + i) * B + b] = up * grc[i];
    }
  }
}

// Deterministic row sums in FP64: row y = blockIdx.y is cut into gridDim.x equal pieces, one block of
// the cluster (gridDim.x, 1, 1) each; a thread adds its piece's elements with 8 loads in flight into 4
// accumulators, a block its threads by butterflies and warps in order, block 0 the blocks' sums in
// order through distributed shared memory. All orders are fixed by (B, gridDim.x).
// Bound: the FP64 pipe (a widening and an addition per element, each holding a sub-partition's unit
// 64 cycles). One block of 256 threads with one load in flight per row kept 6 SMs busy on the 6
// parameter rows of 262,144 states and waited on every load: 195 us of a 485 us gradient pass, which takes
// 328 us with 16 blocks per row (60,001 states and 8 rows: 52 us of 396, now 359).
constexpr int kReduceThreads = 512;  // of a cluster's blocks
template <typename T, int TH>
__global__ void __launch_bounds__(TH) k_reduce_rows(const T* __restrict__ x, int64_t B, double* out) {
  constexpr int NW = TH / 32;
  __shared__ double part[NW];
  __shared__ double total;
  namespace cg = cooperative_groups;
  const int64_t len = (B + gridDim.x - 1) / gridDim.x;
  const int64_t b0 = len * blockIdx.x, b1 = b0 + len < B ? b0 + len : B;
  const T* row = x + (int64_t)blockIdx.y * B;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  int64_t b = b0 + threadIdx.x;
  for (; b + 7 * TH < b1; b += 8 * TH) {
    T v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = row[b + k * TH];
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[k & 3] += double(v[k]);
  }
  if (NW == 1) {  // the last elements: in flight together where no other warp hides their latency
    T v[7];
#pragma unroll
    for (int k = 0; k < 7; ++k) v[k] = b + k * TH < b1 ? row[b + k * TH] : T(0);
#pragma unroll
    for (int k = 0; k < 7; ++k)
      if (b + k * TH < b1) acc[0] += double(v[k]);
  } else {
    for (; b < b1; b += TH) acc[0] += double(row[b]);
  }
  double s = (acc[0] + acc[1]) + (acc[2] + acc[3]);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (NW > 1) {
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    if (NW > 1) {
      s = part[0];
      for (int w = 1; w < NW; ++w) s += part[w];
    }
    total = s;
  }
  if (gridDim.x == 1) {
    if (threadIdx.x == 0) out[blockIdx.y] = s;
    return;
  }
  cg::cluster_group cl = cg::this_cluster();
  cl.sync();
  if (blockIdx.x == 0 && threadIdx.x < 32) {
    double t = threadIdx.x < gridDim.x ? *cl.map_shared_rank(&total, threadIdx.x) : 0.0;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    if (threadIdx.x == 0) out[blockIdx.y] = t;
  }
  cl.sync();  // block 0 has read every block's sum before any of them exits
}

// Whether the current device can hold a cluster of 16 of these blocks, which is more than the 8 that every one
// schedules: a partition of a GPU may not. Asked once per device and type, so that the order of the sums stays fixed.
template <typename T> bool reduce_cluster16_fits() {
  constexpr int kDevices = 64;
  static std::atomic<int> known[kDevices];  // 0: not asked, 1: no, 2: yes
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return false;
  const int k = known[dev].load(std::memory_order_relaxed);
  if (k) return k == 2;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(16, 1, 1);
  cfg.blockDim = dim3(kReduceThreads, 1, 1);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 16;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int clusters = 0;
  const bool fits =
      cudaFuncSetAttribute(k_reduce_rows<T, kReduceThreads>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
          cudaSuccess &&
      cudaOccupancyMaxActiveClusters(&clusters, k_reduce_rows<T, kReduceThreads>, &cfg) == cudaSuccess && clusters > 0;
  if (!fits) (void)cudaGetLastError();
  known[dev].store(fits ? 2 : 1, std::memory_order_relaxed);
  return fits;
}

// Blocks per row: enough for about one block per SM over all rows, a power of two of at most 16 (the
// largest cluster, opt-in; 8 where that does not fit), and at least 2048 elements to a block, below which one
// block's few loads cost less than the cluster's barriers.
template <typename T> int reduce_cluster(int64_t rows, int64_t B) {
  int c = 1;
  while (c < 16 && rows * c < 152 && B >= (int64_t)4096 * c) c *= 2;
  return c > 8 && !reduce_cluster16_fits<T>() ? 8 : c;
}

// Threads of a block: 512 in a cluster. A row that is one block's (many rows, or short ones) takes fewer: every warp
// adds 8 FP64 operations of its own, which bound short rows (100,000 rows of 300 in FP32: 1.45 ms with 512 threads, 0.52
// with 128, 0.23 with a warp). With a warp or more to each of the 4 x 152 sub-partitions a row of up to 8192
// elements is one warp's (1000 rows of 1000: 10 us, 25 with 512 threads); fewer rows have 128 threads (304 rows of 4096: 8
// us, 14 with a warp), and above 16,384 elements 256 keep more loads in flight (1000 rows of 30,000 in FP64: 72 us, 77
// with 128, 80 with 512).
inline int reduce_threads(int c, int64_t rows, int64_t B) {
  if (c > 1) return kReduceThreads;
  if (rows >= 608 && B <= 8192) return 32;
  return B <= 16384 ? 128 : 256;
}

// ------------------------------------------------------------------------------------------------
// Host launchers (instantiated for float and double in separate translation units)
// ------------------------------------------------------------------------------------------------
struct EvalArgs {
  cr_robot robot;
  cr_scene scene;
  cr_task task;
  const void* u;
  int64_t B;
  void *cost, *coll, *gu, *gp, *Tout, *bb, *J;
  const void* upstream;
  cudaStream_t stream;
};

template <typename T> cr_status launch_fk(const EvalArgs& a);
template <typename T> cr_status launch_fk_jac(const EvalArgs& a);
template <typename T> cr_status launch_cost_grad(const EvalArgs& a);
template <typename T> cr_status launch_reduce_rows(const void* x, int64_t rows, int64_t B, double* out,
                                                   cudaStream_t s);

inline unsigned grid_of(int64_t B, int bs) { return (unsigned)((B + bs - 1) / bs); }

template <typename T, int N, int MODEL = CR_MODEL_TENDON> void fk_n(const EvalArgs& a) {
  RobotK<T> rb = crh::robot_k<T>(a.robot);
  k_fk<T, N, MODEL><<<grid_of(a.B, 128), 128, 0, a.stream>>>(rb, (const T*)a.u, a.B, (T*)a.Tout, (T*)a.bb);
}
template <typename T, int N, int MODEL = CR_MODEL_TENDON> void fk_jac_n(const EvalArgs& a) {
  RobotK<T> rb = crh::robot_k<T>(a.robot);
  k_fk_jac<T, N, MODEL><<<grid_of(a.B, 128), 128, 0, a.stream>>>(rb, (const T*)a.u, a.B, (T*)a.J);
}
template <typename T, int N, int MODEL = CR_MODEL_TENDON> void cost_grad_n(const EvalArgs& a) {
  RobotK<T> rb = crh::robot_k<T>(a.robot);
  WeightsK<T> w = crh::weights_k<T>(a.task.w);
  int no = a.scene.n_o, np = a.scene.n_p;
  int mode = a.gp ? 2 : (a.gu ? 1 : 0);
  size_t sm = obstacles_smem<T>(no, np);
  // FP64: the FP32 table behind it; at most 45 + 4 KB = the 48 KB of a launch without opt-in
  if (sizeof(T) == 8) sm = ((sm + 15) & ~(size_t)15) + (size_t)(no + np) * sizeof(Sphere4<float>);
  unsigned g = grid_of(a.B, 128);
#define CR_CG(OB, MO)                                                                              \
  k_cost_grad<T, N, OB, MO, MODEL><<<g, 128, sm, a.stream>>>(rb, w, a.task.kind, a.task.targets,   \
                                                       a.task.n_targets, a.task.seeds_per_target,  \
                                                       a.scene.spheres, no, a.scene.prims, np,     \
                                                       (const T*)a.u, a.B,                         \
                                                       (T*)a.cost, (T*)a.coll, (T*)a.gu, (T*)a.gp, \
                                                       (const T*)a.upstream)
  if (no + np > 0 || a.task.w.rho_s > 0) {  // collision rows: obstacles and / or self-contact
    if (mode == 0) CR_CG(true, 0); else if (mode == 1) CR_CG(true, 1); else CR_CG(true, 2);
  } else {
    if (mode == 0) CR_CG(false, 0); else if (mode == 1) CR_CG(false, 1); else CR_CG(false, 2);
  }
#undef CR_CG
}

// The arc model's launchers (1..CR_MAX_SEG_ARC segments) live in their own translation units.
#define CR_EVAL_ARC(FN, T, a)                  \
  switch ((a).robot.n) {                       \
    case 1: FN<T, 1, CR_MODEL_ARC>(a); break;  \
    case 2: FN<T, 2, CR_MODEL_ARC>(a); break;  \
    case 3: FN<T, 3, CR_MODEL_ARC>(a); break;  \
    default: FN<T, 4, CR_MODEL_ARC>(a); break; \
  }
template <typename T> void launch_eval_arc(const EvalArgs& a, int what) {
  if (what == 0) { CR_EVAL_ARC(fk_n, T, a) }
  else if (what == 1) { CR_EVAL_ARC(fk_jac_n, T, a) }
  else { CR_EVAL_ARC(cost_grad_n, T, a) }
}

// Coupled routing (model B), 1..CR_MAX_SEG segments, in its own translation units.
#define CR_EVAL_COUPLED(FN, T, a)                  \
  switch ((a).robot.n) {                           \
    case 1: FN<T, 1, CR_MODEL_COUPLED>(a); break;  \
    case 2: FN<T, 2, CR_MODEL_COUPLED>(a); break;  \
    case 3: FN<T, 3, CR_MODEL_COUPLED>(a); break;  \
    case 4: FN<T, 4, CR_MODEL_COUPLED>(a); break;  \
    case 5: FN<T, 5, CR_MODEL_COUPLED>(a); break;  \
    default: FN<T, 6, CR_MODEL_COUPLED>(a); break; \
  }
template <typename T> void launch_eval_coupled(const EvalArgs& a, int what) {
  if (what == 0) { CR_EVAL_COUPLED(fk_n, T, a) }
  else if (what == 1) { CR_EVAL_COUPLED(fk_jac_n, T, a) }
  else { CR_EVAL_COUPLED(cost_grad_n, T, a) }
}

template <typename T> cr_status launch_fk(const EvalArgs& a) {
  if (a.robot.model == CR_MODEL_ARC) launch_eval_arc<T>(a, 0);
  else if (a.robot.model == CR_MODEL_COUPLED) launch_eval_coupled<T>(a, 0);
  else CR_DISPATCH_NT(a.robot.n, fk_n, T, a);
  return crh::check_launch("cr_fk");
}
template <typename T> cr_status launch_fk_jac(const EvalArgs& a) {
  if (a.robot.model == CR_MODEL_ARC) launch_eval_arc<T>(a, 1);
  else if (a.robot.model == CR_MODEL_COUPLED) launch_eval_coupled<T>(a, 1);
  else CR_DISPATCH_NT(a.robot.n, fk_jac_n, T, a);
  return crh::check_launch("cr_fk_jac");
}
template <typename T> cr_status launch_cost_grad(const EvalArgs& a) {
  if (a.robot.model == CR_MODEL_ARC) launch_eval_arc<T>(a, 2);
  else if (a.robot.model == CR_MODEL_COUPLED) launch_eval_coupled<T>(a, 2);
  else CR_DISPATCH_NT(a.robot.n, cost_grad_n, T, a);
  return crh::check_launch("cr_cost_grad");
}

#define CR_EVAL_ARC_INSTANTIATE(EXT, T) EXT template void launch_eval_arc<T>(const EvalArgs&, int);
#define CR_EVAL_COUPLED_INSTANTIATE(EXT, T) EXT template void launch_eval_coupled<T>(const EvalArgs&, int);
template <typename T>
cr_status launch_reduce_rows(const void* x, int64_t rows, int64_t B, double* out, cudaStream_t s) {
  const int c = reduce_cluster<T>(rows, B);
  const int th = reduce_threads(c, rows, B);
  auto kernel = th == 32 ? k_reduce_rows<T, 32> : th == 128 ? k_reduce_rows<T, 128>
              : th == 256 ? k_reduce_rows<T, 256> : k_reduce_rows<T, kReduceThreads>;
  for (int64_t r0 = 0; r0 < rows; r0 += 65535) {  // rows along grid.y
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)c, (unsigned)(rows - r0 < 65535 ? rows - r0 : 65535), 1);
    cfg.blockDim = dim3((unsigned)th, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)c;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = c > 1 ? 1 : 0;
    cudaError_t e = cudaSuccess;
    if (c > 8) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, kernel, (const T*)x + r0 * B, B, out + r0);
    if (e != cudaSuccess) {
      (void)cudaGetLastError();
      return crh::fail(CR_ECUDA, "cr_reduce_rows: %s", cudaGetErrorString(e));
    }
  }
  return crh::check_launch("cr_reduce_rows");
}

#define CR_EVAL_INSTANTIATE(EXT, T)                                                              \
  EXT template cr_status launch_fk<T>(const EvalArgs&);                                          \
  EXT template cr_status launch_fk_jac<T>(const EvalArgs&);                                      \
  EXT template cr_status launch_cost_grad<T>(const EvalArgs&);                                   \
  EXT template cr_status launch_reduce_rows<T>(const void*, int64_t, int64_t, double*, cudaStream_t);

}  // namespace crk
