// The coarse tail of the V-cycle (Sec. 5) in one block: every level from the first one that fits
// down to the coarsest is held in shared memory, and one launch runs its pre-relaxation and
// restriction on the way down, the dense coarsest solve, and the correction and post-relaxation
// on the way up. Below a few thousand nodes a level's kernels are bound by launch and ramp
// latency, not by work, so this replaces 2 (L - lt) - 1 launches by one. Each level's operations
// are the ones the per-level kernels perform (hz_level.cuh, fixed-rounding arithmetic), so the
// result is bitwise the same as without the tail (one-sweep Gauss-Seidel levels and every
// Kaczmarz form). In FP64 a cluster's other blocks help with the coarsest solve (coarse_cluster).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "hz_common.cuh"
#include "hz_host.h"
#include "hz_internal.h"
#include "hz_level.cuh"

namespace hz {

namespace {

constexpr int TAIL_THREADS = 1024;

// The coarsest solve of the FP64 tail over a cluster: one SM's FP64 pipe (a warp instruction every 77
// cycles or so) took 19 us for m = 81 rows of m columns, most of the tail. The tail's block and TAIL_CLUSTER - 1
// helpers take ceil(m / TAIL_CLUSTER) rows each: the products of all columns at once, then the additions
// in column order (lvl::coarse_row's bits), a lane per row and component. The helpers hold their rows of
// the inverse before the right-hand side is there and do nothing else; two cluster barriers. The
// tail of n_l = 16 and 8 37.7 -> 25.4 us.
constexpr int TAIL_CLUSTER = 8;
struct CoarseShare {  // shared-memory layout at off_ainv, inside the m * m cells of the whole inverse
  int m, rows;
  double2 *inv, *f;
  double* prod;
  __device__ CoarseShare(unsigned char* base, int m_) : m(m_), rows((m_ + TAIL_CLUSTER - 1) / TAIL_CLUSTER) {
    inv = reinterpret_cast<double2*>(base);
    f = inv + (size_t)m * rows;
    prod = reinterpret_cast<double*>(f + m);
  }
};
// one warp's lanes hold a block's rows, and the layout fits
constexpr bool coarse_share_fits(int m) {
  const int rows = (m + TAIL_CLUSTER - 1) / TAIL_CLUSTER;
  return 2 * rows <= 32 && 2 * rows + 1 <= m;
}
__device__ __forceinline__ void coarse_fetch(const CoarseShare& S, const double2* __restrict__ ainvT, int rank) {
  for (int t = threadIdx.x; t < S.m * S.rows; t += TAIL_THREADS) {
    const int c = t / S.rows, r = min(rank * S.rows + t - c * S.rows, S.m - 1);
    lvl::cp_async<sizeof(double2)>(S.inv + t, ainvT + (long long)c * S.m + r);
  }
}
// u = A^-1 f of the tail's block (rank 0); every thread of the cluster takes part.
__device__ __forceinline__ void coarse_cluster(const CoarseShare& S, double2* u, const double2* f) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), lanes = 2 * S.rows;
  cl.sync();  // f is there
  const double2* f0 = cl.map_shared_rank(const_cast<double2*>(f), 0);
  for (int q = threadIdx.x; q < S.m; q += TAIL_THREADS) S.f[q] = f0[q];
  __syncthreads();
  for (int t = threadIdx.x; t < S.m * lanes; t += TAIL_THREADS) {  // xr::cmul's components
    const int c = t / lanes, x = t - c * lanes, comp = x & 1;
    const double2 a = S.inv[c * S.rows + (x >> 1)], v = S.f[c];
    const double p = xr::mul(a.y, comp ? v.x : v.y);
    S.prod[t] = xr::fma(a.x, comp ? v.y : v.x, comp ? p : -p);
  }
  __syncthreads();
  const int row = rank * S.rows + (int)(threadIdx.x >> 1);
  if ((int)threadIdx.x < lanes && row < S.m) {
    double acc = 0.0;
#pragma unroll 8
    for (int c = 0; c < S.m; ++c) acc = xr::add(acc, S.prod[c * lanes + threadIdx.x]);
    reinterpret_cast<double*>(cl.map_shared_rank(u, 0) + row)[threadIdx.x & 1] = acc;
  }
  cl.sync();  // u is there
}

// CL: the block and its helpers form a cluster (coarse_cluster).
template <class T, bool CL>
__device__ __forceinline__ void tail_body(const TailArgs& A, const int* __restrict__ stop, const Inst& bi) {
  extern __shared__ __align__(16) unsigned char smem[];
  const c2<T>* fin = reinterpret_cast<const c2<T>*>(A.f_in) + blockIdx.z * bi.sf;
  c2<T>* uout = reinterpret_cast<c2<T>*>(A.u_out) + blockIdx.z * bi.so;
  auto U = [&](int l) { return reinterpret_cast<c2<T>*>(smem + A.lv[l].off_u); };
  auto F = [&](int l) { return reinterpret_cast<c2<T>*>(smem + A.lv[l].off_f); };
  auto K = [&](int l) { return reinterpret_cast<T*>(smem + A.lv[l].off_k); };
  auto D = [&](int l) { return reinterpret_cast<c2<T>*>(smem + A.lv[l].off_d); };
  auto V = [&](int l) { return reinterpret_cast<T*>(smem + A.lv[l].off_inv); };
  c2<T>* R = reinterpret_cast<c2<T>*>(smem + A.off_r);
  const int last = A.count - 1;

  // Kaczmarz levels are stored colour-blocked, the others row-major (lvl::Natural, lvl::Blocked)
  auto with_layout = [&](int l, auto&& fn) {
    const int nl = A.lv[l].n;
    if (A.lv[l].kind == TAIL_KACZ)
      fn(lvl::blocked(nl));
    else
      fn(lvl::Natural{nl + 1});
  };

  if constexpr (CL) {
    const CoarseShare S(smem + A.off_ainv, (A.lv[last].n + 1) * (A.lv[last].n + 1));
    const int rank = (int)cooperative_groups::this_cluster().block_rank();
    coarse_fetch(S, reinterpret_cast<const c2<T>*>(A.ainvT), rank);
    if (rank > 0) {
      lvl::cp_async_wait_all();
      pdl_enter();
      if (stop && stop[blockIdx.z * bi.stop_stride]) return;  // the whole cluster
      coarse_cluster(S, U(last), F(last));
      return;
    }
  }

  // Before the wait for the preceding kernel, everything that does not depend on it, so that with
  // programmatic dependent launch it overlaps that kernel: k H of every relaxation level (set up
  // once per problem), copied at once (cp.async, one wait) into K(l) on Gauss-Seidel levels and
  // into the cells of 1/|a|^2 on Kaczmarz levels, where the row constants replace it (plus a
  // row-major copy for the residual when there is room); the zero guess of the Kaczmarz levels.
  for (int l = 0; l < last; ++l) {
    const TailLevel& L = A.lv[l];
    const T* kh = reinterpret_cast<const T*>(L.kh);
    if (L.kind == TAIL_KACZ) {
      for (int q = threadIdx.x; q < lvl::blocked_cells(L.n); q += TAIL_THREADS) U(l)[q] = mk<T>(0, 0);
      T* kres = L.off_kres ? reinterpret_cast<T*>(smem + L.off_kres) : nullptr;
      lvl::for_nodes_blocked(L.n, [&](int q, int i, int j, int p) {
        const T* src = kh + (long long)j * L.pk + i;
        lvl::cp_async<sizeof(T)>(&V(l)[p], src);
        if (kres) lvl::cp_async<sizeof(T)>(&kres[q], src);
      });
    } else {
      const int w = L.n + 1;
      lvl::for_nodes(w, w * w, [&](int q, int i, int j) {
        lvl::cp_async<sizeof(T)>(&K(l)[q], kh + (long long)j * L.pk + i);
      });
    }
  }
  const int mc = (A.lv[last].n + 1) * (A.lv[last].n + 1);
  if (!CL && A.off_ainv) {  // the coarsest inverse, when it fits
    const c2<T>* src = reinterpret_cast<const c2<T>*>(A.ainvT);
    c2<T>* dst = reinterpret_cast<c2<T>*>(smem + A.off_ainv);
    for (int q = threadIdx.x; q < mc * mc; q += TAIL_THREADS) lvl::cp_async<sizeof(c2<T>)>(dst + q, src + q);
  }
  lvl::cp_async_wait_all();
  __syncthreads();
  for (int l = 0; l < last; ++l) {
    const TailLevel& L = A.lv[l];
    if (L.kind == TAIL_KACZ)
      lvl::for_blocked(L.n, [&](int i, int j, int p) {
        lvl::row_consts<T>(V(l)[p], i, j, L.n, (T)L.bA, &D(l)[p], &V(l)[p]);
      });
  }

  pdl_enter();
  if (stop && stop[blockIdx.z * bi.stop_stride]) return;  // the whole block
  // the first level's right-hand side (the preceding kernel's output), and its red nodes if it is
  // a Gauss-Seidel level
  {
    const TailLevel& L = A.lv[0];
    const int w = L.n + 1;
    if (L.kind == TAIL_KACZ)
      lvl::for_nodes_blocked(L.n, [&](int, int i, int j, int p) {
        lvl::cp_async<sizeof(c2<T>)>(&F(0)[p], fin + (long long)j * A.pf + i);
      });
    else
      lvl::for_nodes(w, w * w, [&](int q, int i, int j) {
        lvl::cp_async<sizeof(c2<T>)>(&F(0)[q], fin + (long long)j * A.pf + i);
      });
    lvl::cp_async_wait_all();
    __syncthreads();
    if (L.kind == TAIL_GS) lvl::gs_red<T>(U(0), F(0), K(0), L.n, (T)L.bA);
  }
  __syncthreads();

  // down: relax from a zero guess (a Gauss-Seidel level's red nodes were set by the phase that
  // produced its right-hand side), residual with the (B) operator, full weighting
  for (int l = 0; l < last; ++l) {
    const TailLevel& L = A.lv[l];
    if (L.kind == TAIL_GS) {
      lvl::gs_black<T>(U(l), F(l), K(l), L.n, (T)L.bA);
      lvl::residual<T>(R, U(l), F(l), lvl::Natural{L.n + 1}, K(l), L.n + 1, L.n, (T)L.bB);
    } else {
      lvl::kacz_sweeps<T>(U(l), F(l), D(l), V(l), L.n, L.nu, false);
      if (L.off_kres)
        lvl::residual_blocked<T>(R, U(l), F(l), reinterpret_cast<const T*>(smem + L.off_kres), L.n + 1, L.n, (T)L.bB);
      else
        lvl::residual_blocked<T>(R, U(l), F(l), reinterpret_cast<const T*>(L.kh), L.pk, L.n, (T)L.bB);
    }
    __syncthreads();
    const TailLevel& C = A.lv[l + 1];
    if (C.kind == TAIL_GS)
      lvl::restrict_fw_red<T>(F(l + 1), U(l + 1), K(l + 1), (T)C.bA, R, L.n);
    else
      with_layout(l + 1, [&](auto lc) { lvl::restrict_fw<T>(F(l + 1), lc, R, L.n); });
    __syncthreads();
  }

  // coarsest: u = A^-1 f
  if constexpr (CL) {
    coarse_cluster(CoarseShare(smem + A.off_ainv, mc), U(last), F(last));
  } else {
    const int m = (A.lv[last].n + 1) * (A.lv[last].n + 1);
    const c2<T>* ainvT = A.off_ainv ? reinterpret_cast<const c2<T>*>(smem + A.off_ainv)
                                    : reinterpret_cast<const c2<T>*>(A.ainvT);
    for (int r = threadIdx.x; r < m; r += TAIL_THREADS) U(last)[r] = lvl::coarse_row<T>(ainvT, F(last), m, r);
    __syncthreads();
  }

  // up: bilinear correction, relaxation in the reverse order (fused on Gauss-Seidel levels)
  for (int l = last - 1; l >= 0; --l) {
    const TailLevel& L = A.lv[l];
    if (L.kind == TAIL_GS) {
      with_layout(l + 1, [&](auto le) { lvl::gs_post_corrected<T>(U(l), F(l), K(l), L.n, (T)L.bA, U(l + 1), le); });
    } else {
      with_layout(l + 1, [&](auto le) { lvl::prolong_add<T>(U(l), lvl::blocked(L.n), U(l + 1), le, L.n); });
      __syncthreads();
      lvl::kacz_sweeps<T>(U(l), F(l), D(l), V(l), L.n, L.nu, true);
    }
  }

  const int w = A.lv[0].n + 1;
  if (A.lv[0].kind == TAIL_KACZ)
    lvl::for_nodes_blocked(A.lv[0].n, [&](int, int i, int j, int p) { uout[(long long)j * A.po + i] = U(0)[p]; });
  else
    lvl::for_nodes(w, w * w, [&](int q, int i, int j) { uout[(long long)j * A.po + i] = U(0)[q]; });
}

// The FP32 tail is held to 56 registers a thread, so that its 1024-thread block fits beside the
// deferred solution update (k_update_x, one 128-thread block per SM) that runs during the cycle.
__global__ void __maxnreg__(56) tail_kernel32(const TailArgs A, const int* __restrict__ stop, Inst bi) {
  tail_body<float, false>(A, stop, bi);
}
__global__ void __launch_bounds__(TAIL_THREADS) tail_kernel64(const TailArgs A, const int* __restrict__ stop, Inst bi) {
  tail_body<double, false>(A, stop, bi);
}
__global__ void __launch_bounds__(TAIL_THREADS) tail_cluster_kernel(const TailArgs A, const int* __restrict__ stop, Inst bi) {
  tail_body<double, true>(A, stop, bi);
}

}  // namespace

size_t tail_layout(bool fp32, TailArgs* A) {
  const size_t c = fp32 ? sizeof(float2) : sizeof(double2), r = fp32 ? sizeof(float) : sizeof(double);
  size_t off = 0, rmax = 0;
  auto take = [&](size_t bytes) {
    size_t o = off;
    off += (bytes + 15) & ~(size_t)15;
    return (unsigned)o;
  };
  for (int l = 0; l < A->count; ++l) {
    TailLevel& L = A->lv[l];
    const size_t Nn = (size_t)(L.n + 1) * (L.n + 1);
    const size_t N = L.kind == TAIL_KACZ ? (size_t)lvl::blocked_cells(L.n) : Nn;  // cells of u, f~, d, 1/|a|^2
    L.off_u = take(N * c);
    L.off_f = take(N * c);
    L.off_k = L.off_d = L.off_inv = 0;
    if (L.kind == TAIL_GS) L.off_k = take(N * r);
    if (L.kind == TAIL_KACZ) {
      L.off_d = take(N * c);
      L.off_inv = take(N * r);
    }
    if (L.kind != TAIL_COARSE) rmax = std::max(rmax, Nn);
  }
  for (int l = 0; l + 1 < A->count; ++l) {
    TailLevel& L = A->lv[l];
    const TailLevel& C = A->lv[l + 1];
    L.off_kres = 0;
    // the next level's u and f cells are contiguous; a Kaczmarz next level needs its zeroed u
    const size_t need = (size_t)(L.n + 1) * (L.n + 1) * r;
    const size_t nc = C.kind == TAIL_KACZ ? (size_t)lvl::blocked_cells(C.n) : (size_t)(C.n + 1) * (C.n + 1);
    if (L.kind == TAIL_KACZ && C.kind != TAIL_KACZ && need <= (size_t)(C.off_f - C.off_u) + nc * c) L.off_kres = C.off_u;
  }
  A->lv[A->count - 1].off_kres = 0;
  A->off_r = take(rmax * c);
  const size_t m = (size_t)(A->lv[A->count - 1].n + 1) * (A->lv[A->count - 1].n + 1);
  A->off_ainv = 0;
  if (off + m * m * c <= (size_t)TAIL_MAX_SMEM) A->off_ainv = take(m * m * c);
  return off;
}

namespace {

template <class K>
cudaError_t tail_opt_in(K kernel) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TAIL_MAX_SMEM);
}
cudaError_t cluster_opt_in() {
  static OncePerDevice ready;
  return ready([] { return tail_opt_in(tail_cluster_kernel); });
}
cudaLaunchConfig_t cluster_config(int count, size_t smem, cudaLaunchAttribute (&attr)[2], cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(TAIL_CLUSTER, 1, count);
  cfg.blockDim = dim3(TAIL_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = TAIL_CLUSTER;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cfg;
}

}  // namespace

int tail_max_clusters(const TailArgs& A, size_t smem) {
  const int m = (A.lv[A.count - 1].n + 1) * (A.lv[A.count - 1].n + 1);
  if (!A.off_ainv || m < 25 || !coarse_share_fits(m) || cluster_opt_in() != cudaSuccess) return 0;
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = cluster_config(1, smem, attr, nullptr);
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, tail_cluster_kernel, &cfg) != cudaSuccess) n = 0;
  cudaGetLastError();  // a refused shape leaves no sticky error
  return n;
}

cudaError_t launch_tail(bool fp32, const TailArgs& A, size_t smem, int clusters, const int* stop, cudaStream_t s,
                        const Inst& bi) {
  if (A.count < 2 || A.count > TAIL_MAX_LEVELS || smem > (size_t)TAIL_MAX_SMEM) return cudaErrorInvalidValue;
  static OncePerDevice ready[2];
  cudaError_t e;
  // A cluster per instance while the device holds them all at once (a block of the tail takes an SM, and a
  // cluster's eight lie in one GPC: 15 on 152 SMs) and there is something to share: tails of n_l = 8, 4 (m = 25)
  // 23.2 us in one block, 19.1 with helpers, 10, 5 (m = 36) 25.2 and 20.1, 14, 7 (m = 64) 31.4 and 21.9. A
  // second wave of clusters loses: whole solves (n = 32, six iterations) with and without them 1.69 and 1.72 ms
  // for 15 right-hand sides, 2.20 and 1.79 ms for 16.
  if (!fp32 && bi.count <= clusters) {
    if ((e = cluster_opt_in())) return e;
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = cluster_config(bi.count, smem, attr, s);
    return cudaLaunchKernelEx(&cfg, tail_cluster_kernel, A, stop, bi);
  }
  if ((e = ready[fp32]([&] { return fp32 ? tail_opt_in(tail_kernel32) : tail_opt_in(tail_kernel64); }))) return e;
  dim3 grid(1, 1, bi.count);
  if (fp32)
    pdl_launch(tail_kernel32, grid, TAIL_THREADS, smem, s, A, stop, bi);
  else
    pdl_launch(tail_kernel64, grid, TAIL_THREADS, smem, s, A, stop, bi);
  return cudaGetLastError();
}

}  // namespace hz
