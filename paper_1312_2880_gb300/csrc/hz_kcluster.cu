// A whole FP64 Kaczmarz level in a thread-block cluster (Sec. 4-5: Gauss-Seidel on the normal
// equations): its rows split into bands over up to 16 blocks, each band in its block's shared
// memory with one ghost row on either side, one cluster barrier per colour.
//
// What bounds it: 20 dependent phases per launch, each at least the FP64 instructions of one row action
// (30, at 77 cycles of a sub-partition each) and a cluster barrier. A thread keeps one block of five
// consecutive nodes of a band row for the launch, so a phase finds its node with a few integer
// operations; all reads are local (an action that changes a row which another block holds, its own
// or as a ghost, stores the value there too, and the stores complete in the barrier); and where
// the band has few rows, two lanes take one action, one per component (SPLIT 2): half the FP64
// instructions on the critical path for the same bits. Rows of one colour have disjoint supports,
// so no value is written twice in a phase. Per launch, against reading neighbour rows through
// distributed shared memory and finding every node anew: n_l = 32 (two lanes) 48 -> 30 us, n_l = 60
// (two lanes) 47 -> 32, n_l = 64 48 -> 45, n_l = 128 (two warps of actions per sub-partition: bound by
// the FP64 pipe) 84 -> 82.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <map>
#include <mutex>

#include "hz_common.cuh"
#include "hz_internal.h"
#include "hz_level.cuh"

namespace hz {

namespace {

namespace cgx = cooperative_groups;

// The band of a block: rows r0 .. r1 - 1 (row j at local row j - r0 + 1 of su, the ghosts at 0 and
// r1 - r0 + 1; at j - r0 of the other arrays). Every band but the last has `rows` >= 2 rows.
struct Band {
  double2 *su, *sf, *sd;  // u, f~, diagonal (after the sweeps: the residual)
  double* sinv;           // 1 / |a_p|^2
  int n, w, rows, r0, r1, rank;
  __device__ Band(unsigned char* smem, int n_, int rows_, int rank_) : n(n_), w(n_ + 1), rows(rows_), rank(rank_) {
    r0 = min(rank * rows, w);
    r1 = min(r0 + rows, w);
    su = reinterpret_cast<double2*>(smem);
    sf = su + (rows + 2) * w;
    sd = sf + rows * w;
    sinv = reinterpret_cast<double*>(sd + rows * w);
  }
  // The other copy of grid row j that this band's actions must keep: the owner's of a ghost row, or a
  // neighbour's ghost of the band's first or last row (null: none).
  __device__ double2* mirror(cgx::cluster_group& cl, int j) const {
    if (j == r0 - 1) return cl.map_shared_rank(su, rank - 1) + rows * w;
    if (j == r1) return cl.map_shared_rank(su, rank + 1) + w;
    if (j == r0 && rank > 0) return cl.map_shared_rank(su, rank - 1) + (rows + 1) * w;
    if (j == r1 - 1 && r1 < w) return cl.map_shared_rank(su, rank + 1);
    return nullptr;
  }
};
size_t band_smem(int n, int rows) { return (size_t)(n + 1) * ((rows + 2) * 16 + rows * 40); }

__device__ __forceinline__ void put(double2* row, double2* copy, int i, double2 v) {
  row[i] = v;
  if (copy) copy[i] = v;
}
__device__ __forceinline__ void put(double2* row, double2* copy, int i, int comp, double v) {
  reinterpret_cast<double*>(row + i)[comp] = v;
  if (copy) reinterpret_cast<double*>(copy + i)[comp] = v;
}

// nu sweeps over the colours 0..4 (4..0 when post), a cluster barrier after each colour. The operations
// of lvl::act_update, so the bits are those of every Kaczmarz form.
template <int SPLIT>
__device__ __forceinline__ void band_sweeps(cgx::cluster_group& cl, const Band& B, int nu, bool post) {
  const int M = (B.w + 4) / 5, n = B.n;
  const int s = threadIdx.x / SPLIT, comp = threadIdx.x % SPLIT;
  const int jl = s / M, i0 = 5 * (s - jl * M), j = B.r0 + jl;
  const bool own = jl < B.r1 - B.r0;
  const int pR = own ? n - i0 : -1, pL = i0 == 0 ? 0 : -1;  // positions of the last and first grid columns
  const int jS = j > 0 ? j - 1 : 1, jN = j < n ? j + 1 : n - 1;
  const bool my = jS == jN;
  double2 *rc = nullptr, *rs = nullptr, *rn = nullptr, *cc = nullptr, *cs = nullptr, *cn = nullptr;
  const double2 *f = nullptr, *d = nullptr;
  const double* iv = nullptr;
  if (own) {
    rc = B.su + (jl + 1) * B.w + i0;
    rs = B.su + (jS - B.r0 + 1) * B.w + i0;
    rn = B.su + (jN - B.r0 + 1) * B.w + i0;
    if ((cc = B.mirror(cl, j))) cc += i0;
    if ((cs = B.mirror(cl, jS))) cs += i0;
    if ((cn = B.mirror(cl, jN))) cn += i0;
    f = B.sf + jl * B.w + i0;
    d = B.sd + jl * B.w + i0;
    iv = B.sinv + jl * B.w + i0;
  }
  int pos = (((post ? 4 : 0) - 2 * j) % 5 + 5) % 5;  // of the colour: i + 2 j = colour mod 5
#pragma unroll 1
  for (int k = 0; k < 5 * nu; ++k) {
    const bool on = pos <= pR;
    if (__any_sync(0xffffffffu, on)) {
      const int dW = pos == pL ? 1 : -1, dE = pos == pR ? -1 : 1;
      const bool mx = dW == dE;
      const double cx = mx ? 2.0 : 1.0, cy = my ? 2.0 : 1.0;
      if constexpr (SPLIT == 1) {
        if (on) {
          double2 up = rc[pos], uw = rc[pos + dW], ue = rc[pos + dE], us = rs[pos], un = rn[pos];
          lvl::act_update<double>(up, uw, ue, us, un, f[pos], d[pos], iv[pos], mx, my);
          put(rc, cc, pos, up);
          put(rc, cc, pos + dW, uw);
          if (!mx) put(rc, cc, pos + dE, ue);
          put(rs, cs, pos, us);
          if (!my) put(rn, cn, pos, un);
        }
      } else {
        double own_u = 0, delta = 0, uw = 0, ue = 0, us = 0, un = 0;
        double2 dd = make_double2(0, 0);
        if (on) {
          const double2 uc = rc[pos];
          own_u = comp ? uc.y : uc.x;
          const double oth = comp ? uc.x : uc.y;
          uw = reinterpret_cast<const double*>(rc + pos + dW)[comp];
          ue = reinterpret_cast<const double*>(rc + pos + dE)[comp];
          us = reinterpret_cast<const double*>(rs + pos)[comp];
          un = reinterpret_cast<const double*>(rn + pos)[comp];
          dd = d[pos];
          const double nb = xr::add(xr::add(uw, ue), xr::add(us, un));
          const double t = xr::mul(dd.y, oth);
          const double du = xr::fma(dd.x, own_u, comp ? t : -t);
          delta = xr::mul(xr::sub(reinterpret_cast<const double*>(f + pos)[comp], xr::add(du, nb)), iv[pos]);
        }
        const double other = __shfl_xor_sync(0xffffffffu, delta, 1);
        if (on) {
          const double v = xr::mul(dd.y, other);
          put(rc, cc, pos, comp, xr::add(own_u, xr::fma(dd.x, delta, comp ? -v : v)));
          put(rc, cc, pos + dW, comp, xr::fma(delta, cx, uw));
          if (!mx) put(rc, cc, pos + dE, comp, xr::add(ue, delta));
          put(rs, cs, pos, comp, xr::fma(delta, cy, us));
          if (!my) put(rn, cn, pos, comp, xr::add(un, delta));
        }
      }
    }
    pos = post ? (pos == 0 ? 4 : pos - 1) : (pos == 4 ? 0 : pos + 1);
    cl.sync();
  }
}

__device__ __forceinline__ void band_consts(const Band& B, int q, int i, int j, const double* __restrict__ kh, int pk,
                                            double bA, const Inst& bi) {
  B.sd[q] = xr::diag<double>(kh[(long long)j * pk + i], lvl::sides_at(i, j, B.n), bA);
  B.sinv[q] = bi.inv[(long long)j * bi.pi + i];
}

template <int SPLIT, int CT>
__global__ void __launch_bounds__(CT) cluster64_pre_kernel(double2* __restrict__ u, int pu, double2* __restrict__ fc,
                                                           int pc, const double2* __restrict__ f, int pf,
                                                           const double* __restrict__ kh, int pk, int n, double bA,
                                                           double bB, int nu, int rows, const int* __restrict__ stop,
                                                           Inst bi) {
  extern __shared__ __align__(16) unsigned char smem[];
  cgx::cluster_group cl = cgx::this_cluster();
  const Band B(smem, n, rows, (int)cl.block_rank());
  const int w = B.w, cells = (B.r1 - B.r0) * w;
  // zero guess and row constants do not depend on the preceding kernel
  for (int q = threadIdx.x; q < (rows + 2) * w; q += CT) B.su[q] = make_double2(0, 0);
  for (int q = threadIdx.x; q < cells; q += CT) band_consts(B, q, q % w, B.r0 + q / w, kh, pk, bA, bi);
  pdl_enter();
  if (stop && stop[blockIdx.z * bi.stop_stride]) return;  // the whole cluster (one instance) returns
  u += blockIdx.z * bi.su;
  fc += blockIdx.z * bi.sc;
  f += blockIdx.z * bi.sf;
  for (int q = threadIdx.x; q < cells; q += CT) B.sf[q] = f[(long long)(B.r0 + q / w) * pf + q % w];
  cl.sync();
  band_sweeps<SPLIT>(cl, B, nu, false);
  for (int q = threadIdx.x; q < cells; q += CT) {
    const int j = B.r0 + q / w, i = q % w;
    const double2* row = B.su + (j - B.r0 + 1) * w;
    u[(long long)j * pu + i] = row[i];
    const Nbr b = neighbours(i, j, n);
    const double2 nb = xr::nb4<double>(row[b.iw], row[b.ie], B.su[(b.js - B.r0 + 1) * w + i], B.su[(b.jn - B.r0 + 1) * w + i]);
    B.sd[q] = xr::resid<double>(B.sf[q], row[i], nb, xr::diag<double>(kh[(long long)j * pk + i], b.sides, bB));
  }
  cl.sync();
  // full weighting of the coarse rows whose centre row lies in this band (residual rows of the
  // neighbouring bands through distributed shared memory)
  const int wc = n / 2 + 1, J0 = (B.r0 + 1) / 2, J1 = min((B.r1 + 1) / 2, wc);  // 2J in [r0, r1)
  for (int q = threadIdx.x; q < (J1 - J0) * wc; q += CT) {
    const int J = J0 + q / wc, I = q % wc;
    double2 sum[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int j = reflect(2 * J + b - 1, n), owner = j / rows;
      const double2* r = cl.map_shared_rank(B.sd, owner) + (j - owner * rows) * w;
      sum[b] = xr::fw3<double>(r[reflect(2 * I - 1, n)], r[2 * I], r[reflect(2 * I + 1, n)]);
    }
    fc[(long long)J * pc + I] = xr::cscale<double>(xr::fw3<double>(sum[0], sum[1], sum[2]), 0.25);
  }
  cl.sync();  // no block leaves while others may still read its shared memory
}

template <int SPLIT, int CT>
__global__ void __launch_bounds__(CT) cluster64_post_kernel(double2* __restrict__ u, int pu,
                                                            const double2* __restrict__ ec, int pc,
                                                            const double2* __restrict__ f, int pf,
                                                            const double* __restrict__ kh, int pk, int n, double bA,
                                                            int nu, int rows, const int* __restrict__ stop, Inst bi) {
  extern __shared__ __align__(16) unsigned char smem[];
  cgx::cluster_group cl = cgx::this_cluster();
  const Band B(smem, n, rows, (int)cl.block_rank());
  const int w = B.w, cells = (B.r1 - B.r0) * w;
  for (int q = threadIdx.x; q < cells; q += CT) band_consts(B, q, q % w, B.r0 + q / w, kh, pk, bA, bi);
  pdl_enter();
  if (stop && stop[blockIdx.z * bi.stop_stride]) return;
  u += blockIdx.z * bi.su;
  ec += blockIdx.z * bi.sc;
  f += blockIdx.z * bi.sf;
  for (int q = threadIdx.x; q < cells; q += CT) B.sf[q] = f[(long long)(B.r0 + q / w) * pf + q % w];
  // u_pre + P e_c on the band and its ghost rows
  for (int q = threadIdx.x; q < (cells ? cells + 2 * w : 0); q += CT) {
    const int j = B.r0 - 1 + q / w, i = q % w;
    if (j < 0 || j > n) continue;
    const double2* e0 = ec + (long long)(j >> 1) * pc;
    B.su[q] = xr::cadd<double>(u[(long long)j * pu + i], xr::bilinear<double>(e0, e0 + pc, i >> 1, i & 1, j & 1));
  }
  cl.sync();
  band_sweeps<SPLIT>(cl, B, nu, true);
  for (int q = threadIdx.x; q < cells; q += CT) u[(long long)(B.r0 + q / w) * pu + q % w] = B.su[q + w];
  cl.sync();
}

// Cluster shape of a level: the most blocks (16, 8, 4 or 2; 16 is beyond the portable cluster size)
// whose bands fit CLUSTER_MAX_SMEM, have two rows and one thread (or pair) per block of five nodes,
// and that the device can co-schedule, found once per device and n. c = 0: no cluster form. threads: 256 a
// block, or 1024 where a band has more than 256 blocks of five nodes.
struct Shape {
  int c = 0, rows = 0, split = 1, threads = 256;
  size_t smem = 0;
};
constexpr int CLUSTER_MAX_SMEM = 220 * 1024;
// fn(pre kernel, post kernel) of a shape
template <class F>
auto with_kernels(const Shape& S, F&& fn) {
  if (S.split == 2) return fn(cluster64_pre_kernel<2, 256>, cluster64_post_kernel<2, 256>);
  if (S.threads == 256) return fn(cluster64_pre_kernel<1, 256>, cluster64_post_kernel<1, 256>);
  return fn(cluster64_pre_kernel<1, 1024>, cluster64_post_kernel<1, 1024>);
}

cudaError_t cluster_attrs() {  // the caller holds the lock of cluster_shape
  cudaError_t e = cudaSuccess;
  auto set = [&](auto kernel) {
    if (!e) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, CLUSTER_MAX_SMEM);
    if (!e) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  };
  Shape S;
  for (int k = 0; k < 3; ++k) {
    S.split = k == 0 ? 2 : 1;
    S.threads = k == 2 ? 1024 : 256;
    with_kernels(S, [&](auto pre, auto post) {
      set(pre);
      set(post);
      return 0;
    });
  }
  return e;
}

cudaLaunchConfig_t config(const Shape& S, int batch, cudaLaunchAttribute (&attr)[2], int nattr, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(S.c, 1, batch);
  cfg.blockDim = dim3(S.threads);
  cfg.dynamicSmemBytes = S.smem;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = S.c;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = nattr;
  return cfg;
}

Shape cluster_shape(int n) {
  static std::mutex mu;
  static std::map<std::pair<int, int>, Shape> cache;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return Shape();
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find({dev, n});
  if (it != cache.end()) return it->second;
  Shape best;
  if (!cluster_attrs()) {
    for (int c = 16; c >= 2 && !best.c; c /= 2) {
      Shape S;
      S.c = c;
      S.rows = (n + 1 + c - 1) / c;
      S.smem = band_smem(n, S.rows);
      const int slots = S.rows * ((n + 5) / 5);
      if (S.rows < 2) continue;
      if (S.smem > (size_t)CLUSTER_MAX_SMEM || slots > 1024) break;
      if (slots > 256) S.threads = 1024;
      // FP64 instructions of the busiest sub-partition in a phase: 30 per warp of actions, or 15 per
      // warp of half actions
      auto warps = [](int lanes) { return ((lanes + 31) / 32 + 3) / 4; };
      if (2 * slots <= 256 && 15 * warps(2 * slots) < 30 * warps(slots)) S.split = 2;
      cudaLaunchAttribute attr[2];
      const cudaLaunchConfig_t cfg = config(S, 1, attr, 1, nullptr);
      int a1 = 0, a2 = 0;
      const bool ok = with_kernels(S, [&](auto pre, auto post) {
        return !cudaOccupancyMaxActiveClusters(&a1, pre, &cfg) && !cudaOccupancyMaxActiveClusters(&a2, post, &cfg);
      });
      if (ok && a1 > 0 && a2 > 0) best = S;
    }
    cudaGetLastError();  // an unsupported shape leaves no sticky error
  }
  cache[{dev, n}] = best;
  return best;
}

}  // namespace

bool kacz_cluster64_fits(int n) { return cluster_shape(n).c > 0; }

cudaError_t launch_kacz_cluster64_pre(double2* u, int pu, double2* fc, int pc, const double2* f, int pf,
                                      const double* kh, int pk, int n, double bA, double bB, int nu, const int* stop,
                                      cudaStream_t s, const Inst& bi) {
  const Shape S = cluster_shape(n);
  if (!S.c || !bi.inv) return cudaErrorInvalidValue;
  cudaLaunchAttribute attr[2];
  const cudaLaunchConfig_t cfg = config(S, bi.count, attr, 2, s);
  return with_kernels(S, [&](auto pre, auto) {
    return cudaLaunchKernelEx(&cfg, pre, u, pu, fc, pc, f, pf, kh, pk, n, bA, bB, nu, S.rows, stop, bi);
  });
}

cudaError_t launch_kacz_cluster64_post(double2* u, int pu, const double2* ec, int pc, const double2* f, int pf,
                                       const double* kh, int pk, int n, double bA, int nu, const int* stop,
                                       cudaStream_t s, const Inst& bi) {
  const Shape S = cluster_shape(n);
  if (!S.c || !bi.inv) return cudaErrorInvalidValue;
  cudaLaunchAttribute attr[2];
  const cudaLaunchConfig_t cfg = config(S, bi.count, attr, 2, s);
  return with_kernels(S, [&](auto, auto post) {
    return cudaLaunchKernelEx(&cfg, post, u, pu, ec, pc, f, pf, kh, pk, n, bA, nu, S.rows, stop, bi);
  });
}

}  // namespace hz
