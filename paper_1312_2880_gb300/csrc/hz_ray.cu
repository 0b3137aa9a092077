// Ray correction (Sec. 6; Table 7) on the device, complex FP64 throughout.
//
// The near-kernel error is sought as sum_j exp(i k d_j . x) a_j(x) over the eight directions
// d_j = (cos j pi/4, sin j pi/4), with ray functions a_j bilinear on a ray grid of spacing
// H = m h (every m-th node of the fine vertex grid). With P the fine-grid matrix of these basis
// functions (column 8 C + j: the hat of ray node C times plane wave j), the correction is the
// Galerkin projection x += P (P^H A P)^{-1} P^H r of the residual r.
//
// The ray operator couples ray nodes at most one apart, so ordered by rows of ray nodes it is
// block tridiagonal: block row J holds the 8 (nc + 1) unknowns of ray row J (node-major, eight
// directions inner), with blocks L_J (row J - 1), D_J and U_J (row J + 1). It is factored once by
// a two-sided block LU that eliminates from both ends towards the middle row Mid = Nr / 2:
//   J < Mid: S_0 = D_0,      S_J = D_J - L_J S_{J-1}^{-1} U_{J-1}   (from the row below)
//   J > Mid: S_{Nr-1} = D_{Nr-1}, S_J = D_J - U_J S_{J+1}^{-1} L_{J+1}   (from the row above)
//   S_Mid = D_Mid - L_Mid S_{Mid-1}^{-1} U_{Mid-1} - U_Mid S_{Mid+1}^{-1} L_{Mid+1},
// each S_J inverted by Gauss-Jordan elimination with row pivoting. The solve keeps S_J^{-1}, the
// products that carry a row towards the middle (G: L_J S_{J-1}^{-1} in slot J, U_J S_{J+1}^{-1} in
// slot J + 1) and back (W: S_J^{-1} U_J below the middle, S_J^{-1} L_J above), and runs one step of
// iterative refinement on the block residual. The two chains are independent, so every step of the
// factorisation and of the substitutions works on two block rows at once: half the dependent
// steps of a one-sided elimination, which are what bounds the solve beside the FP64 pipe.
//
// Every kernel here is launched with programmatic stream serialization and starts with pdl_enter()
// (hz_common.cuh): it waits for its predecessor before reading anything.
#include "hz_common.cuh"
#include "hz_internal.h"

namespace hz {
namespace {

constexpr double RAY_S = 0x1.6a09e667f3bcdp-1;  // sqrt(1/2), correctly rounded

__device__ __forceinline__ void ray_dir(int j, double& dx, double& dy) {
  const double a[8] = {1.0, RAY_S, 0.0, -RAY_S, -1.0, -RAY_S, 0.0, RAY_S};
  const double b[8] = {0.0, RAY_S, 1.0, RAY_S, 0.0, -RAY_S, -1.0, -RAY_S};
  dx = a[j];
  dy = b[j];
}

__device__ __forceinline__ double2 zadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// conj(a) * b
__device__ __forceinline__ double2 zmulc(double2 a, double2 b) {
  return make_double2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ double2 zscale(double2 a, double s) { return make_double2(a.x * s, a.y * s); }

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Weight of the bilinear hat of a ray node at fine distance (di, dj); exact for m a power of two.
__device__ __forceinline__ double hat_w(int di, int dj, double rm) {
  return (1.0 - (double)abs(di) * rm) * (1.0 - (double)abs(dj) * rm);
}

// ph[j N + p] = exp(i k (d_x x + d_y y)) at node p = (i, jj), x = i h, y = jj h.
__global__ void ray_phase_kernel(double2* ph, int n, double k) {
  pdl_enter();
  const long long N = (long long)(n + 1) * (n + 1);
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= 8 * N) return;
  const int j = (int)(t / N);
  const long long p = t - j * N;
  const int i = (int)(p % (n + 1)), jj = (int)(p / (n + 1));
  const double h = 1.0 / n;
  double dx, dy;
  ray_dir(j, dx, dy);
  const double arg = __dmul_rn(k, __dadd_rn(__dmul_rn(dx, __dmul_rn((double)i, h)), __dmul_rn(dy, __dmul_rn((double)jj, h))));
  double s, c;
  sincos(arg, &s, &c);
  ph[t] = make_double2(c, s);
}

// One warp per (column ray node C', direction j', neighbouring ray node C): the eight entries
// (8 C + j, 8 C' + j') of P^H A P, j = 0..7. The sum runs over the fine nodes p under the hat of
// C where A applied to the column (hat of C' times plane wave j') can be non-zero; A's rows are
// the scaled 5-point rows with mirrored boundary neighbours (hz_common.cuh), times 1/h^2.
__global__ void __launch_bounds__(256) ray_assemble_kernel(double2* Lb, double2* Db, double2* Ub, const double2* ph,
                                                           const double* kh, int n, int m) {
  pdl_enter();
  const int nc = n / m, Nr = nc + 1, Bs = 8 * Nr;
  const long long Nc = (long long)Nr * Nr;
  const long long wid = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (wid >= Nc * 72) return;
  const int Cp = (int)(wid / 72), rem = (int)(wid % 72);
  const int jp = rem / 9, q9 = rem % 9;
  const int Ip = Cp % Nr, Jp = Cp / Nr;
  const int I = Ip + q9 % 3 - 1, J = Jp + q9 / 3 - 1;
  if (I < 0 || I > nc || J < 0 || J > nc) return;
  const int i0 = max(max(0, I * m - m + 1), Ip * m - m), i1 = min(min(n, I * m + m - 1), Ip * m + m);
  const int j0 = max(max(0, J * m - m + 1), Jp * m - m), j1 = min(min(n, J * m + m - 1), Jp * m + m);
  const long long N = (long long)(n + 1) * (n + 1);
  const double rm = 1.0 / m;
  const double2* phc = ph + jp * N;
  double ar[8], ai[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) ar[j] = ai[j] = 0.0;
  if (i0 <= i1 && j0 <= j1) {
    const int wi = i1 - i0 + 1, cnt = wi * (j1 - j0 + 1);
    auto col = [&](int a, int c) -> double2 {  // hat of C' times plane wave j' at node (a, c)
      const int di = a - Ip * m, dj = c - Jp * m;
      if (abs(di) >= m || abs(dj) >= m) return make_double2(0.0, 0.0);
      return zscale(phc[(long long)c * (n + 1) + a], hat_w(di, dj, rm));
    };
    for (int q = lane; q < cnt; q += 32) {
      const int i = i0 + q % wi, jj = j0 + q / wi;
      const Nbr b = neighbours(i, jj, n);
      const long long p = (long long)jj * (n + 1) + i;
      const double k1 = kh[p];
      const double2 d = make_double2(k1 * k1 - 4.0, 2.0 * b.sides * k1);
      const double2 s = zadd(zadd(col(b.iw, jj), col(b.ie, jj)), zadd(col(i, b.js), col(i, b.jn)));
      const double2 av = zscale(zadd(s, zmul(d, col(i, jj))), hat_w(i - I * m, jj - J * m, rm));
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const double2 e = zmulc(ph[j * N + p], av);
        ar[j] += e.x;
        ai[j] += e.y;
      }
    }
  }
  const double n2 = (double)n * (double)n;
  double2* blk = Jp == J - 1 ? Lb : (Jp == J ? Db : Ub);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const double re = warp_sum(ar[j]), im = warp_sum(ai[j]);
    if (lane == j) blk[((long long)J * Bs + (8 * I + j)) * Bs + (8 * Ip + jp)] = make_double2(re * n2, im * n2);
  }
}

// g[8 C + j] = sum over the hat of ray node C of hat(p) conj(ph_j[p]) r[p]   (g = P^H r). One warp
// per ray node (eight per block of 256 threads).
__global__ void __launch_bounds__(256) ray_restrict_kernel(double2* g, const double2* r, const double2* ph, int n,
                                                           int m) {
  pdl_enter();
  const int nc = n / m, Nr = nc + 1;
  const long long C = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (C >= (long long)Nr * Nr) return;
  const int I = (int)(C % Nr), J = (int)(C / Nr);
  const int i0 = max(0, I * m - m + 1), i1 = min(n, I * m + m - 1);
  const int j0 = max(0, J * m - m + 1), j1 = min(n, J * m + m - 1);
  const int wi = i1 - i0 + 1, cnt = wi * (j1 - j0 + 1);
  const long long N = (long long)(n + 1) * (n + 1);
  const double rm = 1.0 / m;
  double ar[8], ai[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) ar[j] = ai[j] = 0.0;
  for (int q = lane; q < cnt; q += 32) {
    const int i = i0 + q % wi, jj = j0 + q / wi;
    const long long p = (long long)jj * (n + 1) + i;
    const double2 wr = zscale(r[p], hat_w(i - I * m, jj - J * m, rm));
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const double2 e = ph[j * N + p];
      ar[j] = fma(e.x, wr.x, fma(e.y, wr.y, ar[j]));
      ai[j] = fma(e.x, wr.y, fma(-e.y, wr.x, ai[j]));
    }
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const double re = warp_sum(ar[j]), im = warp_sum(ai[j]);
    if (lane == j) g[8 * C + j] = make_double2(re, im);
  }
}

// x[p] += sum_j ph_j[p] * (bilinear interpolation of the ray function z_j at p)   (x += P z)
__global__ void ray_prolong_add_kernel(double2* x, const double2* z, const double2* ph, int n, int m) {
  pdl_enter();
  const long long N = (long long)(n + 1) * (n + 1);
  const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (p >= N) return;
  const int i = (int)(p % (n + 1)), jj = (int)(p / (n + 1));
  const int Nr = n / m + 1;
  const int I = i / m, ti = i - I * m, J = jj / m, tj = jj - J * m;
  const double rm = 1.0 / m;
  const double wx1 = ti * rm, wx0 = 1.0 - wx1, wy1 = tj * rm, wy0 = 1.0 - wy1;
  const double2* z00 = z + 8LL * ((long long)J * Nr + I);
  double2 tot = make_double2(0.0, 0.0);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    double2 e = zscale(z00[j], wx0 * wy0);
    if (ti) e = zadd(e, zscale(z00[8 + j], wx1 * wy0));
    if (tj) {
      e = zadd(e, zscale(z00[8LL * Nr + j], wx0 * wy1));
      if (ti) e = zadd(e, zscale(z00[8LL * Nr + 8 + j], wx1 * wy1));
    }
    tot = zadd(tot, zmul(ph[j * N + p], e));
  }
  x[p] = zadd(x[p], tot);
}

// Step k of the in-place Gauss-Jordan inversion with row pivoting of the Bs x Bs matrix S: the row
// of largest |S[i][k]| (i >= k; the first on ties) is swapped into row k and recorded in perm[k];
// column k is saved in fcol; row k is scaled by 1 / pivot with the pivot's own entry replaced by
// 1 / pivot. A zero or non-finite pivot column sets *status = 1 (the inverse is then meaningless).
// Block b of the launch works on the b-th of up to two matrices (with its own fcol and perm).
struct Pair {
  double2* p[2];
};
__global__ void __launch_bounds__(1024) ray_gj_pivot_kernel(Pair m, int Bs, int k, double2* fcol, int* perm,
                                                            int* status) {
  pdl_enter();
  double2* S = blockIdx.x ? m.p[1] : m.p[0];
  fcol += blockIdx.x * Bs;
  perm += blockIdx.x * Bs;
  __shared__ double sv[32];
  __shared__ int si[32];
  __shared__ int piv;
  double best = -1.0;
  int bi = Bs;
  for (int i = k + threadIdx.x; i < Bs; i += blockDim.x) {
    const double2 a = S[(long long)i * Bs + k];
    const double v = a.x * a.x + a.y * a.y;
    if (v > best) {
      best = v;
      bi = i;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double ov = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ov > best || (ov == best && oi < bi)) {
      best = ov;
      bi = oi;
    }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    sv[warp] = best;
    si[warp] = bi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double b = -1.0;
    int ib = Bs;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      if (sv[w] > b || (sv[w] == b && si[w] < ib)) {
        b = sv[w];
        ib = si[w];
      }
    }
    const bool ok = b > 0.0 && isfinite(b) && ib < Bs;
    if (!ok) *status = 1;
    piv = ok ? ib : k;
    perm[k] = piv;
  }
  __syncthreads();
  const int p = piv;
  if (p != k) {
    for (int c = threadIdx.x; c < Bs; c += blockDim.x) {
      const double2 t = S[(long long)k * Bs + c];
      S[(long long)k * Bs + c] = S[(long long)p * Bs + c];
      S[(long long)p * Bs + c] = t;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < Bs; i += blockDim.x) fcol[i] = S[(long long)i * Bs + k];
  __syncthreads();
  const double2 pv = fcol[k];
  const double d = pv.x * pv.x + pv.y * pv.y;
  const double2 inv = make_double2(pv.x / d, -pv.y / d);
  for (int c = threadIdx.x; c < Bs; c += blockDim.x) {
    const long long q = (long long)k * Bs + c;
    S[q] = c == k ? inv : zmul(S[q], inv);
  }
}

// Rows i != k: S[i][c] = (c == k ? 0 : S[i][c]) - fcol[i] S[k][c]  (row k is only read).
__global__ void ray_gj_elim_kernel(Pair m, int Bs, int k, const double2* fcol) {
  pdl_enter();
  double2* S = blockIdx.z ? m.p[1] : m.p[0];
  fcol += blockIdx.z * Bs;
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = blockIdx.y;
  if (c >= Bs || i == k) return;
  const double2 f = fcol[i];
  if (f.x == 0.0 && f.y == 0.0) return;  // the row already holds its final values (S[i][k] is 0)
  const long long q = (long long)i * Bs + c;
  const double2 a = c == k ? make_double2(0.0, 0.0) : S[q];
  const double2 fr = zmul(f, S[(long long)k * Bs + c]);
  S[q] = make_double2(a.x - fr.x, a.y - fr.y);
}

// Undo the row interchanges on the inverse: columns k and perm[k] swapped, k = Bs-1 .. 0.
__global__ void ray_gj_unpermute_kernel(Pair m, int Bs, const int* perm) {
  pdl_enter();
  double2* S = blockIdx.y ? m.p[1] : m.p[0];
  perm += blockIdx.y * Bs;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Bs) return;
  double2* row = S + (long long)i * Bs;
  for (int k = Bs - 1; k >= 0; --k) {
    const int p = perm[k];
    if (p != k) {
      const double2 t = row[k];
      row[k] = row[p];
      row[p] = t;
    }
  }
}

// C = A B (acc 0) or C = C - A B (acc 1) for Bs x Bs row-major blocks; C aliases neither A nor B.
// A 32 x 32 tile of C per block of 256 threads, each thread 2 x 2 entries, k in steps of 16.
// The z-th of up to two products.
struct GemmJob {
  double2* C;
  const double2 *A, *B;
};
struct GemmJobs {
  GemmJob j[2];
};
__global__ void __launch_bounds__(256) ray_gemm_kernel(GemmJobs jobs, int Bs, int acc) {
  pdl_enter();
  const GemmJob job = blockIdx.z ? jobs.j[1] : jobs.j[0];
  double2* C = job.C;
  const double2 *A = job.A, *B = job.B;
  __shared__ double2 As[32][17];
  __shared__ double2 Bsh[16][33];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int row0 = blockIdx.y * 32, col0 = blockIdx.x * 32;
  double2 c[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) c[a][b] = make_double2(0.0, 0.0);
  for (int k0 = 0; k0 < Bs; k0 += 16) {
    for (int e = threadIdx.x; e < 512; e += 256) {
      const int r = e >> 4, kk = e & 15, gr = row0 + r, gk = k0 + kk;
      As[r][kk] = (gr < Bs && gk < Bs) ? A[(long long)gr * Bs + gk] : make_double2(0.0, 0.0);
      const int kb = e >> 5, cc = e & 31, gk2 = k0 + kb, gc = col0 + cc;
      Bsh[kb][cc] = (gk2 < Bs && gc < Bs) ? B[(long long)gk2 * Bs + gc] : make_double2(0.0, 0.0);
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < 16; ++kk) {
      const double2 a0 = As[ty][kk], a1 = As[ty + 16][kk], b0 = Bsh[kk][tx], b1 = Bsh[kk][tx + 16];
      c[0][0] = zadd(c[0][0], zmul(a0, b0));
      c[0][1] = zadd(c[0][1], zmul(a0, b1));
      c[1][0] = zadd(c[1][0], zmul(a1, b0));
      c[1][1] = zadd(c[1][1], zmul(a1, b1));
    }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int r = row0 + ty + 16 * a, cc = col0 + tx + 16 * b;
      if (r < Bs && cc < Bs) {
        const long long q = (long long)r * Bs + cc;
        C[q] = acc ? make_double2(C[q].x - c[a][b].x, C[q].y - c[a][b].y) : c[a][b];
      }
    }
}

// out = base + sgn (M x + M2 x2) for job blockIdx.y (base and M2 may be null; base may equal out), or,
// with BATCH, job 0 advanced to block row blockIdx.y. One warp per row.
//
// Bound by the FP64 pipe (four FMAs a complex element, 77 cycles a warp instruction on a sub-partition:
// 4.1 us for the two 520 x 520 products of a step at n = 512) and by the latency of the chain. A row's
// elements are factors, fixed since set-up, so a warp loads its first 32 GEMV_PRE of them before it
// waits for the preceding launch, and the launch after it may start as soon as every block has begun:
// the factors' trip from HBM overlaps the step before. The real and imaginary parts are reduced
// together in the two halves of the warp (five additions where two shuffle trees took ten: at 77
// cycles each, four warps per row with a tree apiece spent a third of a step's FP64 time there, and
// 128 threads on 520 columns left one warp twice the work of the others). A solve at n = 512 took
// 2.23 ms with the one-sided elimination and four warps per row, 1.86 ms now; at n = 256 0.71 and
// 0.50 ms; the factorisation 1.21 s and 0.77 s. GEMV_PRE covers rows of 544 elements (n = 512 with ray cells of
// 8 h has 520) at 110 registers a thread; longer rows fetch the rest after the wait and gain less (n = 1024,
// 1032 elements, 10.7 and 10.4 ms).
constexpr int GEMV_WARPS = 4, GEMV_PRE = 17;
struct GemvJob {
  double2* out;
  const double2 *base, *M, *x, *M2, *x2;
};
struct GemvJobs {
  GemvJob j[2];
};
template <bool BATCH>
__global__ void __launch_bounds__(32 * GEMV_WARPS) ray_gemv_kernel(GemvJobs jobs, int Bs, double sgn) {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const GemvJob job = !BATCH && blockIdx.y ? jobs.j[1] : jobs.j[0];
  const long long b = BATCH ? blockIdx.y : 0;
  const int row = blockIdx.x * GEMV_WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const bool live = row < Bs;
  const double2* Mr = job.M + b * Bs * (long long)Bs + (long long)(live ? row : 0) * Bs;
  double2 a[GEMV_PRE];
#pragma unroll
  for (int q = 0; q < GEMV_PRE; ++q) {
    const int c = lane + 32 * q;
    a[q] = c < Bs ? Mr[c] : make_double2(0.0, 0.0);
  }
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  if (!live) return;
  double re = 0.0, im = 0.0;
  auto acc = [&](double2 m, double2 v) {
    re = fma(m.x, v.x, re);
    re = fma(-m.y, v.y, re);
    im = fma(m.x, v.y, im);
    im = fma(m.y, v.x, im);
  };
  const double2* x = job.x + b * Bs;
#pragma unroll
  for (int q = 0; q < GEMV_PRE; ++q) {
    const int c = lane + 32 * q;
    if (32 * q < Bs) acc(a[q], c < Bs ? __ldcg(x + c) : make_double2(0.0, 0.0));
  }
  for (int c = lane + 32 * GEMV_PRE; c < Bs; c += 32) acc(Mr[c], __ldcg(x + c));
  if (!BATCH && job.M2) {
    const double2* M2r = job.M2 + (long long)row * Bs;
    for (int c = lane; c < Bs; c += 32) acc(M2r[c], __ldcg(job.x2 + c));
  }
  // lanes 0 .. 15 reduce the real part, 16 .. 31 the imaginary part
  const bool hi = lane >= 16;
  double v = hi ? im : re;
  v += __shfl_xor_sync(0xffffffffu, hi ? re : im, 16);
#pragma unroll
  for (int o = 8; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((lane & 15) == 0) {
    const double* base = job.base ? reinterpret_cast<const double*>(job.base + b * Bs + row) + hi : nullptr;
    reinterpret_cast<double*>(job.out + b * Bs + row)[hi] = fma(sgn, v, base ? __ldcg(base) : 0.0);
  }
}

// e_J = g_J - (L_J z_{J-1} + D_J z_J + U_J z_{J+1}), one thread per row of the whole system. Row
// 8 I + j of block row J couples only ray nodes I - 1 .. I + 1 of the three ray rows, so only those
// 24 columns of each block are read (the others are zero by construction).
__global__ void __launch_bounds__(128) ray_block_residual_kernel(double2* e, const double2* g, const double2* z,
                                                                 const double2* Lb, const double2* Db,
                                                                 const double2* Ub, int Bs, int Nr) {
  pdl_enter();
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= (long long)Nr * Bs) return;
  const int J = (int)(t / Bs), row = (int)(t % Bs), I = row / 8;
  const int c0 = 8 * max(I - 1, 0), c1 = 8 * min(I + 2, Nr);
  const long long off = (long long)J * Bs * Bs + (long long)row * Bs;
  const double2* zJ = z + (long long)J * Bs;
  double re = 0.0, im = 0.0;
  for (int c = c0; c < c1; ++c) {
    double2 q = zmul(Db[off + c], zJ[c]);
    if (J > 0) q = zadd(q, zmul(Lb[off + c], zJ[c - Bs]));
    if (J < Nr - 1) q = zadd(q, zmul(Ub[off + c], zJ[c + Bs]));
    re += q.x;
    im += q.y;
  }
  e[t] = make_double2(g[t].x - re, g[t].y - im);
}

// dst = src on entries [0, cnt) and [last, last + cnt) (blockIdx.y).
__global__ void ray_copy_kernel(double2* dst, const double2* src, int cnt, int last) {
  pdl_enter();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < cnt) dst[blockIdx.y * last + i] = src[blockIdx.y * last + i];
}

constexpr int RED_BLOCKS = 512, RED_THREADS = 256;

// r = b - v and per-block partial sums of |r|^2 (v null: |b|^2 only, r untouched).
__global__ void __launch_bounds__(RED_THREADS) ray_residual_norm_kernel(double2* r, const double2* b, const double2* v,
                                                                        long long N, double* partials) {
  pdl_enter();
  double s = 0.0;
  for (long long p = blockIdx.x * (long long)RED_THREADS + threadIdx.x; p < N; p += (long long)RED_BLOCKS * RED_THREADS) {
    double2 t = b[p];
    if (v) {
      const double2 w = v[p];
      t = make_double2(t.x - w.x, t.y - w.y);
      r[p] = t;
    }
    s += t.x * t.x + t.y * t.y;
  }
  __shared__ double red[RED_THREADS / 32];
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < RED_THREADS / 32; ++w) t += red[w];
    partials[blockIdx.x] = t;
  }
}

__global__ void ray_sum_kernel(const double* partials, double* out) {
  pdl_enter();
  __shared__ double red[RED_BLOCKS];
  for (int i = threadIdx.x; i < RED_BLOCKS; i += blockDim.x) red[i] = partials[i];
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < RED_BLOCKS; ++i) t += red[i];
    *out = t;
  }
}

__global__ void ray_axpy_kernel(double2* x, const double2* z, long long N) {
  pdl_enter();
  const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (p < N) x[p] = zadd(x[p], z[p]);
}

inline unsigned blocks_for(long long work, int threads) { return (unsigned)((work + threads - 1) / threads); }

}  // namespace

// ---------------------------------------------------------------- launchers

cudaError_t launch_ray_phases(double2* ph, int n, double k, cudaStream_t s) {
  const long long work = 8LL * (n + 1) * (n + 1);
  return pdl_launch(ray_phase_kernel, dim3(blocks_for(work, 256)), dim3(256), 0, s, ph, n, k);
}

cudaError_t launch_ray_assemble(const RayBlocks& B, const double2* ph, const double* kh, cudaStream_t s) {
  const long long warps = 72LL * B.Nr * B.Nr;
  return pdl_launch(ray_assemble_kernel, dim3(blocks_for(warps * 32, 256)), dim3(256), 0, s, B.L, B.D, B.U, ph, kh,
                    B.n, B.m);
}

cudaError_t launch_ray_restrict(double2* g, const double2* r, const double2* ph, int n, int m, cudaStream_t s) {
  const long long Nr = n / m + 1;
  return pdl_launch(ray_restrict_kernel, dim3(blocks_for(32 * Nr * Nr, 256)), dim3(256), 0, s, g, r, ph, n, m);
}

cudaError_t launch_ray_prolong_add(double2* x, const double2* z, const double2* ph, int n, int m, cudaStream_t s) {
  return pdl_launch(ray_prolong_add_kernel, dim3(blocks_for((long long)(n + 1) * (n + 1), 256)), dim3(256), 0, s, x,
                    z, ph, n, m);
}

namespace {

cudaError_t gj_inverse(const Pair& S, int count, int Bs, double2* fcol, int* perm, int* status, cudaStream_t s) {
  const dim3 eg(blocks_for(Bs, 128), Bs, count);
  for (int k = 0; k < Bs; ++k) {
    cudaError_t e = pdl_launch(ray_gj_pivot_kernel, dim3(count), dim3(1024), 0, s, S, Bs, k, fcol, perm, status);
    if (e == cudaSuccess) e = pdl_launch(ray_gj_elim_kernel, eg, dim3(128), 0, s, S, Bs, k, (const double2*)fcol);
    if (e != cudaSuccess) return e;
  }
  return pdl_launch(ray_gj_unpermute_kernel, dim3(blocks_for(Bs, 128), count), dim3(128), 0, s, S, Bs, (const int*)perm);
}

cudaError_t gemm(const GemmJobs& jobs, int count, int Bs, int acc, cudaStream_t s) {
  const dim3 g(blocks_for(Bs, 32), blocks_for(Bs, 32), count);
  return pdl_launch(ray_gemm_kernel, g, dim3(256), 0, s, jobs, Bs, acc);
}

cudaError_t gemv(const GemvJobs& jobs, int count, int Bs, double sgn, cudaStream_t s) {
  return pdl_launch(ray_gemv_kernel<false>, dim3(blocks_for(Bs, GEMV_WARPS), count), dim3(32 * GEMV_WARPS), 0, s, jobs,
                    Bs, sgn);
}

// z = (block LU)^{-1} g; y is scratch of one vector. Both ends move to the middle row, every row is
// multiplied by its inverse, and the middle is carried back to both ends.
cudaError_t block_substitute(const RayBlocks& B, double2* z, const double2* g, double2* y, cudaStream_t s) {
  const int Bs = B.Bs, Nr = B.Nr, mid = Nr / 2, up = Nr - 1 - mid;  // `up` rows above the middle
  const long long bs2 = (long long)Bs * Bs;
  auto at = [&](auto* v, int J) { return v + (long long)J * Bs; };
  cudaError_t e = pdl_launch(ray_copy_kernel, dim3(blocks_for(Bs, 128), 2), dim3(128), 0, s, y, g, Bs, (Nr - 1) * Bs);
  for (int k = 1; k < mid && e == cudaSuccess; ++k) {
    const int J = k, T = Nr - 1 - k;  // y_J = g_J - G_J y_{J-1}, y_T = g_T - G_{T+1} y_{T+1}
    GemvJobs j = {{{at(y, J), at(g, J), B.G + J * bs2, at(y, J - 1), nullptr, nullptr},
                   {at(y, T), at(g, T), B.G + (T + 1) * bs2, at(y, T + 1), nullptr, nullptr}}};
    e = gemv(j, k < up ? 2 : 1, Bs, -1.0, s);
  }
  if (e == cudaSuccess) {
    GemvJobs j = {{{at(y, mid), at(g, mid), B.G + mid * bs2, at(y, mid - 1), up ? B.G + (mid + 1) * bs2 : nullptr,
                    up ? at(y, mid + 1) : nullptr}, {}}};
    e = gemv(j, 1, Bs, -1.0, s);
  }
  if (e == cudaSuccess) {
    GemvJobs j = {{{z, nullptr, B.Sinv, y, nullptr, nullptr}, {}}};
    e = pdl_launch(ray_gemv_kernel<true>, dim3(blocks_for(Bs, GEMV_WARPS), Nr), dim3(32 * GEMV_WARPS), 0, s, j, Bs, 1.0);
  }
  for (int k = 1; k <= mid && e == cudaSuccess; ++k) {
    const int J = mid - k, T = mid + k;  // z_J -= W_J z_{J+1}, z_T -= W_T z_{T-1}
    GemvJobs j = {{{at(z, J), at(z, J), B.W + J * bs2, at(z, J + 1), nullptr, nullptr},
                   {at(z, T), at(z, T), B.W + T * bs2, at(z, T - 1), nullptr, nullptr}}};
    e = gemv(j, k <= up ? 2 : 1, Bs, -1.0, s);
  }
  return e;
}

}  // namespace

cudaError_t ray_factor(const RayBlocks& B, cudaStream_t s) {
  const int Bs = B.Bs, Nr = B.Nr, mid = Nr / 2, up = Nr - 1 - mid;
  const long long bs2 = (long long)Bs * Bs;
  auto blk = [&](double2* a, int J) { return a + J * bs2; };
  // What row J's elimination adds towards the middle: below it W_J, then S_{J+1} -= L_{J+1} W_J and
  // G_{J+1}; above it W_J, then S_{J-1} -= U_{J-1} W_J and the product in slot J.
  auto w_of = [&](int J) {
    return J < mid ? GemmJob{blk(B.W, J), blk(B.Sinv, J), blk(B.U, J)} : GemmJob{blk(B.W, J), blk(B.Sinv, J), blk(B.L, J)};
  };
  auto s_of = [&](int J) {
    return J < mid ? GemmJob{blk(B.Sinv, J + 1), blk(B.L, J + 1), blk(B.W, J)}
                   : GemmJob{blk(B.Sinv, J - 1), blk(B.U, J - 1), blk(B.W, J)};
  };
  auto g_of = [&](int J) {
    return J < mid ? GemmJob{blk(B.G, J + 1), blk(B.L, J + 1), blk(B.Sinv, J)}
                   : GemmJob{blk(B.G, J), blk(B.U, J - 1), blk(B.Sinv, J)};
  };
  cudaError_t e = cudaMemcpyAsync(B.Sinv, B.D, sizeof(double2) * (size_t)(bs2 * Nr), cudaMemcpyDeviceToDevice, s);
  for (int k = 0; k < mid && e == cudaSuccess; ++k) {
    const int J = k, T = Nr - 1 - k, count = k < up ? 2 : 1;
    e = gj_inverse(Pair{{blk(B.Sinv, J), blk(B.Sinv, T)}}, count, Bs, B.fcol, B.perm, B.status, s);
    if (e == cudaSuccess) e = gemm(GemmJobs{{w_of(J), w_of(T)}}, count, Bs, 0, s);
    if (e == cudaSuccess) e = gemm(GemmJobs{{g_of(J), g_of(T)}}, count, Bs, 0, s);
    // both ends reach the middle row in the last steps: its two updates one after the other
    if (e == cudaSuccess && count == 2 && J + 1 == T - 1) {
      e = gemm(GemmJobs{{s_of(J), {}}}, 1, Bs, 1, s);
      if (e == cudaSuccess) e = gemm(GemmJobs{{s_of(T), {}}}, 1, Bs, 1, s);
    } else if (e == cudaSuccess) {
      e = gemm(GemmJobs{{s_of(J), s_of(T)}}, count, Bs, 1, s);
    }
  }
  if (e == cudaSuccess) e = gj_inverse(Pair{{blk(B.Sinv, mid), nullptr}}, 1, Bs, B.fcol, B.perm, B.status, s);
  return e;
}

cudaError_t ray_coarse_solve(const RayBlocks& B, double2* z, const double2* g, cudaStream_t s) {
  cudaError_t e = block_substitute(B, z, g, B.y, s);
  if (e != cudaSuccess) return e;
  // one step of iterative refinement: z += (block LU)^{-1} (g - A_ray z)
  const long long cnt = (long long)B.Bs * B.Nr;
  e = pdl_launch(ray_block_residual_kernel, dim3(blocks_for(cnt, 128)), dim3(128), 0, s, B.e, g, (const double2*)z,
                 (const double2*)B.L, (const double2*)B.D, (const double2*)B.U, B.Bs, B.Nr);
  if (e == cudaSuccess) e = block_substitute(B, B.dz, B.e, B.y, s);
  if (e == cudaSuccess) e = pdl_launch(ray_axpy_kernel, dim3(blocks_for(cnt, 256)), dim3(256), 0, s, z, (const double2*)B.dz, cnt);
  return e;
}

cudaError_t launch_ray_residual_norm(double2* r, const double2* b, const double2* v, long long N, double* partials,
                                     double* out, cudaStream_t s) {
  cudaError_t e = pdl_launch(ray_residual_norm_kernel, dim3(RED_BLOCKS), dim3(RED_THREADS), 0, s, r, b, v, N, partials);
  if (e == cudaSuccess) e = pdl_launch(ray_sum_kernel, dim3(1), dim3(256), 0, s, (const double*)partials, out);
  return e;
}

cudaError_t launch_ray_axpy(double2* x, const double2* z, long long N, cudaStream_t s) {
  return pdl_launch(ray_axpy_kernel, dim3(blocks_for(N, 256)), dim3(256), 0, s, x, z, N);
}

int ray_reduction_blocks() { return RED_BLOCKS; }

}  // namespace hz
