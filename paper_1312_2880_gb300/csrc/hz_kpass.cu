// Whole pre- and post-relaxation passes of an FP32 Kaczmarz level (Sec. 4-5: 4 sweeps of Gauss-Seidel on
// the normal equations each way), transfers included, in launches of independent tiles with four or two
// sweeps each (nu / 4 or nu / 2 launches a pass).
//
// Pre: zero guess, the sweeps (colours 0..4), residual with the (B) operator and full weighting onto the
// coarse level. Post: u_pre + P e_c, the sweeps (colours 4..0). A tile holds a region with the
// dependency cone of all colour phases of the launch (6 columns each side and 6 and 10 rows per
// sweep), so no block waits for another and every value is the one the whole-level sweeps give.
//
// What bounds it: 10 or 20 dependent phases, each a block barrier, and the shared-memory traffic of its
// row actions (92 bytes an action: a phase moves the whole region through shared memory once), 0.4
// to 0.7 us a phase. Boundary tests, the node of a phase's colour and the rows' constants are set up
// once per thread and launch (a thread keeps one or two blocks of five nodes): finding them again in
// every phase took 275 instructions a row action, the ALU pipe 63% busy (24 us a launch of 20 phases
// at n_l = 128 against 18). Recomputing the halo costs two to four times the actions of the level,
// but on SMs that a small level leaves idle, while a cluster pays per phase (cluster barriers and
// distributed shared memory, about 1.3 us) and launches without the transfers pay two more launches.
// Per iteration (four launches or pairs, transfers included, FP32): n_l = 128 114 us (cluster) to
// 93; n_l = 256 139 us (two sweeps per launch and separate transfers) to 105; n_l = 512 176 to 156;
// n_l = 1024 315 to 291.
#include <cuda_runtime.h>

#include "hz_common.cuh"
#include "hz_host.h"
#include "hz_internal.h"
#include "hz_level.cuh"

namespace hz {

namespace {

constexpr int PT = 1024;  // threads per block

// A launch of S sweeps on tiles whose region (the tile plus the dependency cone of the 5 S colour phases) is
// RX x RY nodes, RX = 5 COLS. CAP: the launch also does the pass's transfer (pre: residual and
// restriction after the last sweep; post: bilinear correction before the first). VALID is the square
// of nodes whose values must be right after the last phase: the tile itself, and two more nodes on
// every side where residuals around the tile's coarse nodes read them.
template <int S_, int COLS_, bool POST, bool CAP>
struct PassGeo {
  static constexpr int S = S_, PHASES = 5 * S, COLS = COLS_;
  static constexpr int HX = 6 * S, HN = 6 * S, HF = 10 * S;  // TileGeo's halo
  static constexpr int PAD = (!POST && CAP) ? 2 : 0;
  static constexpr int RX = 5 * COLS, VALID = RX - 2 * HX, KT = VALID - 2 * PAD;
  static constexpr int BELOW = POST ? HF : HN;  // region rows below VALID
  static constexpr int RY = VALID + HN + HF, REG = RX * RY;
  static constexpr int SLOTS = COLS * RY;             // blocks of five nodes of a region row
  static constexpr int NS = (SLOTS + PT - 1) / PT;    // per thread
  // coarse nodes that the bilinear correction of the region reads
  static constexpr int CX = RX / 2 + 2, CY = RY / 2 + 2;
  static constexpr size_t SMEM = (size_t)REG * 20 + (POST && CAP ? (size_t)CX * CY * 8 : 0);
  // Rows of phase ph (R = PHASES - 1 - ph phases follow it) that can still reach the outputs, as in
  // PhaseRect; actions of other rows are skipped. (Columns out of reach are not: they change only
  // values that no output depends on.)
  __host__ __device__ static constexpr int ylo(int R) { return BELOW - 1 - (POST ? 2 : 1) * R; }
  __host__ __device__ static constexpr int rows(int R) { return VALID + 2 + 3 * R; }
  static_assert(ylo(PHASES - 1) >= 1 && ylo(PHASES - 1) + rows(PHASES - 1) <= RY - 1 && HX - PHASES >= 1 && KT > 0,
                "supports inside the region");
  static_assert(NS <= 2, "at most two actions per thread and phase");
};

// A thread's block of five consecutive nodes of region row r: one of them has each colour, at position
// pos for the current phase's colour, one further per phase (one back in the post order). Everything
// a phase needs about the boundary is set up once.
struct Slot {
  int base, r, pos;  // first node's region index, region row, position of the colour
  int dS, dN;        // offsets of the S and N support (mirrored on the first and last grid row)
  unsigned live;     // bit p: node p is in the square and its support is in the region
  int pL, pR;        // position of the node on the first / last grid column (or none)
  float ty, ny;      // boundary terms of the row: 2 per side in the diagonal, 2 or 4 in |a_p|^2
};

template <class G, bool POST>
__device__ __forceinline__ Slot make_slot(int t, int gx, int gy, int n) {
  Slot s;
  s.r = t / G::COLS;
  const int c0 = 5 * (t - s.r * G::COLS), j = gy + s.r, i0 = gx + c0;
  s.base = s.r * G::RX + c0;
  const int colour = POST ? 4 : 0;  // i + 2 j = colour mod 5 at position pos of the row
  s.pos = (((colour - i0 - 2 * j) % 5) + 5) % 5;
  s.dS = j > 0 ? -G::RX : G::RX;
  s.dN = j < n ? G::RX : -G::RX;
  const bool my = j == 0 || j == n;
  s.ty = my ? 2.0f : 0.0f;
  s.ny = my ? 4.0f : 2.0f;
  s.pL = -i0;
  s.pR = n - i0;
  s.live = 0;
  if (t < G::SLOTS && (unsigned)j <= (unsigned)n && s.r >= 1 && s.r <= G::RY - 2)
#pragma unroll
    for (int p = 0; p < 5; ++p)
      if ((unsigned)(i0 + p) <= (unsigned)n && c0 + p >= 1 && c0 + p <= G::RX - 2) s.live |= 1u << p;
  return s;
}

// All colour phases, a barrier after each. A thread reads the supports of both its actions before
// updating either (same-colour supports are disjoint). The operations are those of lvl::row_consts
// and lvl::act_update, so the bits are those of every Kaczmarz form (a mirror node's update
// u + 2 delta is one fma with the exact factor 2).
template <class G, bool POST, bool INNER>
__device__ __forceinline__ void pass_phases(float2* su, const float2* sf, const float* sk, int gx, int gy, int n,
                                            float beta) {
  constexpr int W = G::RX, NS = G::NS;
  Slot sl[NS];
#pragma unroll
  for (int q = 0; q < NS; ++q) sl[q] = make_slot<G, POST>((int)threadIdx.x + q * PT, gx, gy, n);
#pragma unroll 1
  for (int ph = 0; ph < G::PHASES; ++ph) {
    const int R = G::PHASES - 1 - ph, ylo = G::ylo(R), rows = G::rows(R);
    bool on[NS];
    int p[NS], dW[NS], dE[NS];
    float2 up[NS], uw[NS], ue[NS], us[NS], un[NS], f[NS];
    float kh[NS];
#pragma unroll
    for (int q = 0; q < NS; ++q) {
      const Slot& s = sl[q];
      on[q] = (unsigned)(s.r - ylo) < (unsigned)rows && (s.live >> s.pos & 1u);
      p[q] = s.base + s.pos;
      dW[q] = !INNER && s.pos == s.pL ? 1 : -1;
      dE[q] = !INNER && s.pos == s.pR ? -1 : 1;
      if (on[q]) {
        up[q] = su[p[q]];
        uw[q] = su[p[q] + dW[q]];
        ue[q] = su[p[q] + dE[q]];
        us[q] = su[p[q] + (INNER ? -W : s.dS)];
        un[q] = su[p[q] + (INNER ? W : s.dN)];
        f[q] = sf[p[q]];
        kh[q] = sk[p[q]];
      }
    }
#pragma unroll
    for (int q = 0; q < NS; ++q) {
      Slot& s = sl[q];
      if (on[q]) {
        const bool mx = !INNER && dW[q] == dE[q], my = !INNER && s.dS == s.dN;
        const float two_sides = INNER ? 0.0f : s.ty + (mx ? 2.0f : 0.0f);
        const float2 d = xr::diag2<float>(kh[q], two_sides, beta);
        const float inv = xr::rcp(xr::add(xr::cabs2<float>(d), INNER ? 4.0f : s.ny + (mx ? 4.0f : 2.0f)));
        const float2 delta =
            xr::cscale<float>(xr::resid<float>(f[q], up[q], xr::nb4<float>(uw[q], ue[q], us[q], un[q]), d), inv);
        const float cx = mx ? 2.0f : 1.0f, cy = my ? 2.0f : 1.0f;
        su[p[q]] = xr::cadd<float>(up[q], xr::cmulc<float>(d, delta));
        su[p[q] + dW[q]] = make_float2(xr::fma(delta.x, cx, uw[q].x), xr::fma(delta.y, cx, uw[q].y));
        if (!mx) su[p[q] + dE[q]] = xr::cadd<float>(ue[q], delta);
        su[p[q] + (INNER ? -W : s.dS)] = make_float2(xr::fma(delta.x, cy, us[q].x), xr::fma(delta.y, cy, us[q].y));
        if (!my) su[p[q] + (INNER ? W : s.dN)] = xr::cadd<float>(un[q], delta);
      }
      s.pos = POST ? (s.pos == 0 ? 4 : s.pos - 1) : (s.pos == 4 ? 0 : s.pos + 1);
    }
    __syncthreads();
  }
}

// ZERO: from a zero guess (uin unused).
template <class G, bool POST, bool CAP, bool ZERO>
__device__ __forceinline__ void pass_body(const KaczPassArgs& a, const Inst& bi) {
  constexpr int RX = G::RX, RY = G::RY, REG = G::REG, NW = PT / 32, KT = G::KT;
  const int n = a.n;
  extern __shared__ __align__(16) unsigned char smem[];
  float2* su = reinterpret_cast<float2*>(smem);
  float2* sf = su + REG;
  float2* se = sf + REG;  // coarse correction, G::CX x G::CY
  float* sk = reinterpret_cast<float*>(se + (POST && CAP ? G::CX * G::CY : 0));
  const int x0 = blockIdx.x * KT, y0 = blockIdx.y * KT;
  const int gx = x0 - G::PAD - G::HX, gy = y0 - G::PAD - G::BELOW;
  const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
  // k H does not depend on the preceding kernel: fetched before the wait for it, with the zero guess
  for (int r = warp; r < RY; r += NW) {
    const int j = gy + r;
    if ((unsigned)j > (unsigned)n) continue;
    const float* row = a.kh + (long long)j * a.pk;
    for (int c = lane; c < RX; c += 32) {
      const int i = gx + c;
      if ((unsigned)i > (unsigned)n) continue;
      lvl::cp_async<4>(sk + r * RX + c, row + i);
      if (ZERO) su[r * RX + c] = make_float2(0.0f, 0.0f);
    }
  }
  pdl_enter();
  if (a.stop && a.stop[blockIdx.z * bi.stop_stride]) {
    lvl::cp_async_wait_all();
    return;
  }
  float2* uout = a.uout + blockIdx.z * bi.su;
  const float2* f = a.f + blockIdx.z * bi.sf;
  for (int r = warp; r < RY; r += NW) {
    const int j = gy + r;
    if ((unsigned)j > (unsigned)n) continue;
    const float2* frow = f + (long long)j * a.pf;
    const float2* urow = ZERO ? nullptr : a.uin + blockIdx.z * bi.su + (long long)j * a.pu;
    for (int c = lane; c < RX; c += 32) {
      const int i = gx + c;
      if ((unsigned)i > (unsigned)n) continue;
      lvl::cp_async<8>(sf + r * RX + c, frow + i);
      if (!ZERO) lvl::cp_async<8>(su + r * RX + c, urow + i);
    }
  }
  const int I0 = max(gx, 0) >> 1, J0 = max(gy, 0) >> 1, nc = n >> 1;
  if constexpr (POST && CAP) {
    const float2* ec = a.ec + blockIdx.z * bi.sc;
    for (int r = warp; r < G::CY; r += NW) {
      const int J = J0 + r;
      if (J > nc) break;
      for (int c = lane; c < G::CX; c += 32)
        if (I0 + c <= nc) lvl::cp_async<8>(se + r * G::CX + c, ec + (long long)J * a.pc + I0 + c);
    }
  }
  lvl::cp_async_wait_all();
  __syncthreads();
  if constexpr (POST && CAP) {  // u_pre + P e_c, in the operation order of the separate correction
    for (int r = warp; r < RY; r += NW) {
      const int j = gy + r;
      if ((unsigned)j > (unsigned)n) continue;
      const float2* e0 = se + ((j >> 1) - J0) * G::CX;
      for (int c = lane; c < RX; c += 32) {
        const int i = gx + c;
        if ((unsigned)i > (unsigned)n) continue;
        su[r * RX + c] = xr::cadd<float>(su[r * RX + c], xr::bilinear<float>(e0, e0 + G::CX, (i >> 1) - I0, i & 1, j & 1));
      }
    }
    __syncthreads();
  }
  // every node of the region strictly inside the square: no mirrors, no boundary terms
  if (gx >= 1 && gx + RX <= n && gy >= 1 && gy + RY <= n)
    pass_phases<G, POST, true>(su, sf, sk, gx, gy, n, a.bA);
  else
    pass_phases<G, POST, false>(su, sf, sk, gx, gy, n, a.bA);
  // the tile's own nodes back to global memory
  for (int r = warp; r < KT; r += NW) {
    const int j = y0 + r;
    if (j > n) break;
    float2* orow = uout + (long long)j * a.pu;
    const float2* srow = su + (r + G::BELOW + G::PAD) * RX + G::HX + G::PAD;
    for (int c = lane; c < KT && x0 + c <= n; c += 32) orow[x0 + c] = srow[c];
  }
  if constexpr (!POST && CAP) {
    // residual one node around the tile, in place of f~ (a node's residual reads no other f~)
    constexpr int W = RX;
    for (int r = warp; r < KT + 2; r += NW) {
      const int j = y0 - 1 + r;
      if ((unsigned)j > (unsigned)n) continue;
      for (int c = lane; c < KT + 2; c += 32) {
        const int i = x0 - 1 + c;
        if ((unsigned)i > (unsigned)n) continue;
        const int p = (j - gy) * W + (i - gx);
        const float2 nb = xr::nb4<float>(su[p + (i > 0 ? -1 : 1)], su[p + (i < n ? 1 : -1)], su[p + (j > 0 ? -W : W)],
                                         su[p + (j < n ? W : -W)]);
        sf[p] = xr::resid<float>(sf[p], su[p], nb, xr::diag<float>(sk[p], lvl::sides_at(i, j, n), a.bB));
      }
    }
    __syncthreads();
    // full weighting at the coarse nodes whose fine node lies in the tile (xr::fw_node's order)
    float2* fc = a.fc + blockIdx.z * bi.sc;
    const int Ia = (x0 + 1) >> 1, Ja = (y0 + 1) >> 1;
    const float2* r0 = sf - (gy * W + gx);  // node (i, j) at r0[j W + i]
    for (int r = warp; r < KT / 2 + 1; r += NW) {
      const int J = Ja + r;
      if (2 * J >= y0 + KT || J > nc) break;
      for (int c = lane; c < KT / 2 + 1; c += 32) {
        const int I = Ia + c;
        if (2 * I >= x0 + KT || I > nc) break;
        fc[(long long)J * a.pc + I] = xr::fw_node<float>(r0, W, n, I, J);
      }
    }
  }
}

// 56 registers, so that the block fits beside the deferred solution update (k_update_x, one 128-thread
// block per SM) that runs during the cycle.
template <class G, bool POST, bool CAP, bool ZERO>
__global__ void __maxnreg__(56) kacz_pass_kernel(const KaczPassArgs a, Inst bi) {
  pass_body<G, POST, CAP, ZERO>(a, bi);
}

template <int S, int COLS, bool POST, bool CAP, bool ZERO>
cudaError_t launch_one(const KaczPassArgs& a, cudaStream_t s, const Inst& bi) {
  using G = PassGeo<S, COLS, POST, CAP>;
  static OncePerDevice opt_in;
  const cudaError_t e = opt_in([] {
    return cudaFuncSetAttribute(kacz_pass_kernel<G, POST, CAP, ZERO>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)G::SMEM);
  });
  if (e) return e;
  const int t = (a.n + G::KT) / G::KT;
  pdl_launch(kacz_pass_kernel<G, POST, CAP, ZERO>, dim3(t, t, bi.count), PT, G::SMEM, s, a, bi);
  return cudaGetLastError();
}

// The launches of a pass alternate between u and u2 (a tile reads its neighbours' input): the pre pass
// ends in u, the post pass starts from u and ends in u2 after an odd number of launches.
template <int S, int COLS>
cudaError_t run_pass(bool post, int nu, KaczPassArgs a, float2* u, float2* u2, cudaStream_t s, const Inst& bi) {
  const int launches = nu / S;
  for (int k = 0; k < launches; ++k) {
    const bool first = k == 0, last = k == launches - 1;
    a.uout = (post ? k : launches - 1 - k) % 2 == (post ? 1 : 0) ? u : u2;
    cudaError_t e;
    if (post)
      e = first ? launch_one<S, COLS, true, true, false>(a, s, bi) : launch_one<S, COLS, true, false, false>(a, s, bi);
    else if (first)
      e = last ? launch_one<S, COLS, false, true, true>(a, s, bi) : launch_one<S, COLS, false, false, true>(a, s, bi);
    else
      e = last ? launch_one<S, COLS, false, true, false>(a, s, bi) : launch_one<S, COLS, false, false, false>(a, s, bi);
    if (e) return e;
    a.uin = a.uout;
  }
  return cudaSuccess;
}

// Geometries (rules::pass_config): 0, 65 x 81 regions for four sweeps; 1, 65 x 73 regions and 2, 90 x 98
// regions for two.
constexpr int cfg_sweeps(int cfg) { return cfg == 0 ? 4 : 2; }

}  // namespace

bool pass_in_place(int cfg, int nu) { return nu / cfg_sweeps(cfg) % 2 == 0; }

cudaError_t launch_kacz_pass(bool post, int cfg, int nu, const KaczPassArgs& args, float2* u, float2* u2,
                             cudaStream_t s, const Inst& bi) {
  KaczPassArgs a = args;
  a.uin = u;
  switch (cfg) {
    case 0: return run_pass<4, 13>(post, nu, a, u, u2, s, bi);
    case 1: return run_pass<2, 13>(post, nu, a, u, u2, s, bi);
    case 2: return run_pass<2, 18>(post, nu, a, u, u2, s, bi);
  }
  return cudaErrorInvalidValue;
}

}  // namespace hz
