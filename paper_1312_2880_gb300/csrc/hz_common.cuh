// Device-side helpers shared by the kernels: complex arithmetic in the working precision and
// the 5-point Helmholtz row of the paper's discretisation in h^2-scaled form.
//
// Scaled form: every level stores its equations multiplied by H^2, so a row reads
//   u_E + u_W + u_N + u_S + d_p u_p = f~_p,   f~ = H^2 f,
//   d_p = -4 + (k_p H)^2 (1 + i beta_A) + 2 i s_p (k_p H),
// where s_p is the number of sides of the square the node lies on (0 inside, 1 on an edge,
// 2 at a corner). This is L^H (beta_A = 0) or M^H = L^H + i k^2 beta (Eq. 3) with the
// first-order Sommerfeld condition du/dn - i k u = 0 (Sec. 1) closed by a centred difference:
// the ghost value is u_mirror + 2 i k H u_p, so at the boundary the mirror node's coefficient
// becomes 2 and the diagonal gains 2 i k H per side.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace hz {

// Programmatic dependent launch: every kernel is launched allowed to start while its predecessor
// in the stream (or graph) is still running. It first waits until the predecessor has completed
// and its writes are visible (griddepcontrol.wait; nothing is read before), then allows its own
// successor to begin launching, so launch latency overlaps execution. Both are no-ops for a
// kernel launched without the attribute.
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}

template <class T> struct cplx_of;
template <> struct cplx_of<double> { using type = double2; };
template <> struct cplx_of<float> { using type = float2; };
template <class T> using c2 = typename cplx_of<T>::type;

template <class T>
__host__ __device__ __forceinline__ c2<T> mk(T re, T im) {
  c2<T> z;
  z.x = re;
  z.y = im;
  return z;
}

// Conversions between binary64 and binary32 on the integer pipe. GB300 runs hardware float
// conversions on its narrow FP64 pipe, which the FP32 V-cycle would otherwise saturate just
// reading and writing the FP64 Krylov vectors. Written from the IEEE 754 formats: narrowing
// rounds to nearest, ties to even, on the 29 dropped significand bits (a carry into the exponent
// is the correct rounding); results below the binary32 normal range become signed zero;
// overflow gives infinity; NaN stays NaN. Widening is exact for normal numbers and zero
// (subnormal binary32 inputs become signed zero).
__device__ __forceinline__ float f64_to_f32(double d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const unsigned int sign = (unsigned int)(b >> 32) & 0x80000000u;
  const int e = (int)((b >> 52) & 0x7FF);
  if (e == 0x7FF) return __int_as_float((int)(sign | 0x7F800000u | ((b & 0x000FFFFFFFFFFFFFull) ? 0x400000u : 0u)));
  const int ef = e - 1023 + 127;
  if (ef <= 0) return __int_as_float((int)sign);
  const unsigned int m = (unsigned int)((b >> 29) & 0x7FFFFFu);
  const unsigned int rem = (unsigned int)(b & 0x1FFFFFFFu);
  unsigned int mag = ((unsigned int)ef << 23) | m;
  mag += (rem > 0x10000000u || (rem == 0x10000000u && (m & 1u))) ? 1u : 0u;
  if (mag >= 0x7F800000u) mag = 0x7F800000u;
  return __int_as_float((int)(sign | mag));
}
__device__ __forceinline__ double f32_to_f64(float f) {
  const unsigned int u = (unsigned int)__float_as_int(f);
  const unsigned long long sign = (unsigned long long)(u & 0x80000000u) << 32;
  const unsigned int e = (u >> 23) & 0xFF;
  const unsigned long long m = (unsigned long long)(u & 0x7FFFFFu) << 29;
  if (e == 0) return __longlong_as_double((long long)sign);
  const unsigned long long eb = (e == 0xFF) ? 0x7FFull : (unsigned long long)(e - 127 + 1023);
  return __longlong_as_double((long long)(sign | (eb << 52) | m));
}

// Load a complex element stored as double2 or float2 and convert it to precision T.
template <class T>
__device__ __forceinline__ c2<T> ldc(const double2* p, long long i) {
  double2 v = p[i];
  return mk<T>((T)v.x, (T)v.y);
}
template <>
__device__ __forceinline__ c2<float> ldc<float>(const double2* p, long long i) {
  double2 v = p[i];
  return mk<float>(f64_to_f32(v.x), f64_to_f32(v.y));
}
template <class T>
__device__ __forceinline__ c2<T> ldc(const float2* p, long long i) {
  float2 v = p[i];
  return mk<T>((T)v.x, (T)v.y);
}
template <class T>
__device__ __forceinline__ void stc(double2* p, long long i, c2<T> v) {
  p[i] = make_double2((double)v.x, (double)v.y);
}
template <>
__device__ __forceinline__ void stc<float>(double2* p, long long i, c2<float> v) {
  p[i] = make_double2(f32_to_f64(v.x), f32_to_f64(v.y));
}
template <class T>
__device__ __forceinline__ void stc(float2* p, long long i, c2<T> v) {
  p[i] = make_float2((float)v.x, (float)v.y);
}

template <class T> __device__ __forceinline__ c2<T> cadd(c2<T> a, c2<T> b) { return mk<T>(a.x + b.x, a.y + b.y); }
template <class T> __device__ __forceinline__ c2<T> csub(c2<T> a, c2<T> b) { return mk<T>(a.x - b.x, a.y - b.y); }
template <class T> __device__ __forceinline__ c2<T> cscale(c2<T> a, T s) { return mk<T>(a.x * s, a.y * s); }
template <class T>
__device__ __forceinline__ c2<T> cmul(c2<T> a, c2<T> b) {
  return mk<T>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// conj(a) * b
template <class T>
__device__ __forceinline__ c2<T> cmulc(c2<T> a, c2<T> b) {
  return mk<T>(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}
// 1/x: IEEE division in FP64; the correctly rounded single-precision reciprocal in FP32.
__device__ __forceinline__ double rcp(double x) { return 1.0 / x; }
__device__ __forceinline__ float rcp(float x) { return __frcp_rn(x); }

template <class T>
__device__ __forceinline__ c2<T> cdiv(c2<T> a, c2<T> b) {
  T inv = rcp(b.x * b.x + b.y * b.y);
  return mk<T>((a.x * b.x + a.y * b.y) * inv, (a.y * b.x - a.x * b.y) * inv);
}
template <class T> __device__ __forceinline__ T cabs2(c2<T> a) { return a.x * a.x + a.y * a.y; }

// Diagonal of the scaled row at a node with kh = k_p H on `sides` sides of the square.
template <class T>
__device__ __forceinline__ c2<T> row_diag(T kh, int sides, T beta) {
  T kh2 = kh * kh;
  return mk<T>(kh2 - (T)4, beta * kh2 + (T)(2 * sides) * kh);
}

// Neighbour indices of node (i, j) on a grid with n intervals, with out-of-domain neighbours
// replaced by their mirror nodes (ghost elimination).
struct Nbr {
  int iw, ie, js, jn, sides;
};
__device__ __forceinline__ Nbr neighbours(int i, int j, int n) {
  Nbr b;
  b.iw = i > 0 ? i - 1 : 1;
  b.ie = i < n ? i + 1 : n - 1;
  b.js = j > 0 ? j - 1 : 1;
  b.jn = j < n ? j + 1 : n - 1;
  b.sides = (i == 0) + (i == n) + (j == 0) + (j == n);
  return b;
}

__device__ __forceinline__ int reflect(int i, int n) {
  i = i < 0 ? -i : i;
  return i > n ? 2 * n - i : i;
}

// Fixed-rounding complex arithmetic for the fused Gauss-Seidel passes. Every operation is an
// explicit round-to-nearest add, multiply or fused multiply-add, so the compiler cannot contract
// or reorder it differently from one kernel to another: the tile and streaming forms of a pass,
// which share these helpers and take the same operations in the same order on every node, give
// bit-identical results, and the choice between them never changes a solution.
namespace xr {
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma(double a, double b, double c) { return __fma_rn(a, b, c); }
// The correctly rounded FP64 sum a + b on the integer pipe (the bits of __dadd_rn, from the IEEE 754
// formats): order by magnitude, align the smaller significand below the larger with ten guard bits and
// a sticky bit, add or subtract, normalise, round to nearest even. About 50 instructions of the
// integer pipe against 77 cycles of the FP64 pipe, which kernels bound by the latter leave idle:
// there, some of the additions done here run beside the rest. Zeros, subnormal operands or results,
// infinities, NaN and exact cancellation take the hardware addition.
// Out of line: in line, the compiler predicates this addition and issues it for every warp.
static __device__ __noinline__ double add_hw(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double add_int(double a, double b) {
  unsigned ah = (unsigned)__double2hiint(a), al = (unsigned)__double2loint(a);
  unsigned bh = (unsigned)__double2hiint(b), bl = (unsigned)__double2loint(b);
  const unsigned long long ua = ((unsigned long long)(ah & 0x7fffffffu) << 32) | al;
  const unsigned long long ub = ((unsigned long long)(bh & 0x7fffffffu) << 32) | bl;
  if (ub > ua) {
    unsigned t = ah; ah = bh; bh = t;
    t = al; al = bl; bl = t;
  }
  const int ea = (int)(ah >> 20) & 0x7ff, eb = (int)(bh >> 20) & 0x7ff;
  const unsigned long long ma = ((unsigned long long)__funnelshift_l(al, (ah & 0xfffffu) | 0x100000u, 10) << 32) | (al << 10);
  const unsigned long long mb = ((unsigned long long)__funnelshift_l(bl, (bh & 0xfffffu) | 0x100000u, 10) << 32) | (bl << 10);
  const int d = min(ea - eb, 63);
  unsigned long long t = mb >> d;
  t |= (t << d) != mb ? 1ull : 0ull;
  const long long neg = (long long)(int)(ah ^ bh) >> 31;  // all ones: a difference
  unsigned long long r = ma + ((t ^ (unsigned long long)neg) - (unsigned long long)neg);
  const int lz = __clzll((long long)r), e = ea + 1 - lz;
  if (eb == 0 || ea == 0x7ff || (unsigned)(e - 1) >= 0x7feu || r == 0) return add_hw(a, b);
  r <<= lz;
  const unsigned long long p = r >> 11;
  const unsigned up = ((unsigned)r & 0x7ffu) + ((unsigned)p & 1u) > 0x400u ? 1u : 0u;
  const unsigned long long q = p + up + ((unsigned long long)(unsigned)(e - 1) << 52);
  return __hiloint2double((int)((unsigned)(q >> 32) | (ah & 0x80000000u)), (int)(unsigned)q);
}
// FP32: the hardware reciprocal approximation (rcp.approx, about 1 ulp); the divisors here are
// |d|^2 of a Helmholtz diagonal, never denormal. FP64: the correctly rounded reciprocal.
__device__ __forceinline__ float rcp(float a) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ double rcp(double a) { return __drcp_rn(a); }

template <class T> __device__ __forceinline__ c2<T> cadd(c2<T> a, c2<T> b) { return mk<T>(add(a.x, b.x), add(a.y, b.y)); }
template <class T> __device__ __forceinline__ c2<T> csub(c2<T> a, c2<T> b) { return mk<T>(sub(a.x, b.x), sub(a.y, b.y)); }
template <class T> __device__ __forceinline__ c2<T> cscale(c2<T> a, T s) { return mk<T>(mul(a.x, s), mul(a.y, s)); }
// FP32: both components in one packed instruction (the same rounding per component; a - b is formed as
// a + (-1) b with the exact product). Fewer issue slots in kernels bound by them: the coarse tail of
// the n = 512 hierarchy 62.5 -> 60.6 us, the Kaczmarz passes of an n_l = 256 level 108 -> 105 us per
// iteration, the finest smooth_restrict at n = 4096 78 -> 76 us.
template <>
__device__ __forceinline__ float2 cadd<float>(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 p, q;\n\tmov.b64 p, {%2, %3};\n\tmov.b64 q, {%4, %5};\n\tadd.rn.f32x2 p, p, q;\n\t"
      "mov.b64 {%0, %1}, p;\n\t}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
template <>
__device__ __forceinline__ float2 csub<float>(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 p, q, m;\n\tmov.b64 p, {%2, %3};\n\tmov.b64 q, {%4, %5};\n\tmov.b64 m, 0xbf800000bf800000;\n\t"
      "fma.rn.f32x2 p, q, m, p;\n\tmov.b64 {%0, %1}, p;\n\t}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
template <class T>
__device__ __forceinline__ c2<T> cmul(c2<T> a, c2<T> b) {
  return mk<T>(fma(a.x, b.x, -mul(a.y, b.y)), fma(a.x, b.y, mul(a.y, b.x)));
}
// conj(a) * b
template <class T>
__device__ __forceinline__ c2<T> cmulc(c2<T> a, c2<T> b) {
  return mk<T>(fma(a.x, b.x, mul(a.y, b.y)), fma(a.x, b.y, -mul(a.y, b.x)));
}
template <class T> __device__ __forceinline__ T cabs2(c2<T> a) { return fma(a.x, a.x, mul(a.y, a.y)); }
template <class T>
__device__ __forceinline__ c2<T> cdiv(c2<T> a, c2<T> d) {
  const T inv = rcp(fma(d.x, d.x, mul(d.y, d.y)));
  return mk<T>(mul(fma(a.x, d.x, mul(a.y, d.y)), inv), mul(fma(a.y, d.x, -mul(a.x, d.y)), inv));
}
// Scaled-row diagonal (k H)^2 - 4 + i (beta (k H)^2 + 2 sides k H); two_sides = 2 sides.
template <class T>
__device__ __forceinline__ c2<T> diag2(T kh, T two_sides, T beta) {
  const T k2 = mul(kh, kh);
  return mk<T>(sub(k2, (T)4), fma(two_sides, kh, mul(beta, k2)));
}
template <class T>
__device__ __forceinline__ c2<T> diag(T kh, int sides, T beta) { return diag2<T>(kh, (T)(2 * sides), beta); }
// Sum of a node's four neighbours in the order (W + E) + (S + N).
template <class T>
__device__ __forceinline__ c2<T> nb4(c2<T> w, c2<T> e, c2<T> s, c2<T> n) {
  return cadd<T>(cadd<T>(w, e), cadd<T>(s, n));
}
// The same with MIX of its six FP64 additions on the integer pipe (add_int; 0, 1, 2, 4 or 6).
template <int MIX>
__device__ __forceinline__ double2 nb4_mix(double2 w, double2 e, double2 s, double2 n) {
  const double hx = MIX >= 1 ? add_int(w.x, e.x) : add(w.x, e.x), hy = MIX >= 2 ? add_int(w.y, e.y) : add(w.y, e.y);
  const double vx = MIX >= 4 ? add_int(s.x, n.x) : add(s.x, n.x), vy = MIX >= 4 ? add_int(s.y, n.y) : add(s.y, n.y);
  return MIX >= 6 ? mk<double>(add_int(hx, vx), add_int(hy, vy)) : mk<double>(add(hx, vx), add(hy, vy));
}
template <int MIX>
__device__ __forceinline__ float2 nb4_mix(float2 w, float2 e, float2 s, float2 n) { return nb4<float>(w, e, s, n); }
// Gauss-Seidel point update (f - nb) / d and residual f - (d u + nb).
template <class T>
__device__ __forceinline__ c2<T> gs(c2<T> f, c2<T> nb, c2<T> d) { return cdiv<T>(csub<T>(f, nb), d); }
template <class T>
__device__ __forceinline__ c2<T> resid(c2<T> f, c2<T> u, c2<T> nb, c2<T> d) {
  return csub<T>(f, cadd<T>(cmul<T>(d, u), nb));
}
// The same operations for the passes' specialised paths. K says what the compiler may take as known
// of a node's diagonal: DIAG_ANY nothing, DIAG_INNER that the node is inside the square (no boundary
// term), DIAG_REAL that the operator is L there as well, so that d is real. Terms with an exact zero
// factor are left out: the same values (only the sign of a zero can differ). In FP64 the reciprocal
// 1 / |d|^2 is read (inv, stored once per problem): it is eight of the 20 FP64 instructions of a
// quotient, and an FP64 warp instruction takes about 77 cycles of a sub-partition. With both, a node
// of the finest FP64 smooth_restrict takes about 29 FP64 instructions instead of 49 (n = 4096: 1.94
// to 1.19 ms; prolong_smooth 1.16 to 0.85 ms). Chosen at run time per node, by testing d's
// imaginary part, the compiler evaluated both cases and the passes gained nothing.
enum { DIAG_ANY = 0, DIAG_INNER = 1, DIAG_REAL = 2 };
template <class T, int K>
__device__ __forceinline__ c2<T> diag_k(T kh, T two_sides, T beta) {
  if (K == DIAG_ANY) return diag2<T>(kh, two_sides, beta);
  const T k2 = mul(kh, kh);
  return mk<T>(sub(k2, (T)4), K == DIAG_REAL ? (T)0 : mul(beta, k2));
}
template <class T, int K>
__device__ __forceinline__ c2<T> cdiv_k(c2<T> a, c2<T> d, T inv) {
  if constexpr (sizeof(T) == 4) inv = rcp(K == DIAG_REAL ? mul(d.x, d.x) : cabs2<T>(d));
  if (K == DIAG_REAL) return mk<T>(mul(mul(a.x, d.x), inv), mul(mul(a.y, d.x), inv));
  return mk<T>(mul(fma(a.x, d.x, mul(a.y, d.y)), inv), mul(fma(a.y, d.x, -mul(a.x, d.y)), inv));
}
template <class T, int K>
__device__ __forceinline__ c2<T> gs_k(c2<T> f, c2<T> nb, c2<T> d, T inv) { return cdiv_k<T, K>(csub<T>(f, nb), d, inv); }
template <class T, int K>
__device__ __forceinline__ c2<T> resid_k(c2<T> f, c2<T> u, c2<T> nb, c2<T> d) {
  const c2<T> du = K == DIAG_REAL ? cscale<T>(u, d.x) : cmul<T>(d, u);
  return csub<T>(f, cadd<T>(du, nb));
}
// One row of full weighting: (w + e) + 2 c.
template <class T>
__device__ __forceinline__ c2<T> fw3(c2<T> w, c2<T> c, c2<T> e) {
  const c2<T> s = cadd<T>(w, e);
  if constexpr (sizeof(T) == 8)  // 2 c is exact: one FP64 instruction and one rounding, as in an addition
    return mk<T>(fma(c.x, (T)2, s.x), fma(c.y, (T)2, s.y));
  else
    return cadd<T>(s, cscale<T>(c, (T)2));
}
// Full weighting at coarse node (I, J) of a fine array r (row pitch pr, n intervals), fine nodes
// outside the square mirrored: rows (w + e) + 2 c, then across rows the same, times 4/16 (the
// restricted residual is scaled by (2h)^2 / h^2 = 4 for the coarse level's h^2-scaled rows).
template <class T>
__device__ __forceinline__ c2<T> fw_node(const c2<T>* r, int pr, int n, int I, int J) {
  c2<T> row[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    const c2<T>* rr = r + (long long)reflect(2 * J + b - 1, n) * pr;
    row[b] = fw3<T>(rr[reflect(2 * I - 1, n)], rr[2 * I], rr[reflect(2 * I + 1, n)]);
  }
  return cscale<T>(fw3<T>(row[0], row[1], row[2]), (T)0.25);
}
// One component of fw_node<double>: r points at that component of the array's first value.
__device__ __forceinline__ double fw_comp(const double* r, int pr, int n, int I, int J) {
  const int w = 2 * reflect(2 * I - 1, n), c = 4 * I, e = 2 * reflect(2 * I + 1, n);
  double row[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    const double* rr = r + 2ll * reflect(2 * J + b - 1, n) * pr;
    row[b] = fma(rr[c], 2.0, add(rr[w], rr[e]));
  }
  return mul(fma(row[1], 2.0, add(row[0], row[2])), 0.25);
}
// Bilinear interpolation of the coarse correction at fine node (2I + oi, 2J + oj) from coarse rows
// e0 (J) and e1 (J + 1): coincident nodes copy, edge midpoints average two, centres four, in the
// order ((e00 + e10) + (e01 + e11)) / 4.
template <class T>
__device__ __forceinline__ c2<T> bilinear(const c2<T>* e0, const c2<T>* e1, int I, int oi, int oj) {
  if (oi && oj) return cscale<T>(cadd<T>(cadd<T>(e0[I], e1[I]), cadd<T>(e0[I + 1], e1[I + 1])), (T)0.25);
  if (oi) return cscale<T>(cadd<T>(e0[I], e0[I + 1]), (T)0.5);
  if (oj) return cscale<T>(cadd<T>(e0[I], e1[I]), (T)0.5);
  return e0[I];
}
}  // namespace xr

}  // namespace hz
