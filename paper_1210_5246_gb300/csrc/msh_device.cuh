// msh_device.cuh -- per-cell and per-face device arithmetic of the BME Godunov step.
//
// Everything here works on one 10-vector in registers.  The reconstruction and the flux
// are written in the "local frame" of a sweep direction: the normal axis is moved to
// the x slot, the two transverse axes keep their natural order.  In that frame the
// eigen-system is the ten-variable extension of the paper's x-direction system
// (Sec. 3.3, eqs jacobian, eigenvalues, righteigvec, lefteigvec):
//   eigenvalues  u -+ cf, u -+ cs (twice each), u (four contact waves),
//   cf = sqrt(3 P_xx / rho), cs = sqrt(P_xx / rho),
// and the projections below are its closed-form sparse left/right eigenvectors.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace msh {

constexpr int NV = 10;

// Primitive/conserved component that sits at local slot k for sweep direction D.
// D = 0: (rho, u, v, w, Pxx, Pxy, Pxz, Pyy, Pyz, Pzz)
// D = 1: normal y, transverse (x, z);  D = 2: normal z, transverse (x, y).
template <int D> struct Frame;
template <> struct Frame<0> {
  static __device__ __forceinline__ constexpr int g(int k) { return k; }
};
template <> struct Frame<1> {
  static __device__ __forceinline__ constexpr int g(int k) {
    return k == 1 ? 2 : k == 2 ? 1 : k == 4 ? 7 : k == 6 ? 8 : k == 7 ? 4 : k == 8 ? 6 : k;
  }
};
template <> struct Frame<2> {
  static __device__ __forceinline__ constexpr int g(int k) {
    return k == 1 ? 3 : k == 2 ? 1 : k == 3 ? 2 : k == 4 ? 9 : k == 5 ? 6 : k == 6 ? 8
         : k == 7 ? 4 : k == 8 ? 5 : k == 9 ? 7 : k;
  }
};

// ---------------------------------------------------------- fast arithmetic
// FP32: hardware approximate reciprocal and reciprocal square root (a few ulp, far
// inside the FP32 tolerances).  FP64: IEEE division, and CUDA's rsqrt() for the square roots:
// a double-precision warp instruction holds its scheduler's pipe for 64 cycles on GB300, and
// 1 / sqrt(x) took 930 of them where rsqrt(x) takes 377 (measured, independent chains; errors up
// to 1.48 and 0.51 ulp over 2^20 values).
template <typename T> __device__ __forceinline__ T frcp(T x) { return T(1) / x; }
template <> __device__ __forceinline__ float frcp<float>(float x) { return __fdividef(1.0f, x); }
__device__ __forceinline__ float frsqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ double frsqrt(double x) { return rsqrt(x); }
// sqrt(p / r) for p, r > 0.  FP64: p rsqrt(p r), corrected by its residual p - s (s r) (s r with
// its rounding error), where p and p r are far enough from the ends of the range that nothing
// under- or overflows, and otherwise the square root of the quotient: 828 pipe cycles and errors
// up to 0.50 ulp, where the quotient's root takes 1159 (0.85 ulp) and p rsqrt(p r) alone 522 (1.67
// ulp, and infinite or zero once p r under- or overflows).
__device__ __forceinline__ float sqrt_ratio(float p, float r) { return p * rsqrtf(p * r); }
static __device__ __noinline__ double sqrt_quotient(double p, double r) { return sqrt(p / r); }
__device__ __forceinline__ double sqrt_ratio(double p, double r) {
  const double q = p * r;
  const unsigned ep = (unsigned)__double2hiint(p) - 0x04000000u, eq = (unsigned)__double2hiint(q) - 0x04000000u;
  if (__builtin_expect(max(ep, eq) >= 0x78000000u, 0)) return sqrt_quotient(p, r);  // (also p <= 0 and NaN)
  const double y = rsqrt(q), s = p * y, h = s * r, l = fma(s, r, -h);
  const double e = fma(-s, l, fma(-s, h, p));
  return fma(e, __hiloint2double(__double2hiint(y) - 0x00100000, __double2loint(y)), s);  // s + e y / 2
}
// u - c and u + c, and |u| + c, with c = sqrt(3 p / r), q = sqrt(p / r).  FP64 states its multiply-adds: the branch
// of sqrt_ratio leaves the compiler a choice, and every kernel has to round alike.
__device__ __forceinline__ void acoustic(float u, float q, float &lo, float &hi) {
  const float c = 1.7320508075688772f * q;
  lo = u - c;
  hi = u + c;
}
__device__ __forceinline__ void acoustic(double u, double q, double &lo, double &hi) {
  lo = fma(-1.7320508075688772, q, u);
  hi = fma(1.7320508075688772, q, u);
}
__device__ __forceinline__ float signal_speed(float u, float p, float r) {
  return fabsf(u) + 1.7320508075688772f * sqrt_ratio(p, r);
}
__device__ __forceinline__ double signal_speed(double u, double p, double r) {
  return fma(1.7320508075688772, sqrt_ratio(p, r), fabs(u));
}

// x > 0, x >= 0 and min / max.  FP64: on the bit patterns (integer instructions; the
// double-precision compare runs on the 64-cycle pipe).  A NaN is neither > 0 nor >= 0; the
// min / max of a NaN is unspecified (its flux is NaN whatever they return).
__device__ __forceinline__ bool gt0(float x) { return x > 0.0f; }
__device__ __forceinline__ bool gt0(double x) {
  const long long b = __double_as_longlong(x);
  return b > 0 && b <= 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool ge0(float x) { return x >= 0.0f; }
__device__ __forceinline__ bool ge0(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  return b <= 0x7ff0000000000000ull || b == 0x8000000000000000ull;
}
__device__ __forceinline__ long long order_bits(double x) {  // orders like the numbers
  const long long b = __double_as_longlong(x);
  return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ float min_of(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ float max_of(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double min_of(double a, double b) { return order_bits(a) < order_bits(b) ? a : b; }
__device__ __forceinline__ double max_of(double a, double b) { return order_bits(a) > order_bits(b) ? a : b; }

// Sum and product that are never contracted into a fused multiply-add.  Where an expression
// leaves the compiler a choice of what to fuse, the Roe-type scheme states it, so that every
// kernel it is inlined into rounds alike.
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// ------------------------------------------------------- paired FP32 arithmetic
// Componentwise operations on 10-vectors, d_k = a_k s + c_k (v_fma), d_k = a_k s (v_mul),
// d_k = a_k + b_k (v_add) and d_k = a_k - b_k (v_sub).  In FP32 components (k, k+1) go through the packed f32x2 instructions of sm_100
// (__ffma2_rn, __fadd2_rn: two single-precision operations per issued instruction, each
// rounded as its scalar form); FP64 stays scalar.
template <typename T>
__device__ __forceinline__ void v_fma(T (&d)[NV], const T (&a)[NV], T s, const T (&c)[NV]) {
#pragma unroll
  for (int k = 0; k < NV; k++) d[k] = fma(a[k], s, c[k]);
}
template <>
__device__ __forceinline__ void v_fma<float>(float (&d)[NV], const float (&a)[NV], float s, const float (&c)[NV]) {
  const float2 ss = make_float2(s, s);
#pragma unroll
  for (int k = 0; k < NV; k += 2) {
    const float2 r = __ffma2_rn(make_float2(a[k], a[k + 1]), ss, make_float2(c[k], c[k + 1]));
    d[k] = r.x;
    d[k + 1] = r.y;
  }
}
template <typename T> __device__ __forceinline__ void v_mul(T (&d)[NV], const T (&a)[NV], T s) {
#pragma unroll
  for (int k = 0; k < NV; k++) d[k] = a[k] * s;
}
template <> __device__ __forceinline__ void v_mul<float>(float (&d)[NV], const float (&a)[NV], float s) {
  const float2 ss = make_float2(s, s);
#pragma unroll
  for (int k = 0; k < NV; k += 2) {
    const float2 r = __fmul2_rn(make_float2(a[k], a[k + 1]), ss);
    d[k] = r.x;
    d[k + 1] = r.y;
  }
}
template <typename T> __device__ __forceinline__ void v_add(T (&d)[NV], const T (&a)[NV], const T (&b)[NV]) {
#pragma unroll
  for (int k = 0; k < NV; k++) d[k] = a[k] + b[k];
}
template <>
__device__ __forceinline__ void v_add<float>(float (&d)[NV], const float (&a)[NV], const float (&b)[NV]) {
#pragma unroll
  for (int k = 0; k < NV; k += 2) {
    const float2 r = __fadd2_rn(make_float2(a[k], a[k + 1]), make_float2(b[k], b[k + 1]));
    d[k] = r.x;
    d[k + 1] = r.y;
  }
}
template <typename T> __device__ __forceinline__ void v_sub(T (&d)[NV], const T (&a)[NV], const T (&b)[NV]) {
#pragma unroll
  for (int k = 0; k < NV; k++) d[k] = a[k] - b[k];
}
template <>
__device__ __forceinline__ void v_sub<float>(float (&d)[NV], const float (&a)[NV], const float (&b)[NV]) {
#pragma unroll
  for (int k = 0; k < NV; k += 2) {
    const float2 r = __fadd2_rn(make_float2(a[k], a[k + 1]), make_float2(-b[k], -b[k + 1]));
    d[k] = r.x;
    d[k + 1] = r.y;
  }
}

// ---------------------------------------------------------------- conversions
// E_ij = P_ij + rho u_i u_j (Sec. 2).  The FP32 path recomputes a diagonal dispersion
// in FP64 when the kinetic part cancels more than 99.9 % of E_ii, i.e. where P_ii/rho
// approaches realizability loss.
template <typename T> __device__ __forceinline__ T diag_fix(T P, T E, T m, T rho) { return P; }
template <> __device__ __forceinline__ float diag_fix<float>(float P, float E, float m, float rho) {
  if (P < 1.0e-3f * E) {
    double r = (double)E - (double)m * (double)m / (double)rho;
    return (float)r;
  }
  return P;
}

template <typename T>
__device__ __forceinline__ void cons_to_prim(const T (&U)[NV], T (&W)[NV]) {
  const T rho = U[0];
  const T ir = frcp(rho);
  const T u = U[1] * ir, v = U[2] * ir, w = U[3] * ir;
  W[0] = rho; W[1] = u; W[2] = v; W[3] = w;
  W[4] = diag_fix<T>(U[4] - U[1] * u, U[4], U[1], rho);
  W[5] = U[5] - U[1] * v;
  W[6] = U[6] - U[1] * w;
  W[7] = diag_fix<T>(U[7] - U[2] * v, U[7], U[2], rho);
  W[8] = U[8] - U[2] * w;
  W[9] = diag_fix<T>(U[9] - U[3] * w, U[9], U[3], rho);
}

template <typename T>
__device__ __forceinline__ void prim_to_cons(const T (&W)[NV], T (&U)[NV]) {
  const T rho = W[0];
  const T mx = rho * W[1], my = rho * W[2], mz = rho * W[3];
  U[0] = rho; U[1] = mx; U[2] = my; U[3] = mz;
  U[4] = W[4] + mx * W[1];
  U[5] = W[5] + mx * W[2];
  U[6] = W[6] + mx * W[3];
  U[7] = W[7] + my * W[2];
  U[8] = W[8] + my * W[3];
  U[9] = W[9] + mz * W[3];
}

// rho > 0 and P positive definite by its leading principal minors.
template <typename T> __device__ __forceinline__ bool realizable(const T (&W)[NV]) {
  const T m1 = W[4];
  const T m2 = W[4] * W[7] - W[5] * W[5];
  const T m3 = W[4] * (W[7] * W[9] - W[8] * W[8]) - W[5] * (W[5] * W[9] - W[8] * W[6]) +
               W[6] * (W[5] * W[8] - W[7] * W[6]);
  return gt0(W[0]) && gt0(m1) && gt0(m2) && gt0(m3);
}

// ----------------------------------------------------------- reconstruction
// MC limiter on one characteristic amplitude, halved: for differences of the same sign
//   mc(l, r) / 2 = sign(l) min(|l|, |r|, |l + r| / 4),  else 0
// (mc = sign min(2|l|, |l + r| / 2, 2|r|); the factors are powers of two, so the callers, whose
// coefficients carry the factor 2, get exactly the unscaled result).
// FP32: the clamp of 0 between the smallest and the largest of l, r and q = (l + r) / 4, by the
// three-input minimum and maximum of sm_100: four half-rate instructions per amplitude where
// products, signs and selects took five (measured 7.7 against 9.1 cycles per amplitude).
__device__ __forceinline__ float clamp_zero3(float l, float r, float q) {
  float lo, hi;
  asm("min.f32 %0, %1, %2, %3;\n" : "=f"(lo) : "f"(l), "f"(r), "f"(q));
  asm("max.f32 %0, %1, %2, %3;\n" : "=f"(hi) : "f"(l), "f"(r), "f"(q));
  return fminf(fmaxf(0.0f, lo), hi);
}
// FP64: the signs and the two minima on the bit patterns, so that two double-precision
// instructions are left (the pipe's 64 cycles each; with compares and products the limiter was a
// quarter of a reconstruction's time).  A NaN difference gives 0.
__device__ __forceinline__ double mc_half(double dl, double dr) {
  constexpr long long kAbs = 0x7fffffffffffffffll, kInf = 0x7ff0000000000000ll, kSign = ~kAbs;
  const long long bl = __double_as_longlong(dl), br = __double_as_longlong(dr);
  const long long al = bl & kAbs, ar = br & kAbs;
  const long long lo = al < ar ? al : ar, hi = al < ar ? ar : al;
  const long long q = __double_as_longlong(0.25 * (dl + dr)) & kAbs;
  const bool on = (bl ^ br) >= 0 && lo != 0 && hi <= kInf;
  return __longlong_as_double(on ? ((lo < q ? lo : q) | (bl & kSign)) : 0ll);
}

// The halved limiter on every amplitude of a 10-vector (FP32: q in packed f32x2 instructions).
__device__ __forceinline__ void mc_half_v(const double (&dl)[NV], const double (&dr)[NV], double (&m)[NV]) {
#pragma unroll
  for (int k = 0; k < NV; k++) m[k] = mc_half(dl[k], dr[k]);
}
__device__ __forceinline__ void mc_half_v(const float (&dl)[NV], const float (&dr)[NV], float (&m)[NV]) {
#pragma unroll
  for (int k = 0; k < NV; k += 2) {
    const float2 q = __fmul2_rn(make_float2(0.25f, 0.25f),
                                __fadd2_rn(make_float2(dl[k], dl[k + 1]), make_float2(dr[k], dr[k + 1])));
    m[k] = clamp_zero3(dl[k], dr[k], q.x);
    m[k + 1] = clamp_zero3(dl[k + 1], dr[k + 1], q.y);
  }
}

// Eigen-quantities of the local-frame state w0 shared by projection and back-projection.
template <typename T> struct Eig {
  T rho, u, Pxx, Pxy, Pxz, Pyy, Pyz, Pzz;
  T cf, cs, a, b, ip, icf2, ics2;
  __device__ __forceinline__ void init(const T (&w)[NV]) {
    rho = w[0]; u = w[1];
    Pxx = w[4]; Pxy = w[5]; Pxz = w[6]; Pyy = w[7]; Pyz = w[8]; Pzz = w[9];
    ip = frcp(Pxx);
    const T s = frsqrt(Pxx * rho);       // 1 / sqrt(P_xx rho)
    cs = Pxx * s;                        // sqrt(P_xx / rho)
    const T rs = rho * s;                // 1 / cs
    cf = T(1.7320508075688772) * cs;
    a = Pxy * ip;
    b = Pxz * ip;
    icf2 = T(0.28867513459481287) * rs;  // 1 / (2 cf)
    ics2 = T(0.5) * rs;                  // 1 / (2 cs)
  }
  // characteristic amplitudes c = L d in wave order
  // (f-, sv-, sw-, c_rho, c_yy, c_yz, c_zz, sv+, sw+, f+)
  // t = d_xx / (6 P_xx) is the pressure part of both fast waves; the contact amplitudes take
  // 2 t.  The factors of the cell are formed once for its two projections.
  __device__ __forceinline__ void project(const T (&d)[NV], T (&c)[NV]) const {
    const T ip6 = ip * T(1.0 / 6.0), hip = T(0.5) * ip, r2 = T(2) * rho, a2 = T(2) * a, b2 = T(2) * b;
    const T k4 = T(2) * fma(T(4) * a, Pxy, -Pyy), k5 = T(2) * fma(T(4) * a, Pxz, -Pyz),
            k6 = T(2) * fma(T(4) * b, Pxz, -Pzz);
    const T t = d[4] * ip6;
    c[0] = fma(-d[1], icf2, t);
    c[9] = fma(d[1], icf2, t);
    const T qv = fma(-a, d[1], d[2]), rv = fma(-a, d[4], d[5]) * hip;
    c[1] = fma(-qv, ics2, rv);
    c[7] = fma(qv, ics2, rv);
    const T qw = fma(-b, d[1], d[3]), rw = fma(-b, d[4], d[6]) * hip;
    c[2] = fma(-qw, ics2, rw);
    c[8] = fma(qw, ics2, rw);
    c[3] = fma(-r2, t, d[0]);
    c[4] = fma(k4, t, fma(-a2, d[5], d[7]));
    c[5] = fma(k5, t, fma(-a, d[6], fma(-b, d[5], d[8])));
    c[6] = fma(k6, t, fma(-b2, d[6], d[9]));
  }
  // primitive vector R c
  __device__ __forceinline__ void back(const T (&c)[NV], T (&o)[NV]) const {
    const T A = c[9] + c[0], B = (c[9] - c[0]) * cf;
    const T C = c[7] + c[1], Dv = (c[7] - c[1]) * cs;
    const T E = c[8] + c[2], Fw = (c[8] - c[2]) * cs;
    o[0] = rho * A + c[3];
    o[1] = B;
    o[2] = a * B + Dv;
    o[3] = b * B + Fw;
    o[4] = T(3) * Pxx * A;
    o[5] = T(3) * Pxy * A + Pxx * C;
    o[6] = T(3) * Pxz * A + Pxx * E;
    o[7] = (Pyy + T(2) * a * Pxy) * A + T(2) * Pxy * C + c[4];
    o[8] = (Pyz + T(2) * a * Pxz) * A + Pxz * C + Pxy * E + c[5];
    o[9] = (Pzz + T(2) * b * Pxz) * A + T(2) * Pxz * E + c[6];
  }
  // R c and R (s c), s the wave speeds relative to u (-cf, -cs, -cs, 0 x 4, cs, cs, cf),
  // sharing the wave-pair sums: with A = c_f+ + c_f-, B = (c_f+ - c_f-) cf and so on, the
  // speed-weighted amplitudes give A' = B, B' = cf^2 A (cf^2 = 3 cs^2), C' = Dv, Dv' = cs^2 C,
  // E' = Fw, Fw' = cs^2 E, and no contact amplitudes.
  __device__ __forceinline__ void back2(const T (&c)[NV], T (&o)[NV], T (&os)[NV]) const {
    back(c, o);
    const T A = c[9] + c[0], C = c[7] + c[1], E = c[8] + c[2];
    const T A2 = (c[9] - c[0]) * cf, C2 = (c[7] - c[1]) * cs, E2 = (c[8] - c[2]) * cs;
    const T cs2 = cs * cs;
    const T B2 = T(3) * cs2 * A, D2 = cs2 * C, F2 = cs2 * E;
    os[0] = rho * A2;
    os[1] = B2;
    os[2] = a * B2 + D2;
    os[3] = b * B2 + F2;
    os[4] = T(3) * Pxx * A2;
    os[5] = T(3) * Pxy * A2 + Pxx * C2;
    os[6] = T(3) * Pxz * A2 + Pxx * E2;
    os[7] = (Pyy + T(2) * a * Pxy) * A2 + T(2) * Pxy * C2;
    os[8] = (Pyz + T(2) * a * Pxz) * A2 + Pxz * C2 + Pxy * E2;
    os[9] = (Pzz + T(2) * b * Pxz) * A2 + T(2) * Pxz * E2;
  }
};

// ------------------------------------------------- corner transport upwind
// Transverse term of a cell along direction t for the corner-transport-upwind form of the
// unsplit step (the data reconstruction of Lee & Deane 2009, on which FLASH's unsplit
// MUSCL-Hancock solver of Sec. 3.3 is built; the paper prints none of it): the
// quasi-linear transverse derivative -(dt/2) A_t dW/dx_t taken wave by wave from the
// upwind side,
//   T_t = -nu sum_a lam^a (L^a . dW^a) R^a,   dW^a = w0 - wm if lam^a > 0, else wp - w0,
// nu = dt / (2 dx_t), with the eigen-system of the cell along t (local frame of t).  The
// face states along d take sum_{t != d} T_t before the face-state check.
// cl, cr: the amplitudes L (w0 - wm) and L (wp - w0).
template <typename T>
__device__ __forceinline__ void upwind_terms(const Eig<T> &E, const T (&cl)[NV], const T (&cr)[NV], T nu,
                                             T (&o)[NV]) {
  const T s[NV] = {-E.cf, -E.cs, -E.cs, T(0), T(0), T(0), T(0), E.cs, E.cs, E.cf};
  T c[NV];
#pragma unroll
  for (int k = 0; k < NV; k++) {
    const T lam = E.u + s[k];
    c[k] = -nu * lam * (lam > T(0) ? cl[k] : cr[k]);
  }
  E.back(c, o);
}

template <typename T>
__device__ __forceinline__ void transverse(const T (&wm)[NV], const T (&w0)[NV], const T (&wp)[NV], T nu,
                                           T (&o)[NV]) {
  Eig<T> E;
  E.init(w0);
  T d[NV], cl[NV], cr[NV];
#pragma unroll
  for (int k = 0; k < NV; k++) d[k] = w0[k] - wm[k];
  E.project(d, cl);
#pragma unroll
  for (int k = 0; k < NV; k++) d[k] = wp[k] - w0[k];
  E.project(d, cr);
  upwind_terms(E, cl, cr, nu, o);
}

// Face-state check: if a face state has rho <= 0 or P_nn <= 0 both revert to w0 (first
// order).
template <typename T>
__device__ __forceinline__ void face_state_check(const T (&w0)[NV], T (&lo)[NV], T (&hi)[NV]) {
  const bool ok = gt0(hi[0]) && gt0(lo[0]) && gt0(hi[4]) && gt0(lo[4]);
  if (__builtin_expect(!ok, 0)) {
#pragma unroll
    for (int k = 0; k < NV; k++) { hi[k] = w0[k]; lo[k] = w0[k]; }
  }
}

// Reconstruction of one cell along the sweep direction, in the local frame.
//   wm, w0, wp   primitive states of cells i-1, i, i+1
//   nu           dt / (2 dx)
// Output: face states lo (at i-1/2) and hi (at i+1/2):
//   dw^m = R mc(L dw_L, L dw_R);   w0 -+ dw^m/2 - nu A dw^m,   A dw^m = R Lambda mc(...)
// CTU: both face states also take X (the other directions' transverse terms, local frame;
// xget(k) returns X_k) and the cell's own transverse term along this direction is handed to
// tput(k, T_k) (upwind_terms).  Then the face-state check.  The accessors let a kernel keep
// X and T in shared memory, read and written where they are used.
template <typename T, bool CTU, typename XG, typename TP>
__device__ __forceinline__ void reconstruct(const T (&wm)[NV], const T (&w0)[NV], const T (&wp)[NV], T nu,
                                            T (&lo)[NV], T (&hi)[NV], XG &&xget, TP &&tput) {
  Eig<T> E;
  E.init(w0);
  T d[NV], cl[NV], cr[NV];
  v_sub(d, w0, wm);
  E.project(d, cl);
  v_sub(d, wp, w0);
  E.project(d, cr);
  // limited amplitudes, halved (every quantity below up to the predictor is exactly half its
  // unscaled value, so the face states are bit for bit those of the unscaled form)
  T m[NV];
  mc_half_v(cl, cr, m);
  if constexpr (CTU) {
    T o[NV];
    upwind_terms(E, cl, cr, nu, o);
#pragma unroll
    for (int k = 0; k < NV; k++) tput(k, o[k]);
  }
  T dw[NV], g[NV];
  E.back2(m, dw, g);  // dw^m / 2 (dw^m the limited primitive slope) and (A dw^m - u dw^m) / 2
  // hi, lo = w0 -+ dw^m/2 - nu A dw^m = (w0 - 2 nu g) + (+-1 - 2 nu u) dw^m/2
  const T nu2 = T(2) * nu;
  T base[NV];
  v_fma(base, g, -nu2, w0);
  if constexpr (CTU) {
#pragma unroll
    for (int k = 0; k < NV; k++) base[k] += xget(k);
  }
  v_fma(hi, dw, T(1) - nu2 * E.u, base);
  v_fma(lo, dw, T(-1) - nu2 * E.u, base);
  face_state_check(w0, lo, hi);
}

template <typename T>
__device__ __forceinline__ void reconstruct(const T (&wm)[NV], const T (&w0)[NV], const T (&wp)[NV], T nu,
                                            T (&lo)[NV], T (&hi)[NV]) {
  reconstruct<T, false>(wm, w0, wp, nu, lo, hi, [](int) { return T(0); }, [](int, T) {});
}

// Upwind characteristic tracing for the Roe-type flux (Sec. 3.3, eqs 40-43: reference
// states traced with the fastest wave towards each face, then each wave that reaches the
// face corrected to its own speed; no eq 44-45 terms).  Summed per wave a with amplitude
// c_a = (L dw^m)_a and speed lam_a = u + s_a:
//   hi = w0 + sum_a (1/2 - nu x_a) c_a R^a,   x_a = lam_a if lam_a > 0, else max(u + cf, 0)
//   lo = w0 + sum_a (-1/2 - nu y_a) c_a R^a,  y_a = lam_a if lam_a < 0, else min(u - cf, 0)
// (eq 41 read in the mirror form of eq 40).  Same limiter, transverse terms (CTU) and
// face-state check as reconstruct.
template <typename T, bool CTU, typename XG, typename TP>
__device__ __forceinline__ void reconstruct_upwind(const T (&wm)[NV], const T (&w0)[NV], const T (&wp)[NV],
                                                   T nu, T (&lo)[NV], T (&hi)[NV], XG &&xget, TP &&tput) {
  Eig<T> E;
  E.init(w0);
  T d[NV], cl[NV], cr[NV];
#pragma unroll
  for (int k = 0; k < NV; k++) d[k] = w0[k] - wm[k];
  E.project(d, cl);
#pragma unroll
  for (int k = 0; k < NV; k++) d[k] = wp[k] - w0[k];
  E.project(d, cr);
  // halved limited amplitudes: the coefficients below carry the factor 2
  T m[NV];
  mc_half_v(cl, cr, m);
  if constexpr (CTU) {
    T o[NV];
    upwind_terms(E, cl, cr, nu, o);
#pragma unroll
    for (int k = 0; k < NV; k++) tput(k, o[k]);
  }
  const T u = E.u;
  const T s[NV] = {-E.cf, -E.cs, -E.cs, T(0), T(0), T(0), T(0), E.cs, E.cs, E.cf};
  const T xM = fmax(add_rn(u, E.cf), T(0)), y0 = fmin(add_rn(u, -E.cf), T(0)), nu2 = T(2) * nu;
  T ch[NV], cl2[NV];
#pragma unroll
  for (int k = 0; k < NV; k++) {
    const T lam = add_rn(u, s[k]);
    ch[k] = mul_rn(fma(-nu2, lam > T(0) ? lam : xM, T(1)), m[k]);
    cl2[k] = mul_rn(fma(-nu2, lam < T(0) ? lam : y0, T(-1)), m[k]);
  }
  T dh[NV], dl[NV];
  E.back(ch, dh);
  E.back(cl2, dl);
#pragma unroll
  for (int k = 0; k < NV; k++) {
    T base = w0[k];
    if constexpr (CTU) base += xget(k);
    hi[k] = add_rn(base, dh[k]);
    lo[k] = add_rn(base, dl[k]);
  }
  face_state_check(w0, lo, hi);
}

template <typename T>
__device__ __forceinline__ void reconstruct_upwind(const T (&wm)[NV], const T (&w0)[NV], const T (&wp)[NV],
                                                   T nu, T (&lo)[NV], T (&hi)[NV]) {
  reconstruct_upwind<T, false>(wm, w0, wp, nu, lo, hi, [](int) { return T(0); }, [](int, T) {});
}

// A-posteriori fallback: every face that touches a cell whose second-order update was
// not realizable takes first-order states (the cell-centred primitive state).  fm, f0,
// fp: tags of cells i-1, i, i+1 along the sweep.
template <typename T>
__device__ __forceinline__ void first_order_faces(bool fm, bool f0, bool fp, const T (&w0)[NV], T (&lo)[NV],
                                                  T (&hi)[NV]) {
  if (f0 || fm) {
#pragma unroll
    for (int k = 0; k < NV; k++) lo[k] = w0[k];
  }
  if (f0 || fp) {
#pragma unroll
    for (int k = 0; k < NV; k++) hi[k] = w0[k];
  }
}

// Conserved vector and normal flux of a local-frame primitive state (eqs contin,
// moment, dispers: rho u_n; rho u_i u_n + P_in; E_ij u_n + P_in u_j + P_jn u_i).
template <typename T>
__device__ __forceinline__ void phys(const T (&w)[NV], T (&U)[NV], T (&F)[NV]) {
  const T r = w[0], u = w[1], v = w[2], ww = w[3];
  const T Pxx = w[4], Pxy = w[5], Pxz = w[6], Pyy = w[7], Pyz = w[8], Pzz = w[9];
  const T mx = r * u, my = r * v, mz = r * ww;
  U[0] = r; U[1] = mx; U[2] = my; U[3] = mz;
  U[4] = Pxx + mx * u; U[5] = Pxy + mx * v; U[6] = Pxz + mx * ww;
  U[7] = Pyy + my * v; U[8] = Pyz + my * ww; U[9] = Pzz + mz * ww;
  F[0] = mx;
  F[1] = mx * u + Pxx;
  F[2] = my * u + Pxy;
  F[3] = mz * u + Pxz;
  F[4] = (U[4] + T(2) * Pxx) * u;
  F[5] = (U[5] + Pxy) * u + Pxx * v;
  F[6] = (U[6] + Pxz) * u + Pxx * ww;
  F[7] = U[7] * u + T(2) * Pxy * v;
  F[8] = U[8] * u + Pxy * ww + Pxz * v;
  F[9] = U[9] * u + T(2) * Pxz * ww;
}

// HLL flux between local-frame face states wl | wr with signal speeds
// S_L = min(u_L - cf_L, u_R - cf_R), S_R = max(u_L + cf_L, u_R + cf_R).
// The difference U_R - U_L is formed first, so that its term vanishes between equal states; with
// U_L and U_R weighted separately FP64 saves 14 of 98 operations (3 % of a step), but the mass flux
// through a wall or in a gas at rest is then a rounding error of c rho instead of zero.
template <typename T>
__device__ __forceinline__ void hll(const T (&wl)[NV], const T (&wr)[NV], T (&F)[NV]) {
  T lo_l, hi_l, lo_r, hi_r;
  acoustic(wl[1], sqrt_ratio(wl[4], wl[0]), lo_l, hi_l);
  acoustic(wr[1], sqrt_ratio(wr[4], wr[0]), lo_r, hi_r);
  const T SL = min_of(lo_l, lo_r), SR = max_of(hi_l, hi_r);
  // F = a Fl + b Fr + c (Ur - Ul): (1, 0, 0) for SL >= 0, (0, 1, 0) for SR <= 0, else
  // (SR, -SL, SL SR) / (SR - SL); the branch selects three scalars, not ten fluxes
  T a, b, c;
  if (ge0(SL)) {
    a = T(1); b = T(0); c = T(0);
  } else if (ge0(-SR)) {
    a = T(0); b = T(1); c = T(0);
  } else {
    const T inv = frcp(SR - SL);
    a = SR * inv;
    b = -SL * inv;
    c = SL * SR * inv;
  }
  T Ul[NV], Fl[NV], Ur[NV], Fr[NV], t[NV];
  phys(wl, Ul, Fl);
  phys(wr, Ur, Fr);
  v_sub(t, Ur, Ul);
  v_mul(t, t, c);
  v_fma(t, Fr, b, t);
  v_fma(F, Fl, a, t);
}

// ------------------------------------------------------- Kurganov-Tadmor
// Face values of one cell for the central scheme of Sec. 3.2 (local frame): primitive
// variables reconstructed component by component with the MC limiter (w0 -+ mc/2); a face value with rho <= 0 or P_nn <= 0 reverts both
// faces to w0.
template <typename T>
__device__ __forceinline__ void kt_reconstruct(const T (&wm)[NV], const T (&w0)[NV], const T (&wp)[NV],
                                               T (&lo)[NV], T (&hi)[NV]) {
  T dl[NV], dr[NV], s[NV];
  v_sub(dl, w0, wm);
  v_sub(dr, wp, w0);
  mc_half_v(dl, dr, s);
  v_add(hi, w0, s);
  v_sub(lo, w0, s);
  face_state_check(w0, lo, hi);
}

// Central flux H = (f(wl) + f(wr))/2 - a (U(wr) - U(wl))/2 through a face with the value wl
// on its left side and wr on its right side; a = the larger spectral radius of df/du,
// |u_n| + sqrt(3 P_nn / rho), of the two (eqs spectralfreq, soundspeed with gamma = 3).
template <typename T>
__device__ __forceinline__ void kt_flux(const T (&wl)[NV], const T (&wr)[NV], T (&F)[NV]) {
  const T al = signal_speed(wl[1], wl[4], wl[0]), ar = signal_speed(wr[1], wr[4], wr[0]);
  const T h = T(0.5) * fmax(al, ar);
  T Ul[NV], Fl[NV], Ur[NV], Fr[NV];  // after the speeds' branches, so that it rounds alike everywhere
  phys(wl, Ul, Fl);
  phys(wr, Ur, Fr);
  T dU[NV], Fs[NV];
  v_sub(dU, Ur, Ul);
  v_add(Fs, Fl, Fr);
  v_mul(Fs, Fs, T(0.5));
  v_fma(F, dU, -h, Fs);
}

// ------------------------------------------------------------ Roe-type flux
// Linearised characteristic upwind flux (local frame):
//   F = (f(wl) + f(wr)) / 2 - (dU/dW)(wm) R |Lambda| L (wr - wl) / 2,
// with wm = (wl + wr) / 2 (no Roe average is known for the ten-moment system), the
// closed-form eigen-system of wm, and Harten's entropy fix on the two fast waves only:
// |lambda| -> (lambda^2 + delta^2) / (2 delta) below delta = cf / 10.  The shear and contact
// waves are linearly degenerate and keep |lambda|, so a stationary contact is not diffused.
template <typename T>
__device__ __forceinline__ void roe_flux(const T (&wl)[NV], const T (&wr)[NV], T (&F)[NV]) {
  T wm[NV], dw[NV];
#pragma unroll
  for (int k = 0; k < NV; k++) {
    wm[k] = mul_rn(T(0.5), wl[k] + wr[k]);
    dw[k] = wr[k] - wl[k];
  }
  Eig<T> E;
  E.init(wm);
  T c[NV];
  E.project(dw, c);
  const T u = E.u, delta = T(0.1) * E.cf;
  auto fast = [&](T l) {
    const T al = fabs(l);
    return al < delta ? mul_rn(fma(l, l, mul_rn(delta, delta)), mul_rn(T(0.5), frcp(delta))) : al;
  };
  const T am = fabs(add_rn(u, -E.cs)), ap = fabs(add_rn(u, E.cs)), a0 = fabs(u);
  const T w[NV] = {fast(add_rn(u, -E.cf)), am, am, a0, a0, a0, a0, ap, ap, fast(add_rn(u, E.cf))};
#pragma unroll
  for (int k = 0; k < NV; k++) c[k] = mul_rn(c[k], w[k]);
  T d[NV];
  E.back(c, d);  // primitive dissipation R |Lambda| L dw
  const T r = wm[0], ux = wm[1], uy = wm[2], uz = wm[3];
  T dU[NV];      // through the Jacobian of the conserved map at wm
  dU[0] = d[0];
  const T vx = mul_rn(d[0], ux), vy = mul_rn(d[0], uy), vz = mul_rn(d[0], uz);
  dU[1] = fma(r, d[1], vx);
  dU[2] = fma(r, d[2], vy);
  dU[3] = fma(r, d[3], vz);
  dU[4] = fma(r, mul_rn(T(2) * d[1], ux), fma(vx, ux, d[4]));
  dU[5] = fma(r, fma(d[1], uy, mul_rn(ux, d[2])), fma(vx, uy, d[5]));
  dU[6] = fma(r, fma(d[1], uz, mul_rn(ux, d[3])), fma(vx, uz, d[6]));
  dU[7] = fma(r, mul_rn(T(2) * d[2], uy), fma(vy, uy, d[7]));
  dU[8] = fma(r, fma(d[2], uz, mul_rn(uy, d[3])), fma(vy, uz, d[8]));
  dU[9] = fma(r, mul_rn(T(2) * d[3], uz), fma(vz, uz, d[9]));
  T Ul[NV], Fl[NV], Ur[NV], Fr[NV];
  phys(wl, Ul, Fl);
  phys(wr, Ur, Fr);
  T Fs[NV];
  v_add(Fs, Fl, Fr);
  v_sub(Fs, Fs, dU);
  v_mul(F, Fs, T(0.5));
}

// ------------------------------------------------------------------- HLLC
// The part Pi of the normal flux F = u U + Pi (local frame) that depends only on the
// quantities continuous across a contact, u_i and P_ix:
//   Pi = (0; P_ix; P_ix u_j + P_jx u_i).
template <typename T>
__device__ __forceinline__ void pi_terms(T u, T v, T w, T pxx, T pxy, T pxz, T (&P)[NV]) {
  P[0] = T(0);
  P[1] = pxx;
  P[2] = pxy;
  P[3] = pxz;
  P[4] = T(2) * pxx * u;
  P[5] = pxy * u + pxx * v;
  P[6] = pxz * u + pxx * w;
  P[7] = T(2) * pxy * v;
  P[8] = pxy * w + pxz * v;
  P[9] = T(2) * pxz * w;
}

// Three-wave HLLC flux for the ten-moment system (local frame).  Outer waves S_L, S_R as in
// HLL (they carry the fast and shear waves), the contact S_M in between (it carries rho and
// the transverse stresses).  Every pair (u_i, P_ix) takes one star value on both sides of
// the contact, from the momentum jump conditions across S_L and S_R with C_K = rho_K
// (S_K - u_K):  u*_i = (C_R u_i,R - C_L u_i,L - (P_ix,R - P_ix,L)) / (C_R - C_L),
// P*_ix = P_ix,L + C_L (u*_i - u_i,L);  S_M = u*_x.  The star state of side K follows from
// the jump conditions across S_K, U*_K = (U_K (S_K - u_K) + Pi* - Pi_K) / (S_K - S_M), so
// the flux F_K + S_K (U*_K - U_K) of the side of the face that holds x/t = 0 is
//   F = a U_K + b Pi_K + c Pi*,  (a, b, c) = (S_M (S_K - u_K), -S_M, S_K) / (S_K - S_M),
// or (u_K, 1, 0) (the physical flux) when both waves move away from the face.  Where S_M is
// not strictly inside (S_L, S_R) the flux is HLL's.
template <typename T>
__device__ __forceinline__ void hllc_flux(const T (&wl)[NV], const T (&wr)[NV], T (&F)[NV]) {
  T lo_l, hi_l, lo_r, hi_r;
  acoustic(wl[1], sqrt_ratio(wl[4], wl[0]), lo_l, hi_l);
  acoustic(wr[1], sqrt_ratio(wr[4], wr[0]), lo_r, hi_r);
  const T SL = min_of(lo_l, lo_r), SR = max_of(hi_l, hi_r);
  const T CL = wl[0] * (SL - wl[1]), CR = wr[0] * (SR - wr[1]);
  const T inv = frcp(CR - CL);
  T us[3], ps[3];
#pragma unroll
  for (int i = 0; i < 3; i++) {
    us[i] = (CR * wr[1 + i] - CL * wl[1 + i] - (wr[4 + i] - wl[4 + i])) * inv;
    ps[i] = wl[4 + i] + CL * (us[i] - wl[1 + i]);
  }
  const T SM = us[0];
  if (!(SL < SM && SM < SR)) {
    hll(wl, wr, F);
    return;
  }
  const bool left = ge0(SM);
  T wk[NV];
#pragma unroll
  for (int k = 0; k < NV; k++) wk[k] = left ? wl[k] : wr[k];
  const T SK = left ? SL : SR, uk = wk[1];
  T a, b, c;
  if (ge0(SL) || ge0(-SR)) {
    a = uk; b = T(1); c = T(0);
  } else {
    const T i2 = frcp(SK - SM);
    a = SM * (SK - uk) * i2;
    b = -SM * i2;
    c = SK * i2;
  }
  T Uk[NV], Fk[NV], Pk[NV], Ps[NV];
  phys(wk, Uk, Fk);
  pi_terms(wk[1], wk[2], wk[3], wk[4], wk[5], wk[6], Pk);
  pi_terms(us[0], us[1], us[2], ps[0], ps[1], ps[2], Ps);
  T t[NV];
  v_mul(t, Ps, c);
  v_fma(t, Pk, b, t);
  v_fma(F, Uk, a, t);
}

// Scheme of a step kernel: 0 the characteristic MUSCL-Hancock step with HLL (Sec. 3.3);
// 1 and 2 the two Runge-Kutta stages of the Kurganov-Tadmor scheme (Sec. 3.2); 3 the
// characteristic step with upwind tracing and the Roe-type flux; 4 the characteristic step
// with the HLLC flux.  0, 3 and 4 have the a-posteriori fallback.
template <int SCH> constexpr bool kCharacteristic = SCH == 0 || SCH == 3 || SCH == 4;

template <int SCH, typename T>
__device__ __forceinline__ void recon(const T (&wm)[NV], const T (&w0)[NV], const T (&wp)[NV], T nu, T (&lo)[NV],
                                      T (&hi)[NV]) {
  if constexpr (SCH == 0 || SCH == 4) reconstruct(wm, w0, wp, nu, lo, hi);
  else if constexpr (SCH == 3) reconstruct_upwind(wm, w0, wp, nu, lo, hi);
  else kt_reconstruct(wm, w0, wp, lo, hi);
}

// The characteristic schemes' reconstruction with the transverse terms X (local frame,
// xget(k) = X_k) in the face states; the cell's own transverse term along the sweep goes to
// tput(k, T_k).
template <int SCH, typename T, typename XG, typename TP>
__device__ __forceinline__ void recon_ctu(const T (&wm)[NV], const T (&w0)[NV], const T (&wp)[NV], T nu,
                                          XG &&xget, TP &&tput, T (&lo)[NV], T (&hi)[NV]) {
  static_assert(kCharacteristic<SCH>, "transverse terms belong to the characteristic schemes");
  if constexpr (SCH == 3) reconstruct_upwind<T, true>(wm, w0, wp, nu, lo, hi, xget, tput);
  else reconstruct<T, true>(wm, w0, wp, nu, lo, hi, xget, tput);
}

template <int SCH, typename T>
__device__ __forceinline__ void face_flux(const T (&wl)[NV], const T (&wr)[NV], T (&F)[NV]) {
  if constexpr (SCH == 0) hll(wl, wr, F);
  else if constexpr (SCH == 3) roe_flux(wl, wr, F);
  else if constexpr (SCH == 4) hllc_flux(wl, wr, F);
  else kt_flux(wl, wr, F);
}

// Flux through a face in a step pass: in a fallback pass (RETRY) a face with first-order
// states (it touches a tagged cell) takes HLL under the Roe-type and HLLC schemes too.  The
// fallback has to make the update realizable; HLL with bounding wave speeds is positively
// conservative, a linearised Roe flux is not (Einfeldt, Munz, Roe & Sjogreen 1991), and
// HLLC's star states, formed from jump conditions, need not be realizable.
template <int SCH, bool RETRY, typename T>
__device__ __forceinline__ void face_flux(const T (&wl)[NV], const T (&wr)[NV], bool first, T (&F)[NV]) {
  if constexpr ((SCH == 3 || SCH == 4) && RETRY) {
    if (first) hll(wl, wr, F);
    else face_flux<SCH>(wl, wr, F);
  } else {
    face_flux<SCH>(wl, wr, F);
  }
}

// float -> double on the bit patterns: a conversion instruction holds the 64-cycle FP64 pipe, and
// the totals convert ten values per cell or thread.  Denormals, infinities and NaNs convert.
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) {
  const unsigned b = __float_as_uint(x), a = b & 0x7fffffffu;
  if (a - 0x00800000u < 0x7f000000u)  // normal
    return __hiloint2double((int)((b & 0x80000000u) | ((a >> 3) + 0x38000000u)), (int)(b << 29));
  return a == 0u ? __hiloint2double((int)b, 0) : (double)x;
}

// ---------------------------------------------------------- accumulators
// Per-thread running sums of the conserved totals over the cells one thread updates.  FP64
// states add in FP64.  FP32 states add in FP32 per thread (relative rounding error of a
// k-term sum below k 2^-24, random in sign across threads), in pairs of floats over a warp
// (warp_sum10) and in FP64 from there on, so the totals need no FP64 arithmetic per cell (FP64 throughput is a small
// fraction of FP32 on this GPU).  The 3D step moves a thread's FP32 sum into FP64 block
// totals every 64 planes of a stretch and at its end, so one FP32 sum spans at most 64
// cells; 2D strips and 1D tiles stream one chunk.
template <typename T> struct Acc {
  using Sum = double;  // what a thread hands to the warp's sum
  double v[NV];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int k = 0; k < NV; k++) v[k] = 0.0;
  }
  __device__ __forceinline__ void add(const T (&x)[NV]) {
#pragma unroll
    for (int k = 0; k < NV; k++) v[k] += x[k];
  }
  __device__ __forceinline__ void get(double (&o)[NV]) const {
#pragma unroll
    for (int k = 0; k < NV; k++) o[k] = v[k];
  }
};
template <> struct Acc<float> {
  using Sum = float;
  float v[NV];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int k = 0; k < NV; k++) v[k] = 0.f;
  }
  __device__ __forceinline__ void add(const float (&x)[NV]) {
#pragma unroll
    for (int k = 0; k < NV; k += 2) {
      const float2 r = __fadd2_rn(make_float2(v[k], v[k + 1]), make_float2(x[k], x[k + 1]));
      v[k] = r.x;
      v[k + 1] = r.y;
    }
  }
  __device__ __forceinline__ void get(float (&o)[NV]) const {
#pragma unroll
    for (int k = 0; k < NV; k++) o[k] = v[k];
  }
};

// ------------------------------------------------------------- boundaries
enum { BC_PERIODIC = 0, BC_OUTFLOW = 1, BC_REFLECT = 2 };

// Map a (possibly ghost) index onto the grid.  mirror = reflect image.  The result is
// clamped into [0, n) so that tile overhang beyond the ghost layers stays in bounds.
__device__ __forceinline__ int map_index(int i, int n, int bclo, int bchi, bool &mirror) {
  mirror = false;
  if (i < 0) {
    if (bclo == BC_PERIODIC) i += n;
    else if (bclo == BC_OUTFLOW) i = 0;
    else { i = -1 - i; mirror = true; }
  } else if (i >= n) {
    if (bchi == BC_PERIODIC) i -= n;
    else if (bchi == BC_OUTFLOW) i = n - 1;
    else { i = 2 * n - 1 - i; mirror = true; }
  }
  return min(max(i, 0), n - 1);
}

// Sign flips of a mirrored image across a face normal to d: m_d and E_dt (t != d).
__device__ __forceinline__ unsigned flip_mask(int d) {
  return d == 0 ? ((1u << 1) | (1u << 5) | (1u << 6))
       : d == 1 ? ((1u << 2) | (1u << 5) | (1u << 8))
                : ((1u << 3) | (1u << 6) | (1u << 8));
}

}  // namespace msh
