// Device-side building blocks of the coupled step: D2Q9 lattice, Peng-Robinson EOS, boundary
// closures, moment transforms and the two MRT collisions. Every kernel of liblbpc composes these,
// so that the split and fused kernels compute the same arithmetic.
//
// D2Q9 order: e0=(0,0) e1=(1,0) e2=(0,1) e3=(-1,0) e4=(0,-1) e5=(1,1) e6=(-1,1) e7=(-1,-1) e8=(1,-1);
// weights 4/9, 1/9, 1/36 (Sec. II B). Moments (rho, e, eps, jx, qx, jy, qy, pxx, pxy): the orthogonal
// MRT basis of Eqs. 42-43, whose thermal equilibria are Eq. 53.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>
#include <string.h>

#include "lbpc_dw.cuh"

namespace lbpc {

enum { BC_PERIODIC = 0, BC_WALL = 1, BC_PRESSURE = 2 };
enum { ST_RHO_LE0 = 1, ST_RHO_POLE = 2, ST_T_LE0 = 3, ST_PSI2_NEG = 4, ST_NONFINITE = 5, ST_TIMEOUT = 6 };

__host__ __device__ constexpr int EX(int a) { return a == 1 || a == 5 || a == 8 ? 1 : (a == 3 || a == 6 || a == 7 ? -1 : 0); }
__host__ __device__ constexpr int EY(int a) { return a == 2 || a == 5 || a == 6 ? 1 : (a == 4 || a == 7 || a == 8 ? -1 : 0); }

// Real-valued parameters in the arithmetic type of a kernel, folded on the host, so that a kernel
// never converts between FP64 and FP32 (on GB300 those conversions run at the FP64 rate).
//
// The flow relaxation in the form each arithmetic uses. Binary32 takes it in increments with the rates as
// they are. Binary64 and double-word arithmetic, whose step is bound by the number of such operations, take
// it with the back-transform's scale c of each moment folded in: c = (1/36, 1/36, 1/12, 1/12, 1/4, 1/4) for the
// moments (e, eps, qx, qy, pxx, pxy).
template <class R> struct FlowRates {
  R s_f[9];
  R hf[9];      // 1 - s_f[k]/2, the forcing weights of (I - Lambda/2) S_F
};
template <class R> struct FoldedFlowRates {
  R A[6], H[6];  // (1 - s) c, (1 - s/2) c; H[4] (pxx) carries the factor 2 of its S_F
  R B[4];        // s c of qx, qy, pxx, pxy
  R E[2];        // 3 s c of e and eps: the weights of rho v^2 in their equilibria
  R w0, wa, wd;  // weights of rho in f0, in f1..f4 and in f5..f8 that the zeroth moment and those equilibria add
  // further constants of these steps, with the scales of the unscaled differences (12 grad, 6 lap) folded in
  R kappa1, kappa_Tc;           // 1 + kappa, kappa / T_c
  R G12, qG144, inv_cV12;       // -G/12, qG2/144, 1/(12 c_V)
  R lambda2, kdiff6, chi6, chi144;  // 2 lambda, kdiff/6, (chi - kdiff)/6, chi/144
};
template <> struct FlowRates<double> : FoldedFlowRates<double> {};
template <> struct FlowRates<dw> : FoldedFlowRates<dw> {};

template <class R> struct Coefs {
  R T_bc[4], T_strip;
  R rho_bc_lo, rho_bc_hi;
  R a, b, R_gas, G, kappa;
  R s_g[9];
  FlowRates<R> flow;
  R lambda, chi, cV, kdiff;  // kdiff = (1/s_g3 - 1/2) c_s^2
  R gx, gy, G_wall;
  R c3, c5;     // (1 - s3/2) s4, (1 - s5/2) s6 of Eqs. 54-55
  R inv_Tc;     // 1 / T_c
  R qG2;        // 12 sigma / (1/s_e - 1/2) * G^2: Q = qcoef |F_int|^2 / psi^2 = qG2 |sum_a w psi e|^2
  R inv_cV;     // 1 / c_V
  R psi_scale;  // 2 / G: psi^2 = (2/G) (p - rho c_s^2)
  R cV_chi;     // c_V chi
  R wf[9];      // rest-state equilibrium weights of f: M^{-1} m_eq(1, v = 0) = (4/9, 1/9 x4, 1/36 x4)
  R wg[9];      // rest-state equilibrium weights of g: M^{-1} m_eq(T = 1, v = 0) of the thermal model
};

// Everything a kernel needs, derived once on the host from lbpc_params and passed by value. The
// coefficient sets start on 16-byte boundaries so that a kernel can copy the header and the one set
// it uses with 16-byte asynchronous copies.
struct alignas(16) DevParams {
  int nx, ny;
  long long N;       // pitch * ny: elements of a plane, the stride between planes
  int yper;          // y periodic
  int ybc_lo, ybc_hi;
  int tbc[4];
  int strip_x0, strip_x1;
  int model;         // 0 improved, 1 compromised
  int lambda_mode;   // 0 const, 1 rho cV chi
  int buoyancy;
  int heat_unit_rates;  // s_g[1..8] all 1: the thermal relaxation sets every non-conserved moment to m_eq
  int pitch;         // elements of a stored row: nx, or nx rounded up to whole 16-byte pieces (row_pitch)
  alignas(16) Coefs<double> cd;
  alignas(16) Coefs<float> cf;
  alignas(16) Coefs<dw> cw;  // double-word arithmetic (LBPC_DF64)
};

template <class R> __host__ __device__ __forceinline__ const Coefs<R>& coefs(const DevParams& P);
template <> __host__ __device__ __forceinline__ const Coefs<double>& coefs<double>(const DevParams& P) { return P.cd; }
template <> __host__ __device__ __forceinline__ const Coefs<float>& coefs<float>(const DevParams& P) { return P.cf; }
template <> __host__ __device__ __forceinline__ const Coefs<dw>& coefs<dw>(const DevParams& P) { return P.cw; }

// The header of DevParams with the one coefficient set of arithmetic R: what a kernel of that arithmetic
// reads, in a third of the bytes, for parameters that are copied per launch (the batch's per-tile
// launches). The device helpers take either form (template parameter PT).
template <class R> struct alignas(16) DevParamsOf {
  int nx, ny;
  long long N;
  int yper;
  int ybc_lo, ybc_hi;
  int tbc[4];
  int strip_x0, strip_x1;
  int model;
  int lambda_mode;
  int buoyancy;
  int heat_unit_rates;
  int pitch;
  alignas(16) Coefs<R> c;
};
static_assert(offsetof(DevParamsOf<float>, c) == offsetof(DevParams, cd) &&
                  offsetof(DevParamsOf<float>, pitch) == offsetof(DevParams, pitch),
              "DevParamsOf repeats the header of DevParams");
template <class R> __host__ __device__ __forceinline__ const Coefs<R>& coefs(const DevParamsOf<R>& P) { return P.c; }
template <class R> inline DevParamsOf<R> params_of(const DevParams& P) {
  DevParamsOf<R> q;
  memcpy(&q, &P, offsetof(DevParams, cd));  // the common header
  q.c = coefs<R>(P);
  return q;
}

// First call of every kernel launched with launch_pdl, by every thread, before it reads or writes device memory:
// wait until all earlier work of the stream is complete and visible. Returns threadIdx.x (NTH: the block's
// threads, a power of two), read after the wait: addresses formed from it cannot be loaded from before the wait,
// not even by read-only loads, which the compiler may otherwise move across it.
template <int NTH> __device__ __forceinline__ int pdl_wait() {
  static_assert((NTH & (NTH - 1)) == 0, "power of two");
  int t;
  asm volatile("griddepcontrol.wait;\n mov.u32 %0, %%tid.x;" : "=r"(t)::"memory");
  return t & (NTH - 1);
}
// A value that an earlier kernel of the stream wrote, at an address that no thread index enters.
__device__ __forceinline__ double load_after_wait(const double* p) { return *(const volatile double*)p; }

// ------------------------------------------------------------------------------------------------
// moment transforms: m = M x and x = M^{-1} m with M^{-1} = M^T diag(1/9,1/36,1/36,1/6,1/12,1/6,1/12,1/4,1/4)
// ------------------------------------------------------------------------------------------------
template <class R> __device__ __forceinline__ void to_moments(const R x[9], R m[9]) {
  const R s14 = x[1] + x[2] + x[3] + x[4];
  const R s58 = x[5] + x[6] + x[7] + x[8];
  const R d13 = x[1] - x[3], d24 = x[2] - x[4];
  const R px = x[5] - x[6] - x[7] + x[8];
  const R py = x[5] + x[6] - x[7] - x[8];
  m[0] = x[0] + s14 + s58;
  m[1] = x[0] * -4 - s14 + s58 * 2;
  m[2] = x[0] * 4 - s14 * 2 + s58;
  m[3] = d13 + px;
  m[4] = d13 * -2 + px;
  m[5] = d24 + py;
  m[6] = d24 * -2 + py;
  m[7] = x[1] - x[2] + x[3] - x[4];
  m[8] = x[5] - x[6] + x[7] - x[8];
}

template <class R> __device__ __forceinline__ void from_moments(const R m[9], R x[9]) {
  const R u0 = m[0] * R(1.0 / 9.0), u1 = m[1] * R(1.0 / 36.0), u2 = m[2] * R(1.0 / 36.0);
  const R u3 = m[3] * R(1.0 / 6.0), u4 = m[4] * R(1.0 / 12.0), u5 = m[5] * R(1.0 / 6.0);
  const R u6 = m[6] * R(1.0 / 12.0), u7 = m[7] * R(0.25), u8 = m[8] * R(0.25);
  const R ax = u0 - u1 - u2 * 2;  // common to e1..e4
  const R dg = u0 + u1 * 2 + u2;  // common to e5..e8
  const R qx = u3 - u4 * 2, qy = u5 - u6 * 2;
  const R sx = u3 + u4, sy = u5 + u6;
  x[0] = u0 - u1 * 4 + u2 * 4;
  x[1] = ax + qx + u7;
  x[2] = ax + qy - u7;
  x[3] = ax - qx + u7;
  x[4] = ax - qy - u7;
  x[5] = dg + sx + sy + u8;
  x[6] = dg - sx + sy - u8;
  x[7] = dg - sx - sy + u8;
  x[8] = dg + sx - sy - u8;
}

// x = M^{-1} m for the post-collision populations. In binary32 arithmetic the rest population is taken
// as x0 = m0 - (x1 + ... + x8), so that the populations sum to the zeroth moment up to one rounding:
// the scale 1/9 of m0 rounds up by 7.5e-9 in binary32, and the plain transform would scale each node's
// mass (or heat) by 9 fl(1/9) in every collision, a steady drift of about 1e-8 per step. In binary64
// and double-word arithmetic that drift is about 5e-17 per step, and the plain transform is kept (the
// double-word type's lazy additions lose accuracy in the longer sum).
template <class R> __device__ __forceinline__ void from_moments_conserving(const R m[9], R x[9]) {
  from_moments(m, x);
  if constexpr (sizeof(R) == 4) x[0] = m[0] - (((x[1] + x[2]) + (x[3] + x[4])) + ((x[5] + x[6]) + (x[7] + x[8])));
}

// Reciprocal and roots. Binary32 takes the hardware's approximations without the compiler's handling of
// subnormal and huge arguments (a test, a select and two products each, about 4 % of the fused step's
// instructions): the same bits for normal arguments, and a state with others is outside the equation of state's range.
template <class R> __device__ R inverse_of(R x);  // float, double and dw
template <> __device__ __forceinline__ float inverse_of<float>(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float inverse_root_of(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ------------------------------------------------------------------------------------------------
// Peng-Robinson EOS (Eq. 56) and (dp/dT)_rho
// ------------------------------------------------------------------------------------------------
// In binary32 (eos_psi_squared: the wider types).
template <class R, class PT> __device__ __forceinline__ void eos(R rho, R T, const PT& P, R& p, R& dpdT, R* inv_rho = nullptr) {
  static_assert(sizeof(R) == 4, "binary32");
  const Coefs<R>& C = coefs<R>(P);
  // theta(T) = [1 + kappa (1 - sqrt(T/T_c))]^2 and d theta/dT = -kappa [..] / sqrt(T T_c); one rsqrt
  // gives both sqrt(T/T_c) = t rsqrt(t) and 1/sqrt(T T_c) = rsqrt(t) / T_c with t = T/T_c.
  const R t = T * C.inv_Tc;
  const R rs = inverse_root_of(t);
  const R sq = t * rs;
  const R th1 = R(1) + C.kappa * (R(1) - sq);
  const R theta = th1 * th1;
  const R dtheta = -C.kappa * th1 * rs * C.inv_Tc;
  // 1/(1 - b rho) and 1/(1 + 2 b rho - b^2 rho^2) (and 1/rho if asked) from one reciprocal
  const R br = C.b * rho;
  const R d1 = R(1) - br;
  const R d2 = R(1) + br * 2 - br * br;
  const R d12 = d1 * d2;
  R r12;
  if (inv_rho) {
    const R r = inverse_of(rho * d12);
    *inv_rho = d12 * r;
    r12 = rho * r;
  } else {
    r12 = inverse_of(d12);
  }
  const R inv1 = d2 * r12, inv2 = d1 * r12;
  const R r2 = rho * rho;
  p = rho * C.R_gas * T * inv1 - C.a * theta * r2 * inv2;
  dpdT = rho * C.R_gas * inv1 - C.a * dtheta * r2 * inv2;
}

template <> __device__ __forceinline__ dw inverse_of<dw>(dw x) {  // binary32 reciprocal, corrected once
  x = dw_norm(x);
  const float r = __frcp_rn(x.hi);
  const dw p = dw_two_prod(r, x.hi);
  const float d = __fsub_rn(__fsub_rn(__fsub_rn(1.0f, p.hi), p.lo), __fmul_rn(r, x.lo));  // 1 - r x
  return dw_fast_two_sum(r, __fmul_rn(d, r));
}
// Binary64 reciprocal and roots from the hardware's approximations, which see and give the upper 32 bits of a number,
// by one step of the third-order iteration (Householder 1970; for the reciprocal, r (1 + e + e^2) with
// e = 1 - x r). |e| is at most 2^-18 by those two truncations (over 2^-1000 to 2^1000 measured 2^-19.98 for the reciprocal,
// 2^-19.06 for the root's 1 - x y^2), so the step leaves e^3 <= 2^-54, or 5/16 of that for the roots, of a last place of 2^-53
// or more. With the roundings 1/x is within 1 ulp (measured 0.501), sqrt(x) within 1 (0.744) and 1/sqrt(x) within 1.25
// (0.922); CUDA states 0.5, 0.5 and 1 for its own, which take more than these 3 and 5 operations of the pipe that bounds
// the step. Arguments are normal numbers here (a state outside the equation of state's range is reported by classify,
// whatever these return for it).
template <> __device__ __forceinline__ double inverse_of<double>(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
// 1/sqrt(x) and sqrt(x) of x > 0
__device__ __forceinline__ void roots_of(double x, double& inv_root, double& root) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double s = x * y;
  const double e = fma(-s, y, 1.0);
  const double pe = fma(0.375, e, 0.5) * e;
  inv_root = fma(pe, y, y);
  root = fma(pe, s, s);
}
__device__ __forceinline__ void roots_of(dw x, dw& inv_root, dw& root) {
  inv_root = rsqrt(x);
  root = x * inv_root;
}
// psi = sqrt(max(psi^2, 0)), a NaN counting as 0; the tests of the binary64 form run on the integer pipe.
template <class R> __device__ __forceinline__ R psi_of(R psi2) { return sqrt(fmax(psi2, R(0))); }
template <> __device__ __forceinline__ float psi_of<float>(float psi2) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(::fmaxf(psi2, 0.0f)));
  return y;
}
template <> __device__ __forceinline__ double psi_of<double>(double psi2) {
  const long long b = __double_as_longlong(psi2);
  double inv_root, root;
  roots_of(psi2, inv_root, root);
  return b >= 0x0010000000000000LL && b < 0x7ff0000000000000LL ? root : (b == 0x7ff0000000000000LL ? psi2 : 0.0);
}
// eos and psi^2 for binary64 and double-word arithmetic, arranged for the fewest operations (their step is bound by
// the arithmetic pipe): psi^2, (dp/dT)_rho and 1/rho from one reciprocal and one reciprocal square root.
// With u = rho R / (1 - b rho), A = a rho^2 / (1 + 2 b rho - b^2 rho^2) and h = 1 + kappa (1 - sqrt(T/T_c)):
// p = u T - A h^2 and dp/dT = u + A h kappa / sqrt(T T_c).
template <class R, class PT>
__device__ __forceinline__ R eos_psi_squared(R rho, R T, const PT& P, R& dpdT, R& inv_rho) {
  const Coefs<R>& C = coefs<R>(P);
  const R t = T * C.inv_Tc;
  R rs, sq;
  roots_of(t, rs, sq);
  const R h = C.flow.kappa1 - C.kappa * sq;
  const R br = C.b * rho;
  const R d1 = R(1) - br;
  const R d2 = br * (R(2) - br) + R(1);
  const R d12 = d1 * d2;
  const R r = inverse_of(rho * d12);
  inv_rho = d12 * r;
  const R z = rho * (rho * r);  // rho / d12
  const R u = (d2 * z) * C.R_gas;
  const R Ah = ((C.a * rho) * (d1 * z)) * h;
  dpdT = u + (Ah * rs) * C.flow.kappa_Tc;
  const R p = u * T - Ah * h;
  return C.psi_scale * (p - rho * R(1.0 / 3.0));
}

// ------------------------------------------------------------------------------------------------
// zeroth moments and the pseudopotential in binary32
// ------------------------------------------------------------------------------------------------
// In binary32 a plain sum of nine populations rounds up to eight times at the scale of the result.
// Near rest the populations stand in fixed ratios to the rest population (D2Q9 flow weights: f_a = f0/4
// on the axes, 4 f_a = f0/4 on the diagonals; thermal weights of the improved model, g0 = 5T/9 and
// g_a = T/18 = g0/10, within a factor 2 of g0/8), and a difference of two binary32 numbers within a
// factor 2 of each other is exact (Sterbenz). The sums below take every population relative to that ratio first, so
// the large part is one exact product of the rest population and the rounding falls on small
// deviations. Binary64 and double-word arithmetic keep the plain sums (flow_moments, heat_of).
__device__ __forceinline__ float density_of(const float f[9]) {
  const float q = f[0] * 0.25f;
  const float A = ((f[1] - q) + (f[2] - q)) + ((f[3] - q) + (f[4] - q));
  const float B = (fmaf(4.f, f[5], -q) + fmaf(4.f, f[6], -q)) + (fmaf(4.f, f[7], -q) + fmaf(4.f, f[8], -q));
  return fmaf(2.25f, f[0], A + B * 0.25f);  // rho = 9 f0/4 + A + B/4
}

// Temperature T = sum g. In binary32 also its rounding residual lo (T + lo is the sum of the deviations
// to within their own small roundings): the liquid's pressure changes with T about 30 times faster than
// with rho in lattice units, so the residual is carried into psi^2 (psi_squared).
template <class R> __device__ __forceinline__ R heat_of(const R g[9], R& lo) {
  if constexpr (sizeof(R) == 4) {
    const R q = g[0] * 0.125f;
    const R E = (((g[1] - q) + (g[2] - q)) + ((g[3] - q) + (g[4] - q))) +
                (((g[5] - q) + (g[6] - q)) + ((g[7] - q) + (g[8] - q)));
    const R t2 = g[0] * 2.f;
    const R T = t2 + E;  // T = 2 g0 + sum (g_a - g0/8)
    lo = E - (T - t2);   // exact residual (Fast2Sum: |2 g0| > |E|)
    return T;
  } else {
    lo = R(0);
    return g[0] + g[1] + g[2] + g[3] + g[4] + g[5] + g[6] + g[7] + g[8];
  }
}

// psi^2 = (2/G)(p_EOS - rho c_s^2) (reading of Ref. [48]) in binary32, with p_EOS first moved by (dp/dT)_rho Tlo
// for the residual of the temperature.
__device__ __forceinline__ float psi_squared(float p, float dpdT, float Tlo, float rho, const Coefs<float>& C) {
  return C.psi_scale * ((p + dpdT * Tlo) - rho * float(1.0 / 3.0));
}

// psi^2 and (dp/dT)_rho of a node in the form its arithmetic takes (Tlo: the residual of a binary32 T).
template <class R, class PT>
__device__ __forceinline__ R node_psi_squared(R rho, R T, R Tlo, const PT& P, R& dpdT) {
  if constexpr (sizeof(R) == 4) {
    R p;
    eos(rho, T, P, p, dpdT);
    return psi_squared(p, dpdT, Tlo, rho, coefs<R>(P));
  } else {
    R inv_rho;
    return eos_psi_squared(rho, T, P, dpdT, inv_rho);
  }
}

// ------------------------------------------------------------------------------------------------
// population storage
// ------------------------------------------------------------------------------------------------
// One population set (f or g) in one buffer: SoA [9][N] of the storage type S. With S = __half the
// stored value is the deviation of the post-collision population from the rest-state equilibrium
// w_a * ref of the node that stored it, ref being that node's density (f) or post-collision
// temperature (g), held in an FP32 plane beside the populations. The collision conserves the zeroth
// moment, so the deviations are of order |u| w rho and keep binary16's 11 bits relative to them.
//
// A flow buffer also carries the force on its wall rows (`wall`, FP64 [edge y-/y+][Fx/Fy][nx]), written
// by the step that stored the populations: the next step's wall closure sets j = -F/2 from it.
template <class S> struct PopBuf {
  S* p;
  float* ref;    // FP16 storage only
  double* wall;  // flow buffers: wall-row forces (null where unused; aggregate init leaves it null)
};

// nodes of a domain
template <class PT> __host__ __device__ __forceinline__ double node_count(const PT& P) { return (double)P.nx * (double)P.ny; }

// Index of a wall row's entries in PopBuf::wall: edge 0 = y-, 1 = y+; component 0 = Fx, 1 = Fy.
__host__ __device__ __forceinline__ long long wall_slot(int nx, int edge, int comp, int x) {
  return (long long)(2 * edge + comp) * nx + x;
}
// doubles of one wall-force buffer (one parity)
__host__ __device__ __forceinline__ long long wall_doubles(int nx) { return 4LL * nx; }

template <class S> struct is_half_t { static constexpr bool value = false; };
template <> struct is_half_t<__half> { static constexpr bool value = true; };

// P.pitch as the index arithmetic of a storage type takes it. A product of signed 32-bit numbers cannot overflow by the
// language's rules, so the compiler widens a row's nine sources to 64-bit addresses early; unsigned ones stay 32-bit
// until they are used. The FP16 tiles, which hold a reference's address beside each population's, are short of
// registers and take the unsigned form: 12 FP16 instances of 60^2 to 77^2 13.97 us a step signed, 10.8 unsigned; 24 of
// 64^2 to 512^2 119, 110. FP32 is better off with the wide addresses (4096^2 421 us, 434 unsigned; small ones alike).
template <class S, class PT> __device__ __forceinline__ auto pitch_of(const PT& P) {
  if constexpr (is_half_t<S>::value) return (unsigned)P.pitch;
  else return P.pitch;
}

// double(x) from the bits, exact for every x (NaN stays NaN): a conversion instruction runs at the FP64 pipe's rate,
// a seventieth of the integer and binary32 ones. A subnormal is scaled into the normal numbers first. A dozen
// instructions more per value in flight, so it pays where the FP64 pipe and not latency sets the time (launch_sums).
__host__ __device__ __forceinline__ double widen(float x) {
  union { float f; unsigned u; } v;
  v.f = x;
  const bool tiny = (v.u & 0x7f800000u) == 0;
  v.f = x * (tiny ? 4294967296.0f : 1.0f);
  unsigned bias = tiny ? 0x38000000u - (32u << 20) : 0x38000000u;
  if ((v.u & 0x7f800000u) == 0x7f800000u) bias = 0x70000000u;
  if ((v.u & 0x7fffffffu) == 0) bias = 0;
  const unsigned hi = ((unsigned)((int)v.u >> 3) & 0x8fffffffu) + bias;
  union { unsigned long long u; double d; } r;
  r.u = ((unsigned long long)hi << 32) | (v.u << 29);
  return r.d;
}
template <class R, bool BITS> __device__ __forceinline__ R widen_to(float x) {
  if constexpr (BITS) return widen(x);
  else return R(x);
}

// IX is the index type: long long in general; int where the caller guarantees that every population
// index of the buffer (9 N) fits in 31 bits, which turns each address into one 32-bit multiply-add.
// BITS (R = double): narrower storage widened from its bits, see widen.
template <class S, class R, class IX = long long, bool BITS = false>
__device__ __forceinline__ R pop_load(const PopBuf<S>& b, IX N, int a, IX idx, const R* w) {
  if constexpr (is_half_t<S>::value) {
    return widen_to<R, BITS>(__half2float(__ldg(b.p + ((IX)a * N + idx)))) +
           w[a] * widen_to<R, BITS>(__ldg(b.ref + idx));
  } else if constexpr (is_dw_t<S>::value) {
    const dw v = ldgv(b.p + ((IX)a * N + idx));
    if constexpr (BITS) return widen(v.hi) + widen(v.lo);
    else return R(v);
  } else {
    if constexpr (BITS && sizeof(S) == 4) return widen(__ldg(b.p + ((IX)a * N + idx)));
    else return R(__ldg(b.p + ((IX)a * N + idx)));
  }
}

// Store the post-collision populations v of node i; refval is the node's zeroth moment after the
// collision (rho for f, T + S0 for g), the reference of the FP16 deviation.
template <class S, class R, class IX = long long>
__device__ __forceinline__ void pop_store(const PopBuf<S>& b, IX N, IX i, const R v[9], R refval, const R* w) {
  if constexpr (is_half_t<S>::value) {
#pragma unroll
    for (int a = 0; a < 9; ++a) b.p[(IX)a * N + i] = __float2half_rn(float(v[a] - w[a] * refval));
    b.ref[i] = float(refval);
  } else {
#pragma unroll
    for (int a = 0; a < 9; ++a) b.p[(IX)a * N + i] = (S)v[a];
  }
}

// pop_store through explicitly global stores, for buffer pointers that the compiler cannot place in
// the global space (descriptors read from shared memory).
template <class S, class R, class IX = long long>
__device__ __forceinline__ void pop_store_global(const PopBuf<S>& b, IX N, IX i, const R v[9], R refval,
                                                 const R* w) {
  if constexpr (is_half_t<S>::value) {
#pragma unroll
    for (int a = 0; a < 9; ++a) __stwb(b.p + ((IX)a * N + i), __float2half_rn(float(v[a] - w[a] * refval)));
    __stwb(b.ref + i, float(refval));
  } else {
#pragma unroll
    for (int a = 0; a < 9; ++a) __stwb(b.p + ((IX)a * N + i), (S)v[a]);
  }
}

// ------------------------------------------------------------------------------------------------
// pull-stream with the boundary closures applied at the pulling node
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ int wrapx(int x, int nx) { return x < 0 ? x + nx : (x >= nx ? x - nx : x); }

// Post-stream populations at (x, y): src holds post-collision populations (SoA [9][N]); a
// population whose source node lies beyond a non-periodic y edge is unknown and returned as 0.
//
// The nine source nodes (x - e_a) share three columns and three rows; PullSrc holds them once per node
// (x, y inside the grid), wrapped on the periodic axes. Entry k of each array is the source for e = k - 1.
struct PullSrc {
  int col[3];  // x + 1, x, x - 1 (wrapped)
  int row[3];  // y + 1, y, y - 1 (wrapped when y is periodic; -1 beyond a non-periodic y edge)
};
template <class PT> __device__ __forceinline__ PullSrc pull_src(const PT& P, int x, int y) {
  PullSrc s;
  s.col[0] = x == P.nx - 1 ? 0 : x + 1;
  s.col[1] = x;
  s.col[2] = x == 0 ? P.nx - 1 : x - 1;
  s.row[0] = y == P.ny - 1 ? (P.yper ? 0 : -1) : y + 1;
  s.row[1] = y;
  s.row[2] = y == 0 ? (P.yper ? P.ny - 1 : -1) : y - 1;
  return s;
}

template <class S, class R, class IX = long long, class PT = DevParams, bool BITS = false>
__device__ __forceinline__ void pull_from(const PopBuf<S>& src, const R* w, const PT& P, const PullSrc& s,
                                          R v[9]) {
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    const int r = s.row[EY(a) + 1];
    v[a] = r >= 0 ? pop_load<S, R, IX, BITS>(src, (IX)P.N, a, (IX)r * pitch_of<S>(P) + s.col[EX(a) + 1], w) : R(0);
  }
}

template <class S, class R, class PT>
__device__ __forceinline__ void pull(const PopBuf<S>& src, const R* w, const PT& P, int x, int y, R v[9]) {
  pull_from<S, R>(src, w, P, pull_src(P, x, y), v);
}

// Zou-He closure of the unknown f on a non-periodic y edge. Wall: the momentum is set to j = -F/2, F
// being the wall row's force of the step that stored the populations (`wall`, see PopBuf), so that the
// forcing scheme's velocity v = (j + F/2)/rho vanishes on the wall (a null `wall` reads as F = 0).
// Pressure: rho = rho_bc, u_x = 0.
template <class R, class PT>
__device__ __forceinline__ void flow_closure(R f[9], const PT& P, int x, int y, const double* wall) {
  if (P.yper) return;
  const Coefs<R>& C = coefs<R>(P);
  const R d13 = f[1] - f[3];
  if (y == 0) {
    if (P.ybc_lo == BC_WALL) {  // f2 - f4 = 2/3 j_y; f5 - f6 closes j_x
      const R jx = wall ? R(wall[wall_slot(P.nx, 0, 0, x)]) * -0.5f : R(0);
      const R jy = wall ? R(wall[wall_slot(P.nx, 0, 1, x)]) * -0.5f : R(0);
      f[2] = f[4] + R(2.0 / 3.0) * jy;
      f[5] = f[7] - d13 * 0.5f + jx * 0.5f + jy * R(1.0 / 6.0);
      f[6] = f[8] + d13 * 0.5f - jx * 0.5f + jy * R(1.0 / 6.0);
    } else {
      const R ru = C.rho_bc_lo - (f[0] + f[1] + f[3] + (f[4] + f[7] + f[8]) * 2);  // rho_bc u_y
      f[2] = f[4] + R(2.0 / 3.0) * ru;
      f[5] = f[7] - d13 * 0.5f + ru * R(1.0 / 6.0);
      f[6] = f[8] + d13 * 0.5f + ru * R(1.0 / 6.0);
    }
  } else if (y == P.ny - 1) {
    if (P.ybc_hi == BC_WALL) {
      const R jx = wall ? R(wall[wall_slot(P.nx, 1, 0, x)]) * -0.5f : R(0);
      const R jy = wall ? R(wall[wall_slot(P.nx, 1, 1, x)]) * -0.5f : R(0);
      f[4] = f[2] - R(2.0 / 3.0) * jy;
      f[7] = f[5] + d13 * 0.5f - jx * 0.5f - jy * R(1.0 / 6.0);
      f[8] = f[6] - d13 * 0.5f + jx * 0.5f - jy * R(1.0 / 6.0);
    } else {
      const R ru = (f[0] + f[1] + f[3] + (f[2] + f[5] + f[6]) * 2) - C.rho_bc_hi;  // rho_bc u_y
      f[4] = f[2] - R(2.0 / 3.0) * ru;
      f[7] = f[5] + d13 * 0.5f - ru * R(1.0 / 6.0);
      f[8] = f[6] - d13 * 0.5f - ru * R(1.0 / 6.0);
    }
  }
}

// Thermal equilibrium moments (Eq. 53 for the improved model, Eq. 44 for the compromised one, and for
// the Gong-Cheng model the moments of Eq. 14: the second-order equilibrium with rho replaced by T).
template <class R> __device__ __forceinline__ void heat_meq(R T, R vx, R vy, int model, R n[9]) {
  if (model == 2) {
    const R v2 = vx * vx + vy * vy;
    n[0] = T;
    n[1] = T * (R(-2) + v2 * 3);
    n[2] = T * (R(1) - v2 * 3);
    n[3] = T * vx;
    n[4] = -T * vx;
    n[5] = T * vy;
    n[6] = -T * vy;
    n[7] = T * (vx * vx - vy * vy);
    n[8] = T * vx * vy;
    return;
  }
  n[0] = T;
  n[1] = T * -2;
  n[2] = model == 0 ? T * 2 : T;
  n[3] = T * vx;
  n[4] = -T * vx;
  n[5] = T * vy;
  n[6] = -T * vy;
  n[7] = R(0);
  n[8] = R(0);
}

// Thermal boundary step. On a non-periodic y edge the unknown g are closed by bounce-back:
// g_a = -g_opp(a) + 2 g_a^eq(T_bc, 0) where the edge holds T_bc (anti-bounce-back; heat enters through
// the wall), g_a = g_opp(a) otherwise (zero heat flux). A Dirichlet edge of a periodic axis (a ring
// inside a periodic domain) resets the node to g := M^{-1} m_eq(T_bc, 0): x edges, then y edges.
template <class R, class PT> __device__ __forceinline__ void heat_closure(R g[9], const PT& P, int x, int y) {
  const Coefs<R>& C = coefs<R>(P);
  if (!P.yper) {
    if (y == 0) {
      if (P.tbc[2]) {
        const R Tb = (x >= P.strip_x0 && x < P.strip_x1) ? C.T_strip : C.T_bc[2];
        R n[9], e[9];
        heat_meq(Tb, R(0), R(0), P.model, n);
        from_moments(n, e);
        g[2] = e[2] * 2 - g[4];
        g[5] = e[5] * 2 - g[7];
        g[6] = e[6] * 2 - g[8];
      } else {
        g[2] = g[4]; g[5] = g[7]; g[6] = g[8];
      }
    }
    if (y == P.ny - 1) {
      if (P.tbc[3]) {
        R n[9], e[9];
        heat_meq(C.T_bc[3], R(0), R(0), P.model, n);
        from_moments(n, e);
        g[4] = e[4] * 2 - g[2];
        g[7] = e[7] * 2 - g[5];
        g[8] = e[8] * 2 - g[6];
      } else {
        g[4] = g[2]; g[7] = g[5]; g[8] = g[6];
      }
    }
  }
  bool set = false;
  R Tb = R(0);
  if (x == 0 && P.tbc[0]) { set = true; Tb = C.T_bc[0]; }
  if (x == P.nx - 1 && P.tbc[1]) { set = true; Tb = C.T_bc[1]; }
  if (P.yper) {
    if (y == 0 && P.tbc[2]) { set = true; Tb = (x >= P.strip_x0 && x < P.strip_x1) ? C.T_strip : C.T_bc[2]; }
    if (y == P.ny - 1 && P.tbc[3]) { set = true; Tb = C.T_bc[3]; }
  }
  if (set) {
    R n[9];
    heat_meq(Tb, R(0), R(0), P.model, n);
    from_moments(n, g);
  }
}

// Post-stream, post-boundary f and g at (x, y).
template <class S, class R, class IX = long long, class PT = DevParams, bool BITS = false>
__device__ __forceinline__ void pull_closed(const PopBuf<S>& fsrc, const PopBuf<S>& gsrc, const PT& P, int x,
                                            int y, R f[9], R g[9]) {
  const Coefs<R>& C = coefs<R>(P);
  const PullSrc src = pull_src(P, x, y);  // f and g read the same nine source nodes
  pull_from<S, R, IX, PT, BITS>(fsrc, C.wf, P, src, f);
  pull_from<S, R, IX, PT, BITS>(gsrc, C.wg, P, src, g);
  flow_closure(f, P, x, y, fsrc.wall);
  heat_closure(g, P, x, y);
}

// Keep the force of a wall-row node for the next step's closure (into the destination flow buffer).
template <class R, class PT>
__device__ __forceinline__ void wall_force_store(double* wall, const PT& P, int x, int y, R Fx, R Fy) {
  if (P.yper || !wall) return;
  const int edge = (y == 0 && P.ybc_lo == BC_WALL) ? 0 : (y == P.ny - 1 && P.ybc_hi == BC_WALL) ? 1 : -1;
  if (edge < 0) return;
  wall[wall_slot(P.nx, edge, 0, x)] = double(Fx);
  wall[wall_slot(P.nx, edge, 1, x)] = double(Fy);
}

// ------------------------------------------------------------------------------------------------
// collisions
// ------------------------------------------------------------------------------------------------
// Density, momentum and the non-conserved flow moments m = (e, eps, qx, qy, pxx, pxy) of f in binary64 and
// double-word arithmetic: 24 additions, the sums and differences of opposite populations shared by all of them.
template <class R> __device__ __forceinline__ R flow_moments(const R f[9], R& jx, R& jy, R m[6]) {
  const R s13 = f[1] + f[3], s24 = f[2] + f[4], s57 = f[5] + f[7], s68 = f[6] + f[8];
  const R d13 = f[1] - f[3], d24 = f[2] - f[4], a = f[5] - f[7], b = f[8] - f[6];
  const R s14 = s13 + s24, s58 = s57 + s68;
  const R c = a + b, d = a - b;
  jx = d13 + c;
  jy = d24 + d;
  m[0] = s58 * 2 - s14 - f[0] * 4;
  m[1] = f[0] * 4 - s14 * 2 + s58;
  m[2] = c - d13 * 2;
  m[3] = d - d24 * 2;
  m[4] = s13 - s24;
  m[5] = s57 - s68;
  return f[0] + s14 + s58;
}

// Post-collision f from those moments: c_k m_k* = (1 - s) c_k m_k + s c_k m_k,eq + (1 - s/2) c_k S_F,k for the
// six relaxed moments (FlowRates), m0* = rho and j* = j + F whatever the rates (S_F,0 = 0, m0_eq = rho,
// m_eq,3 = j + F/2), and the back-transform. 57 binary64 instructions.
template <class R>
__device__ __forceinline__ void relax_flow(const R m[6], R jx, R jy, R rho, R vx, R vy, R Fx, R Fy, R Q, const Coefs<R>& C,
                                           R f[9]) {
  const auto& K = C.flow;
  const R rvx = rho * vx, rvy = rho * vy;
  const R rxx = rvx * vx, ryy = rvy * vy;
  const R r3 = rxx + ryy;                      // rho v^2: m1_eq = 3 r3 - 2 rho, m2_eq = rho - 3 r3
  const R xF = vx * Fx, yF = vy * Fy;
  const R t = (xF + yF) * 6 + Q;               // S_F,1 = -S_F,2
  // energy moments without the parts of their equilibria linear in rho, which w0, wa and wd carry
  const R u1 = K.A[0] * m[0] + (K.E[0] * r3 + K.H[0] * t);
  const R u2 = K.A[1] * m[1] - (K.E[1] * r3 + K.H[1] * t);
  const R u4 = K.A[2] * m[2] - (K.B[0] * rvx + K.H[2] * Fx);
  const R u6 = K.A[3] * m[3] - (K.B[1] * rvy + K.H[3] * Fy);
  const R u7 = K.A[4] * m[4] + (K.B[2] * (rxx - ryy) + K.H[4] * (xF - yF));
  const R u8 = K.A[5] * m[5] + (K.B[3] * (rvx * vy) + K.H[5] * (vx * Fy + vy * Fx));
  const R ax = (K.wa * rho - u1) - u2 * 2;  // common to e1..e4
  const R dg = (K.wd * rho + u2) + u1 * 2;  // common to e5..e8
  R sx, sy, qx, qy;                         // j*/6 plus the fluxes, on the diagonals and on the axes
  if constexpr (is_dw_t<R>::value) {        // a scale by 2 costs a double-word less than one by 3
    const R w3 = (jx + Fx) * R(1.0 / 6.0), w5 = (jy + Fy) * R(1.0 / 6.0);
    sx = w3 + u4; qx = w3 - u4 * 2;
    sy = w5 + u6; qy = w5 - u6 * 2;
  } else {
    sx = (jx + Fx) * R(1.0 / 6.0) + u4; qx = sx - u4 * 3;
    sy = (jy + Fy) * R(1.0 / 6.0) + u6; qy = sy - u6 * 3;
  }
  const R a1 = ax + u7, a2 = ax - u7, g5 = dg + u8, g6 = dg - u8, k5 = sx + sy, k6 = sy - sx;
  f[0] = K.w0 * rho + (u2 - u1) * 4;
  f[1] = a1 + qx;
  f[2] = a2 + qy;
  f[3] = a1 - qx;
  f[4] = a2 - qy;
  f[5] = g5 + k5;
  f[6] = g6 + k6;
  f[7] = g5 - k5;
  f[8] = g6 - k6;
}

// Flow MRT collision with forcing (reading of the improved pseudopotential model, Refs. [13,29]):
// m* = m - Lambda (m - m_eq) + (I - Lambda/2) S_F, S_F with the sigma term Q in the energy moments.
//
// Binary32 takes the collision in increments, f* = f + M^{-1} (m* - m), so that every stored population
// is rounded once at its own scale. Rebuilding f* from all nine post-collision moments rounds several
// times at the scale of the populations, and the roundings of the opposite pair e_a, -e_a differ, which
// moves momentum at random. The non-equilibrium parts m - m_eq of the energy and stress moments come
// from the populations' exact deviations from their rest-state ratios (see density_of), not from moments
// of size about 2 rho that cancel. This function is binary32's; binary64 and double-word arithmetic rebuild f* from m*
// (relax_flow).
template <class R, class PT>
__device__ __forceinline__ void collide_flow(R f[9], R rho, R vx, R vy, R Fx, R Fy, R Q, const PT& P) {
  static_assert(sizeof(R) == 4, "binary32");
  const Coefs<R>& C = coefs<R>(P);
  const R vxx = vx * vx, vyy = vy * vy;
  const R v2 = vxx + vyy;
  const R vF = vx * Fx + vy * Fy;
  const R q = f[0] * 0.25f;
  const R d1 = f[1] - q, d2 = f[2] - q, d3 = f[3] - q, d4 = f[4] - q;
  const R d5 = fmaf(4.f, f[5], -q), d6 = fmaf(4.f, f[6], -q), d7 = fmaf(4.f, f[7], -q), d8 = fmaf(4.f, f[8], -q);
  const R A = (d1 + d2) + (d3 + d4), B = (d5 + d6) + (d7 + d8);
  const R e_dev = A + B;                       // m1 + 2 rho
  const R eps_dev = A * -3.f;                  // m2 - rho
  const R pxx = (d1 + d3) - (d2 + d4);         // m7
  const R pxy = ((d5 + d7) - (d6 + d8)) * 0.25f;  // m8
  const R qx = (f[1] - f[3]) * -2.f + ((f[5] - f[6]) + (f[8] - f[7]));  // m4
  const R qy = (f[2] - f[4]) * -2.f + ((f[5] - f[7]) + (f[6] - f[8]));  // m6
  const R r3v2 = rho * v2 * 3.f;
  R dm[9], df[9];
  dm[0] = R(0);  // S_F,0 = 0 and m0_eq = rho
  dm[3] = Fx;    // j* = j + F whatever s_j (m_eq,3 = j + F/2)
  dm[5] = Fy;
  dm[1] = C.flow.hf[1] * (vF * 6 + Q) - C.flow.s_f[1] * (e_dev - r3v2);  // m1 - m1_eq = (m1 + 2 rho) - 3 rho v^2
  dm[2] = C.flow.hf[2] * (vF * -6 - Q) - C.flow.s_f[2] * (eps_dev + r3v2);  // m2 - m2_eq = (m2 - rho) + 3 rho v^2
  dm[4] = C.flow.hf[4] * -Fx - C.flow.s_f[4] * (qx + rho * vx);
  dm[6] = C.flow.hf[6] * -Fy - C.flow.s_f[6] * (qy + rho * vy);
  dm[7] = C.flow.hf[7] * ((vx * Fx - vy * Fy) * 2) - C.flow.s_f[7] * (pxx - rho * (vxx - vyy));
  dm[8] = C.flow.hf[8] * (vx * Fy + vy * Fx) - C.flow.s_f[8] * (pxy - rho * vx * vy);
  from_moments(dm, df);
#pragma unroll
  for (int a = 0; a < 9; ++a) f[a] = f[a] + df[a];
}

// The thermal moments n4, n6 (the fluxes qx, qy of g) in binary64 and double-word arithmetic.
template <class R> __device__ __forceinline__ void heat_fluxes(const R g[9], R& n4, R& n6) {
  const R a = g[5] - g[7], b = g[8] - g[6];
  n4 = (a + b) - (g[1] - g[3]) * 2;
  n6 = (a - b) - (g[2] - g[4]) * 2;
}

// Post-collision g of the improved model when every rate s_k, k >= 1, is 1, from n4 and n6 alone.
template <class R>
__device__ __forceinline__ void relax_heat_unit(R n4, R n6, R T, R vx, R vy, R S0, R g[9]) {
  const R TS = T + S0;
  const R Tvx = T * vx, Tvy = T * vy;
  const R h4 = n4 * R(1.0 / 12.0), h6 = n6 * R(1.0 / 12.0);
  const R X = Tvx * R(5.0 / 12.0) + h4, Xd = Tvx * R(1.0 / 6.0) + h4;
  const R Y = Tvy * R(5.0 / 12.0) + h6, Yd = Tvy * R(1.0 / 6.0) + h6;
  const R B = TS * R(1.0 / 9.0) - T * R(1.0 / 18.0);
  const R P1 = B + Xd, P2 = B - Xd;
  g[1] = B + X;
  g[3] = B - X;
  g[2] = B + Y;
  g[4] = B - Y;
  g[5] = P1 + Yd;
  g[8] = P1 - Yd;
  g[6] = P2 + Yd;
  g[7] = P2 - Yd;
  // binary32 keeps the heat of the node to one rounding (see from_moments_conserving)
  if constexpr (sizeof(R) == 4) g[0] = TS - (((g[1] + g[2]) + (g[3] + g[4])) + ((g[5] + g[6]) + (g[7] + g[8])));
  else g[0] = B + T * 0.5f;
}

// Thermal MRT collision of the improved model: Eq. 45 with m_eq of Eq. 53 and S = (S0, 0, ..., 0)
// (Eq. 46), then m3* += (1 - s3/2) s4 (m4 - m4_eq) and m5* += (1 - s5/2) s6 (m6 - m6_eq) (Eqs. 54-55).
template <class R, class PT>
__device__ __forceinline__ void collide_heat(R g[9], R T, R vx, R vy, R S0, const PT& P, R tau_inv = R(0)) {
  const Coefs<R>& C = coefs<R>(P);
  R ns[9];
  if (P.model == 2) {
    // Gong-Cheng (Eqs. 12-14): BGK with the local 1/tau_g, source G_a = w_a phi, whose moments are
    // phi (1, -2, 1, 0, ..., 0)
    R n[9], neq[9];
    to_moments(g, n);
    heat_meq(T, vx, vy, 2, neq);
#pragma unroll
    for (int k = 0; k < 9; ++k) ns[k] = n[k] - tau_inv * (n[k] - neq[k]);
    ns[0] += S0;
    ns[1] += S0 * -2;
    ns[2] += S0;
  } else if (P.heat_unit_rates && P.model == 0) {
    // s_k = 1 for k >= 1 (so c3 = c5 = 1/2): every non-conserved moment takes its Eq. 53 value and
    // n* = (T + S0, -2T, 2T, T vx + (n4 + T vx)/2, -T vx, T vy + (n6 + T vy)/2, -T vy, 0, 0). Its
    // back-transform M^{-1} n* in closed form: the axes and the diagonals share the base
    // B = (T + S0)/9 - T/18, the axes add +-X (+-Y) with X = 5 T vx/12 + n4/12, the diagonals +-X' +-Y'
    // with X' = T vx/6 + n4/12, and the rest population is B + T/2.
    R n4, n6;
    if constexpr (sizeof(R) == 4) {
      n4 = (g[1] - g[3]) * -2 + (g[5] - g[6] - g[7] + g[8]);
      n6 = (g[2] - g[4]) * -2 + (g[5] + g[6] - g[7] - g[8]);
    } else {
      heat_fluxes(g, n4, n6);
    }
    relax_heat_unit(n4, n6, T, vx, vy, S0, g);
    return;
  } else if (P.heat_unit_rates) {
    // compromised model with s_k = 1 for k >= 1: every non-conserved moment relaxes to its equilibrium,
    // so only the zeroth moment (T) is needed.
    heat_meq(T, vx, vy, P.model, ns);  // Eq. 44: n7 = n8 = 0
    ns[0] = T + S0;
  } else {
    R n[9], neq[9];
    to_moments(g, n);
    heat_meq(T, vx, vy, P.model, neq);
    ns[0] = n[0] + S0;  // n0_eq = T = n0: the relaxation leaves the zeroth moment, the source adds S0
#pragma unroll
    for (int k = 1; k < 9; ++k) ns[k] = n[k] - C.s_g[k] * (n[k] - neq[k]);
    if (P.model == 0) {
      ns[3] += C.c3 * (n[4] - neq[4]);
      ns[5] += C.c5 * (n[6] - neq[6]);
    }
  }
  from_moments_conserving(ns, g);
}

// ------------------------------------------------------------------------------------------------
// block reduction (fixed order: warp shuffle tree, then warp 0 over the warp sums)
// ------------------------------------------------------------------------------------------------
template <int BLOCK> __device__ __forceinline__ double block_sum(double v, double* smem) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) smem[w] = v;
  __syncthreads();
  double s = 0.0;
  if (w == 0) {
    s = lane < BLOCK / 32 ? smem[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  }
  __syncthreads();
  return s;  // valid in thread 0
}

// Record the first non-physical node (step, x, y, code); later reports are dropped.
__device__ __forceinline__ void report(long long* status, long long step, int x, int y, int code) {
  if (atomicCAS((unsigned long long*)status, 0ull, 1ull) == 0ull) {
    status[1] = step;
    status[2] = x;
    status[3] = y;
    status[4] = code;
  }
}

template <class R, class PT> __device__ __forceinline__ int classify(R rho, R T, R psi2, const PT& P) {
  if constexpr (sizeof(R) == 8 && !is_dw_t<R>::value) {
    // binary64: the same tests on the bit patterns, on the integer pipe (the FP64 pipe bounds this step).
    // A finite double is positive exactly when its bits, read as a signed integer, are; b rho >= 1 for
    // a positive finite b rho exactly when its bits are at least those of 1.0; -0.0 counts as >= 0.
    const long long EXP = 0x7ff0000000000000LL;
    const long long ir = __double_as_longlong(rho), iT = __double_as_longlong(T), ip = __double_as_longlong(psi2);
    if ((ir & EXP) == EXP || (iT & EXP) == EXP || (ip & EXP) == EXP) return ST_NONFINITE;
    if (ir <= 0) return ST_RHO_LE0;
    if (__double_as_longlong(coefs<R>(P).b * rho) >= 0x3ff0000000000000LL) return ST_RHO_POLE;
    if (iT <= 0) return ST_T_LE0;
    if (ip < 0 && ip != (long long)0x8000000000000000ULL) return ST_PSI2_NEG;
    return 0;
  }
  if (!isfinite(rho) || !isfinite(T) || !isfinite(psi2)) return ST_NONFINITE;
  if (!(rho > R(0))) return ST_RHO_LE0;
  if (!(coefs<R>(P).b * rho < R(1))) return ST_RHO_POLE;
  if (!(T > R(0))) return ST_T_LE0;
  if (!(psi2 >= R(0))) return ST_PSI2_NEG;
  return 0;
}

// Report a node that is not physical. Binary32 first tests everything at once (a NaN fails every comparison) and
// classifies only what fails.
template <class R, class PT>
__device__ __forceinline__ void check_node(R rho, R T, R psi2, const PT& P, long long* status, const long long* step_at,
                                           long long step, int x, int y) {
  if constexpr (sizeof(R) == 4) {
    const R top = R(3.402823466e38);
    if (rho > R(0) && coefs<R>(P).b * rho < R(1) && T > R(0) && T <= top && psi2 >= R(0) && psi2 <= top) return;
  }
  const int bad = classify(rho, T, psi2, P);
  if (bad) report(status, step_at ? *step_at : step, x, y, bad);  // step_at: read only to report
}

}  // namespace lbpc
