// dg_common.cuh -- shared device definitions of the GB300 modal DG solver
// (arXiv:1602.09079, Sect. 2): table layout, ideal-gas physics, HLLC flux,
// positivity limiter, launch geometry.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

// a device function that is called, not inlined (no such keyword in host builds)
#ifdef __CUDACC__
#define DG_NOINLINE __noinline__
#else
#define DG_NOINLINE
#endif

namespace dg {

// First statement of every kernel that is launched with programmatic stream
// serialisation (launch_after): the kernel may be set up while its predecessor
// in the stream still runs; this waits until that one has completed and its
// writes are visible, before anything is read or written.
__device__ __forceinline__ void stream_wait() {
#ifdef __CUDA_ARCH__
  asm volatile("griddepcontrol.wait;" ::: "memory");
#endif
}

// adds 1 to a counter and returns the old value; this thread's earlier atomics are
// visible to whoever sees the addition, and those of the earlier counts to this thread
__device__ __forceinline__ unsigned count_done(unsigned* p) {
#ifdef __CUDA_ARCH__
  unsigned r;
  asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(r) : "l"(__cvta_generic_to_global(p)) : "memory");
  return r;
#else
  return __atomic_fetch_add(p, 1u, __ATOMIC_ACQ_REL);
#endif
}

// ------------------------------------------------------------- sizes
__host__ __device__ constexpr int nmodes(int k) { return (k + 1) * (k + 2) * (k + 3) / 6; }
__host__ __device__ constexpr int gll_m(int k) { return k <= 1 ? 2 : 3; }
// index of the tangential pair (a, b), a + b <= k, in the order a
// ascending, b ascending
__host__ __device__ constexpr int pair_index(int k, int a, int b) {
  int j = 0;
  for (int ap = 0; ap < a; ++ap) j += k - ap + 1;
  return j + b;
}
// index of mode (u, v, w) in the exchange order (total degree ascending,
// then u descending, then v descending)
__host__ __device__ constexpr int mode_index(int u, int v, int w) {
  const int D = u + v + w;
  int idx = D > 0 ? nmodes(D - 1) : 0;
  for (int up = D; up > u; --up) idx += D - up + 1;
  return idx + (D - u - v);
}

// (u, v, w) of mode l in the canonical order (degree ascending, u then v
// descending).
__device__ __forceinline__ void mode_uvw(int l, int& u, int& v, int& w) {
  int D = 0;
  while (l >= nmodes(D)) ++D;
  int r = l - (D > 0 ? nmodes(D - 1) : 0);
  u = D;
  while (r > D - u) {
    r -= D - u + 1;
    --u;
  }
  v = D - u - r;
  w = D - u - v;
}

// 8 x 8 matrices of 16-bit elements from shared memory in the fragment layout of
// mma.sync (PTX ldmatrix): lane l gives the address of row l % 8 of matrix l / 8;
// lane (g, t) = (l / 4, l % 4) receives elements [g][2t], [g][2t + 1] of every
// matrix, transposed [2t][g], [2t + 1][g]. Rows are 16-byte aligned.
#ifdef __CUDA_ARCH__
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p))
               : "memory");
}
__device__ __forceinline__ void ldsm4_t(uint32_t (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p))
               : "memory");
}
__device__ __forceinline__ void ldsm2_t(uint32_t (&r)[2], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];"
               : "=r"(r[0]), "=r"(r[1])
               : "r"((uint32_t)__cvta_generic_to_shared(p))
               : "memory");
}
#endif

// Per-degree basis/quadrature tables (Sect. 2.2-2.5), all values at the
// method's point sets, offsets in elements. Weights are folded in so the
// kernels only multiply and add.
template <int K>
struct Tab {
  static constexpr int Q = K + 1;
  static constexpr int Q2 = Q * Q;
  static constexpr int Q3 = Q * Q * Q;
  static constexpr int N = nmodes(K);
  static constexpr int M = gll_m(K);
  static constexpr int NL = 3 * M * Q2;  // positivity point set S
  // phi_l(xi_q) at volume Gauss points, [Q3][N]
  static constexpr int VPHI = 0;
  // dphi_l/dxi_a (xi_q) * omega_q / 4, [3][Q3][N]
  static constexpr int VDPHI = VPHI + Q3 * N;
  // phi_l(xi_q) * omega_q / 8, [Q3][N]
  static constexpr int VPHIW = VDPHI + 3 * Q3 * N;
  // phi_l at face points of face (a, s), s = 0 low (xi_a = -1) / 1 high, [3][2][Q2][N]
  static constexpr int FPHI = VPHIW + Q3 * N;
  // same times omega_2D / 4, [3][2][Q2][N]
  static constexpr int FPHIW = FPHI + 6 * Q2 * N;
  // phi_l at the limiter points, [NL][N]
  static constexpr int LPHI = FPHIW + 6 * Q2 * N;
  // max over S of |phi_l|, [N]
  static constexpr int LMAX = LPHI + NL * N;
  // tangential products Pt_a(x_t1) Pt_b(x_t2) at the face points, pairs
  // (a, b) with a + b <= K in the order a ascending, b ascending, [Q2][T]
  static constexpr int T = (K + 1) * (K + 2) / 2;
  static constexpr int F2D = LMAX + N;
  // Pt_e(-1) and Pt_e(+1), [2][K+1]
  static constexpr int FEND = F2D + Q2 * T;
  // 1D tables at the Gauss points for sum factorisation, [K+1][Q] each:
  // Pt_u(x_a), Pt_u(x_a) w_a, Pt_u'(x_a) w_a
  static constexpr int P1 = FEND + 2 * (K + 1);
  static constexpr int P1W = P1 + (K + 1) * Q;
  static constexpr int D1W = P1W + (K + 1) * Q;
  // 1D Gauss nodes and weights, [Q] each
  static constexpr int GX = D1W + (K + 1) * Q;
  static constexpr int GW = GX + Q;
  // max over S and the volume Gauss points of |phi_l|, [N]
  static constexpr int LMAXV = GW + Q;
  static constexpr int SIZE = LMAXV + N;
};
constexpr int TAB_STRIDE = 16384;  // >= Tab<3>::SIZE
static_assert(Tab<3>::SIZE <= TAB_STRIDE, "table stride");

// ------------------------------------------------------------ error word
enum : unsigned {
  ERRB_NONFINITE = 1u,
  ERRB_POSITIVITY = 2u,
  ERRB_NEWTON = 4u,
};

// Control block at the start of the scratch buffer. The queue counters: every stage
// (and the energy reset) clears n_deep before its cells are queued; n_flag is 0
// between the stages and between the calls (the limiter's last pass clears it, and
// a call that fails before that does on the stream); the unfused stages' face kernels
// clear it in any case.
struct Ctrl {
  unsigned long long cfl_max_bits;  // max over cells of the wave-speed sum (bits of a double >= 0): the result
  unsigned int err;                 // sticky ERRB_* bits
  unsigned int n_flag;              // cells queued for the full limiter
  unsigned long long n_limited;     // limiter count
  unsigned int n_gate;              // queued cells the indicator passes on
  unsigned int n_deep;              // queued cells the FP32 point screen does not clear
  unsigned long long n_queued_total;  // cells that failed the limiter screen (all stages)
  unsigned long long n_full_total;    // cells that went through the full limiter
  unsigned long long cfl_running;     // of the reduction under way; 0 between the calls, like
  unsigned int cfl_blocks;            // the number of its blocks that are done
  double sums[8];                     // results of the host-facing sums, read back with the error word
};

struct Geo {
  int nx, ny, nz;
  long long nc;  // cells
  double dx[3];
  double inv_dx[3];
  double gamma;
  double eps_rho, eps_p;
  int lim_vol;  // limiter point set: 0 = S, 1 = S and the volume Gauss points
};

// --------------------------------------------------------------- physics
template <typename T>
__device__ __forceinline__ T pressure_of(const T* U, T gm1) {
  T ke = T(0.5) * (U[1] * U[1] + U[2] * U[2] + U[3] * U[3]) / U[0];
  return gm1 * (U[4] - ke);
}

// Euler flux along direction d from conserved U, given velocity and pressure.
template <typename T>
__device__ __forceinline__ void euler_flux(int d, const T* U, const T* v, T p, T* F) {
  T mn = U[1 + d];
  F[0] = mn;
  F[1] = mn * v[0];
  F[2] = mn * v[1];
  F[3] = mn * v[2];
  F[1 + d] += p;
  F[4] = (U[4] + p) * v[d];
}

// HLLC numerical flux across a face with normal +e_d, left = lower cell
// (Sect. 2.3, the approximate HLLC Riemann solver): Einfeldt wave-speed
// estimates from Roe averages, middle wave and star states from the
// Rankine-Hugoniot conditions across the three waves (Toro's formulation).
// ------------------------------------------- IEEE 754 conversions
// binary32 <-> binary64 from the format definitions (sign, biased exponent,
// fraction) on the integer pipe, for the FP32 path's FP64 stage epilogue:
// GB300 issues the hardware conversions on its FP64 unit, which the FP32
// volume kernel otherwise keeps 45 % busy. Exact for every input: values
// outside the fast range (zeros, subnormals, infinities, NaNs) take the
// hardware conversion. dg_selftest_conversions compares both with the
// hardware.

// binary32 -> binary64: exponent rebias 127 -> 1023, fraction widened
__device__ __forceinline__ double f32_to_f64(float x) {
  const unsigned u = __float_as_uint(x);
  const unsigned e = (u >> 23) & 0xffu;
  if (e == 0u || e == 0xffu) return (double)x;
  const unsigned hi = (u & 0x80000000u) | ((e + 896u) << 20) | ((u & 0x7fffffu) >> 3);
  return __hiloint2double((int)hi, (int)(u << 29));
}

// binary64 -> binary32, round to nearest, ties to even: results in the
// binary32 normal range (biased exponents 897..1150) and magnitudes below
// 2^-150 (round to a signed zero) on the integer pipe
__device__ __forceinline__ float f64_to_f32(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned e = (hi >> 20) & 0x7ffu;
  if (e - 897u <= 253u) {
    unsigned f = (hi & 0x80000000u) | ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
    const unsigned rem = lo & 0x1fffffffu;  // the 29 dropped fraction bits
    f += (rem > 0x10000000u || (rem == 0x10000000u && (f & 1u))) ? 1u : 0u;
    return __uint_as_float(f);
  }
  if (e < 873u) return __uint_as_float(hi & 0x80000000u);
  return (float)x;
}

// finite test on the exponent field (integer pipe)
__device__ __forceinline__ bool finite64(double x) {
  return (((unsigned)__double2hiint(x) >> 20) & 0x7ffu) != 0x7ffu;
}

__device__ __forceinline__ float rsq(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsq(double x) { return rsqrt(x); }

template <typename T>
__device__ __forceinline__ void hllc_flux(int d, const T* UL, const T* UR, T gamma, T* F) {
  const T gm1 = gamma - T(1);
  // one reciprocal square root per side gives 1/rho and sqrt(rho)
  const T rL = rsq(UL[0]), rR = rsq(UR[0]);
  const T irL = rL * rL, irR = rR * rR;
  T vL[3] = {UL[1] * irL, UL[2] * irL, UL[3] * irL};
  T vR[3] = {UR[1] * irR, UR[2] * irR, UR[3] * irR};
  T pL = gm1 * (UL[4] - T(0.5) * UL[0] * (vL[0] * vL[0] + vL[1] * vL[1] + vL[2] * vL[2]));
  T pR = gm1 * (UR[4] - T(0.5) * UR[0] * (vR[0] * vR[0] + vR[1] * vR[1] + vR[2] * vR[2]));
  // a face pressure at the positivity floor can round to <= 0 (FP32 traces
  // of an FP64-limited state; FP64 near vacuum when gamma - 1 is small): the
  // sound speed is then 0, the limit p -> 0+
  const T cL = sqrt(fmax(gamma * pL * irL, T(0)));
  const T cR = sqrt(fmax(gamma * pR * irR, T(0)));
  const T sL = UL[0] * rL, sR = UR[0] * rR;
  T iss = T(1) / (sL + sR);
  T vt[3], v2 = T(0);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    vt[a] = (sL * vL[a] + sR * vR[a]) * iss;
    v2 += vt[a] * vt[a];
  }
  T Ht = (rL * (UL[4] + pL) + rR * (UR[4] + pR)) * iss;
  T c2t = gm1 * (Ht - T(0.5) * v2);
  T ct = c2t > T(0) ? sqrt(c2t) : T(0);
  T uL = vL[d], uR = vR[d];
  T SL = fmin(uL - cL, vt[d] - ct);
  T SR = fmax(uR + cR, vt[d] + ct);
  if (SL >= T(0)) {
    euler_flux(d, UL, vL, pL, F);
    return;
  }
  if (SR <= T(0)) {
    euler_flux(d, UR, vR, pR, F);
    return;
  }
  T aL = UL[0] * (SL - uL), aR = UR[0] * (SR - uR);
  T Ss = (pR - pL + uL * aL - uR * aR) / (aL - aR);
  // both sound speeds 0 in a receding flow: S_L = u_L and S_R = u_R, so
  // aL = aR = 0. Take S* = 0; the flux is then (0, p e_d, 0), the flux at a
  // vacuum interface.
  if (aL - aR == T(0)) Ss = T(0);
  // the side of the contact, selected by value (no pointer into either
  // side's arrays, which would put them in local memory)
  const bool left = Ss >= T(0);
  T U[5], v[3];
#pragma unroll
  for (int i = 0; i < 5; ++i) U[i] = left ? UL[i] : UR[i];
#pragma unroll
  for (int a = 0; a < 3; ++a) v[a] = left ? vL[a] : vR[a];
  T p = left ? pL : pR;
  T S = left ? SL : SR;
  T ak = left ? aL : aR;  // rho_K (S_K - u_K)
  T ir = left ? irL : irR;
  T uk = left ? uL : uR;
  euler_flux(d, U, v, p, F);
  // star state: chi = rho_K (S_K - u_K) / (S_K - S*), and
  // E* = chi (E_K / rho_K + (S* - u_K) (S* + p_K / (rho_K (S_K - u_K))))
  const T isd = T(1) / (S - Ss);
  T chi = ak * isd;
  T Us[5];
  Us[0] = chi;
  Us[1] = chi * v[0];
  Us[2] = chi * v[1];
  Us[3] = chi * v[2];
  Us[1 + d] = chi * Ss;
  Us[4] = chi * (U[4] * ir + (Ss - uk) * Ss) + (Ss - uk) * p * isd;
#pragma unroll
  for (int i = 0; i < 5; ++i) F[i] += S * (Us[i] - U[i]);
}

// Exact zeros of the 1D tables: a Gauss rule with an odd number of points
// has a node at 0, where the odd Legendre polynomials and the derivatives of
// the even ones vanish, and Pt_0' = 0 everywhere. The multiply-adds by them
// are dropped at compile time (the loops are unrolled); for finite operands
// the sums are unchanged, bit for bit.
template <int K>
__host__ __device__ constexpr bool zero_p(int u, int q) {
  return K % 2 == 0 && 2 * q == K && u % 2 == 1;
}
template <int K>
__host__ __device__ constexpr bool zero_d(int u, int q) {
  return u == 0 || (K % 2 == 0 && 2 * q == K && u % 2 == 0);
}

// mode index of the exponents along (normal, tangential 1, tangential 2) of a
// face normal to axis D (tangential axes in ascending order)
template <int D>
__host__ __device__ constexpr int face_mode(int e, int a, int b) {
  return D == 0 ? mode_index(e, a, b) : (D == 1 ? mode_index(a, e, b) : mode_index(a, b, e));
}

// an upper bound of |x| in binary32 from the high word of x (20 fraction
// bits, rounded up: at most 2^-20 above |x|); magnitudes below 2^-126 map to
// 2^-126, huge and non-finite values to infinity
__device__ __forceinline__ float abs_up(double x) {
  unsigned u = (unsigned)__double2hiint(x) & 0x7fffffffu;
  u = min(max(u, 0x38100000u), 0x47efffffu);
  return __uint_as_float(((u - 0x38000000u) << 3) + 8u);
}

// binary64 -> binary32 on the integer pipe (no FP64-unit conversion):
// rounded to nearest on the 29 dropped fraction bits (ties away from zero,
// which differs from ties-to-even only when they are exactly 2^28);
// magnitudes below 2^-126 give a signed zero, magnitudes of 2^128 and above,
// infinities and NaNs a signed infinity (the stage's screen then queues the
// cell and the full limiter reports the non-finite state)
__device__ __forceinline__ float f64_to_f32_q(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned mag = hi & 0x7fffffffu;
  unsigned r = (__funnelshift_l(lo, hi, 3) - 0xC0000000u) + ((lo >> 28) & 1u);
  r = mag < 0x38100000u ? 0u : r;
  r = mag >= 0x47f00000u ? 0x7f800000u : r;
  return __uint_as_float(r | (hi & 0x80000000u));
}

// binary32 -> binary64 on the integer pipe: exact for normal numbers,
// subnormals give a signed zero, infinities and NaNs stay what they are
__device__ __forceinline__ double f32_to_f64_q(float x) {
  const unsigned u = __float_as_uint(x), mag = u & 0x7fffffffu, sg = u & 0x80000000u;
  unsigned hi = sg | ((mag >> 3) + 0x38000000u);
  unsigned lo = u << 29;
  hi = mag >= 0x7f800000u ? (hi | 0x7ff00000u) : hi;
  hi = mag < 0x00800000u ? sg : hi;
  lo = mag < 0x00800000u ? 0u : lo;
  return __hiloint2double((int)hi, (int)lo);
}

// approximate reciprocal and reciprocal square root (one MUFU operation
// each, subnormals flushed to zero: relative error of a few ulp)
__device__ __forceinline__ float rcp_fast(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.f / x;
#endif
}
__device__ __forceinline__ float rsqrt_fast(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.f / std::sqrt(x);
#endif
}
// Pressure part of the limiter's FP32 screens: true when gm1 (E - |m|^2 / (2
// rho)) clears ep for every rho >= rlo > 0, E >= elo and |m_j| <= mh_j,
// multiplied through by the density bound, with a 1e-5 margin relative to eabs >=
// |E|, which covers the FP32 rounding of the inputs and of the test. The products
// rho E and m^2 leave the range of binary32 in units as common as g / cm^3 (and 0
// >= 0 would hold): where the margin itself is not well inside it, the test is made
// on rho, E and m scaled by powers of two 2^a, 2^b and 2^((a + b) / 2) that bring rlo
// and eabs near 1. Bounds below 2^-103 or above 2^125, zeros, infinities and
// NaNs then fail: the caller's next, FP64 test decides.
__device__ __forceinline__ bool pressure_clear_f32(float rlo, float elo, float eabs, const float (&mh)[3], float gm1,
                                                   float ep) {
  float k2 = 0.f;
#pragma unroll
  for (int a = 0; a < 3; ++a) k2 = fmaf(mh[a], mh[a], k2);
  k2 *= 0.5f;
  float mg = 1e-5f * gm1 * fmaf(eabs, rlo, k2);
  if (!(mg >= 1e-30f && mg <= 1e30f)) {
    // biased exponents (a set sign makes them large), their sum made even
    const int xr = (int)(__float_as_uint(rlo) >> 23), x4 = (int)(__float_as_uint(eabs) >> 23);
    if ((unsigned)(xr - 24) > 228u || (unsigned)(x4 - 24) > 228u) return false;
    const int xe = x4 + ((xr + x4) & 1);
    const float sr = __uint_as_float((unsigned)(254 - xr) << 23), se = __uint_as_float((unsigned)(254 - xe) << 23);
    const float sm = __uint_as_float((unsigned)(254 - (xr + xe) / 2) << 23);
    rlo *= sr;
    elo *= se;
    ep *= se;
    k2 = 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) k2 = fmaf(mh[a] * sm, mh[a] * sm, k2);
    k2 *= 0.5f;
    mg = 1e-5f * gm1 * fmaf(eabs * se, rlo, k2);
  }
  return gm1 * fmaf(elo, rlo, -k2) >= fmaf(ep, rlo, mg);
}

// Sufficient limiter screen in FP32 from the cell means m and the excursion
// bounds s_i >= sum_{l>=1} |w_il| max|phi_l|: true when the density and the
// pressure provably stay above the floors at every point of the limiter's
// point set (same bounds as the FP64 screen, with a 1e-5 relative margin that
// covers the FP32 rounding of the inputs and of the test). NaN inputs fail, and
// so do states outside the range of pressure_clear_f32.
__device__ __forceinline__ bool screen_f32(const float* m, const float* s, float gm1, float er, float ep) {
  const float r = m[0];
  const float rlo = r - s[0];
  if (!(rlo >= er + 1e-5f * (fabsf(r) + s[0]))) return false;
  const float mh[3] = {fabsf(m[1]) + s[1], fabsf(m[2]) + s[2], fabsf(m[3]) + s[3]};
  return pressure_clear_f32(rlo, m[4] - s[4], fabsf(m[4]) + s[4], mh, gm1, ep);
}

// position of conserved variable i in the frame of a face normal to axis d:
// (rho, m_n, m_t1, m_t2, E) with t1 < t2 the other two axes. Traces and
// fluxes are stored in this order, so the numerical flux is evaluated with
// a compile-time normal and no reordering.
__device__ __forceinline__ int face_var(int d, int i) {
  if (i == 0 || i == 4) return i;
  const int ax = i - 1, t1 = d == 0 ? 1 : 0;
  return ax == d ? 1 : (ax == t1 ? 2 : 3);
}

// ------------------------------------------------- 64-bit fixed point
// The FP64 path's contractions with the 1D tables (point values, face traces,
// projections) run in 64-bit fixed point on the integer pipe: a GB300 SM
// retires 2 FP64 FMAs per clock (measured 1.98 lanes) but 59 32 x 32 -> 64 bit
// multiply-adds, and the sums of these contractions need one common exponent,
// not one per operand. A block of numbers (a variable's coefficients of one
// cell, its fluxes at the points of a slice) shares the exponent B of a bound
// of every sum formed from it: x = X 2^(B - 1083), |X| < 2^61, so a unit is
// 2^-61 of the bound, where an FP64 sum of that size rounds at 2^-53. An
// operand is two limbs, X = h 2^30 + l, a table entry c = C 2^-58, C = ch 2^30
// + cl with |cl| <= 2^29; a product takes three multiply-adds (h ch into hi,
// h cl + l ch into mid; l cl stays below one unit), a sum one shift at its
// end. Partial sums may wrap, sums may not: the bounds stand at each caller.
struct Fx {
  int h, l;  // value h 2^30 + l, 0 <= l < 2^30 (fx_split_signed: |l| <= 2^29)
};
struct FxAcc {
  long long hi, mid;  // value (hi 2^60 + mid 2^30) 2^-58
};
__device__ __forceinline__ Fx fx_split(long long r) { return {(int)(r >> 30), (int)(r & 0x3fffffff)}; }
// the same with -2^29 <= l < 2^29, for |r| < 2^60.9: where many products go into
// one sum, low limbs that are never negative would not cancel in its mid
__device__ __forceinline__ Fx fx_split_signed(long long r) {
  return {(int)((r + 0x20000000) >> 30), (int)((unsigned)r << 2) >> 2};
}
__device__ __forceinline__ long long fx_join(Fx x) { return (long long)x.h * (1 << 30) + x.l; }
__device__ __forceinline__ void fx_mad(FxAcc& a, Fx x, int ch, int cl) {
  a.hi += (long long)x.h * ch;
  a.mid += (long long)x.h * cl;
  a.mid += (long long)x.l * ch;
}
__device__ __forceinline__ long long fx_val(FxAcc a) { return a.hi * 4 + ((a.mid + (1 << 27)) >> 28); }

// biased exponent of |x| from a high word
__device__ __forceinline__ int bexp(unsigned hi) { return (int)((hi >> 20) & 0x7ffu); }

// x in units of 2^(B - 1083), truncated; needs bexp(x) <= B (|X| < 2^61), or a
// smaller |X| where the caller's bound asks for it. Exponents B are at least
// kFxTiny, so that zeros and subnormals (whose implicit bit is not one) are
// shifted out.
constexpr int kFxTiny = 64;
__device__ __forceinline__ long long fx_from(double x, int B) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int bx = bexp(hi);
  const int d = min(B - bx, 63);
  unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 40) | ((unsigned long long)lo << 8);
  m >>= d;
  return (hi >> 31) ? -(long long)m : (long long)m;
}

// the same of a binary32 value (biased exponent + 896 <= B)
__device__ __forceinline__ long long fx_from(float x, int B) {
  const unsigned u = __float_as_uint(x);
  const int e = (int)((u >> 23) & 0xffu);
  const int d = e ? min(B - 896 - e, 63) : 63;
  const unsigned long long m = ((unsigned long long)((u & 0x7fffffu) | 0x800000u) << 37) >> d;
  return (u >> 31) ? -(long long)m : (long long)m;
}

__device__ __forceinline__ int clz64(unsigned long long m) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)m);
#else
  return m ? __builtin_clzll(m) : 64;
#endif
}

// r 2^(B - 1083) as a double, rounded to nearest (ties up in magnitude);
// results below 2^-1022 give 0
__device__ __forceinline__ double fx_to_double(long long r, int B) {
  const unsigned long long s = (unsigned long long)r & 0x8000000000000000ull;
  unsigned long long m = s ? 0ull - (unsigned long long)r : (unsigned long long)r;
  const int lz = clz64(m);
  const int b = B + 2 - lz;  // biased exponent less the implicit bit
  m <<= lz & 63;
  m = (m >> 11) + ((m >> 10) & 1u);
  const unsigned long long bits = s | (((unsigned long long)(unsigned)b << 52) + m);
  return (lz < 64 && b >= 0) ? __longlong_as_double((long long)bits) : 0.0;
}

// exponent B of a cell variable's coefficients: sum_l |w_l| max |phi_l| <
// 2^(B - 1022) (max |phi_l| over the cell, the product of sqrt(2u + 1)), which
// bounds the variable and every partial sum of its contractions everywhere in
// the cell. Summed in FP32 from the high words relative to the largest one
// (each rounded up by 2^-20; the 1e-4 covers the sum's own rounding).
template <int K>
__device__ __forceinline__ int fx_bound(const double (&w)[nmodes(K)]) {
  constexpr int N = nmodes(K);
  unsigned mx = 0;
#pragma unroll
  for (int l = 0; l < N; ++l) mx = max(mx, (unsigned)__double2hiint(w[l]) & 0x7fffffffu);
  const int top = (int)(mx & 0x7ff00000u) - (127 << 20);
  float s = 0.f;
#pragma unroll
  for (int u = 0; u <= K; ++u)
#pragma unroll
    for (int v = 0; u + v <= K; ++v)
#pragma unroll
      for (int ww = 0; u + v + ww <= K; ++ww) {
        const int f = (int)((unsigned)__double2hiint(w[mode_index(u, v, ww)]) & 0x7fffffffu) - top;
        // sqrt(2u + 1) rounded up: 1, 1.7321, 2.2361, 2.6458
        constexpr float r[4] = {1.f, 1.7321f, 2.2361f, 2.6458f};
        const float bl = (u == 0 ? r[0] : u == 1 ? r[1] : u == 2 ? r[2] : r[3]) *
                         (v == 0 ? r[0] : v == 1 ? r[1] : v == 2 ? r[2] : r[3]) *
                         (ww == 0 ? r[0] : ww == 1 ? r[1] : ww == 2 ? r[2] : r[3]);
        s = fmaf(__uint_as_float((unsigned)max(f, 0) * 8u + 8u), bl, s);
      }
  return max(kFxTiny, bexp(mx) + (int)(__float_as_uint(s * 1.0001f) >> 23) - 127);
}
// a block whose exponent reaches kFxHuge holds an infinity or a NaN (or values
// whose squares overflow): its results are NaN
constexpr int kFxHuge = 2000;

// Integer tables {ch, cl} of degree K at fx_base(K), KQ = (K + 1)^2 (round(c 2^58)
// of the exact values, from 60-digit arithmetic): Pt_u(x_q) at FXP + u Q + q;
// Pt_u(x_q) w_q / 2 at FXW; Pt_u'(x_q) w_q / 16 at FXD; Pt_e(-1), Pt_e(+1) at
// FXE + e, FXE + K + 1 + e; the same / 16 at FXF.
__host__ __device__ constexpr int fx_base(int k) { return k == 0 ? 0 : k == 1 ? 7 : k == 2 ? 27 : 66; }
template <int K>
struct FxTab {
  static constexpr int KQ = (K + 1) * (K + 1);
  static constexpr int P = fx_base(K), W = P + KQ, D = W + KQ, E = D + KQ, F = E + 2 * (K + 1);
};
static __constant__ int c_fx[130][2] = {
    // degree 0
    {268435456, 0}, {268435456, 0}, {0, 0}, {268435456, 0}, {268435456, 0}, {16777216, 0}, {16777216, 0},
    // degree 1
    {268435456, 0}, {268435456, 0}, {-268435456, 0}, {268435456, 0}, {134217728, 0}, {134217728, 0}, {-134217728, 0},
    {134217728, 0}, {0, 0}, {0, 0}, {29058991, -513723734}, {29058991, -513723734}, {268435456, 0},
    {-464943848, -370354845}, {268435456, 0}, {464943848, 370354845}, {16777216, 0}, {-29058991, 513723734},
    {16777216, 0}, {29058991, -513723734},
    // degree 2
    {268435456, 0}, {268435456, 0}, {268435456, 0}, {-360143956, -335321274}, {0, 0}, {360143956, 335321274},
    {240095971, -134366425}, {-300119964, 436393488}, {240095971, -134366425}, {74565404, 477218588},
    {119304647, 119304647}, {74565404, 477218588}, {-100039988, 145464496}, {0, 0}, {100039988, -145464496},
    {66693325, 260937611}, {-133386650, -521875221}, {66693325, 260937611}, {0, 0}, {0, 0}, {0, 0},
    {16143884, -404706722}, {25830214, -218034025}, {16143884, -404706722}, {-48431651, 140378341}, {0, 0},
    {48431651, -140378341}, {268435456, 0}, {-464943848, -370354845}, {600239927, 200954849}, {268435456, 0},
    {464943848, 370354845}, {600239927, 200954849}, {16777216, 0}, {-29058991, 513723734}, {37514995, 482321726},
    {16777216, 0}, {29058991, -513723734}, {37514995, 482321726},
    // degree 3
    {268435456, 0}, {268435456, 0}, {268435456, 0}, {268435456, 0}, {-400380031, 362829381}, {-158072095, 248394076},
    {158072095, -248394076}, {400380031, -362829381}, {367547088, -91861811}, {-196049966, 149277482},
    {-196049966, 149277482}, {367547088, -91861811}, {-216435411, 534292416}, {292414767, 87758746},
    {-292414767, -87758746}, {216435411, -534292416}, {46688287, -12733607}, {87529441, 12733607},
    {87529441, 12733607}, {46688287, -12733607}, {-69637067, 235101179}, {-51542975, -387813052},
    {51542975, 387813052}, {69637067, -235101179}, {63926518, -350468200}, {-63926518, 350468200},
    {-63926518, 350468200}, {63926518, -350468200}, {-37644053, -108756140}, {95348437, -234821281},
    {-95348437, 234821281}, {37644053, 108756140}, {0, 0}, {0, 0}, {0, 0}, {0, 0}, {10108311, -378250125},
    {18950680, -135473609}, {18950680, -135473609}, {10108311, -378250125}, {-33712900, 10506446},
    {-24953136, 377443648}, {24953136, -377443648}, {33712900, -10506446}, {62714997, -90867394},
    {-18326656, 335695376}, {-18326656, 335695376}, {62714997, -90867394}, {268435456, 0}, {-464943848, -370354845},
    {600239927, 200954849}, {-710213460, 377719588}, {268435456, 0}, {464943848, 370354845}, {600239927, 200954849},
    {710213460, -377719588}, {16777216, 0}, {-29058991, 513723734}, {37514995, 482321726}, {-44388341, -244827982},
    {16777216, 0}, {29058991, -513723734}, {37514995, 482321726}, {44388341, 244827982},
};
__device__ __forceinline__ void fx_madt(FxAcc& a, Fx x, int t) { fx_mad(a, x, c_fx[t][0], c_fx[t][1]); }

// Values at the Q Gauss nodes of the line with the coefficients x[u], u < M.
// Nodes come in pairs +-x_r: the even and the odd modes are summed once for
// both (3 products instead of 5 at degree 2, 6 instead of 12 at degree 3).
template <int K, int M>
__device__ __forceinline__ void fx_values(const Fx (&x)[M], long long (&o)[K + 1]) {
  constexpr int Q = K + 1, P = FxTab<K>::P;
  const long long x0 = fx_join(x[0]);  // Pt_0 = 1
#pragma unroll
  for (int r = Q - Q / 2; r < Q; ++r) {
    FxAcc e{0, 0}, d{0, 0};
#pragma unroll
    for (int u = 2; u < M; u += 2) fx_madt(e, x[u], P + u * Q + r);
#pragma unroll
    for (int u = 1; u < M; u += 2) fx_madt(d, x[u], P + u * Q + r);
    const long long ev = M > 2 ? fx_val(e) + x0 : x0, od = M > 1 ? fx_val(d) : 0;
    o[r] = ev + od;
    o[Q - 1 - r] = ev - od;
  }
  if (Q % 2) {
    FxAcc e{0, 0};
#pragma unroll
    for (int u = 2; u < M; u += 2) fx_madt(e, x[u], P + u * Q + Q / 2);
    o[Q / 2] = M > 2 ? fx_val(e) + x0 : x0;
  }
}

// G[u] += sum_q f(q) W_u(q), u = 0 .. K, or with the derivatives' table D
// (DER; G[0] is left alone), from the sums and differences of the node pairs.
// |f| < 2^60, so that these stay below 2^61.
template <int K, bool DER>
__device__ __forceinline__ void fx_project(const long long (&f)[K + 1], FxAcc (&G)[K + 1]) {
  constexpr int Q = K + 1, W = DER ? FxTab<K>::D : FxTab<K>::W;
#pragma unroll
  for (int r = Q - Q / 2; r < Q; ++r) {
    const Fx s = fx_split(f[r] + f[Q - 1 - r]), d = fx_split(f[r] - f[Q - 1 - r]);
#pragma unroll
    for (int u = DER ? 1 : 0; u <= K; ++u) fx_madt(G[u], (u + DER) % 2 ? d : s, W + u * Q + r);
  }
  if (Q % 2) {
    const Fx m = fx_split(f[Q / 2]);
#pragma unroll
    for (int u = DER ? 1 : 0; u <= K; u += 2) fx_madt(G[u], m, W + u * Q + Q / 2);
  }
}

// ------------------------------------- FP64 reciprocal and square roots
// One MUFU approximation y0 of the significand m (|1 - m y0| < 2^-21), then one
// third-order Householder iteration (A. S. Householder, The Numerical Treatment
// of a Single Nonlinear Equation, 1970), y0 (1 + r + r^2) with r = 1 - m y0 and
// y0 (1 + r/2 + 3 r^2 / 8) with r = 1 - m y0^2, on the integer pipe: the exact
// product gives r in units of 2^-82, the result has 60 bits before it is rounded
// (within 0.51 units in the last place). In FP64 operations the iterations take
// 3 and 5 of a pipe that retires two per clock and SM, which bounds the face
// kernel (128^3, degree 2: 11.1 ms per stage so, now 9.15). Arguments near the ends of the exponent range, zeros,
// infinities, NaNs (and x < 0 for the root) take the library function.

// y0 (1 + c) rounded to a double's significand: y0 in units of 2^-30 (2^29 to
// 2^30), c in units of 2^-60; e: biased exponent of the result for 0.5 <= y < 1,
// less one
__device__ __forceinline__ double root_finish(unsigned y0, long long c, unsigned e, unsigned sign) {
  const long long p = (long long)((unsigned long long)y0 * (unsigned)c >> 30) + (long long)(int)(c >> 32) * (int)y0 * 4;
  const unsigned long long y = ((unsigned long long)y0 << 30) + (unsigned long long)p;
  const unsigned long long bits = ((unsigned long long)e << 52) + ((y + 64) >> 7);
  return __longlong_as_double((long long)(bits | ((unsigned long long)sign << 32)));
}

__device__ __forceinline__ double rcp64(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int bx = bexp(hi);
  if ((unsigned)(bx - 64) > 1900u) return 1.0 / x;
  const unsigned mh = (hi & 0xfffffu) | 0x100000u;  // significand, 53 bits
  // (0.5, 1] in units of 2^-30
  const unsigned y0 = (unsigned)(rcp_fast(__uint_as_float(0x3f800000u | ((hi & 0xfffffu) << 3) | (lo >> 29))) * 0x1p30f);
  // 1 - m y0 in units of 2^-82 (the product is 2^82 less this, modulo 2^64)
  const long long r = -(long long)((unsigned long long)lo * y0 + ((unsigned long long)(mh * y0) << 32));
  const int h = (int)(r >> 41);
  return root_finish(y0, (r >> 22) + ((long long)h * h >> 22), (unsigned)(2044 - bx), hi & 0x80000000u);
}
__device__ __forceinline__ double rsqrt64(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int bx = (int)(hi >> 20);
  if ((unsigned)(bx - 64) > 1900u) return rsq(x);
  const unsigned odd = (unsigned)(bx - 1023) & 1u;
  const int half = (bx - 1023 - (int)odd) >> 1;
  const unsigned f = ((127u + odd) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
  // in units of 2^-24: below 0.5 (significands just under 4) the approximation has a
  // bit more, which the residual could not see
  const unsigned y0 = (unsigned)(rsqrt_fast(__uint_as_float(f)) * 0x1p30f) & ~63u;
  // significand in [1, 4), 54 bits
  const unsigned long long m = (((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo) << odd;
  const unsigned a0 = (unsigned)m, a1 = (unsigned)(m >> 32);
  const unsigned k = y0 >> 6;
  const unsigned long long s = (unsigned long long)k * k;
  const unsigned s0 = (unsigned)s, s1 = (unsigned)(s >> 32);
  // 1 - m y0^2 in units of 2^-82, modulo 2^64
  const unsigned long long t = (((unsigned long long)a0 * s0) >> 18) +
                               (((unsigned long long)a0 * s1 + (unsigned long long)a1 * s0) << 14) +
                               ((unsigned long long)(a1 * s1) << 46);
  const long long r = -(long long)t;
  const int h = (int)(r >> 41);
  return root_finish(y0, (r >> 23) + ((long long)(3 * h) * h >> 25), (unsigned)(1021 - half), 0u);
}
// sqrt(max(x, 0))
__device__ __forceinline__ double sqrt64(double x) { return __double2hiint(x) > 0 ? x * rsqrt64(x) : 0.0; }
// x^(2/3) = z z^(-1/3) 2^(2q) for x = z 2^(3q), 1 <= z < 8: FP32 logarithm and
// exponential (2^-20), then one third-order Householder iteration of z^(-1/3),
// y (1 + e/3 + 2 e^2 / 9) with e = 1 - z y^3, in 7 FP64 operations (cbrt and a
// square take about 30). x <= 0 and the ends of the exponent range take cbrt.
__device__ __forceinline__ double pow_2_3(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int bx = (int)(hi >> 20);
  if ((unsigned)(bx - 64) > 1900u) {
    const double c = cbrt(x);
    return c * c;
  }
  const int q = (bx - 1023 + 1200) / 3 - 400, s = bx - 1023 - 3 * q;
  const double z = __hiloint2double((int)((hi & 0xfffffu) | ((unsigned)(1023 + s) << 20)), (int)lo);
  const float f = __uint_as_float(((unsigned)(127 + s) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
  const double y = f32_to_f64_q(exp2f(log2f(f) * (-1.f / 3.f)));
  const double e = fma(-(z * y), y * y, 1.0);
  const double c = z * fma(y * e, fma(e, 2.0 / 9.0, 1.0 / 3.0), y);
  return __hiloint2double(__double2hiint(c) + q * 0x200000, __double2loint(c));
}
// a < b in the total order of the bit patterns (integer pipe)
__device__ __forceinline__ bool less64(double a, double b) {
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
  return (x ^ (long long)((unsigned long long)(x >> 63) >> 1)) < (y ^ (long long)((unsigned long long)(y >> 63) >> 1));
}

// HLLC flux of the face frame in FP64 (same algorithm as hllc_flux: Einfeldt
// wave speeds, sound speed 0 at pressures <= 0, S* = 0 for a receding vacuum
// interface), arranged for few FP64 operations, about 70 a point instead of
// 190 (105 before the roots moved to the integer pipe): the Roe sound speed from the average of the sides' c^2 and the velocity
// jump, c~^2 = <c^2> + (gamma - 1)/2 w (1 - w) |dv|^2 with the Roe weight w
// (the same as through the total enthalpy); the flux of the star region as F(U*)
// with the contact's speed and the star pressure (the jump conditions across
// S_K make it F_K + S_K (U* - U_K)); comparisons on the integer pipe.
__device__ __forceinline__ void hllc64_x(const double* UL, const double* UR, double gamma, double* F) {
  const double gm1 = gamma - 1.0;
  const double rL = rsqrt64(UL[0]), rR = rsqrt64(UR[0]);
  const double irL = rL * rL, irR = rR * rR;
  const double vL[3] = {UL[1] * irL, UL[2] * irL, UL[3] * irL};
  const double vR[3] = {UR[1] * irR, UR[2] * irR, UR[3] * irR};
  const double kL = fma(UL[1], vL[0], fma(UL[2], vL[1], UL[3] * vL[2]));
  const double kR = fma(UR[1], vR[0], fma(UR[2], vR[1], UR[3] * vR[2]));
  const double pL = gm1 * fma(-0.5, kL, UL[4]), pR = gm1 * fma(-0.5, kR, UR[4]);
  const double a2L = gamma * pL * irL, a2R = gamma * pR * irR;
  const double cL = sqrt64(a2L), cR = sqrt64(a2R);
  const double sL = UL[0] * rL, sR = UR[0] * rR;
  const double w = sL * rcp64(sL + sR);
  const double d0 = vL[0] - vR[0], d1 = vL[1] - vR[1], d2 = vL[2] - vR[2];
  const double ut = fma(w, d0, vR[0]);
  const double dv2 = fma(d0, d0, fma(d1, d1, d2 * d2));
  const double ct = sqrt64(fma(0.5 * gm1 * fma(-w, w, w), dv2, fma(w, a2L - a2R, a2R)));
  const double uL = vL[0], uR = vR[0];
  const double S1 = uL - cL, S2 = ut - ct, S3 = uR + cR, S4 = ut + ct;
  // like fmin and fmax: a NaN Roe state is passed over; a NaN of the side
  // itself is neither case below and makes the flux NaN
  const bool roe = finite64(S2);
  const double SL = roe && less64(S2, S1) ? S2 : S1, SR = roe && less64(S3, S4) ? S4 : S3;
  const bool supL = (unsigned)__double2hiint(SL) < 0x7ff00000u;
  const bool supR = __double_as_longlong(SR) <= 0 && finite64(SR);
  if (supL || supR) {
    const double u = supL ? uL : uR, p = supL ? pL : pR;
    const double mn = supL ? UL[1] : UR[1];
    F[0] = mn;
    F[1] = fma(mn, u, p);
    F[2] = mn * (supL ? vL[1] : vR[1]);
    F[3] = mn * (supL ? vL[2] : vR[2]);
    F[4] = ((supL ? UL[4] : UR[4]) + p) * u;
    return;
  }
  const double sdL = SL - uL, sdR = SR - uR;
  const double aL = UL[0] * sdL, aR = UR[0] * sdR;
  const double den = aL - aR;
  const double Ss = (unsigned long long)__double_as_longlong(den) << 1 == 0ull ? 0.0 : fma(uL, aL, fma(-uR, aR, pR - pL)) * rcp64(den);
  const bool left = __double2hiint(Ss) >= 0;
  const double p = left ? pL : pR, u = left ? uL : uR, ak = left ? aL : aR;
  const double isd = rcp64((left ? SL : SR) - Ss);
  const double ps = fma(ak, Ss - u, p);           // star pressure
  const double mn = ak * isd * Ss;                // star mass flux
  const double Es = fma(left ? sdL : sdR, left ? UL[4] : UR[4], fma(ps, Ss, -p * u)) * isd;
  F[0] = mn;
  F[1] = fma(mn, Ss, ps);
  F[2] = mn * (left ? vL[1] : vR[1]);
  F[3] = mn * (left ? vL[2] : vR[2]);
  F[4] = (Es + ps) * Ss;
}

// ------------------------------------------------- exact Riemann solver
// Godunov flux from the exact solution of the Riemann problem (the exact
// option of Sect. 2.3 next to HLLC): the star pressure p* is the root of
// f_L(p) + f_R(p) + u_R - u_L, where f_K is the velocity jump across the
// wave of side K (shock branch from the Rankine-Hugoniot conditions for
// p > p_K, rarefaction branch from the Riemann invariant for p <= p_K);
// Newton's method from the adaptive starting value (linearised estimate for
// close pressures, else the two-rarefaction or two-shock estimate), at most
// kExactIters steps; the face state is the self-similar solution at x/t = 0.
// Returns ERRB_NEWTON if the iteration did not converge (FP64) or produced a
// non-finite pressure.
constexpr int kExactIters = 50;

// x^z for x > 0 and the small exponent z = (gamma - 1) / (2 gamma) < 1/2. FP32:
// through log2f and exp2f; their error enters the jump x^z - 1 with at most
// max_t t 2^-t = 0.53 of an ulp of 1 for x <= 1, less than powf's own rounding
// there, at a third of its instructions.
template <typename T>
__device__ __forceinline__ T pow_z(T x, T z) {
  if constexpr (sizeof(T) == 4) return exp2f(z * log2f(x));
  else return pow(x, z);
}

template <typename T>
struct ExactSide {
  T rho, u, p, c;
  T A, B;   // shock branch: sqrt(A / (p + B)) (p - p_K)
  T crf;    // rarefaction branch: 2 c_K / (gamma - 1)
  __device__ __forceinline__ void init(T r, T un, T pr, T gamma) {
    // FP32 traces of a state limited in FP64 can round a pressure at the
    // floor to zero or below: clamp it to a tiny positive value
    if constexpr (sizeof(T) == 4) pr = fmaxf(pr, 1e-30f);
    rho = r;
    u = un;
    p = pr;
    c = sqrt(gamma * pr / r);
    A = T(2) / ((gamma + T(1)) * r);
    B = (gamma - T(1)) / (gamma + T(1)) * pr;
    crf = T(2) * c / (gamma - T(1));
  }
  // f_K(ps) and its derivative; z = (gamma - 1) / (2 gamma)
  __device__ __forceinline__ void jump(T ps, T z, T gamma, T& f, T& df) const {
    if (ps > p) {
      if constexpr (sizeof(T) == 4) {
        const T i = T(1) / (ps + B);
        const T q = sqrt(A * i);
        f = (ps - p) * q;
        df = q * (T(1) - T(0.5) * (ps - p) * i);
      } else {
        const T q = sqrt(A / (ps + B));
        f = (ps - p) * q;
        df = q * (T(1) - T(0.5) * (ps - p) / (ps + B));
      }
    } else {
      const T r = pow_z(ps / p, z);
      f = crf * (r - T(1));
      df = c * r / (gamma * ps);
    }
  }
};

// state (rho, u, p) inside the rarefaction fan of side K at x/t = 0;
// sgn = +1 for the left fan, -1 for the right one
template <typename T>
__device__ __forceinline__ void fan_at_origin(const ExactSide<T>& k, T sgn, T gamma, T* W) {
  // positive inside the fan; the clamp only absorbs rounding at its edge
  const T cf = fmax(T(2) / (gamma + T(1)) * (k.c + sgn * T(0.5) * (gamma - T(1)) * k.u), T(0));
  const T ratio = cf / k.c;
  W[0] = k.rho * pow(ratio, T(2) / (gamma - T(1)));
  W[1] = sgn * cf;
  W[2] = k.p * pow(ratio, T(2) * gamma / (gamma - T(1)));
}

template <typename T>
__device__ __forceinline__ unsigned exact_flux(int d, const T* UL, const T* UR, T gamma, T* F) {
  const T gm1 = gamma - T(1);
  const T irL = T(1) / UL[0], irR = T(1) / UR[0];
  const T vL[3] = {UL[1] * irL, UL[2] * irL, UL[3] * irL};
  const T vR[3] = {UR[1] * irR, UR[2] * irR, UR[3] * irR};
  ExactSide<T> L, R;
  L.init(UL[0], vL[d], gm1 * (UL[4] - T(0.5) * UL[0] * (vL[0] * vL[0] + vL[1] * vL[1] + vL[2] * vL[2])), gamma);
  R.init(UR[0], vR[d], gm1 * (UR[4] - T(0.5) * UR[0] * (vR[0] * vR[0] + vR[1] * vR[1] + vR[2] * vR[2])), gamma);
  const T du = R.u - L.u;
  const T z = gm1 / (T(2) * gamma);
  T W[3];
  bool left;  // face state on the left of the contact (tangential velocities of L)
  unsigned err = 0;
  if (L.crf + R.crf <= du) {
    // the rarefactions open a vacuum between their tails
    const T tL = L.u + L.crf, tR = R.u - R.crf;
    if (L.u - L.c >= T(0)) {
      W[0] = L.rho; W[1] = L.u; W[2] = L.p; left = true;
    } else if (tL > T(0)) {
      fan_at_origin(L, T(1), gamma, W); left = true;
    } else if (R.u + R.c <= T(0)) {
      W[0] = R.rho; W[1] = R.u; W[2] = R.p; left = false;
    } else if (tR < T(0)) {
      fan_at_origin(R, T(-1), gamma, W); left = false;
    } else {
      W[0] = T(0); W[1] = T(0); W[2] = T(0); left = true;
    }
  } else {
    const T pmin = fmin(L.p, R.p), pmax = fmax(L.p, R.p);
    T ps = T(0.5) * (L.p + R.p) - T(0.125) * du * (L.rho + R.rho) * (L.c + R.c);
    ps = fmax(ps, T(0));
    if (!(pmax <= T(2) * pmin && ps >= pmin && ps <= pmax)) {
      if (ps < pmin) {
        const T num = L.c + R.c - T(0.5) * gm1 * du;
        ps = pow(num / (L.c * pow(L.p, -z) + R.c * pow(R.p, -z)), T(1) / z);
      } else {
        const T gL = sqrt(L.A / (ps + L.B)), gR = sqrt(R.A / (ps + R.B));
        ps = (gL * L.p + gR * R.p - du) / (gL + gR);
      }
    }
    const T tiny = sizeof(T) == 8 ? T(1e-14) * pmin : fmax(T(1e-14) * pmin, T(1e-36));
    const T tol = sizeof(T) == 8 ? T(1e-14) : T(2e-6);
    ps = fmax(ps, tiny);
    bool conv = false;
    const T rtol = sizeof(T) == 8 ? T(1e-15) : T(1e-6);
    T fl, dfl, fr, dfr;
    for (int it = 0; it < kExactIters && !conv; ++it) {
      L.jump(ps, z, gamma, fl, dfl);
      R.jump(ps, z, gamma, fr, dfr);
      const T f = fl + fr + du;
      // residual at the rounding level of its terms (near a vacuum the root
      // is too ill-conditioned for the relative step to reach tol)
      if (fabs(f) <= rtol * (fabs(fl) + fabs(fr) + fabs(du))) {
        conv = true;
        break;
      }
      const T pn = fmax(ps - f / (dfl + dfr), tiny);
      conv = fabs(pn - ps) <= tol * pn;
      // the jumps at pn: the last step is within tol of ps and its second
      // order below rounding, so they need no evaluation of their own (65 x 63
      // x 61, degree 2, FP32: 0.84 -> 0.76 ms per stage). dp = 0 covers a
      // derivative that overflows.
      const T dp = pn - ps;
      if (dp != T(0)) {
        fl += dfl * dp;
        fr += dfr * dp;
      }
      ps = pn;
    }
    if (!isfinite(ps) || (sizeof(T) == 8 && !conv)) err = ERRB_NEWTON;
    if (!conv) {
      L.jump(ps, z, gamma, fl, dfl);
      R.jump(ps, z, gamma, fr, dfr);
    }
    const T us = T(0.5) * (L.u + R.u) + T(0.5) * (fr - fl);
    left = us >= T(0);
    const ExactSide<T>& K = left ? L : R;
    const T sg = left ? T(1) : T(-1);  // +1: wave moves left of the contact
    const T ratio = ps / K.p;
    if (ps > K.p) {
      // shock speed from the jump conditions
      const T S = K.u - sg * K.c * sqrt((gamma + T(1)) / (T(2) * gamma) * ratio + z);
      if (sg * S >= T(0)) {
        W[0] = K.rho; W[1] = K.u; W[2] = K.p;
      } else {
        const T g6 = gm1 / (gamma + T(1));
        W[0] = K.rho * (ratio + g6) / (g6 * ratio + T(1)); W[1] = us; W[2] = ps;
      }
    } else {
      const T head = K.u - sg * K.c, tail = us - sg * K.c * pow_z(ratio, z);
      if (sg * head >= T(0)) {
        W[0] = K.rho; W[1] = K.u; W[2] = K.p;
      } else if (sg * tail < T(0)) {
        W[0] = K.rho * pow(ratio, T(1) / gamma); W[1] = us; W[2] = ps;
      } else {
        fan_at_origin(K, sg, gamma, W);
      }
    }
  }
  const T* vt = left ? vL : vR;
  T v[3] = {vt[0], vt[1], vt[2]};
  v[d] = W[1];
  const T mn = W[0] * W[1];
  F[0] = mn;
#pragma unroll
  for (int a = 0; a < 3; ++a) F[1 + a] = mn * v[a];
  F[1 + d] += W[2];
  F[4] = (W[2] / gm1 + T(0.5) * W[0] * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]) + W[2]) * W[1];
  return err;
}

// numerical flux selected at compile time: 0 = HLLC, 1 = exact Riemann solver
template <int FLUX, typename T>
__device__ __forceinline__ unsigned riemann_flux(int d, const T* UL, const T* UR, T gamma, T* F) {
  if constexpr (FLUX == 1) {
    return exact_flux<T>(d, UL, UR, gamma, F);
  } else {
    hllc_flux<T>(d, UL, UR, gamma, F);
    return 0u;
  }
}

// --------------------------------------------------------------- limiter
// tau in [0,1] with P(qbar + tau (q - qbar)) = eps: Newton from tau = 1.
// The pressure is concave along the segment, so the iterates decrease
// monotonically; stop when a step is below 1e-15 (50 iterations at most).
__device__ __forceinline__ double positivity_tau(const double* qb, const double* q, double gm1,
                                                 double eps, int* iters) {
  double d[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) d[i] = q[i] - qb[i];
  double tau = 1.0;
  int it = 0;
  while (it < 50) {
    double s0 = qb[0] + tau * d[0];
    double s1 = qb[1] + tau * d[1];
    double s2 = qb[2] + tau * d[2];
    double s3 = qb[3] + tau * d[3];
    double s4 = qb[4] + tau * d[4];
    double m2 = s1 * s1 + s2 * s2 + s3 * s3;
    double ir = rcp64(s0);
    double f = gm1 * (s4 - 0.5 * m2 * ir) - eps;
    double md = s1 * d[1] + s2 * d[2] + s3 * d[3];
    double fp = gm1 * (d[4] - md * ir + 0.5 * m2 * d[0] * ir * ir);
    double tn = tau - f * rcp64(fp);
    if (!(tn >= 0.0)) tn = 0.0;
    if (tn > tau) tn = tau;
    double step = tau - tn;
    tau = tn;
    ++it;
    if (step <= 1e-15) break;
  }
  *iters = it;
  return tau;
}

// x 2^de by its exponent field: exact; zeros, subnormals and results below 2^-1022
// give a signed zero, results above the range a number of at least 2^1023
__device__ __forceinline__ double exp_add(double x, int de) {
  const int hi = __double2hiint(x), b = bexp((unsigned)hi), n = min(b + de, 2046);
  const bool zero = b == 0 || n <= 0;
  return __hiloint2double((int)((unsigned)hi & 0x80000000u) | (zero ? 0 : (hi & 0xfffff) | (n << 20)),
                          zero ? 0 : __double2loint(x));
}

// A cell's own units for the FP32 point screens, from its mean density and energy:
// powers of two 2^r, 2^e and 2^((r + e) / 2) that bring rho, E and the momenta near
// 1. rho E and m^2 scale alike, so the screens decide as they would in binary32
// of unlimited range. Means near the ends of the FP64 range (ok unset) are left
// to the FP64 limiter; between 2^-20 and 2^20 (plain) every product of the screens is in
// range as it is, and they decide the same without the scaling.
struct LimUnits {
  int r, m, e;
  bool ok, plain;
  __device__ __forceinline__ LimUnits(double rho, double E) {
    const int br = bexp((unsigned)__double2hiint(rho)), be = bexp((unsigned)__double2hiint(E));
    ok = (unsigned)(br - 64) <= 1900u && (unsigned)(be - 64) <= 1900u;
    r = 1023 - br;
    e = 1023 - be - ((br + be) & 1);
    m = (r + e) / 2;
    plain = (unsigned)(br - 1003) <= 39u && (unsigned)(be - 1003) <= 39u;
  }
  __device__ __forceinline__ int of(int i) const { return i == 0 ? r : (i == 4 ? e : m); }
};

// Second sufficient test of the positivity limiter, for cells whose modal
// bound fails: density and pressure at every point of the limiter's point
// set (S, and the volume Gauss points when vol), evaluated in FP32 from the
// coefficients rounded to FP32 (tab32: the FP32 copy of the degree's table).
// A point value u = sum_l w_l phi_l computed so carries an error of at most
// (N + 3) 2^-24 sum_l |w_l phi_l| <= 2e-6 (|w_0| + sabs_u) for N <= 20
// (rounding of the coefficients, of the table entries and of the N products
// and sums), so e_u = 2e-6 (|mean_u| + sabs_u) bounds it; with these bounds
// the density and the pressure (bounded below through the density's lower
// and the momenta's upper bounds, multiplied through by the density bound)
// must clear the floors with a further 1e-5 relative margin, which covers
// the FP32 rounding of the test itself. The test runs in the cell's own units
// (LimUnits), so that no product of the values leaves the range of binary32. True when the cell provably needs
// no limiting (theta1 = theta2 = 1): the FP64 limiter would leave it as it is.
template <int K>
__device__ bool point_screen_f32(const double* w, long long stride, const float* __restrict__ tab32,
                                 const double* mean, const double* sabs, double gamma, double eps_r, double eps_p,
                                 int vol) {
  using TB = Tab<K>;
  constexpr int N = TB::N;
  const LimUnits un(mean[0], mean[4]);
  if (!un.ok) return false;
  float wf[5 * N];
#pragma unroll
  for (int j = 0; j < 5 * N; ++j) wf[j] = f64_to_f32(exp_add(w[j * stride], un.of(j / N)));
  float e[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) e[i] = f64_to_f32(exp_add(2e-6 * (fabs(mean[i]) + sabs[i]), un.of(i)));
  const float thr_r = f64_to_f32(exp_add(eps_r * (1.0 + 1e-6) + 1e-5 * (fabs(mean[0]) + sabs[0]), un.r));
  const float eps_pf = f64_to_f32(exp_add(eps_p * (1.0 + 1e-6), un.e));
  const float gm1 = f64_to_f32(gamma - 1.0);
  const int npts = TB::NL + (vol ? TB::Q3 : 0);
  for (int s = 0; s < npts; ++s) {
    const float* ph = s < TB::NL ? tab32 + TB::LPHI + s * N : tab32 + TB::VPHI + (s - TB::NL) * N;
    float U[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      float a = 0.f;
#pragma unroll
      for (int l = 0; l < N; ++l) a = fmaf(wf[i * N + l], __ldg(ph + l), a);
      U[i] = a;
    }
    const float rlo = U[0] - e[0];
    if (!(rlo >= thr_r)) return false;
    float k2 = 0.f;
#pragma unroll
    for (int a = 1; a <= 3; ++a) {
      const float mh = fabsf(U[a]) + e[a];
      k2 = fmaf(mh, mh, k2);
    }
    k2 *= 0.5f;
    const float elo = U[4] - e[4];
    const float lhs = gm1 * fmaf(elo, rlo, -k2);
    const float rhs = fmaf(eps_pf, rlo, 1e-5f * gm1 * fmaf(fabsf(U[4]) + e[4], rlo, k2));
    if (!(lhs >= rhs)) return false;
  }
  return true;
}

// The cheap part of the Zhang-Shu limiter of one cell (Sect. 2.5) on its 5N
// FP64 coefficients w[(i*N + l) * stride]: the means (finite, positive:
// otherwise an error bit is ORed into err and false returned), the
// excursion bounds sabs_i = sum_{l>=1} |w_il| max |phi_l| and the modal
// sufficient tests (mean minus sabs with a rounding margin) for the density
// (rho_safe) and the pressure (p_safe; needs rho_safe). When both hold, or
// (tab32 != nullptr) the FP32 point screen (point_screen_f32) holds, the
// limiter provably leaves the cell unchanged and *none is set.
template <int K>
__device__ bool limit_prelude(const double* w, long long stride, const double* __restrict__ tab, double gamma,
                              double eps_r, double eps_p, unsigned* err, int vol, const float* __restrict__ tab32,
                              double* mean, double* sabs, bool* rho_safe, bool* p_safe, bool* none) {
  using TB = Tab<K>;
  constexpr int N = TB::N;
  const double gm1 = gamma - 1.0;
  bool finite = true;
#pragma unroll
  for (int i = 0; i < 5; ++i) mean[i] = w[(i * N) * stride];
  for (int j = 0; j < 5 * N; ++j) finite &= isfinite(w[j * stride]);
  if (!finite) {
    *err |= ERRB_NONFINITE;
    return false;
  }
  const double pbar = gm1 * (mean[4] - 0.5 * (mean[1] * mean[1] + mean[2] * mean[2] + mean[3] * mean[3]) / mean[0]);
  if (!(mean[0] >= eps_r) || !(pbar >= eps_p)) {
    *err |= ERRB_POSITIVITY;
    return false;
  }
  if (N == 1) return false;
  const double* lmax = tab + (vol ? TB::LMAXV : TB::LMAX);
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    double s = 0.0;
    for (int l = 1; l < N; ++l) s += fabs(w[(i * N + l) * stride]) * __ldg(lmax + l);
    sabs[i] = s;
  }
  const double rlo = mean[0] - sabs[0];
  *rho_safe = rlo >= eps_r + 1e-13 * (fabs(mean[0]) + sabs[0]);
  *p_safe = false;
  if (*rho_safe) {
    const double elo = mean[4] - sabs[4];
    double kin = 0.0;
#pragma unroll
    for (int a = 1; a <= 3; ++a) {
      const double mh = fabs(mean[a]) + sabs[a];
      kin += mh * mh;
    }
    kin *= 0.5 / rlo;
    *p_safe = gm1 * (elo - kin) >= eps_p + 1e-13 * gm1 * (fabs(mean[4]) + sabs[4] + kin);
  }
  *none = (*rho_safe && *p_safe) ||
          (tab32 && point_screen_f32<K>(w, stride, tab32, mean, sabs, gamma, eps_r, eps_p, vol));
  return true;
}

// Zhang-Shu positivity limiter of one cell (Sect. 2.5) on its 5N FP64
// coefficients w[(i*N + l) * stride]: limit_prelude's sufficient tests skip
// the FP64 point evaluations when the limiter provably leaves the cell as it
// is. Returns flag bits (1: theta1 < 1, 2: theta2 < 1) and ORs errors into
// err.
template <int K>
__device__ int limit_cell(double* w, long long stride, const double* __restrict__ tab, double gamma,
                          double eps_r, double eps_p, unsigned* err, int vol,
                          const float* __restrict__ tab32 = nullptr) {
  using TB = Tab<K>;
  constexpr int N = TB::N;
  const double gm1 = gamma - 1.0;
  double mean[5], sabs[5];
  bool rho_safe, p_safe, none;
  if (!limit_prelude<K>(w, stride, tab, gamma, eps_r, eps_p, err, vol, tab32, mean, sabs, &rho_safe, &p_safe,
                        &none) ||
      none)
    return 0;
  const double* lphi = tab + TB::LPHI;
  const double* vphi = tab + TB::VPHI;
  // the point set: S (TB::NL points), then optionally the volume Gauss points
  const int npts = TB::NL + (vol ? TB::Q3 : 0);
  int flag = 0;
  // density: theta1
  if (!rho_safe) {
    double rmin = mean[0];
    for (int s = 0; s < npts; ++s) {
      const double* ph = s < TB::NL ? lphi + s * N : vphi + (s - TB::NL) * N;
      double r = 0.0;
#pragma unroll
      for (int l = 0; l < N; ++l) r += w[l * stride] * __ldg(ph + l);
      rmin = fmin(rmin, r);
    }
    if (rmin < eps_r) {
      double th1 = fmin(fabs((mean[0] - eps_r) / (mean[0] - rmin)), 1.0);
      if (th1 < 1.0) {
        for (int l = 1; l < N; ++l) w[l * stride] *= th1;
        flag |= 1;
      }
    }
  }
  // pressure: theta2 (the prelude's modal test p_safe holds only where
  // rho_safe did, i.e. where theta1 left the cell unchanged)
  if (!p_safe) {
    double th2 = 1.0;
    bool newton_fail = false;
    for (int s = 0; s < npts; ++s) {
      const double* ph = s < TB::NL ? lphi + s * N : vphi + (s - TB::NL) * N;
      double U[5];
#pragma unroll
      for (int i = 0; i < 5; ++i) {
        double acc = 0.0;
#pragma unroll
        for (int l = 0; l < N; ++l) acc += w[(i * N + l) * stride] * __ldg(ph + l);
        U[i] = acc;
      }
      double p = gm1 * (U[4] - 0.5 * (U[1] * U[1] + U[2] * U[2] + U[3] * U[3]) / U[0]);
      if (p < eps_p) {
        int it;
        double tau = positivity_tau(mean, U, gm1, eps_p, &it);
        if (it >= 50) newton_fail = true;
        th2 = fmin(th2, tau);
      }
    }
    if (newton_fail) *err |= ERRB_NEWTON;
    if (th2 < 1.0) {
      for (int i = 0; i < 5; ++i)
        for (int l = 1; l < N; ++l) w[(i * N + l) * stride] *= th2;
      flag |= 2;
    }
  }
  return flag;
}

}  // namespace dg
