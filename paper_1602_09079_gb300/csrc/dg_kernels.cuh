// dg_kernels.cuh -- CUDA kernels of the modal DG hot path (arXiv:1602.09079,
// Sect. 2.3-2.5, 3.1-3.2), templated on the polynomial degree K and the
// quadrature type T (double: plain FP64 path; float: mixed path whose RK
// accumulation, limiter and reductions stay FP64).
//
// State layout: y[(i*N + l) * nc + c], rows contiguous over cells (x-fastest),
// so every per-row access of a warp over consecutive cells is coalesced.
//
// One RHS evaluation = a face kernel (one Riemann flux per face point, face
// owned by its upper cell, written once) + a volume kernel (volume
// quadrature, flux projection onto the basis gradients, the two face fluxes
// of each direction projected onto the face traces, and an epilogue: R, or
// the SSP-RK3 stage combination in FP64 followed by the limiter screen of
// the next stage's input).
#pragma once
#include "dg_common.cuh"

namespace dg {

// threads per CTA of the tiled kernels: a multiple of the 5 (k + 1) (cell,
// variable, slice) roles per cell of volume_sf_kernel at every degree
constexpr int kThreads = 240;

enum VolMode { MODE_RHS = 0, MODE_STAGE = 1 };

// Cells per CTA of the volume kernel: the flux staging buffer
// (15 Q^3 values per cell) stays near 128 KB of shared memory.
template <int K, typename T>
struct VolCfg {
  static constexpr int Q3 = (K + 1) * (K + 1) * (K + 1);
  static constexpr int raw = (128 * 1024) / (15 * Q3 * (int)sizeof(T));
  static constexpr int C = raw >= 128 ? 128 : raw >= 64 ? 64 : raw >= 32 ? 32 : 16;
  static constexpr int N = nmodes(K);
  static constexpr size_t smem(bool force) {
    return sizeof(T) * (size_t)(5 * N * C)            // sW: stage input
           + sizeof(T) * (size_t)(15 * Q3 * C)        // sF: volume fluxes
           + (force ? sizeof(T) * (size_t)(4 * Q3 * C) : 0)  // sS: source
           + sizeof(double) * (size_t)(5 * N * C);    // sY: FP64 stage output
  }
};

struct StageArgs {
  const double* ys;  // stage input y^(s)
  const double* y0;  // y^(0) of the step
  double* out;       // stage output (may alias ys or y0; cells are CTA-private)
  double a0, b0, dt; // out = a0 y0 + b0 (ys - dt R(ys))
  int* list;         // cells whose limiter screen failed
  float* yf;         // FP32 shadow of the stage state (FP32 path): read for
                     // this CTA's cells, then overwritten with the output
};

// the queue's counter, by the face kernels: the volume kernel after them queues cells
__device__ __forceinline__ void clear_queue(Ctrl* ctrl) {
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) ctrl->n_flag = 0u;
}

// first thing in every kernel that queues cells: the second pass's counter
__device__ __forceinline__ void clear_deep(Ctrl* ctrl) {
  if (blockIdx.x == 0 && threadIdx.x == 0) ctrl->n_deep = 0u;
}

__device__ __forceinline__ void cell_xyz(long long c, const Geo& g, int& ix, int& iy, int& iz) {
  int cc = (int)c;
  ix = cc % g.nx;
  int r = cc / g.nx;
  iy = r % g.ny;
  iz = r / g.ny;
}

__device__ __forceinline__ long long neighbour(const Geo& g, int ix, int iy, int iz, int d, int s) {
  if (d == 0) ix = (ix + s + g.nx) % g.nx;
  else if (d == 1) iy = (iy + s + g.ny) % g.ny;
  else iz = (iz + s + g.nz) % g.nz;
  return ((long long)iz * g.ny + iy) * g.nx + ix;
}

// ------------------------------------------------------------ face fluxes
// Face (d, c) joins the lower cell c - e_d (left state, its high face) and
// cell c (right state, its low face), fh[((d*5 + i)*Q2 + p)*nc + c]; the
// kernels (face_sf64_kernel, face_flux_f32_kernel) follow the FP32 section.

// Screen of the positivity limiter from a cell's FP64 means and the sums
// sabs_i = sum_{l>=1} |w_il| max_S |phi_l| (same test and margins as
// limit_cell): true when the cell provably needs no limiting.
template <int K>
__device__ __forceinline__ bool limiter_screen(const double* mean, const double* sabs, bool finite, double gamma,
                                               double eps_r, double eps_p) {
  if (!finite) return false;
  const double gm1 = gamma - 1.0;
  const double r = mean[0];
  const double pbar = gm1 * (mean[4] - 0.5 * (mean[1] * mean[1] + mean[2] * mean[2] + mean[3] * mean[3]) / r);
  if (!(r >= eps_r) || !(pbar >= eps_p)) return false;
  if (nmodes(K) == 1) return true;
  const double rlo = r - sabs[0];
  if (!(rlo >= eps_r + 1e-13 * (fabs(r) + sabs[0]))) return false;
  const double elo = mean[4] - sabs[4];
  double kin = 0.0;
#pragma unroll
  for (int a = 1; a <= 3; ++a) {
    const double mh = fabs(mean[a]) + sabs[a];
    kin += mh * mh;
  }
  kin *= 0.5 / rlo;
  const double plo = gm1 * (elo - kin);
  return plo >= eps_p + 1e-13 * gm1 * (fabs(mean[4]) + sabs[4] + kin);
}

// --------------------------------------------------------------- volume
template <int K, typename T, int MODE, bool FORCE>
__global__ void __launch_bounds__(kThreads) volume_kernel(const double* __restrict__ yin, const T* __restrict__ fh,
                                                          const T* __restrict__ field, const T* __restrict__ tab,
                                                          const double* __restrict__ tab64, Geo g, StageArgs st,
                                                          double* __restrict__ R, Ctrl* ctrl) {
  stream_wait();
  using TB = Tab<K>;
  using CF = VolCfg<K, T>;
  constexpr int N = TB::N, Q2 = TB::Q2, Q3 = TB::Q3, C = CF::C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* sY = reinterpret_cast<double*>(smem_raw);
  T* sW = reinterpret_cast<T*>(sY + 5 * N * C);
  T* sF = sW + 5 * N * C;
  T* sS = sF + 15 * Q3 * C;
  if (MODE == MODE_STAGE) clear_deep(ctrl);
  const long long nc = g.nc;
  const long long c0 = (long long)blockIdx.x * C;
  const int tid = threadIdx.x;
  const double* ysrc = (MODE == MODE_STAGE) ? st.ys : yin;

  // phase 1: stage input -> shared (converted to T), coalesced rows
  for (int it = tid; it < 5 * N * C; it += kThreads) {
    const int c = it % C, r = it / C;
    const long long cell = c0 + c;
    sW[r * C + c] = cell < nc ? (T)ysrc[(size_t)r * nc + cell] : T(0);
  }
  __syncthreads();

  // phase 2: values at the volume Gauss points, Euler fluxes, source
  const T gm1 = (T)(g.gamma - 1.0);
  const T idx0 = (T)g.inv_dx[0], idx1 = (T)g.inv_dx[1], idx2 = (T)g.inv_dx[2];
  for (int it = tid; it < Q3 * C; it += kThreads) {
    const int c = it % C, q = it / C;
    const long long cell = c0 + c;
    if (cell >= nc) continue;
    const T* ph = tab + TB::VPHI + q * N;
    T U[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      T a = T(0);
#pragma unroll
      for (int l = 0; l < N; ++l) a += sW[(i * N + l) * C + c] * __ldg(ph + l);
      U[i] = a;
    }
    const T ir = T(1) / U[0];
    const T v[3] = {U[1] * ir, U[2] * ir, U[3] * ir};
    const T p = gm1 * (U[4] - T(0.5) * U[0] * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]));
    const T idx[3] = {idx0, idx1, idx2};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      T F[5];
      euler_flux<T>(d, U, v, p, F);
#pragma unroll
      for (int i = 0; i < 5; ++i) sF[((d * 5 + i) * Q3 + q) * C + c] = F[i] * idx[d];
    }
    if (FORCE) {
      T a[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) a[d] = __ldg(field + ((size_t)d * Q3 + q) * nc + cell);
      sS[(0 * Q3 + q) * C + c] = U[0] * a[0];
      sS[(1 * Q3 + q) * C + c] = U[0] * a[1];
      sS[(2 * Q3 + q) * C + c] = U[0] * a[2];
      sS[(3 * Q3 + q) * C + c] = U[1] * a[0] + U[2] * a[1] + U[3] * a[2];
    }
  }
  __syncthreads();

  // phase 3: projection onto the basis (volume, source, faces): dw/dt
  for (int it = tid; it < 5 * C; it += kThreads) {
    const int c = it % C, i = it / C;
    const long long cell = c0 + c;
    if (cell >= nc) continue;
    T acc[N];
#pragma unroll
    for (int l = 0; l < N; ++l) acc[l] = T(0);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      for (int q = 0; q < Q3; ++q) {
        const T f = sF[((d * 5 + i) * Q3 + q) * C + c];
        const T* dp = tab + TB::VDPHI + (d * Q3 + q) * N;
#pragma unroll
        for (int l = 0; l < N; ++l) acc[l] += f * __ldg(dp + l);
      }
    }
    if (FORCE && i > 0) {
      for (int q = 0; q < Q3; ++q) {
        const T s = sS[((i - 1) * Q3 + q) * C + c];
        const T* pw = tab + TB::VPHIW + q * N;
#pragma unroll
        for (int l = 0; l < N; ++l) acc[l] += s * __ldg(pw + l);
      }
    }
    int ix, iy, iz;
    cell_xyz(cell, g, ix, iy, iz);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const long long cu = neighbour(g, ix, iy, iz, d, +1);
      const T idx = (T)g.inv_dx[d];
      for (int p = 0; p < Q2; ++p) {
        const size_t base = ((size_t)(d * 5 + i) * Q2 + p) * nc;
        const T fm = __ldg(fh + base + cell) * idx;  // low face of this cell
        const T fp = __ldg(fh + base + cu) * idx;    // high face (owned by the upper cell)
        const T* wl = tab + TB::FPHIW + ((d * 2 + 0) * Q2 + p) * N;
        const T* wh = tab + TB::FPHIW + ((d * 2 + 1) * Q2 + p) * N;
#pragma unroll
        for (int l = 0; l < N; ++l) acc[l] += fm * __ldg(wl + l) - fp * __ldg(wh + l);
      }
    }
    if (MODE == MODE_RHS) {
#pragma unroll
      for (int l = 0; l < N; ++l) R[(size_t)(i * N + l) * nc + cell] = -(double)acc[l];
    } else {
#pragma unroll
      for (int l = 0; l < N; ++l) {
        const size_t a = (size_t)(i * N + l) * nc + cell;
        sY[(i * N + l) * C + c] = st.a0 * st.y0[a] + st.b0 * (st.ys[a] + st.dt * (double)acc[l]);
      }
    }
  }
  if (MODE == MODE_RHS) return;
  __syncthreads();

  // phase 4: limiter screen of the next stage's input (FP64); cells that
  // fail it are queued for the full limiter
  for (int it = tid; it < 5 * N * C; it += kThreads) {
    const int c = it % C, r = it / C;
    const long long cell = c0 + c;
    if (cell < nc) st.out[(size_t)r * nc + cell] = sY[r * C + c];
  }
  if (tid < C) {
    const long long cell = c0 + tid;
    if (cell < nc) {
      double m[5], a[5];
      bool fin = true;
#pragma unroll
      for (int i = 0; i < 5; ++i) {
        m[i] = sY[(i * N) * C + tid];
        double sa = 0.0;
        for (int l = 1; l < N; ++l) sa += fabs(sY[(i * N + l) * C + tid]) * __ldg(tab64 + (g.lim_vol ? TB::LMAXV : TB::LMAX) + l);
        a[i] = sa;
        for (int l = 0; l < N; ++l) fin &= isfinite(sY[(i * N + l) * C + tid]);
      }
      if (!limiter_screen<K>(m, a, fin, g.gamma, g.eps_rho, g.eps_p)) {
        const unsigned slot = atomicAdd(&ctrl->n_flag, 1u);
        st.list[slot] = (int)cell;
      }
    }
  }
}

// ============================================================ FP32 path

// FP32 copy of this degree's tables in constant memory: with the point and
// mode loops unrolled, every table value is a compile-time offset into the
// constant bank and becomes an FMA operand (no load instruction).
namespace {
__constant__ float c_tab32[Tab<3>::SIZE];
// 1D tables of the sum-factorised kernels for this translation unit's
// degree (KQ = (k+1)^2): Pt_u(x_a) at [u*Q + a], Pt_u(x_a) w_a at KQ + [u*Q + a],
// Pt_u'(x_a) w_a at 2 KQ + [u*Q + a], Pt_e(-1) at 3 KQ + e, Pt_e(+1) at
// 3 KQ + (k+1) + e. With unrolled loops every entry is a constant-bank operand.
__constant__ float c_sf32[3 * 16 + 8];
__constant__ double c_sf64[3 * 16 + 8];
}

template <typename T>
__device__ __forceinline__ T sfc(int i);
template <>
__device__ __forceinline__ float sfc<float>(int i) { return c_sf32[i]; }
template <>
__device__ __forceinline__ double sfc<double>(int i) { return c_sf64[i]; }

// Face fluxes, FP32 (from the FP32 shadow of the state): tiles of 32
// consecutive cells, warp d computes the low
// face in direction d of each cell (left state = the lower neighbour's high
// face, right state = the cell's own low face). Traces are sum-factorised:
// the coefficients are first contracted with Pt_e(+-1) along the normal into
// the tangential coefficients E[i][(a,b)], which then give the values at all
// Q^2 face points through the tangential products (constant tables).
template <int K, int D, int FLUX>
__device__ __forceinline__ unsigned face_f32_dir(const float* __restrict__ yf, float* __restrict__ fh, const Geo& g,
                                                 long long c, int ix, int iy, int iz) {
  using TB = Tab<K>;
  constexpr int N = TB::N, Q2 = TB::Q2, T = TB::T;
  const long long nc = g.nc;
  const long long cl = neighbour(g, ix, iy, iz, D, -1);
  float EL[5 * T], ER[5 * T];
#pragma unroll
  for (int j = 0; j < 5 * T; ++j) {
    EL[j] = 0.f;
    ER[j] = 0.f;
  }
  // exponents along (normal, tangential 1, tangential 2) -> (u, v, w)
#pragma unroll
  for (int a = 0, j = 0; a <= K; ++a)
#pragma unroll
    for (int b = 0; a + b <= K; ++b, ++j)
#pragma unroll
      for (int e = 0; e + a + b <= K; ++e) {
        const int m = D == 0 ? mode_index(e, a, b) : (D == 1 ? mode_index(a, e, b) : mode_index(a, b, e));
        const float pl = c_tab32[TB::FEND + (K + 1) + e];  // lower cell: its high face, xi_d = +1
        const float pr = c_tab32[TB::FEND + e];            // own cell: its low face, xi_d = -1
#pragma unroll
        for (int i = 0; i < 5; ++i) {
          EL[i * T + j] += __ldg(yf + (size_t)(i * N + m) * nc + cl) * pl;
          ER[i * T + j] += __ldg(yf + (size_t)(i * N + m) * nc + c) * pr;
        }
      }
  const float gamma = (float)g.gamma;
  unsigned err = 0;
#pragma unroll 1
  for (int p = 0; p < Q2; ++p) {
    float UL[5], UR[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      float aL = 0.f, aR = 0.f;
#pragma unroll
      for (int j = 0; j < T; ++j) {
        const float t2 = c_tab32[TB::F2D + p * T + j];
        aL += EL[i * T + j] * t2;
        aR += ER[i * T + j] * t2;
      }
      UL[i] = aL;
      UR[i] = aR;
    }
    float F[5];
    err |= riemann_flux<FLUX, float>(D, UL, UR, gamma, F);
#pragma unroll
    for (int i = 0; i < 5; ++i) fh[((size_t)(D * 5 + i) * Q2 + p) * nc + c] = F[i];
  }
  return err;
}

// Face fluxes, FP64: tile of 32 cells, one direction after the other. One
// (cell, variable) per thread (warp = variable) contracts the coefficients of
// its cell and of the lower neighbour along the normal with Pt_e(-+1) into the
// tangential coefficients E, then along t2 and t1 to the values at the face's
// Q^2 points, all in 64-bit fixed point (dg_common.cuh): both sides' values go
// to shared memory in the face's frame. Then one numerical flux per face point
// in FP64, which with the integer work is what bounds the kernel (27 HLLC fluxes of
// about 70 FP64 operations per cell at degree 2, 2 operations per clock and SM). The fluxes go
// out as their T = (K+1)(K+2)/2 moments with the tangential modes,
// [3][5][T][n_cells], once for the two cells that need them (MOMENTS; for the
// dense volume_kernel the fluxes at the points, [3][5][Q^2][n_cells]). With FP64 contractions
// and the 190-operation HLLC the kernel took 21.5 ms at 128^3, degree 2, now
// 8.74 (the FP64 operations alone: 6.2).
template <int K>
struct FaceSF64 {
  static constexpr int C = 32, THREADS = 5 * C;
  static constexpr int Q2 = (K + 1) * (K + 1), T = (K + 1) * (K + 2) / 2;
  // CTAs per SM the register budget is sized for (128^3, degree 2: 8.74 ms with
  // 5, 8.85 with 4; 64^3, degree 3: 2.36, 2.41)
  static constexpr int MINB = 5;
  // values [side][variable][point][cell]
  static constexpr size_t smem() { return sizeof(double) * 2 * 5 * Q2 * C; }
};

// index of the mode with the exponents (e, a, b) along (normal, tangential 1,
// tangential 2) of a face normal to d, by the index of (e, a, b) as (u, v, w)
static __constant__ unsigned char c_face_order[3][20] = {
    {0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16, 17, 18, 19},
    {0, 2, 1, 3, 7, 5, 8, 4, 6, 9, 16, 13, 17, 11, 14, 18, 10, 12, 15, 19},
    {0, 3, 1, 2, 9, 6, 8, 4, 5, 7, 19, 15, 18, 12, 14, 17, 10, 11, 13, 16}};

// coefficients of one (cell, variable) in fixed point, exponent B; row stride nc
// (order: the modes' order along the face's axes)
template <int K>
__device__ __forceinline__ void fx_load(const double* __restrict__ p, size_t nc, Fx (&x)[nmodes(K)], int& B,
                                        const unsigned char* order = nullptr) {
  constexpr int N = nmodes(K);
  double w[N];
#pragma unroll
  for (int l = 0; l < N; ++l) w[l] = __ldg(p + (size_t)(order ? order[l] : l) * nc);
  B = fx_bound<K>(w);
#pragma unroll
  for (int l = 0; l < N; ++l) x[l] = fx_split(fx_from(w[l], B));
}

// rows of a triangle E[(a, b)] at the nodes along b: H[q][a] = sum_b E[(a, b)] Pt_b(q)
template <int K, int A>
__device__ __forceinline__ void fx_rows(const Fx (&E)[(K + 1) * (K + 2) / 2], Fx (&H)[K + 1][K + 1]) {
  if constexpr (A <= K) {
    Fx e[K + 1 - A];
    long long v[K + 1];
#pragma unroll
    for (int b = 0; b + A <= K; ++b) e[b] = E[pair_index(K, A, b)];
    fx_values<K, K + 1 - A>(e, v);
#pragma unroll
    for (int q = 0; q <= K; ++q) H[q][A] = fx_split(v[q]);
    fx_rows<K, A + 1>(E, H);
  }
}

// values on the face at xi = -1 (S = 0) or +1 (S = 1) of the first axis at the
// points t1 + Q t2, rows of 32 cells apart
template <int K, int S>
__device__ __forceinline__ void fx_trace(const Fx (&x)[nmodes(K)], int B, double* dst) {
  using FT = FxTab<K>;
  constexpr int Q = K + 1, T = (K + 1) * (K + 2) / 2;
  const double bad = __longlong_as_double(0x7ff8000000000000LL);
  Fx E[T];
#pragma unroll
  for (int a = 0, j = 0; a <= K; ++a)
#pragma unroll
    for (int b = 0; a + b <= K; ++b, ++j) {
      FxAcc s{0, 0};
#pragma unroll
      for (int e = 1; e + a + b <= K; ++e) fx_madt(s, x[mode_index(e, a, b)], FT::E + S * (K + 1) + e);
      // Pt_0 = 1
      E[j] = fx_split(fx_val(s) + fx_join(x[mode_index(0, a, b)]));
    }
  Fx H[Q][K + 1];  // [t2][a]
  fx_rows<K, 0>(E, H);
#pragma unroll
  for (int t2 = 0; t2 < Q; ++t2) {
    long long v[Q];
    fx_values<K, K + 1>(H[t2], v);
#pragma unroll
    for (int t1 = 0; t1 < Q; ++t1) dst[(t1 + Q * t2) * 32] = B < kFxHuge ? fx_to_double(v[t1], B) : bad;
  }
}

// T moments sum_{t1,t2} F(t1 + Q t2) P'_a(t1) P'_b(t2), P' = Pt w / 2, of the
// flux values f (Q^2 rows of 32 cells), to m (rows nc apart)
template <int K>
__device__ __forceinline__ void fx_moments(const double* f, double* __restrict__ m, size_t nc) {
  constexpr int Q = K + 1, Q2 = Q * Q;
  unsigned mx = 0;
#pragma unroll
  for (int p = 0; p < Q2; ++p) mx = max(mx, (unsigned)__double2hiint(f[p * 32]) & 0x7fffffffu);
  const int B = max(kFxTiny, bexp(mx) + 1);
  const double bad = __longlong_as_double(0x7ff8000000000000LL);
  long long G[K + 1][Q];  // [a][t2]
#pragma unroll
  for (int t2 = 0; t2 < Q; ++t2) {
    long long v[Q];
#pragma unroll
    for (int t1 = 0; t1 < Q; ++t1) v[t1] = fx_from(f[(t1 + Q * t2) * 32], B);
    FxAcc g[K + 1];
#pragma unroll
    for (int a = 0; a <= K; ++a) g[a] = {0, 0};
    fx_project<K, false>(v, g);
#pragma unroll
    for (int a = 0; a <= K; ++a) G[a][t2] = fx_val(g[a]);
  }
#pragma unroll
  for (int a = 0, j = 0; a <= K; ++a) {
    FxAcc h[K + 1];
#pragma unroll
    for (int b = 0; b <= K; ++b) h[b] = {0, 0};
    fx_project<K, false>(G[a], h);
#pragma unroll
    for (int b = 0; a + b <= K; ++b, ++j) m[(size_t)j * nc] = B < kFxHuge ? fx_to_double(fx_val(h[b]), B) : bad;
  }
}

template <int K, int FLUX, bool MOMENTS = (K >= 2)>
__global__ void __launch_bounds__(FaceSF64<K>::THREADS, FaceSF64<K>::MINB) face_sf64_kernel(const double* __restrict__ y,
                                                                         double* __restrict__ fh, Geo g, Ctrl* ctrl) {
  stream_wait();
  using CF = FaceSF64<K>;
  constexpr int N = nmodes(K), C = CF::C, Q2 = CF::Q2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* sU = reinterpret_cast<double*>(smem_raw);
  const long long nc = g.nc, c0 = (long long)blockIdx.x * C;
  const int c = threadIdx.x % C, i = threadIdx.x / C;  // i: conserved variable, warp-uniform
  clear_queue(ctrl);
  const long long cell = c0 + c;
  const bool live = cell < nc;
  int ix = 0, iy = 0, iz = 0;
  if (live) cell_xyz(cell, g, ix, iy, iz);
  const double* yi = y + (size_t)(i * N) * nc;
  unsigned err = 0;
  // directions blockIdx.y, + gridDim.y, ...: all in one CTA, or one per CTA
  // where a mesh has too few tiles to fill the chip. The coefficients are read
  // in the order of the face's axes, so that one copy of the trace code serves
  // the three directions (three copies missed the instruction cache: 9.15 ms per
  // stage at 128^3, degree 2, one 8.85)
#pragma unroll 1
  for (int d = blockIdx.y; d < 3; d += gridDim.y) {
    if (live) {
      // row of this variable in the face's frame (rho, m_n, m_t1, m_t2, E)
      double* dst = sU + face_var(d, i) * Q2 * C + c;
      Fx x[N];
      int B;
      fx_load<K>(yi + neighbour(g, ix, iy, iz, d, -1), nc, x, B, c_face_order[d]);
      fx_trace<K, 1>(x, B, dst);
      fx_load<K>(yi + cell, nc, x, B, c_face_order[d]);
      fx_trace<K, 0>(x, B, dst + 5 * Q2 * C);
    }
    __syncthreads();
#pragma unroll 1
    for (int it = threadIdx.x; it < Q2 * C; it += CF::THREADS) {
      const int p = it / C, cc = it % C;
      if (c0 + cc < nc) {
        double UL[5], UR[5], F[5];
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          UL[v] = sU[(v * Q2 + p) * C + cc];
          UR[v] = sU[((5 + v) * Q2 + p) * C + cc];
        }
        if constexpr (FLUX == 1) err |= exact_flux<double>(0, UL, UR, g.gamma, F);
        else hllc64_x(UL, UR, g.gamma, F);
        // the flux takes the left values' place (or goes out as it is)
#pragma unroll
        for (int v = 0; v < 5; ++v) {
          if constexpr (MOMENTS) {
            sU[(v * Q2 + p) * C + cc] = F[v];
          } else {
            // position of the frame's component v among (rho, m_x, m_y, m_z, E)
            const int ax = v == 1 ? d : (v == 2 ? (d == 0 ? 1 : 0) : (d == 2 ? 1 : 2));
            fh[((size_t)(d * 5 + ((v == 0 || v == 4) ? v : 1 + ax)) * Q2 + p) * nc + c0 + cc] = F[v];
          }
        }
      }
    }
    if constexpr (MOMENTS) {
      __syncthreads();
      if (live)
        fx_moments<K>(sU + face_var(d, i) * Q2 * C + c, fh + (size_t)(d * 5 + i) * CF::T * nc + cell, nc);
    }
    __syncthreads();
  }
  if (err) atomicOr(&ctrl->err, err);
}

// CTAs per SM the face kernel's register budget is sized for (measured at
// degree 2, 128^3: 4 CTAs 0.82 ms, 6 CTAs 0.92 ms, 8 CTAs 1.06 ms)
template <int K>
struct FaceF32 {
  static constexpr int MINB = 4;
};

template <int K, int FLUX>
__global__ void __launch_bounds__(96, FaceF32<K>::MINB) face_flux_f32_kernel(const float* __restrict__ yf, float* __restrict__ fh,
                                                              Geo g, Ctrl* ctrl) {
  stream_wait();
  clear_queue(ctrl);
  const long long c = (long long)blockIdx.x * 32 + (threadIdx.x & 31);
  if (c >= g.nc) return;
  const int d = threadIdx.x >> 5;  // warp-uniform direction
  int ix, iy, iz;
  cell_xyz(c, g, ix, iy, iz);
  unsigned e;
  if (d == 0) e = face_f32_dir<K, 0, FLUX>(yf, fh, g, c, ix, iy, iz);
  else if (d == 1) e = face_f32_dir<K, 1, FLUX>(yf, fh, g, c, ix, iy, iz);
  else e = face_f32_dir<K, 2, FLUX>(yf, fh, g, c, ix, iy, iz);
  if (e) atomicOr(&ctrl->err, e);
}

// Volume quadrature, FP32, tiled in two phases over a tile of C cells:
//  A) one warp per group of PG volume points (warp-uniform group, so the
//     point loop unrolls against compile-time constant-table offsets): the
//     cell's coefficients in registers, values at the points, Euler fluxes
//     (and the driving source) to shared memory;
//  B) one warp per conserved variable: the N accumulators of one (cell,
//     variable) in registers, the flux projection onto the basis gradients,
//     the source projection and the six face fluxes projected onto the face
//     traces, every table value a constant-bank operand; then R, or the FP64
//     SSP-RK3 stage combination and the limiter screen (cells failing it are
//     queued for the full limiter).
template <int K>
struct VolF32 {
  static constexpr int Q3 = (K + 1) * (K + 1) * (K + 1);
  static constexpr int N = nmodes(K);
  static constexpr int C = K >= 2 ? 32 : 64;  // cells per tile (a multiple of 32)
  static constexpr int NW = K >= 2 ? 3 : (K == 1 ? 2 : 1);  // warps of phase A (point subgroups)
  static constexpr int NCH = K >= 2 ? 3 : 1;                // point chunks (phase A/B rounds)
  static constexpr int PC = Q3 / NCH;                       // points per chunk
  static constexpr int PW = PC / NW;                        // points per phase-A warp and chunk
  static constexpr int THREADS = 5 * C;
  // CTAs per SM the register budget is sized for (degree 2: 56 registers,
  // no spills; 7 CTAs also fill the shared memory). Measured at 128^3,
  // degree 2: 5 CTAs 3.49 ms, 6 3.13, 7 3.00, 8 3.12
  static constexpr int MINB = K >= 2 ? 7 : 3;
  static constexpr size_t smem(bool force) {
    return sizeof(float) * (size_t)(5 * N * C + 15 * PC * C + (force ? 4 * PC * C : 0)) +
           sizeof(double) * (size_t)(10 * C);
  }
  static_assert(K > 2 || (Q3 % NCH == 0 && PC % NW == 0), "point chunks");
};

// phase A of one chunk for one warp: points q = CH*PC + W*PW + j
template <int K, int CH, int W, bool FORCE>
__device__ __forceinline__ void vol_f32_points(const float* sW, float* sF, float* sS, const float* __restrict__ field,
                                               int c, long long cell, long long nc, float gm1, const float* idx) {
  using TB = Tab<K>;
  using CF = VolF32<K>;
  constexpr int N = TB::N, Q3 = TB::Q3, C = CF::C, PC = CF::PC, PW = CF::PW;
  // one point at a time: the coefficients are re-read from shared memory
  // for each point, so no more than the point's five values stay live (the
  // kernel then fits its register budget without spilling)
#pragma unroll
  for (int j = 0; j < PW; ++j) {
    const int ql = W * PW + j;  // point within the chunk
    const int q = CH * PC + ql;
    float U[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      float a = 0.f;
#pragma unroll
      for (int l = 0; l < N; ++l) a += sW[(i * N + l) * C + c] * c_tab32[TB::VPHI + q * N + l];
      U[i] = a;
    }
    const float ir = 1.f / U[0];
    const float v[3] = {U[1] * ir, U[2] * ir, U[3] * ir};
    const float p = gm1 * (U[4] - 0.5f * U[0] * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]));
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      float F[5];
      euler_flux<float>(d, U, v, p, F);
#pragma unroll
      for (int i = 0; i < 5; ++i) sF[((d * 5 + i) * PC + ql) * C + c] = F[i] * idx[d];
    }
    if (FORCE) {
      float a[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) a[d] = __ldg(field + ((size_t)d * Q3 + q) * nc + cell);
      sS[(0 * PC + ql) * C + c] = U[0] * a[0];
      sS[(1 * PC + ql) * C + c] = U[0] * a[1];
      sS[(2 * PC + ql) * C + c] = U[0] * a[2];
      sS[(3 * PC + ql) * C + c] = U[1] * a[0] + U[2] * a[1] + U[3] * a[2];
    }
    // without the driving-field loads the scheduler hoists the next points'
    // shared loads over this one and spills (ptxas: 836 B per thread); a
    // compiler memory barrier keeps one point live at a time
    if (!FORCE) asm volatile("" ::: "memory");
  }
}

// phase B of one chunk: accumulate the projections of its points
template <int K, int CH, bool FORCE>
__device__ __forceinline__ void vol_f32_project(const float* sF, const float* sS, int c, int i, float (&acc)[nmodes(K)]) {
  using TB = Tab<K>;
  using CF = VolF32<K>;
  constexpr int N = TB::N, Q3 = TB::Q3, C = CF::C, PC = CF::PC;
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int ql = 0; ql < PC; ++ql) {
      const int q = CH * PC + ql;
      const float f = sF[((d * 5 + i) * PC + ql) * C + c];
#pragma unroll
      for (int l = 0; l < N; ++l) acc[l] += f * c_tab32[TB::VDPHI + (d * Q3 + q) * N + l];
    }
  if (FORCE && i > 0) {
#pragma unroll
    for (int ql = 0; ql < PC; ++ql) {
      const int q = CH * PC + ql;
      const float sv = sS[((i - 1) * PC + ql) * C + c];
#pragma unroll
      for (int l = 0; l < N; ++l) acc[l] += sv * c_tab32[TB::VPHIW + q * N + l];
    }
  }
}

template <int K, int CH, bool FORCE>
__device__ __forceinline__ void vol_f32_chunk(const float* sW, float* sF, float* sS, const float* __restrict__ field,
                                              long long c0, long long nc, float gm1, const float* idx,
                                              float (&acc)[nmodes(K)]) {
  using CF = VolF32<K>;
  constexpr int C = CF::C;
  const int tid = threadIdx.x;
  {
    const int c = tid % C, wg = tid / C;  // warp-uniform phase-A role
    const long long cell = c0 + c;
    const long long cellc = cell < nc ? cell : nc - 1;  // ragged tail: in-bounds field reads
    if (wg == 0) vol_f32_points<K, CH, 0, FORCE>(sW, sF, sS, field, c, cellc, nc, gm1, idx);
    if (CF::NW > 1 && wg == 1) vol_f32_points<K, CH, (CF::NW > 1 ? 1 : 0), FORCE>(sW, sF, sS, field, c, cellc, nc, gm1, idx);
    if (CF::NW > 2 && wg == 2) vol_f32_points<K, CH, (CF::NW > 2 ? 2 : 0), FORCE>(sW, sF, sS, field, c, cellc, nc, gm1, idx);
  }
  __syncthreads();
  vol_f32_project<K, CH, FORCE>(sF, sS, tid % C, tid / C, acc);
  __syncthreads();
}

// Volume quadrature, FP32, over a tile of C cells in NCH chunks of points:
//  A) NW warps, each on a fixed subgroup of the chunk's points (warp-uniform,
//     so the point loop unrolls against compile-time constant-table offsets):
//     the cell's coefficients, values at the points, Euler fluxes (and the
//     driving source) to shared memory;
//  B) one warp per conserved variable: the N accumulators of one (cell,
//     variable) in registers, projection onto the basis gradients (and the
//     source onto the basis), every table value a constant-bank operand.
// After the last chunk, the six face fluxes are projected onto the face
// traces; then R, or the FP64 SSP-RK3 stage combination and the limiter
// screen (cells failing it are queued for the full limiter).
template <int K, int MODE, bool FORCE>
__global__ void __launch_bounds__(VolF32<K>::THREADS, VolF32<K>::MINB) volume_f32_kernel(
    const float* yfin, const float* __restrict__ fh, const float* __restrict__ field,
    const double* __restrict__ tab64, Geo g, StageArgs st, double* __restrict__ R, Ctrl* ctrl) {
  stream_wait();
  using TB = Tab<K>;
  using CF = VolF32<K>;
  constexpr int N = TB::N, Q2 = TB::Q2, C = CF::C;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* sM = reinterpret_cast<double*>(smem_raw);  // [5][C] stage means
  double* sA = sM + 5 * C;                            // [5][C] sum |w_l| max|phi_l|
  float* sW = reinterpret_cast<float*>(sA + 5 * C);   // [5N][C]
  float* sF = sW + 5 * N * C;                         // [15][PC][C]
  float* sS = sF + 15 * CF::PC * C;                   // [4][PC][C]
  if (MODE == MODE_STAGE) clear_deep(ctrl);
  const long long nc = g.nc;
  const long long c0 = (long long)blockIdx.x * C;
  const int tid = threadIdx.x;
  const float* ysrc = (MODE == MODE_STAGE) ? st.yf : yfin;
  for (int it = tid; it < 5 * N * C; it += CF::THREADS) {
    const int c = it % C, r = it / C;
    const long long cell = c0 + c;
    sW[r * C + c] = cell < nc ? ysrc[(size_t)r * nc + cell] : (r == 0 ? 1.f : 0.f);
  }
  __syncthreads();
  const float idx[3] = {(float)g.inv_dx[0], (float)g.inv_dx[1], (float)g.inv_dx[2]};
  const float gm1 = (float)(g.gamma - 1.0);
  float acc[N];
#pragma unroll
  for (int l = 0; l < N; ++l) acc[l] = 0.f;
  vol_f32_chunk<K, 0, FORCE>(sW, sF, sS, field, c0, nc, gm1, idx, acc);
  if (CF::NCH > 1) vol_f32_chunk<K, (CF::NCH > 1 ? 1 : 0), FORCE>(sW, sF, sS, field, c0, nc, gm1, idx, acc);
  if (CF::NCH > 2) vol_f32_chunk<K, (CF::NCH > 2 ? 2 : 0), FORCE>(sW, sF, sS, field, c0, nc, gm1, idx, acc);
  const int c = tid % C, i = tid / C;  // i: conserved variable, warp-uniform
  const long long cell = c0 + c;
  const bool live = cell < nc;
  if (live) {
    int ix, iy, iz;
    cell_xyz(cell, g, ix, iy, iz);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const long long cu = neighbour(g, ix, iy, iz, d, +1);
#pragma unroll
      for (int p = 0; p < Q2; ++p) {
        const size_t base = ((size_t)(d * 5 + i) * Q2 + p) * nc;
        const float fm = __ldg(fh + base + cell) * idx[d];
        const float fp = __ldg(fh + base + cu) * idx[d];
#pragma unroll
        for (int l = 0; l < N; ++l)
          acc[l] += fm * c_tab32[TB::FPHIW + ((d * 2 + 0) * Q2 + p) * N + l] -
                    fp * c_tab32[TB::FPHIW + ((d * 2 + 1) * Q2 + p) * N + l];
      }
    }
  }
  if (MODE == MODE_RHS) {
    if (live) {
#pragma unroll
      for (int l = 0; l < N; ++l) R[(size_t)(i * N + l) * nc + cell] = -f32_to_f64(acc[l]);
    }
    return;
  }
  double mean = 0.0;
  float sabsf = 0.f;
  bool finite = true;
  // first stage (a0 = 0, b0 = 1): out = y_s + dt dw/dt exactly, without
  // reading y_0
  const bool first = st.a0 == 0.0 && st.b0 == 1.0;
  if (live) {
#pragma unroll
    for (int l = 0; l < N; ++l) {
      const size_t a = (size_t)(i * N + l) * nc + cell;
      const double inc = __ldcg(st.ys + a) + st.dt * f32_to_f64(acc[l]);
      const double v = first ? inc : st.a0 * __ldcg(st.y0 + a) + st.b0 * inc;
      st.out[a] = v;
      const float vf = f64_to_f32(v);
      st.yf[a] = vf;
      finite &= finite64(v);
      if (l == 0) mean = v;
      else sabsf += fabsf(vf) * (g.lim_vol ? c_tab32[TB::LMAXV + l] : c_tab32[TB::LMAX + l]);
    }
  }
  // the screen's excursion sums are taken in FP32 from the rounded values
  // (relative error below 1e-6); a relative margin of 1e-5 keeps the test a
  // sufficient one
  const double sabs = (double)sabsf * (1.0 + 1e-5);
  sM[i * C + c] = finite ? mean : __longlong_as_double(0x7ff8000000000000LL);  // NaN marks non-finite
  sA[i * C + c] = sabs;
  __syncthreads();
  if (tid < C && live) {
    double m[5], a[5];
    bool fin = true;
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      m[j] = sM[j * C + tid];
      a[j] = sA[j * C + tid];
      fin &= isfinite(m[j]);
    }
    if (!limiter_screen<K>(m, a, fin, g.gamma, g.eps_rho, g.eps_p)) {
      const unsigned slot = atomicAdd(&ctrl->n_flag, 1u);
      st.list[slot] = (int)cell;
    }
  }
}

// Full positivity limiter on the cells queued by a stage kernel (list of
// *count cells), in two passes. The first (limit_screen_list_kernel) runs
// limit_cell's sufficient tests, the modal bounds and then the FP32 point
// screen; the cells that fail both go to a second list (*n_deep), which the
// second pass (limit_list_kernel) limits: compacting these cells keeps its warps
// full. A thread (long queues) or a warp copies its cell's 5N coefficients to
// shared memory once and works on them there: the tests and the point
// evaluations read every coefficient several times (once per point), and from
// global memory the scattered cells of a warp would pull a 128-byte line per
// coefficient and thread through L1 again at every read. Limited cells are
// written back.
template <int K>
struct ListLim {
  static constexpr int N = nmodes(K);
  static constexpr int THREADS = 128;
  static constexpr int MINB = K >= 3 ? 2 : 4;  // 5 N doubles per thread: 100 KB per block at degree 3
  static constexpr size_t smem() { return (size_t)5 * N * THREADS * sizeof(double); }
  // second pass: a cell's coefficients per warp, as they are and in fixed point
  static constexpr size_t smem_deep() { return (size_t)2 * 5 * N * (THREADS / 32) * sizeof(double); }
};

__device__ __forceinline__ void warp_sync() {
#ifdef __CUDA_ARCH__
  __syncwarp();
#else
  (void)__shfl_xor_sync(0xffffffffu, 0, 1);
#endif
}

// Screen of one queued cell by a warp, lanes over the points (point_screen_f32's
// test; w: the cell's coefficients in shared memory, wf: room for 5 N + 6
// floats). True when the cell needs the FP64 limiter; ORs the errors limit_cell
// would report into err.
template <int K>
__device__ bool warp_screen(const double* w, float* wf, const double* __restrict__ tab64,
                            const float* __restrict__ tab32, const Geo& g, int lane, unsigned* err) {
  using TB = Tab<K>;
  constexpr int N = TB::N;
  const double gm1 = g.gamma - 1.0;
  const LimUnits un(w[0], w[4 * N]);
  bool bad = false;
  // the scaling in a branch of its own: a pass over 3,400 queued cells of degree 1 takes
  // 38 us so, 39.6 with it for every cell, 36 without units
  if (un.plain) {
    for (int r = lane; r < 5 * N; r += 32) {
      bad |= !finite64(w[r]);
      wf[r] = f64_to_f32(w[r]);
    }
  } else {
    for (int r = lane; r < 5 * N; r += 32) {
      bad |= !finite64(w[r]);
      wf[r] = f64_to_f32(exp_add(w[r], un.of(r / N)));
    }
  }
  float* e = wf + 5 * N;  // error bounds of the five values, density threshold
  if (lane < 5) {
    const double* lmax = tab64 + (g.lim_vol ? TB::LMAXV : TB::LMAX);
    double s = fabs(w[lane * N]);
    for (int l = 1; l < N; ++l) s += fabs(w[lane * N + l]) * __ldg(lmax + l);
    double el = 2e-6 * s, er = g.eps_rho * (1.0 + 1e-6) + 1e-5 * s;
    if (!un.plain) {
      el = exp_add(el, un.of(lane));
      er = exp_add(er, un.r);
    }
    e[lane] = f64_to_f32(el);
    if (lane == 0) e[5] = f64_to_f32(er);
  }
  // any lane: 1 not finite, 2 some point fails
  unsigned any = bad ? 1u : 0u;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) any |= __shfl_xor_sync(0xffffffffu, any, o);
  warp_sync();
  if (any) {
    *err |= ERRB_NONFINITE;
    return false;
  }
  const double r = w[0], m1 = w[N], m2 = w[2 * N], m3 = w[3 * N];
  const double pbar = gm1 * (w[4 * N] - 0.5 * (m1 * m1 + m2 * m2 + m3 * m3) / r);
  if (!(r >= g.eps_rho) || !(pbar >= g.eps_p)) {
    *err |= ERRB_POSITIVITY;
    return false;
  }
  if (N == 1) return false;
  if (!un.ok) return true;
  float eps_pf = f64_to_f32(g.eps_p * (1.0 + 1e-6));
  const float gm1f = f64_to_f32(gm1);
  if (!un.plain) eps_pf = f64_to_f32(exp_add(g.eps_p * (1.0 + 1e-6), un.e));
  const int npts = TB::NL + (g.lim_vol ? TB::Q3 : 0);
  for (int s = lane; s < npts; s += 32) {
    const float* ph = s < TB::NL ? tab32 + TB::LPHI + s * N : tab32 + TB::VPHI + (s - TB::NL) * N;
    float U[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int l = 0; l < N; ++l) {
      const float p = __ldg(ph + l);
#pragma unroll
      for (int i = 0; i < 5; ++i) U[i] = fmaf(wf[i * N + l], p, U[i]);
    }
    const float rlo = U[0] - e[0];
    float k2 = 0.f;
#pragma unroll
    for (int a = 1; a <= 3; ++a) {
      const float mh = fabsf(U[a]) + e[a];
      k2 = fmaf(mh, mh, k2);
    }
    k2 *= 0.5f;
    const float lhs = gm1f * fmaf(U[4] - e[4], rlo, -k2);
    const float rhs = fmaf(eps_pf, rlo, 1e-5f * gm1f * fmaf(fabsf(U[4]) + e[4], rlo, k2));
    if (!(rlo >= e[5]) || !(lhs >= rhs)) any = 2u;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) any |= __shfl_xor_sync(0xffffffffu, any, o);
  return any != 0u;
}

template <int K>
__global__ void __launch_bounds__(ListLim<K>::THREADS, ListLim<K>::MINB)
    limit_screen_list_kernel(const double* __restrict__ y, const int* __restrict__ list, const unsigned* count,
                             const double* __restrict__ tab64, const float* __restrict__ tab32, Geo g, Ctrl* ctrl,
                             int count_queued, int* __restrict__ deep) {
  stream_wait();
  constexpr int N = nmodes(K), LT = ListLim<K>::THREADS;
  extern __shared__ __align__(16) double ws[];
  const unsigned n = *count;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    atomicAdd(&ctrl->n_full_total, (unsigned long long)n);
    if (count_queued) atomicAdd(&ctrl->n_queued_total, (unsigned long long)n);
  }
  unsigned e = 0;
  if (n <= gridDim.x * LT) {
    // a queue of at most one cell per thread: a warp per cell, so that a short
    // one does not wait for one thread's 81 points (one cell at degree 2: 35 us;
    // 128^3 with 77,000 queued: 78 us instead of 85)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double* w = ws + warp * 2 * (5 * N + 4);
    float* wf = reinterpret_cast<float*>(w + 5 * N);
    for (unsigned i = blockIdx.x * (LT / 32) + warp; i < n; i += gridDim.x * (LT / 32)) {
      const int cell = list[i];
      for (int r = lane; r < 5 * N; r += 32) w[r] = y[(size_t)r * g.nc + cell];
      warp_sync();
      if (warp_screen<K>(w, wf, tab64, tab32, g, lane, &e) && lane == 0) deep[atomicAdd(&ctrl->n_deep, 1u)] = cell;
      warp_sync();
    }
    if (e && lane == 0) atomicOr(&ctrl->err, e);
    return;
  }
  double* w = ws + threadIdx.x;  // this thread's column, stride LT
  for (unsigned i = blockIdx.x * LT + threadIdx.x; i < n; i += gridDim.x * LT) {
    const int cell = list[i];
    for (int r = 0; r < 5 * N; ++r) w[r * LT] = y[(size_t)r * g.nc + cell];
    double mean[5], sabs[5];
    bool rho_safe, p_safe, none;
    if (limit_prelude<K>(w, LT, tab64, g.gamma, g.eps_rho, g.eps_p, &e, g.lim_vol, tab32, mean, sabs, &rho_safe,
                         &p_safe, &none) &&
        !none)
      deep[atomicAdd(&ctrl->n_deep, 1u)] = cell;
  }
  if (e) atomicOr(&ctrl->err, e);
}

// coefficients of variable i of a cell, w[5 N] in shared memory, in fixed point
// to x (lanes: modes); returns the exponent. sum_l |phi_l| over the cell stays
// below 2^3, 2^5 and 2^6 at degrees 1 to 3, so that |x| < 2^55 at degree 3 and a
// point value stays below 2^61. The N - 1 products of a point value go into one
// FxAcc: with signed limbs on both sides |mid| <= sum_l |x.l ch| + |x.h cl| <=
// 2^29 2^28 sum_l |phi_l| + (N - 1) 2^25 2^29 <= 40.7 2^57 + 19 2^54 < 2^62.5.
// (Low limbs that are never negative reached 40.7 2^58 > 2^63 where all phi_l
// are positive.)
template <int K>
__device__ __forceinline__ int fx_cell(const double* w, Fx* x, int lane) {
  constexpr int N = nmodes(K);
  unsigned mx = 0;
  for (int l = 0; l < N; ++l) mx = max(mx, (unsigned)__double2hiint(w[l]) & 0x7fffffffu);
  const int B = max(kFxTiny, bexp(mx) + (K == 1 ? 3 : K == 2 ? 5 : 6));
  if (lane < N) x[lane] = fx_split_signed(fx_from(w[lane], B));
  return B;
}

// Second pass: one warp per cell, lanes over the points of the limiter's point
// set. The point values come from fixed-point sums (dg_common.cuh; 15 integer
// multiply-adds per point and mode, where the FP64 sums took 5 operations of a
// pipe 30 times slower); theta1, the pressure and the Newton iteration of the
// points below the floor are FP64, as in limit_cell. With a thread per cell and
// its points one after the other both passes took 120 us per step for one
// troubled cell (6 x 8 x 7, degree 2), now 37 (25 of them the launches); Sod
// tube, 128^3: 1.52 ms per step, now 0.92.
template <int K>
__global__ void __launch_bounds__(ListLim<K>::THREADS)
    limit_list_kernel(double* __restrict__ y, const int* __restrict__ list, const unsigned* count,
                      const double* __restrict__ tab64, Geo g, Ctrl* ctrl, float* __restrict__ yf,
                      const double* __restrict__ y0, float* __restrict__ dinc) {
  stream_wait();
  using TB = Tab<K>;
  constexpr int N = nmodes(K), LT = ListLim<K>::THREADS, NW = LT / 32;
  extern __shared__ __align__(16) double ws[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double* w = ws + warp * 5 * N;
  Fx* x = reinterpret_cast<Fx*>(ws + NW * 5 * N) + warp * 5 * N;
  const unsigned n = *count;
  // the queue that led here is done with
  if (blockIdx.x == 0 && threadIdx.x == 0) ctrl->n_flag = 0u;
  const long long nc = g.nc;
  const double gm1 = g.gamma - 1.0;
  const double* lphi = tab64 + TB::LPHI;
  const double* vphi = tab64 + TB::VPHI;
  const int npts = TB::NL + (g.lim_vol ? TB::Q3 : 0);
  unsigned err = 0;
  for (unsigned it = blockIdx.x * NW + warp; it < n; it += gridDim.x * NW) {
    const long long cell = list[it];
    for (int r = lane; r < 5 * N; r += 32) w[r] = y[(size_t)r * nc + cell];
    warp_sync();
    double mean[5];
    int B[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      mean[i] = w[i * N];
      B[i] = fx_cell<K>(w + i * N, x + i * N, lane);
    }
    warp_sync();
    bool limited = false;
    // density: theta1
    double rmin = mean[0];
    for (int s = lane; s < npts; s += 32) {
      const double* ph = s < TB::NL ? lphi + s * N : vphi + (s - TB::NL) * N;
      FxAcc a{0, 0};
#pragma unroll
      for (int l = 1; l < N; ++l) {
        const Fx p = fx_split_signed(fx_from(__ldg(ph + l), 1025));  // units of 2^-58
        fx_mad(a, x[l], p.h, p.l);
      }
      const double r = fx_to_double(fx_val(a) + fx_join(x[0]), B[0]);
      if (less64(r, rmin)) rmin = r;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double q = __shfl_xor_sync(0xffffffffu, rmin, o);
      if (less64(q, rmin)) rmin = q;
    }
    if (rmin < g.eps_rho) {
      const double th1 = fmin(fabs((mean[0] - g.eps_rho) / (mean[0] - rmin)), 1.0);
      if (th1 < 1.0) {
        if (lane > 0 && lane < N) w[lane] *= th1;
        warp_sync();
        B[0] = fx_cell<K>(w, x, lane);
        warp_sync();
        limited = true;
      }
    }
    // pressure: theta2 = min over the points of tau. The pressure is concave
    // along the segment from the mean, so a point whose pressure at the lane's
    // tau so far clears the floor has a larger tau: no iteration for it
    double th2 = 1.0;
    for (int s = lane; s < npts; s += 32) {
      const double* ph = s < TB::NL ? lphi + s * N : vphi + (s - TB::NL) * N;
      FxAcc a[5];
#pragma unroll
      for (int i = 0; i < 5; ++i) a[i] = {0, 0};
#pragma unroll
      for (int l = 1; l < N; ++l) {
        const Fx p = fx_split_signed(fx_from(__ldg(ph + l), 1025));
#pragma unroll
        for (int i = 0; i < 5; ++i) fx_mad(a[i], x[i * N + l], p.h, p.l);
      }
      double U[5];
#pragma unroll
      for (int i = 0; i < 5; ++i) U[i] = fx_to_double(fx_val(a[i]) + fx_join(x[i * N]), B[i]);
      double p = gm1 * fma(-0.5, fma(U[1], U[1], fma(U[2], U[2], U[3] * U[3])) * rcp64(U[0]), U[4]);
      if (p < g.eps_p && th2 < 1.0) {
        double V[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) V[i] = fma(th2, U[i] - mean[i], mean[i]);
        p = gm1 * fma(-0.5, fma(V[1], V[1], fma(V[2], V[2], V[3] * V[3])) * rcp64(V[0]), V[4]);
      }
      if (p < g.eps_p) {
        int k;
        const double tau = positivity_tau(mean, U, gm1, g.eps_p, &k);
        if (k >= 50) err |= ERRB_NEWTON;
        th2 = fmin(th2, tau);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) th2 = fmin(th2, __shfl_xor_sync(0xffffffffu, th2, o));
    if (th2 < 1.0) {
      for (int r = lane; r < 5 * N; r += 32)
        if (r % N) w[r] *= th2;
      limited = true;
    }
    warp_sync();
    if (limited) {
      for (int r = lane; r < 5 * N; r += 32) {
        const double v = w[r];
        y[(size_t)r * nc + cell] = v;
        if (yf) yf[(size_t)r * nc + cell] = (float)v;
        if (dinc) dinc[(size_t)r * nc + cell] = (float)(v - y0[(size_t)r * nc + cell]);
      }
    }
    warp_sync();
  }
  if (err) atomicOr(&ctrl->err, err);
}

// screen[c] = 1 when cell c fails the limiter screen (capture of training data)
template <int K>
__global__ void __launch_bounds__(kThreads) screen_kernel(const double* __restrict__ y, uint8_t* __restrict__ screen,
                                                          const double* __restrict__ tab64, Geo g) {
  constexpr int N = nmodes(K);
  const long long cell = (long long)blockIdx.x * kThreads + threadIdx.x;
  if (cell >= g.nc) return;
  double m[5], a[5];
  bool fin = true;
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    m[i] = y[(size_t)(i * N) * g.nc + cell];
    double sa = 0.0;
    for (int l = 1; l < N; ++l) {
      const double v = y[(size_t)(i * N + l) * g.nc + cell];
      sa += fabs(v) * __ldg(tab64 + (g.lim_vol ? Tab<K>::LMAXV : Tab<K>::LMAX) + l);
      fin &= isfinite(v);
    }
    fin &= isfinite(m[i]);
    a[i] = sa;
  }
  screen[cell] = limiter_screen<K>(m, a, fin, g.gamma, g.eps_rho, g.eps_p) ? 0 : 1;
}

// ============================================== sum-factorised volume kernel
// The tensor-product structure of the complete-degree basis turns each
// contraction over the Q^3 points into three one-dimensional ones (sum
// factorisation). Multiply-adds per cell and variable at degree 2: 165 for the
// values, 465 for the projection, 55 per face (dense quadrature: 270, 810, 90).
template <int K, typename T>
struct VolSF {
  static constexpr int Q = K + 1, KP = K + 1, Q2 = Q * Q, Q3 = Q * Q * Q, N = nmodes(K), TP = (K + 1) * (K + 2) / 2;
  static constexpr int mx(int a, int b) { return a > b ? a : b; }
  static constexpr int MT0 = 14 * TP * Q;  // offset of the face moments Mt in buffer 2
  // buffer 1: A1, U, H, M; buffer 2: A2, fluxes, (J, I2, SI | Mt)
  static constexpr int BUF1 = mx(mx(5 * TP * Q, 5 * Q3), mx(19 * KP * Q2, 30 * TP));
  static constexpr int BUF2 = mx(mx(5 * KP * Q2, 19 * Q3), MT0 + 30 * KP * Q);
  static constexpr int C = 8;
  static constexpr size_t smem() { return (size_t)C * (8 * (5 * N + 10) + sizeof(T) * (BUF1 + BUF2)); }
};
// FP64: one (cell, variable, slice of constant z) per thread
template <int K>
struct VolSF<K, double> {
  static constexpr int Q = K + 1, Q3 = Q * Q * Q, N = nmodes(K), T = (K + 1) * (K + 2) / 2;
  static constexpr int NL = nmodes(K - 1);  // modes with an exponent above 0 along a given axis
  static constexpr int C = kThreads / (5 * Q);
  // shared memory in doubles: values [5][Q3][C], fluxes and sources [13][Q3][C];
  // then, over both, 64-bit integers: the slices' sums of each direction
  // [Q][3][5][NL][C], their source sums of the modes u = 0 [Q][4][T][C], the faces' sums
  // [3][5][N][C]; exponents (int) of the slices' [Q][4][5][C] and of the faces'
  // [3][5][C], and the screen's [Q + 1][5][C] (float)
  static constexpr int U = 0, F = 5 * Q3 * C;
  static constexpr int SRC = Q * 15 * NL * C, FACE = SRC + Q * 4 * T * C, EXPS = FACE + 15 * N * C;
  static constexpr int SCREEN = EXPS + ((Q * 20 + 15) * C + 1) / 2;
  static constexpr int A = 18 * Q3 * C, B = SCREEN + ((Q + 1) * 5 * C + 1) / 2, END = A > B ? A : B;
  static constexpr size_t smem() { return sizeof(double) * END; }
  // CTAs per SM the register budget is sized for (128^3, degree 2: 5.5 ms with 3, 7.1
  // with 2; 64^3, degree 1: 0.219 ms with 4, 0.215 with 3, driven 0.271 and 0.305;
  // degree 3 has no shared memory for a third)
  static constexpr int MINB = K == 1 ? 4 : (K == 2 ? 3 : 2);
  // directions whose faces one slice's threads take
  static constexpr int NF = (2 + Q) / Q;
};

// index of the mode with the exponent along an axis lowered by one (255: it is 0)
static __constant__ unsigned char c_lower[3][20] = {
    {255, 0, 255, 255, 1, 2, 3, 255, 255, 255, 4, 5, 6, 7, 8, 9, 255, 255, 255, 255},
    {255, 255, 0, 255, 255, 1, 255, 2, 3, 255, 255, 4, 255, 5, 6, 255, 7, 8, 9, 255},
    {255, 255, 255, 0, 255, 255, 1, 255, 2, 3, 255, 255, 4, 255, 5, 6, 255, 7, 8, 9}};
// index among the modes u = 0 (0 for the others); (v, w) has (v + w)(v + w + 1)/2 + w
static __constant__ unsigned char c_flat[20] = {0, 0, 1, 2, 0, 0, 0, 3, 4, 5, 0, 0, 0, 0, 0, 0, 6, 7, 8, 9};

template <int K>
__device__ __forceinline__ void pair_uv(int j, int& u, int& v) {
  u = 0;
  while (j > K - u) {
    j -= K - u + 1;
    ++u;
  }
  v = j;
}


// raises the accumulators' exponent A to B (never lowers it)
template <int N>
__device__ __forceinline__ void fx_raise(long long (&acc)[N], int& A, int B) {
  if (B > A) {
    const int d = min(B - A, 63);
#pragma unroll
    for (int m = 0; m < N; ++m) acc[m] >>= d;
    A = B;
  }
}

// The two faces normal to D of one (cell, variable), from the moments of their
// fluxes (low face at ml, high face at mh, rows nc apart; face_sf64_kernel):
// Pt_e(-1) M_low - Pt_e(+1) M_high for the mode e along D, Pt_e(-1) = (-1)^e
// Pt_e(+1). With the moments' exponent A: the modes e = 0 as M_low - M_high in units
// of A, exactly 0 where the flow does not change along D; e > 0 divided by 16.
template <int K, int D>
__device__ __forceinline__ void fx_apply(const long long (&even)[(K + 1) * (K + 2) / 2],
                                         const long long (&odd)[(K + 1) * (K + 2) / 2],
                                         long long (&acc)[nmodes(K)]) {
  constexpr int F = FxTab<K>::F + K + 1;
#pragma unroll
  for (int a = 0, j = 0; a <= K; ++a)
#pragma unroll
    for (int b = 0; a + b <= K; ++b, ++j) {
      acc[face_mode<D>(0, a, b)] = even[j];
      const Fx ev = fx_split(even[j]), od = fx_split(odd[j]);
#pragma unroll
      for (int e = 1; e + a + b <= K; ++e) {
        FxAcc t{0, 0};
        fx_madt(t, e % 2 ? od : ev, F + e);
        acc[face_mode<D>(e, a, b)] = e % 2 ? -fx_val(t) : fx_val(t);
      }
    }
}
template <int K>
__device__ __forceinline__ void fx_faces(int d, const double* __restrict__ ml, const double* __restrict__ mh,
                                         size_t nc, long long (&acc)[nmodes(K)], int& A) {
  constexpr int T = (K + 1) * (K + 2) / 2;
  double l[T], h[T];
  unsigned mx = 0;
#pragma unroll
  for (int j = 0; j < T; ++j) {
    l[j] = __ldg(ml + (size_t)j * nc);
    h[j] = __ldg(mh + (size_t)j * nc);
    mx = max(mx, max((unsigned)__double2hiint(l[j]) & 0x7fffffffu, (unsigned)__double2hiint(h[j]) & 0x7fffffffu));
  }
  A = max(kFxTiny, bexp(mx) + 1);
  long long even[T], odd[T];
#pragma unroll
  for (int j = 0; j < T; ++j) {
    const long long a = fx_from(l[j], A), b = fx_from(h[j], A);
    even[j] = a - b;
    odd[j] = a + b;
  }
  if (d == 0) fx_apply<K, 0>(even, odd, acc);
  else if (d == 1) fx_apply<K, 1>(even, odd, acc);
  else fx_apply<K, 2>(even, odd, acc);
}

// H[(u, v)] = sums over a slice's points qx + Q qy (rows C apart) of the values f
// of direction D's flux in units of the exponent A, weighted by D'/8 along D (for z
// that follows later) and by P' along the others; only the modes that the flux
// along D contributes to (an exponent above 0 along D) are formed. Rows in pairs +-y.
// With D = 0 the source fs (SRC and src; exponent As <= A - 2, see volume_sf_kernel)
// joins H for the modes u > 0, weighted by P' throughout; its modes u = 0 go to H0[v]
// in units of As.
template <int K, int D, int C, bool SRC = false>
__device__ __forceinline__ void fx_slice(const double* f, int A, long long (&H)[(K + 1) * (K + 2) / 2],
                                         const double* fs = nullptr, bool src = false, int As = 0,
                                         long long* H0 = nullptr) {
  using FT = FxTab<K>;
  constexpr int Q = K + 1, U0 = D == 0 ? 1 : 0, V0 = D == 1 ? 1 : 0, UV = D == 2 ? K - 1 : K;
  constexpr int TY = D == 1 ? FT::D : FT::W, PY = D == 1 ? 1 : 0;
  auto row = [&](int qy, long long (&g)[K + 1]) {
    FxAcc G[K + 1];
    long long v[Q];
#pragma unroll
    for (int u = 0; u <= K; ++u) G[u] = {0, 0};
#pragma unroll
    for (int q = 0; q < Q; ++q) v[q] = fx_from(f[(q + Q * qy) * C], A);
    fx_project<K, D == 0>(v, G);
    if constexpr (SRC)
      if (src) {
        const int d = min(A - As, 63);
#pragma unroll
        for (int q = 0; q < Q; ++q) v[q] = fx_from(fs[(q + Q * qy) * C], As);
        FxAcc z{0, 0};
#pragma unroll
        for (int r = Q - Q / 2; r < Q; ++r) fx_madt(z, fx_split(v[r] + v[Q - 1 - r]), FT::W + r);
        if (Q % 2) fx_madt(z, fx_split(v[Q / 2]), FT::W + Q / 2);
        g[0] = fx_val(z);
#pragma unroll
        for (int q = 0; q < Q; ++q) v[q] >>= d;
        fx_project<K, false>(v, G);
      }
#pragma unroll
    for (int u = U0; u <= K; ++u) g[u] = fx_val(G[u]);
  };
#pragma unroll
  for (int j = 0; j < (K + 1) * (K + 2) / 2; ++j) H[j] = 0;
  if constexpr (SRC)
#pragma unroll
    for (int v = 0; v <= K; ++v) H0[v] = 0;
  if (Q % 2) {
    long long g[K + 1];
    row(Q / 2, g);
#pragma unroll
    for (int u = U0; u <= UV; ++u) {
      const Fx x = fx_split(g[u]);
#pragma unroll
      for (int v = PY; u + v <= UV; v += 2) {  // the others' weights are 0 at y = 0
        FxAcc h{0, 0};
        fx_madt(h, x, TY + v * Q + Q / 2);
        H[pair_index(K, u, v)] += fx_val(h);
      }
    }
    if constexpr (SRC)
      if (src) {
        const Fx x = fx_split(g[0]);
#pragma unroll
        for (int v = 0; v <= K; v += 2) {
          FxAcc h{0, 0};
          fx_madt(h, x, FT::W + v * Q + Q / 2);
          H0[v] += fx_val(h);
        }
      }
  }
#pragma unroll 1
  for (int r = Q - Q / 2; r < Q; ++r) {
    long long a[K + 1], b[K + 1];
    row(r, a);
    row(Q - 1 - r, b);
#pragma unroll
    for (int u = U0; u <= UV; ++u) {
      const Fx s = fx_split(a[u] + b[u]), d = fx_split(a[u] - b[u]);
#pragma unroll
      for (int v = V0; u + v <= UV; ++v) {
        FxAcc h{0, 0};
        fx_madt(h, (v + PY) % 2 ? d : s, TY + v * Q + r);
        H[pair_index(K, u, v)] += fx_val(h);
      }
    }
    if constexpr (SRC)
      if (src) {
        const Fx s = fx_split(a[0] + b[0]), d = fx_split(a[0] - b[0]);
#pragma unroll
        for (int v = 0; v <= K; ++v) {
          FxAcc h{0, 0};
          fx_madt(h, v % 2 ? d : s, FT::W + v * Q + r);
          H0[v] += fx_val(h);
        }
      }
  }
}

// Volume integral, surface integral and stage update, FP64. One (cell,
// variable, slice of constant z) per thread for the contractions, which run in
// 64-bit fixed point (dg_common.cuh) with one exponent per variable's
// coefficients and one per direction of the fluxes and for the source; one (cell,
// point) per thread for the Euler fluxes and the driving source, in FP64; then
// one (cell, variable) and every Q-th mode per thread for the sum over the
// slices and the stage update:
//   dw/dt = sum_d 1/dx_d [16 (sum_q F_d(q) (D'/8) P' P' + sum_faces +- (P' P'
//           moments) Pt_e / 16)] + 1/dx_x [16 sum_q (dx_x / 16) S(q) P' P' P'],
// P' = P w / 2 and D' = (dP/dxi) w / 2 (sums of |P'| <= 1, of |D'| / 8 <= 0.61),
// the bracket of a direction in fixed point, the brackets added in FP64: a direction
// whose fluxes are far above another's contributes exactly 0 to the modes constant
// along it where the flow does not change along it, and must not cut the other's
// terms. The source joins the x flux in the modes that this contributes to and has
// an exponent of its own in the others. Inputs take 60 bits and the source there 58,
// so that no intermediate reaches 2^61 and no sum 2^63. Integer issue bounds it on large
// meshes (128^3, degree 2: 5.5 ms per stage, 7.1 with driving; with one exponent for
// the three directions and the source, two CTAs per SM, 6.9 and 7.6, with FP64
// contractions 33.6; 64^3, degree 3: 2.28 and 2.67, before 2.16 and 2.61) and one
// thread's chain on small ones, which is why a slice is a thread's work: a thread per
// (cell, variable) was 7 % faster at 128^3, but 8 x 8 x 8 at degree 1 or 33 x 32 x 31
// fill the chip with three or four times the threads (8^3: 12 us, the dense kernel
// took 84).
template <int K, typename T, int MODE, bool FORCE>
__global__ void __launch_bounds__(kThreads, VolSF<K, double>::MINB)
    volume_sf_kernel(const double* __restrict__ yin, const float* __restrict__ yf32, const T* __restrict__ fh,
                     const T* __restrict__ field, const T* __restrict__ tab, const double* __restrict__ tab64, Geo g,
                     StageArgs st, double* __restrict__ R, Ctrl* ctrl) {
  stream_wait();
  static_assert(sizeof(T) == 8, "fixed-point form: FP64 path only");
  using TB = Tab<K>;
  using CF = VolSF<K, double>;
  using FT = FxTab<K>;
  constexpr int N = TB::N, Q = K + 1, Q2 = Q * Q, Q3 = TB::Q3, C = CF::C, T2 = CF::T, NL = CF::NL;
  static_assert(kThreads == 5 * Q * C, "one (cell, variable, slice) per thread");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* sm64 = reinterpret_cast<double*>(smem_raw);
  if (MODE == MODE_STAGE) clear_deep(ctrl);
  const long long nc = g.nc;
  const long long c0 = (long long)blockIdx.x * C;
  const int tid = threadIdx.x;
  const int c = tid % C, i = (tid / C) % 5, qz = tid / (5 * C);
  const long long cell = c0 + c;
  const bool live = cell < nc;
  const long long cellc = live ? cell : nc - 1;  // ragged tail: in-bounds reads, nothing written
  const double* ysrc = (MODE == MODE_STAGE) ? st.ys : yin;
  bool huge = false;  // values or fluxes that have no exponent (kFxHuge): the result is NaN
  // --------------------------------------------- values at the slice's points
  {
    Fx x[N];
    int B;
    fx_load<K>(ysrc + (size_t)(i * N) * nc + cellc, nc, x, B);
    huge = B >= kFxHuge;
    Fx pz[K + 1];  // Pt_w at the slice
#pragma unroll
    for (int ww = 1; ww <= K; ++ww) pz[ww] = {c_fx[FT::P + ww * Q + qz][0], c_fx[FT::P + ww * Q + qz][1]};
    Fx A1[T2];
#pragma unroll
    for (int u = 0, j = 0; u <= K; ++u)
#pragma unroll
      for (int v = 0; u + v <= K; ++v, ++j) {
        FxAcc s{0, 0};
#pragma unroll
        for (int ww = 1; u + v + ww <= K; ++ww) fx_mad(s, x[mode_index(u, v, ww)], pz[ww].h, pz[ww].l);
        const long long x0 = fx_join(x[mode_index(u, v, 0)]);
        A1[j] = fx_split(u + v < K ? fx_val(s) + x0 : x0);
      }
    Fx A2[Q][K + 1];  // [qy][u]
    fx_rows<K, 0>(A1, A2);
    double* u = sm64 + CF::U + (i * Q3 + qz * Q2) * C + c;
#pragma unroll
    for (int qy = 0; qy < Q; ++qy) {
      long long v[Q];
      fx_values<K, K + 1>(A2[qy], v);
#pragma unroll
      for (int qx = 0; qx < Q; ++qx) u[(qx + Q * qy) * C] = fx_to_double(v[qx], B);
    }
  }
  // the faces of the directions qz, qz + Q, ...
  long long facc[CF::NF][N];
  int fexp[CF::NF];
  {
    int ix, iy, iz;
    cell_xyz(cellc, g, ix, iy, iz);
#pragma unroll
    for (int n = 0; n < CF::NF; ++n) {
      const int d = qz + n * Q;
      if (d < 3) {
        const double* f = fh + (size_t)((d * 5 + i) * T2) * nc;
        fx_faces<K>(d, f + cellc, f + neighbour(g, ix, iy, iz, d, 1), nc, facc[n], fexp[n]);
      }
    }
  }
  __syncthreads();
  // ------------------------------ Euler fluxes and the driving source, FP64
  const double gm1 = g.gamma - 1.0;
  {
    const double* sU = sm64 + CF::U;
    double* sF = sm64 + CF::F;
    constexpr int R3 = Q3 * C;
#pragma unroll 1
    for (int it = tid; it < R3; it += kThreads) {
      double a[3];
      if (FORCE) {
        const int q = it / C, cc = it % C;
        const T* ap = field + (size_t)q * nc + (c0 + cc < nc ? c0 + cc : nc - 1);
#pragma unroll
        for (int d = 0; d < 3; ++d) a[d] = 0.0625 * g.dx[0] * __ldg(ap + (size_t)d * Q3 * nc);
      }
      const double r = sU[it], m0 = sU[R3 + it], m1 = sU[2 * R3 + it], m2 = sU[3 * R3 + it], E = sU[4 * R3 + it];
      const double ir = rcp64(r);
      const double v0 = m0 * ir, v1 = m1 * ir, v2 = m2 * ir;
      const double p = gm1 * fma(-0.5, fma(m0, v0, fma(m1, v1, m2 * v2)), E);
      const double h = E + p;
      sF[it] = fma(m0, v0, p);
      sF[R3 + it] = m0 * v1;
      sF[2 * R3 + it] = m0 * v2;
      sF[3 * R3 + it] = fma(m1, v1, p);
      sF[4 * R3 + it] = m1 * v2;
      sF[5 * R3 + it] = fma(m2, v2, p);
      sF[6 * R3 + it] = h * v0;
      sF[7 * R3 + it] = h * v1;
      sF[8 * R3 + it] = h * v2;
      if (FORCE) {
        sF[9 * R3 + it] = r * a[0];
        sF[10 * R3 + it] = r * a[1];
        sF[11 * R3 + it] = r * a[2];
        sF[12 * R3 + it] = fma(m0, a[0], fma(m1, a[1], m2 * a[2]));
      }
    }
  }
  __syncthreads();
  // -------------------- projection onto the basis gradients (and the source)
  const bool src = FORCE && i > 0;
  // by direction, modes by their index with the exponent along it lowered by one
  long long V[3][NL], S[FORCE ? T2 : 1];  // S: the source's modes (0, v, w)
  int ex[3], es = kFxTiny;
  {
    // where this variable's fluxes along x, y, z and its source lie: the mass
    // flux is the momentum itself, the momentum flux is symmetric
    const int sym[3] = {i == 1 ? 0 : i == 2 ? 1 : 2, i == 1 ? 1 : i == 2 ? 3 : 4, i == 1 ? 2 : i == 2 ? 4 : 5};
    const double* fd[3];
#pragma unroll
    for (int d = 0; d < 3; ++d)
      fd[d] = (i == 0 ? sm64 + CF::U + (1 + d) * Q3 * C : sm64 + CF::F + (i == 4 ? 6 + d : sym[d]) * Q3 * C) +
              qz * Q2 * C + c;
    const double* fs = sm64 + CF::F + ((9 + (i > 0 ? i - 1 : 0)) * Q3 + qz * Q2) * C + c;
    unsigned mx[3] = {0, 0, 0}, ms = 0;
#pragma unroll
    for (int q = 0; q < Q2; ++q) {
#pragma unroll
      for (int d = 0; d < 3; ++d) mx[d] = max(mx[d], (unsigned)__double2hiint(fd[d][q * C]) & 0x7fffffffu);
      if (src) ms = max(ms, (unsigned)__double2hiint(fs[q * C]) & 0x7fffffffu);
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) ex[d] = max(kFxTiny, bexp(mx[d]) + 1);
    long long H[T2];
    if constexpr (FORCE) {
      es = max(kFxTiny, bexp(ms) + 1);
      if (src) ex[0] = max(ex[0], es + 2);
      long long H0[K + 1];
      fx_slice<K, 0, C, true>(fd[0], ex[0], H, fs, src, es, H0);
      if (src) {
#pragma unroll
        for (int ww = 0; ww <= K; ++ww) {
          const int h = c_fx[FT::W + ww * Q + qz][0], l = c_fx[FT::W + ww * Q + qz][1];
#pragma unroll
          for (int v = 0; v + ww <= K; ++v) {
            FxAcc t{0, 0};
            fx_mad(t, fx_split(H0[v]), h, l);
            S[(v + ww) * (v + ww + 1) / 2 + ww] = fx_val(t);
          }
        }
      }
    } else {
      fx_slice<K, 0, C>(fd[0], ex[0], H);
    }
#pragma unroll
    for (int ww = 0; ww <= K; ++ww) {
      const int h = c_fx[FT::W + ww * Q + qz][0], l = c_fx[FT::W + ww * Q + qz][1];
#pragma unroll
      for (int u = 1; u + ww <= K; ++u)
#pragma unroll
        for (int v = 0; u + v + ww <= K; ++v) {
          FxAcc t{0, 0};
          fx_mad(t, fx_split(H[pair_index(K, u, v)]), h, l);
          V[0][mode_index(u - 1, v, ww)] = fx_val(t);
        }
    }
    fx_slice<K, 1, C>(fd[1], ex[1], H);
#pragma unroll
    for (int ww = 0; ww <= K; ++ww) {
      const int h = c_fx[FT::W + ww * Q + qz][0], l = c_fx[FT::W + ww * Q + qz][1];
#pragma unroll
      for (int u = 0; u + ww <= K; ++u)
#pragma unroll
        for (int v = 1; u + v + ww <= K; ++v) {
          FxAcc t{0, 0};
          fx_mad(t, fx_split(H[pair_index(K, u, v)]), h, l);
          V[1][mode_index(u, v - 1, ww)] = fx_val(t);
        }
    }
    fx_slice<K, 2, C>(fd[2], ex[2], H);
#pragma unroll
    for (int ww = 1; ww <= K; ++ww) {
      const int h = c_fx[FT::D + ww * Q + qz][0], l = c_fx[FT::D + ww * Q + qz][1];
#pragma unroll
      for (int u = 0; u + ww <= K; ++u)
#pragma unroll
        for (int v = 0; u + v + ww <= K; ++v) {
          FxAcc t{0, 0};
          fx_mad(t, fx_split(H[pair_index(K, u, v)]), h, l);
          V[2][mode_index(u, v, ww - 1)] = fx_val(t);
        }
    }
  }
  __syncthreads();
  // ------------------------- sum over the slices; R, or the FP64 stage update
  long long* sAcc = reinterpret_cast<long long*>(smem_raw);
  int* sExp = reinterpret_cast<int*>(sm64 + CF::EXPS);
  float* sScr = reinterpret_cast<float*>(sm64 + CF::SCREEN);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
#pragma unroll
    for (int m = 0; m < NL; ++m) sAcc[(((qz * 3 + d) * 5 + i) * NL + m) * C + c] = V[d][m];
    sExp[((qz * 4 + d) * 5 + i) * C + c] = huge ? kFxHuge : ex[d];
  }
  if constexpr (FORCE)
    if (src) {
#pragma unroll
      for (int j = 0; j < T2; ++j) sAcc[CF::SRC + ((qz * 4 + i - 1) * T2 + j) * C + c] = S[j];
      sExp[((qz * 4 + 3) * 5 + i) * C + c] = es;
    }
#pragma unroll
  for (int n = 0; n < CF::NF; ++n) {
    const int d = qz + n * Q;
    if (d < 3) {
#pragma unroll
      for (int l = 0; l < N; ++l) sAcc[CF::FACE + ((d * 5 + i) * N + l) * C + c] = facc[n][l];
      sExp[((Q * 4 + d) * 5 + i) * C + c] = fexp[n];
    }
  }
  __syncthreads();
  // per direction: the largest exponent and the shifts to it of the slices (and,
  // last, of the faces); per slice that of the source
  int xm[3], fe[3], sh[3][Q + 1], xs = 0, shs[Q], top = 0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    xm[d] = 0;
#pragma unroll
    for (int z = 0; z <= Q; ++z) {
      sh[d][z] = sExp[((z * 4 + d) * 5 + i) * C + c];
      xm[d] = max(xm[d], sh[d][z]);
    }
    fe[d] = sh[d][Q];
#pragma unroll
    for (int z = 0; z <= Q; ++z) sh[d][z] = min(xm[d] - sh[d][z], 63);
    top = max(top, xm[d]);
  }
  if (src) {
#pragma unroll
    for (int z = 0; z < Q; ++z) {
      shs[z] = sExp[((z * 4 + 3) * 5 + i) * C + c];
      xs = max(xs, shs[z]);
    }
#pragma unroll
    for (int z = 0; z < Q; ++z) shs[z] = min(xs - shs[z], 63);
    top = max(top, xs);
  }
  float sab = 0.f;
  if (live) {
#pragma unroll 1
    for (int l = qz; l < N; l += Q) {
      const size_t at = (size_t)(i * N + l) * nc + cell;
      double a = 0.0;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const int low = c_lower[d][l];
        long long t = sAcc[CF::FACE + ((d * 5 + i) * N + l) * C + c];
        int x = fe[d];  // e = 0: the faces' difference in their own units
        if (low != 255) {
          t >>= sh[d][Q];
#pragma unroll
          for (int z = 0; z < Q; ++z) t += sAcc[(((z * 3 + d) * 5 + i) * NL + low) * C + c] >> sh[d][z];
          x = xm[d] + 4;
        }
        a = fma(g.inv_dx[d], fx_to_double(t, x), a);
      }
      if (src && c_lower[0][l] == 255) {
        long long t = 0;
#pragma unroll
        for (int z = 0; z < Q; ++z) t += sAcc[CF::SRC + ((z * 4 + i - 1) * T2 + c_flat[l]) * C + c] >> shs[z];
        a = fma(g.inv_dx[0], fx_to_double(t, xs + 4), a);
      }
      if (top >= kFxHuge) a = __longlong_as_double(0x7ff8000000000000LL);
      if (MODE == MODE_RHS) {
        R[at] = -a;
      } else {
        // the first stage (a0 = 0, b0 = 1) does not read y_0
        double v = fma(st.dt, a, __ldcg(st.ys + at));
        if (st.a0 != 0.0) v = st.a0 * __ldcg(st.y0 + at) + st.b0 * v;
        st.out[at] = v;
        if (l == 0) sScr[(Q * 5 + i) * C + c] = f64_to_f32_q(v);
        else sab = fmaf(abs_up(v), c_tab32[(g.lim_vol ? TB::LMAXV : TB::LMAX) + l], sab);
      }
    }
  }
  if (MODE == MODE_RHS) return;
  // limiter screen of the next stage's input: FP32 (sufficient) for all cells,
  // FP64 for those it does not clear, so that dg_limiter_counts and the
  // indicator's input are decided in FP64; what fails both is queued for the full
  // limiter. The FP64 sums are taken by the threads that hold the modes: one thread
  // reading 5 N coefficients one after the other took 10 us.
  sScr[(qz * 5 + i) * C + c] = sab * (1.f + 1e-5f);
  __syncthreads();
  int* sTest = reinterpret_cast<int*>(smem_raw);  // [C]; the sums before are done with
  double* sSum = sm64 + C;                        // [Q][5][C]
  bool test = false;
  if (tid < C) {
    float m[5], s[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      m[v] = sScr[(Q * 5 + v) * C + tid];
      s[v] = 0.f;
#pragma unroll
      for (int z = 0; z < Q; ++z) s[v] += sScr[(z * 5 + v) * C + tid];
    }
    test = live && !screen_f32(m, s, (float)gm1, (float)g.eps_rho, (float)g.eps_p);
    sTest[tid] = test;
  }
  __syncthreads();
  if (sTest[c]) {
    double s = 0.0;
#pragma unroll
    for (int j = 0; j * Q < N; ++j) {
      const int l = qz + j * Q;
      if (l > 0 && l < N)
        s += fabs(st.out[(size_t)(i * N + l) * nc + cell]) * __ldg(tab64 + (g.lim_vol ? TB::LMAXV : TB::LMAX) + l);
    }
    sSum[(qz * 5 + i) * C + c] = s;
  }
  __syncthreads();
  if (test) {
    double m[5], s[5];
    bool fin = true;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      m[v] = st.out[(size_t)(v * N) * nc + cell];
      s[v] = 0.0;
#pragma unroll
      for (int z = 0; z < Q; ++z) s[v] += sSum[(z * 5 + v) * C + tid];
      fin &= finite64(m[v]) && finite64(s[v]);
    }
    if (!limiter_screen<K>(m, s, fin, g.gamma, g.eps_rho, g.eps_p)) {
      const unsigned slot = atomicAdd(&ctrl->n_flag, 1u);
      st.list[slot] = (int)cell;
    }
  }
}

// Register-blocked form (FP32): an item loads its inputs along the
// contracted index once and produces all outputs along the new index, the
// 1D tables as constant-bank operands. Triangular ranges become predicated
// unrolled loops, which costs nothing where the FP32 pipe is not the bound.
template <int K, typename T, int MODE, bool FORCE>
__global__ void __launch_bounds__(kThreads) volume_sfb_kernel(const double* __restrict__ yin,
                                                             const float* __restrict__ yf32, const T* __restrict__ fh,
                                                             const T* __restrict__ field, const T* __restrict__ tab,
                                                             const double* __restrict__ tab64, Geo g, StageArgs st,
                                                             double* __restrict__ R, Ctrl* ctrl) {
  stream_wait();
  static_assert(sizeof(T) == 4, "register-blocked form: FP32 path only");
  using TB = Tab<K>;
  using CF = VolSF<K, T>;
  constexpr int N = TB::N, Q = CF::Q, Q2 = CF::Q2, Q3 = CF::Q3, TP = CF::TP, C = CF::C, KP = K + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* sV = reinterpret_cast<double*>(smem_raw);  // stage output (FP64)
  double* sM = sV + 5 * N * C;
  double* sA = sM + 5 * C;
  T* sW = reinterpret_cast<T*>(sV);  // stage input (T), read only by the first pass
  T* b1 = reinterpret_cast<T*>(sA + 5 * C);
  T* b2 = b1 + CF::BUF1 * C;
  if (MODE == MODE_STAGE) clear_deep(ctrl);
  const long long nc = g.nc;
  const long long c0 = (long long)blockIdx.x * C;
  const int tid = threadIdx.x;
  // stage input: FP64 state (T = double) or its FP32 shadow (T = float)
  const double* ysrc = (MODE == MODE_STAGE) ? st.ys : yin;
  const float* yfsrc = (MODE == MODE_STAGE) ? st.yf : yf32;
  for (int it = tid; it < 5 * N * C; it += kThreads) {
    const int c = it % C, r = it / C;
    const long long cell = c0 + c;
    T v = r == 0 ? T(1) : T(0);
    if (cell < nc) {
      if constexpr (sizeof(T) == 4) v = yfsrc[(size_t)r * nc + cell];
      else v = ysrc[(size_t)r * nc + cell];
    }
    sW[r * C + c] = v;
  }
  __syncthreads();
  // Every pass below is a register-blocked 1D contraction: an item loads
  // its inputs along the contracted index once and produces all outputs
  // along the new index, the 1D table entries being constant-bank operands
  // (loops unrolled over compile-time indices).
  constexpr int OP = 0, OPW = KP * Q, ODW = 2 * KP * Q;  // P, P w, P' w in c_sf*
  // A1[i][pair(u,v)][qc] = sum_w w_i,uvw P_w(qc) -> b1
  for (int it = tid; it < 5 * TP * C; it += kThreads) {
    const int c = it % C, r = it / C, j = r % TP, i = r / TP;
    int u, v;
    pair_uv<K>(j, u, v);
    T acc[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) acc[q] = T(0);
#pragma unroll
    for (int w = 0; w <= K; ++w)
      if (w <= K - u - v) {
        const T x = sW[(i * N + mode_index(u, v, w)) * C + c];
#pragma unroll
        for (int q = 0; q < Q; ++q) acc[q] += x * sfc<T>(OP + w * Q + q);
      }
#pragma unroll
    for (int q = 0; q < Q; ++q) b1[((i * TP + j) * Q + q) * C + c] = acc[q];
  }
  __syncthreads();
  // A2[i][u][qb + Q qc] = sum_v A1[i][pair(u,v)][qc] P_v(qb) -> b2
  for (int it = tid; it < 5 * KP * Q * C; it += kThreads) {
    const int c = it % C, r = it / C, qc = r % Q, u = (r / Q) % KP, i = r / (Q * KP);
    T acc[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) acc[q] = T(0);
#pragma unroll
    for (int v = 0; v <= K; ++v)
      if (v <= K - u) {
        const T x = b1[((i * TP + pair_index(K, u, v)) * Q + qc) * C + c];
#pragma unroll
        for (int q = 0; q < Q; ++q) acc[q] += x * sfc<T>(OP + v * Q + q);
      }
#pragma unroll
    for (int q = 0; q < Q; ++q) b2[((i * KP + u) * Q2 + q + Q * qc) * C + c] = acc[q];
  }
  __syncthreads();
  // U[i][qa + Q bc] = sum_u A2[i][u][bc] P_u(qa) -> b1
  for (int it = tid; it < 5 * Q2 * C; it += kThreads) {
    const int c = it % C, r = it / C, bc = r % Q2, i = r / Q2;
    T acc[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) acc[q] = T(0);
#pragma unroll
    for (int u = 0; u <= K; ++u) {
      const T x = b2[((i * KP + u) * Q2 + bc) * C + c];
#pragma unroll
      for (int q = 0; q < Q; ++q) acc[q] += x * sfc<T>(OP + u * Q + q);
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) b1[(i * Q3 + q + Q * bc) * C + c] = acc[q];
  }
  __syncthreads();
  // fluxes G[d*5+i][q] = F_d / (4 dx_d), source S[i-1][q] = S / 8 -> b2
  const T gm1 = (T)(g.gamma - 1.0);
  for (int it = tid; it < Q3 * C; it += kThreads) {
    const int c = it % C, q = it / C;
    T U[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) U[i] = b1[(i * Q3 + q) * C + c];
    const T ir = T(1) / U[0];
    const T v[3] = {U[1] * ir, U[2] * ir, U[3] * ir};
    const T p = gm1 * (U[4] - T(0.5) * U[0] * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]));
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      T F[5];
      euler_flux<T>(d, U, v, p, F);
      const T sc = (T)(0.25 * g.inv_dx[d]);
#pragma unroll
      for (int i = 0; i < 5; ++i) b2[((d * 5 + i) * Q3 + q) * C + c] = F[i] * sc;
    }
    if (FORCE) {
      const long long cell = c0 + c < nc ? c0 + c : nc - 1;  // ragged tail: in-bounds reads
      T a[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) a[d] = __ldg(field + ((size_t)d * Q3 + q) * nc + cell);
      const T e8 = T(0.125);
      b2[((15 + 0) * Q3 + q) * C + c] = U[0] * a[0] * e8;
      b2[((15 + 1) * Q3 + q) * C + c] = U[0] * a[1] * e8;
      b2[((15 + 2) * Q3 + q) * C + c] = U[0] * a[2] * e8;
      b2[((15 + 3) * Q3 + q) * C + c] = (U[1] * a[0] + U[2] * a[1] + U[3] * a[2]) * e8;
    }
  }
  __syncthreads();
  // H[comp][u][bc] = sum_qa G[comp][qa + Q bc] X(u, qa), X = P' w for the
  // x-fluxes (comp < 5), P w otherwise -> b1
  constexpr int NCP = FORCE ? 19 : 15;
  for (int it = tid; it < NCP * Q2 * C; it += kThreads) {
    const int c = it % C, r = it / C, bc = r % Q2, comp = r / Q2;
    T gq[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) gq[q] = b2[(comp * Q3 + q + Q * bc) * C + c];
    if (comp < 5) {
#pragma unroll
      for (int u = 0; u <= K; ++u) {
        T a = T(0);
#pragma unroll
        for (int q = 0; q < Q; ++q) a += gq[q] * sfc<T>(ODW + u * Q + q);
        b1[((comp * KP + u) * Q2 + bc) * C + c] = a;
      }
    } else {
#pragma unroll
      for (int u = 0; u <= K; ++u) {
        T a = T(0);
#pragma unroll
        for (int q = 0; q < Q; ++q) a += gq[q] * sfc<T>(OPW + u * Q + q);
        b1[((comp * KP + u) * Q2 + bc) * C + c] = a;
      }
    }
  }
  __syncthreads();
  // rows 0..4: J_i[pair(u,v)][qc] = sum_b H_{0,i}[u][b,qc] Pw(v,b) + H_{1,i} Dw(v,b);
  // rows 5..9: I2_i = sum_b H_{2,i} Pw; rows 10..13: SI = sum_b SH Pw -> b2.
  // Face moments Mt[d*2+side][i][a][t2] = sum_t1 Fhat Pw(a, t1) -> b2 + MT0
  constexpr int NR = FORCE ? 14 : 10;
  constexpr int NJ = NR * KP * Q * C;
  for (int it = tid; it < NJ + 30 * Q * C; it += kThreads) {
    if (it < NJ) {
      const int c = it % C, r = it / C, qc = r % Q, u = (r / Q) % KP, row = r / (Q * KP);
      const int comp = row < 5 ? row : (row < 10 ? 10 + (row - 5) : 15 + (row - 10));
      T h0[Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) h0[q] = b1[((comp * KP + u) * Q2 + q + Q * qc) * C + c];
      if (row < 5) {
        T h1[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) h1[q] = b1[(((5 + row) * KP + u) * Q2 + q + Q * qc) * C + c];
#pragma unroll
        for (int v = 0; v <= K; ++v)
          if (v <= K - u) {
            T a = T(0);
#pragma unroll
            for (int q = 0; q < Q; ++q) a += h0[q] * sfc<T>(OPW + v * Q + q) + h1[q] * sfc<T>(ODW + v * Q + q);
            b2[((row * TP + pair_index(K, u, v)) * Q + qc) * C + c] = a;
          }
      } else {
#pragma unroll
        for (int v = 0; v <= K; ++v)
          if (v <= K - u) {
            T a = T(0);
#pragma unroll
            for (int q = 0; q < Q; ++q) a += h0[q] * sfc<T>(OPW + v * Q + q);
            b2[((row * TP + pair_index(K, u, v)) * Q + qc) * C + c] = a;
          }
      }
    } else {
      const int jt = it - NJ;
      const int c = jt % C, r = jt / C, t2 = r % Q, i = (r / Q) % 5, ds = r / (5 * Q);
      const int d = ds >> 1, side = ds & 1;
      const long long cell = c0 + c;
      T m[KP];
#pragma unroll
      for (int a = 0; a <= K; ++a) m[a] = T(0);
      if (cell < nc) {
        long long fc = cell;  // low face: this cell's; high face: the upper cell's
        if (side) {
          int ix, iy, iz;
          cell_xyz(cell, g, ix, iy, iz);
          fc = neighbour(g, ix, iy, iz, d, +1);
        }
        const T* fp = fh + ((size_t)(d * 5 + i) * Q2 + Q * t2) * nc + fc;
#pragma unroll
        for (int t1 = 0; t1 < Q; ++t1) {
          const T f = __ldg(fp + (size_t)t1 * nc);
#pragma unroll
          for (int a = 0; a <= K; ++a) m[a] += f * sfc<T>(OPW + a * Q + t1);
        }
      }
#pragma unroll
      for (int a = 0; a <= K; ++a) b2[CF::MT0 * C + (((ds * 5 + i) * KP + a) * Q + t2) * C + c] = m[a];
    }
  }
  __syncthreads();
  // M[d*2+side][i][pair(a,b)] = +-(1/(4 dx_d)) sum_t2 Mt[a][t2] Pw(b, t2) -> b1
  for (int it = tid; it < 30 * KP * C; it += kThreads) {
    const int c = it % C, r = it / C, a = r % KP, i = (r / KP) % 5, ds = r / (5 * KP);
    const int d = ds >> 1, side = ds & 1;
    T mt[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) mt[q] = b2[CF::MT0 * C + (((ds * 5 + i) * KP + a) * Q + q) * C + c];
    const T sc = side == 0 ? (T)(0.25 * g.inv_dx[d]) : (T)(-0.25 * g.inv_dx[d]);
#pragma unroll
    for (int b = 0; b <= K; ++b)
      if (b <= K - a) {
        T m = T(0);
#pragma unroll
        for (int q = 0; q < Q; ++q) m += mt[q] * sfc<T>(OPW + b * Q + q);
        b1[((ds * 5 + i) * TP + pair_index(K, a, b)) * C + c] = m * sc;
      }
  }
  __syncthreads();
  // dw/dt per (cell, variable, (u,v)) for all w: volume + source + six faces
  for (int it = tid; it < 5 * TP * C; it += kThreads) {
    const int c = it % C, r = it / C, j = r % TP, i = r / TP;
    const long long cell = c0 + c;
    int u, v;
    pair_uv<K>(j, u, v);
    T jr[Q], i2[Q], sr[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      jr[q] = b2[((i * TP + j) * Q + q) * C + c];
      i2[q] = b2[(((5 + i) * TP + j) * Q + q) * C + c];
      sr[q] = (FORCE && i > 0) ? b2[(((10 + i - 1) * TP + j) * Q + q) * C + c] : T(0);
    }
    const T* Mi = b1 + (i * TP) * C + c;  // M[ds][i][pair] at Mi[(ds*5*TP + pair) * C]
#pragma unroll
    for (int w = 0; w <= K; ++w)
      if (w <= K - u - v) {
        T a = T(0);
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          a += jr[q] * sfc<T>(OPW + w * Q + q) + i2[q] * sfc<T>(ODW + w * Q + q);
          if (FORCE) a += sr[q] * sfc<T>(OPW + w * Q + q);
        }
        // faces: along x the normal exponent is u and the tangential pair
        // (v, w); along y v and (u, w); along z w and (u, v)
        const int jx = pair_index(K, v, w), jy = pair_index(K, u, w);
        a += Mi[((0 * 5) * TP + jx) * C] * __ldg(tab + TB::FEND + u) +
             Mi[((1 * 5) * TP + jx) * C] * __ldg(tab + TB::FEND + KP + u);
        a += Mi[((2 * 5) * TP + jy) * C] * __ldg(tab + TB::FEND + v) +
             Mi[((3 * 5) * TP + jy) * C] * __ldg(tab + TB::FEND + KP + v);
        a += Mi[((4 * 5) * TP + j) * C] * sfc<T>(3 * KP * Q + w) +
             Mi[((5 * 5) * TP + j) * C] * sfc<T>(3 * KP * Q + KP + w);
        if (cell < nc) {
          const int l = mode_index(u, v, w);
          const size_t at = (size_t)(i * N + l) * nc + cell;
          if (MODE == MODE_RHS) {
            R[at] = -f32_to_f64(a);
          } else {
            const double inc = st.ys[at] + st.dt * f32_to_f64(a);
            const double vv = (st.a0 == 0.0 && st.b0 == 1.0) ? inc : st.a0 * st.y0[at] + st.b0 * inc;
            st.out[at] = vv;
            st.yf[at] = f64_to_f32(vv);
            sV[(i * N + l) * C + c] = vv;
          }
        }
      }
  }
  if (MODE == MODE_RHS) return;
  __syncthreads();
  // limiter screen of the next stage's input (FP64); cells that fail it are
  // queued for the full limiter
  for (int it = tid; it < 5 * C; it += kThreads) {
    const int c = it % C, i = it / C;
    if (c0 + c >= nc) continue;
    const double* row = sV + (i * N) * C + c;
    double sa = 0.0;
    bool fin = isfinite(row[0]);
    for (int l = 1; l < N; ++l) {
      sa += fabs(row[l * C]) * __ldg(tab64 + (g.lim_vol ? TB::LMAXV : TB::LMAX) + l);
      fin &= isfinite(row[l * C]);
    }
    sM[it] = fin ? row[0] : __longlong_as_double(0x7ff8000000000000LL);
    sA[it] = sa;
  }
  __syncthreads();
  if (tid < C && c0 + tid < nc) {
    double m[5], a[5];
    bool fin = true;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      m[i] = sM[i * C + tid];
      a[i] = sA[i * C + tid];
      fin &= isfinite(m[i]);
    }
    if (!limiter_screen<K>(m, a, fin, g.gamma, g.eps_rho, g.eps_p)) {
      const unsigned slot = atomicAdd(&ctrl->n_flag, 1u);
      st.list[slot] = (int)(c0 + tid);
    }
  }
}

// ------------------------------------------------------ standalone limiter
template <int K>
__global__ void __launch_bounds__(kThreads) limit_kernel(double* __restrict__ y, int8_t* __restrict__ flags,
                                                         const double* __restrict__ tab64, Geo g, Ctrl* ctrl,
                                                         const float* __restrict__ tab32) {
  __shared__ unsigned s_err;
  __shared__ unsigned s_cnt;
  if (threadIdx.x == 0) {
    s_err = 0u;
    s_cnt = 0u;
  }
  __syncthreads();
  const long long cell = (long long)blockIdx.x * kThreads + threadIdx.x;
  if (cell < g.nc) {
    unsigned e = 0;
    int f = limit_cell<K>(y + cell, g.nc, tab64, g.gamma, g.eps_rho, g.eps_p, &e, g.lim_vol, tab32);
    if (flags) flags[cell] = (int8_t)f;
    if (f) atomicAdd(&s_cnt, 1u);
    if (e) atomicOr(&s_err, e);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_err) atomicOr(&ctrl->err, s_err);
    if (s_cnt) atomicAdd(&ctrl->n_limited, (unsigned long long)s_cnt);
  }
}

// ------------------------------------------------------------ CFL (max s)
// s_K = sum_a (|v_a| + c) / dx_a from the cell means; the result is the FP64
// maximum over cells, bit for bit what the plain FP64 loop gives, but the
// FP64 division and square root (the FP64 pipe is about 1/64 of the FP32
// rate) run for a few cells per block only. One cell per thread: s in FP32
// first (means converted on the integer pipe, correctly rounded reciprocal
// and square root), then the block's FP32 maximum over the trusted cells; the cells
// within a relative 1e-3 of it and the untrusted ones (means not finite or
// not clearly positive, pressure from a cancellation E - kin with kin above
// 0.99 E) are evaluated in FP64, and the FP64 maximum of those is the
// block's maximum. A trusted cell's FP32 s is within a relative 1e-4 of its
// FP64 s (a few roundings, the pressure's amplified at most 199x by the
// cancellation, halved by the square root), so the cell holding the
// block's FP64 maximum is always among the re-evaluated ones. Blocks combine
// by one atomicMax on the bit pattern of the non-negative double; inside a
// block the maxima are compared as bit patterns too, because a warp's FP64
// comparison holds the FP64 pipe for 16 clocks. 128^3: 39 us, from 60 us with
// FP64 comparisons and blocks of 1024 (bit patterns and 1024: 42; the means at
// the HBM rate: 12); degree 3, 160^3: 67 us from 106 (512 threads: 70).
constexpr int kCflThreads = 256;

template <int K>
__global__ void __launch_bounds__(kCflThreads) cfl_kernel(const double* __restrict__ y, Geo g, Ctrl* ctrl) {
  stream_wait();
  constexpr int N = nmodes(K);
  const long long nc = g.nc;
  const long long c = (long long)blockIdx.x * kCflThreads + threadIdx.x;
  double r = 1.0, m1 = 0.0, m2 = 0.0, m3 = 0.0, E = 0.0;
  float sf = 0.f;
  bool trusted = false;
  if (c < nc) {
    r = y[c];
    m1 = y[(size_t)N * nc + c];
    m2 = y[(size_t)2 * N * nc + c];
    m3 = y[(size_t)3 * N * nc + c];
    E = y[(size_t)4 * N * nc + c];
    const float rf = f64_to_f32(r), m1f = f64_to_f32(m1), m2f = f64_to_f32(m2), m3f = f64_to_f32(m3);
    const float Ef = f64_to_f32(E);
    const float irf = __frcp_rn(rf);
    const float kin = 0.5f * (m1f * m1f + m2f * m2f + m3f * m3f) * irf;
    const float prf = f64_to_f32(g.gamma - 1.0) * (Ef - kin);
    const float csf = sqrtf(f64_to_f32(g.gamma) * prf * irf);
    sf = (fabsf(m1f) * irf + csf) * f64_to_f32(g.inv_dx[0]) + (fabsf(m2f) * irf + csf) * f64_to_f32(g.inv_dx[1]) +
         (fabsf(m3f) * irf + csf) * f64_to_f32(g.inv_dx[2]);
    trusted = rf >= 1e-30f && rf <= 1e30f && Ef <= 1e30f && kin <= 0.99f * Ef && prf >= 1e-30f && sf <= 3e38f;
  }
  __shared__ float s_wf[kCflThreads / 32];
  __shared__ unsigned long long s_w[kCflThreads / 32];
  __shared__ unsigned s_err;
  float mf = trusted ? sf : 0.f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mf = fmaxf(mf, __shfl_xor_sync(0xffffffffu, mf, o));
  if (threadIdx.x == 0) s_err = 0u;
  if ((threadIdx.x & 31) == 0) s_wf[threadIdx.x >> 5] = mf;
  __syncthreads();
  mf = s_wf[0];
#pragma unroll
  for (int w = 1; w < kCflThreads / 32; ++w) mf = fmaxf(mf, s_wf[w]);
  // the FP64 maxima as bit patterns (non-negative doubles order like integers): the
  // FP64 pipe takes 16 clocks for a warp's comparison
  unsigned long long smax = 0ull;
  unsigned e = 0;
  if (c < nc && (!trusted || sf >= mf * (1.f - 1e-3f))) {
    const double ir = 1.0 / r;
    const double pr = (g.gamma - 1.0) * (E - 0.5 * (m1 * m1 + m2 * m2 + m3 * m3) * ir);
    if (!(r > 0.0) || !(pr > 0.0)) {
      e = (isfinite(r) && isfinite(pr)) ? ERRB_POSITIVITY : ERRB_NONFINITE;
    } else {
      const double cs = sqrt(g.gamma * pr * ir);
      const double sd = (fabs(m1) * ir + cs) * g.inv_dx[0] + (fabs(m2) * ir + cs) * g.inv_dx[1] +
                        (fabs(m3) * ir + cs) * g.inv_dx[2];
      if (sd > 0.0) smax = (unsigned long long)__double_as_longlong(sd);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long v = __shfl_xor_sync(0xffffffffu, smax, o);
    if (v > smax) smax = v;
  }
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = smax;
  if (e) atomicOr(&s_err, e);
  __syncthreads();
  if (threadIdx.x < 32) {
    unsigned long long v = threadIdx.x < kCflThreads / 32 ? s_w[threadIdx.x] : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long u = __shfl_xor_sync(0xffffffffu, v, o);
      if (u > v) v = u;
    }
    if (threadIdx.x == 0) {
      if (s_err) atomicOr(&ctrl->err, s_err);
      // the block that ends last hands the maximum over and leaves 0 for the next
      // reduction, so that no call depends on another one having run (a memset
      // before the kernel: 5 us of a host-bound loop on small meshes)
      atomicMax(&ctrl->cfl_running, v);
      if (count_done(&ctrl->cfl_blocks) == gridDim.x - 1) {
        ctrl->cfl_max_bits = atomicMax(&ctrl->cfl_running, 0ull);
        ctrl->cfl_running = 0ull;
        ctrl->cfl_blocks = 0u;
      }
    }
  }
}

// ------------------------------------------------------- energy reset
// Sect. 3.2: at every volume point rho eps = c^2/(gamma-1) rho (rho/rho0)^(gamma-1),
// E_q = 1/2 |m_q|^2 / rho_q + rho_q eps_q, energy modes re-projected (one
// thread per (cell, mode)); only the energy rows are written back. Cells
// that then fail the limiter screen are queued (list / ctrl->n_flag) for the
// full limiter. part[blockIdx.x] receives the block's sum of
// (e_before - e_after), e = E - |m|^2 / (2 rho) from the means.
// Constants of the energy reset in the kernel's arithmetic type, prepared
// on the host (the FP32 kernel then does no per-thread FP64 set-up work).
template <typename T>
struct ResetConsts {
  T c2g, inv_rho0, gm1;  // c^2/(gamma-1), 1/rho0, gamma-1
  int two_thirds;        // gamma - 1 within 1e-15 of 2/3
};

// Energy reset with sum-factorised point values and projection (the same
// sums as a dense evaluation, reordered): one thread per (cell, variable)
// for rho and the momenta loads the variable's N coefficients once and
// evaluates them at the Q^3 Gauss points along z, then y, then x (the 1D
// tables of the sum-factorised kernels), writing rows of Q^3 values per cell
// to shared memory with 16-byte stores; one thread per (cell, point) forms
// E_q; the projection of E contracts x first (one (cell, qz, qy) per
// thread), then y and z per mode. Rows are padded to a multiple of 16 bytes
// whose stride spreads the 8 rows of a quarter warp over all 32 banks. The
// screen sums of rho and the momenta come from the coefficients the value
// threads hold; those of E from the new modes. FP64: values and projection in
// fixed point (dg_common.cuh), a slice at a time, and x^(2/3) by one iteration:
// 128^3, degree 2: 7.05 -> 2.23 ms.
template <int K, typename T>
struct ResetSF {
  static constexpr int C = 32;  // cells per block: one warp per variable
  static constexpr int THREADS = 4 * C;
  static constexpr int Q = K + 1, Q3 = Q * Q * Q, N = nmodes(K);
  static constexpr int V = 16 / (int)sizeof(T);  // elements per 16-byte access
  // row length: at least Q^3, a multiple of V, and (in 4-byte words) an odd
  // multiple of 4 modulo 32 apart from row to row
  static constexpr int ROWW = ((Q3 * (int)sizeof(T) / 4 + 3) / 4) * 4;  // words, multiple of 4
  static constexpr int ROW = ((ROWW / 4) % 2 == 1 ? ROWW : ROWW + 4) * 4 / (int)sizeof(T);
  // dynamic shared memory: point values [4][C][ROW] and E [C][ROW]
  static constexpr size_t smem() { return (size_t)5 * C * ROW * sizeof(T); }
  // CTAs per SM the register budget is sized for: what the kernel takes without
  // reset_screen, which runs for few cells
  static constexpr int MINB = sizeof(T) == 4 ? (K <= 2 ? 16 : 9) : (K <= 1 ? 10 : K == 2 ? 8 : 4);
};

// The FP64 test of a reset cell that the FP32 screen does not clear. m, sa: means and
// sums of rho and the momenta, en: energy modes (all 32 = C apart), whose sum is taken
// in T's precision (FP32: widened). Not inlined and within the kernel's own
// registers (MINB), which it would otherwise raise from 30 to 56: reset and limiter at
// 100 x 90 x 84, degree 1, mixed, 73 us instead of 59 (57 without it).
template <int K, typename T>
__device__ DG_NOINLINE bool reset_screen(const double* m, const double* sa, const double* en,
                                         const T* __restrict__ tab, int vol, double gamma, double eps_r,
                                         double eps_p) {
  using TB = Tab<K>;
  constexpr int C = ResetSF<K, T>::C, N = TB::N;
  const int lmax = vol ? TB::LMAXV : TB::LMAX;
  double md[5], ad[5];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    md[i] = m[i * C];
    ad[i] = sa[i * C];
  }
  md[4] = en[0];
  if constexpr (sizeof(T) == 8) {
    ad[4] = 0.0;
#pragma unroll 1
    for (int l = 1; l < N; ++l) ad[4] += fabs(en[l * C]) * __ldg(tab + lmax + l);
  } else {
    float se = 0.f;
#pragma unroll 1
    for (int l = 1; l < N; ++l) se += fabsf(f64_to_f32(en[l * C])) * c_tab32[lmax + l];
    ad[4] = (double)se * (1.0 + 1e-5);
  }
  return limiter_screen<K>(md, ad, true, gamma, eps_r, eps_p);
}

template <int K, typename T>
__global__ void __launch_bounds__(ResetSF<K, T>::THREADS, ResetSF<K, T>::MINB) energy_reset_sf_kernel(
    double* __restrict__ y, const T* __restrict__ tab, Geo g, ResetConsts<T> rc, double* __restrict__ part,
    int* __restrict__ list, Ctrl* ctrl, float* __restrict__ yf) {
  stream_wait();
  using RS = ResetSF<K, T>;
  using TB = Tab<K>;
  constexpr int C = RS::C, Q = RS::Q, Q3 = RS::Q3, N = RS::N, ROW = RS::ROW, V = RS::V;
  struct alignas(16) Vec {
    T v[V];
  };
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sU = reinterpret_cast<T*>(smem_raw);  // [variable][cell][point]
  T* sE = sU + 4 * C * ROW;                // [cell][point]
  __shared__ double sEn[N * C];                // new energy modes [mode][cell]
  __shared__ double sM[5 * C];                 // means (old energy mean in row 4)
  __shared__ double sA[5 * C];                 // sum_l |w_il| max |phi_l|
  __shared__ int sFin[(4 + Q) * C];            // finite flags; FP64: the slices' exponents
  clear_deep(ctrl);
  const long long nc = g.nc;
  const long long c0 = (long long)blockIdx.x * C;
  const int tid = threadIdx.x;
  const bool from_shadow = sizeof(T) == 4 && yf != nullptr;
  // ------------------------------------------------ point values of rho, m
  {
    const int i = tid / C, c = tid % C;  // warp = variable
    const long long cell = c0 + c;
    const bool in = cell < nc;
    if constexpr (sizeof(T) == 8) {
      // FP64: sum-factorised in fixed point (dg_common.cuh), a slice at a time
      using FT = FxTab<K>;
      constexpr int T2 = (K + 1) * (K + 2) / 2, Q2 = Q * Q;
      double w[N];
#pragma unroll
      for (int l = 0; l < N; ++l) w[l] = in ? y[(size_t)(i * N + l) * nc + cell] : (i == 0 && l == 0 ? 1.0 : 0.0);
      sM[i * C + c] = w[0];
      if (tid < C) sM[4 * C + c] = in ? y[(size_t)(4 * N) * nc + cell] : 0.0;
      // screen sum (FP32 of the rounded coefficients, widened by a relative
      // 1e-5, still an upper bound)
      float sa = 0.f;
      bool fin = finite64(w[0]);
#pragma unroll
      for (int l = 1; l < N; ++l) {
        sa = fmaf(abs_up(w[l]), c_tab32[(g.lim_vol ? TB::LMAXV : TB::LMAX) + l], sa);
        fin &= finite64(w[l]);
      }
      sA[i * C + c] = f32_to_f64_q(sa * (1.f + 1e-5f));
      sFin[i * C + c] = (int)fin;
      const int B = fx_bound<K>(w);
      Fx x[N];
#pragma unroll
      for (int l = 0; l < N; ++l) x[l] = fx_split(fx_from(w[l], B));
      T* out = sU + (i * C + c) * ROW;
#pragma unroll 1
      for (int qz = 0; qz < Q; ++qz) {
        Fx A1[T2];
#pragma unroll
        for (int u = 0, j = 0; u <= K; ++u)
#pragma unroll
          for (int v = 0; u + v <= K; ++v, ++j) {
            FxAcc s{0, 0};
#pragma unroll
            for (int ww = 1; u + v + ww <= K; ++ww) fx_madt(s, x[mode_index(u, v, ww)], FT::P + ww * Q + qz);
            const long long x0 = fx_join(x[mode_index(u, v, 0)]);
            A1[j] = fx_split(u + v < K ? fx_val(s) + x0 : x0);
          }
        Fx A2[Q][K + 1];
        fx_rows<K, 0>(A1, A2);
#pragma unroll
        for (int qy = 0; qy < Q; ++qy) {
          long long v[Q];
          fx_values<K, K + 1>(A2[qy], v);
#pragma unroll
          for (int qx = 0; qx < Q; ++qx)
            out[qz * Q2 + qy * Q + qx] = B < kFxHuge ? fx_to_double(v[qx], B) : __longlong_as_double(0x7ff8000000000000LL);
        }
      }
    } else {
      T w[N];
      double mean = in ? y[(size_t)(i * N) * nc + cell] : (i == 0 ? 1.0 : 0.0);
      w[0] = f64_to_f32(mean);
#pragma unroll
      for (int l = 1; l < N; ++l) {
        if (!in) w[l] = T(0);
        else if (from_shadow) w[l] = (T)yf[(size_t)(i * N + l) * nc + cell];
        else w[l] = (T)y[(size_t)(i * N + l) * nc + cell];
      }
      sM[i * C + c] = mean;
      if (tid < C) sM[4 * C + c] = in ? y[(size_t)(4 * N) * nc + cell] : 0.0;
      // screen sums of this variable from the coefficients held (FP32: of the
      // rounded coefficients, widened by a relative 1e-5, still an upper bound)
      {
        T sa = T(0);
        bool fin = true;
#pragma unroll
        for (int l = 1; l < N; ++l) {
          const T lm = g.lim_vol ? c_tab32[TB::LMAXV + l] : c_tab32[TB::LMAX + l];
          sa += fabs(w[l]) * lm;
          fin &= isfinite(w[l]);
        }
        sA[i * C + c] = in ? (double)sa * (1.0 + 1e-5) : 0.0;
        sFin[i * C + c] = in ? (int)fin : 1;
      }
      // values at q = qx + Q (qy + Q qz): contract z, then y, then x with
      // Pt_u(x_a) (sfc<T>(u Q + a))
      T vals[Q3];
#pragma unroll
      for (int qz = 0; qz < Q; ++qz) {
        T A1[(K + 1) * (K + 2) / 2];
#pragma unroll
        for (int u = 0, j = 0; u <= K; ++u)
#pragma unroll
          for (int v = 0; u + v <= K; ++v, ++j) {
            T s = T(0);
#pragma unroll
            for (int ww = 0; u + v + ww <= K; ++ww) s += w[mode_index(u, v, ww)] * sfc<T>(ww * Q + qz);
            A1[j] = s;
          }
#pragma unroll
        for (int qy = 0; qy < Q; ++qy) {
          T A2[K + 1];
#pragma unroll
          for (int u = 0, j = 0; u <= K; ++u) {
            T s = T(0);
#pragma unroll
            for (int v = 0; u + v <= K; ++v, ++j) s += A1[j] * sfc<T>(v * Q + qy);
            A2[u] = s;
          }
#pragma unroll
          for (int qx = 0; qx < Q; ++qx) {
            T s = T(0);
#pragma unroll
            for (int u = 0; u <= K; ++u) s += A2[u] * sfc<T>(u * Q + qx);
            vals[qx + Q * (qy + Q * qz)] = s;
          }
        }
      }
      Vec* out = reinterpret_cast<Vec*>(sU + (i * C + c) * ROW);
#pragma unroll
      for (int k = 0; k < ROW / V; ++k) {
        Vec t;
#pragma unroll
        for (int e = 0; e < V; ++e) t.v[e] = k * V + e < Q3 ? vals[k * V + e] : T(0);
        out[k] = t;
      }
    }
  }
  __syncthreads();
  // --------------------------------------------------- E at the points
  const T gm1 = rc.gm1;
  const bool two_thirds = rc.two_thirds != 0;
  const T tc2g = rc.c2g, tir0 = rc.inv_rho0;
  for (int it = tid; it < Q3 * C; it += RS::THREADS) {
    const int c = it / Q3, q = it - c * Q3;  // consecutive threads: consecutive points of a cell
    const T r = sU[(0 * C + c) * ROW + q];
    const T m1 = sU[(1 * C + c) * ROW + q], m2 = sU[(2 * C + c) * ROW + q], m3 = sU[(3 * C + c) * ROW + q];
    // gamma = 5/3 (gamma - 1 within 1e-15 of 2/3): x^(2/3) as cbrt(x)^2
    const T x = r * tir0;
    T xg;
    if constexpr (sizeof(T) == 8) {
      xg = two_thirds ? pow_2_3(x) : pow(x, gm1);
      sE[c * ROW + q] = fma(0.5 * fma(m1, m1, fma(m2, m2, m3 * m3)), rcp64(r), r * (tc2g * xg));
    } else {
      if (two_thirds) {
        const T cx = cbrt(x);
        xg = cx * cx;
      } else {
        xg = pow(x, gm1);
      }
      sE[c * ROW + q] = T(0.5) * (m1 * m1 + m2 * m2 + m3 * m3) / r + r * (tc2g * xg);
    }
  }
  __syncthreads();
  // --------------------------------------------------- projection of E
  // sum-factorised: G[(qz, qy)][u] = sum_qx E Pt_u(x_qx) w_qx (one (cell,
  // qz, qy) per thread, into the dead point-value rows), then every mode
  // (u, v, w) as sum_qz Pt_w w_qz sum_qy Pt_v w_qy G[(qz, qy)][u] (one
  // (cell, mode) per thread); Pt w from the 1D tables (sfc<T>(KQ + u Q + a))
  if constexpr (sizeof(T) == 8) {
    // FP64: one (cell, slice) per thread in fixed point, the slices summed per
    // mode
    using FT = FxTab<K>;
    long long* sAcc = reinterpret_cast<long long*>(smem_raw);  // [slice][mode][cell]
    int* sExp = sFin + 4 * C;                                  // [slice][cell]
    if (tid < Q * C) {
      const int qz = tid / C, c = tid % C;
      const T* e = sE + c * ROW + qz * Q * Q;
      unsigned mx = 0;
#pragma unroll
      for (int q = 0; q < Q * Q; ++q) mx = max(mx, (unsigned)__double2hiint(e[q]) & 0x7fffffffu);
      const int A = max(kFxTiny, bexp(mx) + 1);
      long long G[K + 1][Q];  // [u][qy]
#pragma unroll
      for (int qy = 0; qy < Q; ++qy) {
        long long v[Q];
        FxAcc r[K + 1];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          v[q] = fx_from(e[qy * Q + q], A);
          r[q] = {0, 0};
        }
        fx_project<K, false>(v, r);
#pragma unroll
        for (int u = 0; u <= K; ++u) G[u][qy] = fx_val(r[u]);
      }
#pragma unroll
      for (int u = 0; u <= K; ++u) {
        FxAcc h[K + 1];
#pragma unroll
        for (int v = 0; v <= K; ++v) h[v] = {0, 0};
        fx_project<K, false>(G[u], h);
#pragma unroll
        for (int v = 0; u + v <= K; ++v) {
          const Fx hx = fx_split(fx_val(h[v]));
#pragma unroll
          for (int ww = 0; u + v + ww <= K; ++ww) {
            FxAcc t{0, 0};
            fx_mad(t, hx, c_fx[FT::W + ww * Q + qz][0], c_fx[FT::W + ww * Q + qz][1]);
            sAcc[(qz * N + mode_index(u, v, ww)) * C + c] = fx_val(t);
          }
        }
      }
      sExp[qz * C + c] = bexp(mx) < kFxHuge ? A : 2 * kFxHuge;
    }
    __syncthreads();
    for (int it = tid; it < N * C; it += RS::THREADS) {
      const int l = it / C, c = it - l * C;
      int A = 0;
#pragma unroll
      for (int z = 0; z < Q; ++z) A = max(A, sExp[z * C + c]);
      long long t = 0;
#pragma unroll
      for (int z = 0; z < Q; ++z) t += sAcc[(z * N + l) * C + c] >> min(A - sExp[z * C + c], 63);
      sEn[it] = A < kFxHuge ? fx_to_double(t, A) : __longlong_as_double(0x7ff8000000000000LL);
    }
  } else {
    // rows of G an odd number of words apart: lanes over cells hit different banks
    // (degree 3, 160^3: 5.4 ms with 64 words, 1.8 with 65)
    constexpr int KQ = (K + 1) * Q, GROW = Q * Q * (K + 1) | 1;
    T* sG = sU;  // [cell][(qz Q + qy) (K + 1) + u]
    for (int it = tid; it < Q * Q * C; it += RS::THREADS) {
      const int c = it / (Q * Q), r = it - c * (Q * Q);  // r = qz Q + qy
      const T* e = sE + c * ROW + r * Q;
      T ev[Q];
      if constexpr (Q == V) {
        const Vec t = *reinterpret_cast<const Vec*>(e);  // a row of four points is 16 bytes
#pragma unroll
        for (int qx = 0; qx < Q; ++qx) ev[qx] = t.v[qx];
      } else {
#pragma unroll
        for (int qx = 0; qx < Q; ++qx) ev[qx] = e[qx];
      }
#pragma unroll
      for (int u = 0; u <= K; ++u) {
        T s = T(0);
#pragma unroll
        for (int qx = 0; qx < Q; ++qx) s += ev[qx] * sfc<T>(KQ + u * Q + qx);
        sG[c * GROW + r * (K + 1) + u] = s;
      }
    }
    __syncthreads();
    for (int it = tid; it < N * C; it += RS::THREADS) {
      const int l = it / C, c = it - l * C;  // a warp: one mode of 32 cells
      int u, v, ww;
      mode_uvw(l, u, v, ww);
      T pv[Q], pz[Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        pv[q] = sfc<T>(KQ + v * Q + q);
        pz[q] = sfc<T>(KQ + ww * Q + q);
      }
      const T* gc = sG + c * GROW + u;
      T acc = T(0);
#pragma unroll
      for (int qz = 0; qz < Q; ++qz) {
        T h = T(0);
#pragma unroll
        for (int qy = 0; qy < Q; ++qy) h += gc[(qz * Q + qy) * (K + 1)] * pv[qy];
        acc += h * pz[qz];
      }
      acc *= T(0.125);  // the reference cell's volume 8: w_l = 1/8 sum_q E phi_l w_q
      sEn[l * C + c] = f32_to_f64(acc);
    }
  }
  __syncthreads();
  // ------------------------------- screen of the reset state, dissipation
  double diss = 0.0;
  bool queue = false, test = false;
  if (tid < C && c0 + tid < nc) {
    const int c = tid;
    bool fin = finite64(sEn[c]);
    float sf = 0.f;
#pragma unroll
    for (int l = 1; l < N; ++l) {
      sf = fmaf(abs_up(sEn[l * C + c]), g.lim_vol ? c_tab32[TB::LMAXV + l] : c_tab32[TB::LMAX + l], sf);
      fin &= finite64(sEn[l * C + c]);
    }
    // the kinetic energy of the means stays: the drop of the internal energy is
    // that of the total
    diss = sM[4 * C + c] - sEn[c];
    // FP32 screen first (the FP64 one takes two divisions and some 30 further FP64
    // operations per cell: reset and limiter at 128^3, degree 2, FP32-mixed, 0.41
    // ms with it for every cell, 0.35 so)
    float m[5], a[5];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      m[i] = f64_to_f32_q(sM[i * C + c]);
      a[i] = f64_to_f32_q(sA[i * C + c]) * (1.f + 1e-6f);
      fin &= sFin[i * C + c] != 0;
    }
    m[4] = f64_to_f32_q(sEn[c]);
    a[4] = sf * (1.f + 1e-5f);
    queue = !fin;
    test = fin && !screen_f32(m, a, (float)(g.gamma - 1.0), (float)g.eps_rho, (float)g.eps_p);
  }
  if (tid < C) sFin[tid] = test;
  // block sum of the dissipation: the C = 32 cells are warp 0's (fixed
  // shuffle order: deterministic)
  if (tid < 32) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) diss += __shfl_xor_sync(0xffffffffu, diss, o);
    if (tid == 0) part[blockIdx.x] = diss;
  }
  for (int it = tid; it < N * C; it += RS::THREADS) {
    const int l = it / C, c = it - l * C;
    const long long cell = c0 + c;
    if (cell < nc) {
      y[(size_t)(4 * N + l) * nc + cell] = sEn[l * C + c];
      if (yf) yf[(size_t)(4 * N + l) * nc + cell] = f64_to_f32(sEn[l * C + c]);
    }
  }
  // cells that the FP32 screen does not clear: FP64 sums of rho and the momenta (a
  // warp per variable), then the FP64 test
  if constexpr (sizeof(T) == 8) {
    __syncthreads();
    const int i = tid / C, c = tid % C;
    if (sFin[c]) {
      double sa = 0.0;
#pragma unroll
      for (int l = 1; l < N; ++l)
        sa += fabs(y[(size_t)(i * N + l) * nc + c0 + c]) * __ldg(tab + (g.lim_vol ? TB::LMAXV : TB::LMAX) + l);
      sA[i * C + c] = sa;
    }
    __syncthreads();
  }
  if (test)
    queue = !reset_screen<K, T>(sM + tid, sA + tid, sEn + tid, tab, g.lim_vol, g.gamma, g.eps_rho, g.eps_p);
  if (queue) {
    const unsigned slot = atomicAdd(&ctrl->n_flag, 1u);
    list[slot] = (int)(c0 + tid);
  }
}

// ------------------------------------------------------------- projection
// w_l = 1/8 sum_q f(x_q) phi_l(xi_q) omega_q (Sect. 2.3), f canonical
// [nc][5][Q^3]. One thread per (cell, variable).
// Cells first .. first + count - 1; f holds their point values only.
template <int K>
__global__ void __launch_bounds__(kThreads) project_kernel(const double* __restrict__ f, double* __restrict__ y,
                                                           const double* __restrict__ tab64, Geo g, long long first,
                                                           long long count) {
  using TB = Tab<K>;
  constexpr int N = TB::N, Q3 = TB::Q3;
  const long long nc = g.nc;
  const long long it = (long long)blockIdx.x * kThreads + threadIdx.x;
  if (it >= 5 * count) return;
  const long long local = it % count;
  const long long cell = first + local;
  const int i = (int)(it / count);
  double acc[N];
#pragma unroll
  for (int l = 0; l < N; ++l) acc[l] = 0.0;
  for (int q = 0; q < Q3; ++q) {
    const double v = f[((size_t)local * 5 + i) * Q3 + q];
    const double* pw = tab64 + TB::VPHIW + q * N;
#pragma unroll
    for (int l = 0; l < N; ++l) acc[l] += v * __ldg(pw + l);
  }
#pragma unroll
  for (int l = 0; l < N; ++l) y[(size_t)(i * N + l) * nc + cell] = acc[l];
}

// --------------------------------------------------------- forcing field
// a(x_q) = sum_j Re a_j cos(k_j.x) - Im a_j sin(k_j.x), k_j = 2 pi n_j / L
// (Sect. 3.1), cached at every volume point: field[(d*Q3 + q)*nc + c].
// modes: [n][9] = n_x, n_y, n_z (as doubles), Re a (3), Im a (3).
// Turbulence diagnostics (Sect. 4.1 rms Mach number, Sect. 4.2 injected
// energy): per-block partial sums, in a fixed order, of the per-cell
// (|m|/rho / c)^2 and |m|^2/(2 rho) of the cell means and, with forcing, the
// injected power density sum_q (m . a)(xi_q) omega_q / 8 (the state
// polynomial's momentum at the volume Gauss points times the cached driving
// field) as sum_l m_l a_l with the driving field's projection a_l = sum_q a
// phi_l omega_q / 8, sum-factorised in fixed point: the field is read once and
// 3 N FP64 multiply-adds remain of 3 Q^3 (N + 1). 64^3, degree 2, FP32 field:
// 107 us, the dense FP64 sums took 470. Registers for 3 CTAs per SM (2: 125
// us; 4: 107).
// part[j * gridDim.x + b], j = 0, 1, 2.
template <int K, typename T>
__global__ void __launch_bounds__(256, 3) diag_partial_kernel(const double* __restrict__ y, const T* __restrict__ field,
                                                           const double* __restrict__ tab64, Geo g, int force,
                                                           double* __restrict__ part) {
  using TB = Tab<K>;
  constexpr int N = TB::N, Q = K + 1, Q2 = Q * Q, Q3 = TB::Q3, W = FxTab<K>::W;
  __shared__ double s[3][256];
  const long long nc = g.nc;
  double acc[3] = {0.0, 0.0, 0.0};
  // items: (direction, cell); direction 0 also takes the means
  const long long items = force ? 3 * nc : nc;
  for (long long e = (long long)blockIdx.x * 256 + threadIdx.x; e < items; e += (long long)gridDim.x * 256) {
    const int d = e < nc ? 0 : (e < 2 * nc ? 1 : 2);
    const long long c = e - d * nc;
    if (d == 0) {
      const double rho = y[c], E = y[(size_t)4 * N * nc + c];
      double mm = 0.0;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const double m = y[(size_t)(1 + j) * N * nc + c];
        mm = fma(m, m, mm);
      }
      const double ir = rcp64(rho), k2 = mm * ir;
      const double pr = (g.gamma - 1.0) * fma(-0.5, k2, E);
      acc[0] += k2 * rcp64(g.gamma * pr);  // (mm / rho^2) / (gamma p / rho)
      acc[1] = fma(0.5, k2, acc[1]);
    }
    if (force) {
      const T* f = field + (size_t)d * Q3 * nc + c;
      long long a[N];
#pragma unroll
      for (int l = 0; l < N; ++l) a[l] = 0;
      int A = kFxTiny, top = 0;
#pragma unroll 1
      for (int qz = 0; qz < Q; ++qz) {
        T v[Q2];
        unsigned mx = 0;
#pragma unroll
        for (int q = 0; q < Q2; ++q) {
          v[q] = f[(size_t)(qz * Q2 + q) * nc];
          if constexpr (sizeof(T) == 4) mx = max(mx, __float_as_uint(v[q]) & 0x7fffffffu);
          else mx = max(mx, (unsigned)__double2hiint(v[q]) & 0x7fffffffu);
        }
        const int bx = sizeof(T) == 8 ? bexp(mx) : (mx >= 0x7f800000u ? kFxHuge : (int)(mx >> 23) + 896);
        top = max(top, bx);
        fx_raise(a, A, bx + 1);
        long long G[K + 1][Q];  // [u][qy]
#pragma unroll
        for (int qy = 0; qy < Q; ++qy) {
          long long x[Q];
          FxAcc r[K + 1];
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            x[q] = fx_from(v[q + Q * qy], A);
            r[q] = {0, 0};
          }
          fx_project<K, false>(x, r);
#pragma unroll
          for (int u = 0; u <= K; ++u) G[u][qy] = fx_val(r[u]);
        }
#pragma unroll
        for (int u = 0; u <= K; ++u) {
          FxAcc h[K + 1];
#pragma unroll
          for (int v1 = 0; v1 <= K; ++v1) h[v1] = {0, 0};
          fx_project<K, false>(G[u], h);
#pragma unroll
          for (int v1 = 0; u + v1 <= K; ++v1) {
            const Fx hx = fx_split(fx_val(h[v1]));
#pragma unroll
            for (int ww = 0; u + v1 + ww <= K; ++ww) {
              FxAcc t{0, 0};
              fx_madt(t, hx, W + ww * Q + qz);
              a[mode_index(u, v1, ww)] += fx_val(t);
            }
          }
        }
      }
      const double* m = y + (size_t)((1 + d) * N) * nc + c;
      double pw = top < kFxHuge ? 0.0 : __longlong_as_double(0x7ff8000000000000LL);
#pragma unroll
      for (int l = 0; l < N; ++l) pw = fma(m[(size_t)l * nc], fx_to_double(a[l], A), pw);
      acc[2] += pw;
    }
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) s[j][threadIdx.x] = acc[j];
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o)
#pragma unroll
      for (int j = 0; j < 3; ++j) s[j][threadIdx.x] += s[j][threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x < 3) part[threadIdx.x * gridDim.x + blockIdx.x] = s[threadIdx.x][0];
}

template <int K, typename T>
__global__ void __launch_bounds__(kThreads) forcing_field_kernel(T* __restrict__ field, const double* __restrict__ modes,
                                                                 int n_modes, const double* __restrict__ tab64, Geo g,
                                                                 double L0, double L1, double L2) {
  using TB = Tab<K>;
  constexpr int Q = TB::Q, Q3 = TB::Q3;
  const long long nc = g.nc;
  const long long cell = (long long)blockIdx.x * kThreads + threadIdx.x;
  if (cell >= nc) return;
  const int q = blockIdx.y;
  const int a = q % Q, b = (q / Q) % Q, cz = q / (Q * Q);
  int ix, iy, iz;
  cell_xyz(cell, g, ix, iy, iz);
  const double* gx = tab64 + TB::GX;
  const double x = (ix + 0.5) * g.dx[0] + 0.5 * g.dx[0] * gx[a];
  const double yy = (iy + 0.5) * g.dx[1] + 0.5 * g.dx[1] * gx[b];
  const double z = (iz + 0.5) * g.dx[2] + 0.5 * g.dx[2] * gx[cz];
  const double tp = 6.283185307179586476925286766559;
  double acc[3] = {0.0, 0.0, 0.0};
  for (int j = 0; j < n_modes; ++j) {
    const double* m = modes + 9 * j;
    const double ph = tp * (m[0] * x / L0 + m[1] * yy / L1 + m[2] * z / L2);
    double s, c;
    sincos(ph, &s, &c);
#pragma unroll
    for (int d = 0; d < 3; ++d) acc[d] += m[3 + d] * c - m[6 + d] * s;
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) field[((size_t)d * Q3 + q) * nc + cell] = (T)acc[d];
}

}  // namespace dg
