// dg_spectrum.cu -- velocity power spectrum (arXiv:1602.09079, Sect. 3.3):
// E_w(k) is the shell average of |w_hat(k)|^2 scaled so that its integral
// over k equals the mean square of w. Here the velocity of the state
// polynomial is sampled at sub^3 points per cell (cell-centred sub-cells),
// each component is transformed by a 3D real-to-complex FFT on a
// caller-provided work area (own passes in fixed point for grids of 32 to 1024
// points a side, a power of two; cuFFT for the others), and the power of every
// wave vector n is added to the shell round(|n|).
#include "dg_spectrum.h"

#include <cufft.h>

#include <cmath>

#include "dg_common.cuh"

namespace dg {
namespace spec {
namespace {

inline size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

// sqrt(2u+1) P_u(x) by the three-term recurrence
__device__ __forceinline__ double scaled_legendre(int u, double x) {
  double pm = 1.0, p = x;
  if (u == 0) return 1.0;
  for (int j = 2; j <= u; ++j) {
    const double pn = ((2 * j - 1) * x * p - (j - 1) * pm) / j;
    pm = p;
    p = pn;
  }
  return sqrt(2.0 * u + 1.0) * p;
}

// Samples of the state polynomial at the centres of sub^3 sub-cells per cell,
// sum-factorised in 64-bit fixed point (dg_common.cuh): a thread takes one cell
// and one z of its sub-cells (lanes: cells along x, so that a row of samples is
// written in one piece), contracts the coefficients along z once, along y per
// sub-cell row and along x per sample. tab: Pt_u at the sub-cell centres in
// units of 2^-58, [u][8]. What bounds it is the integer pipe and, for the
// velocity, the 4 FP64 operations of a division per sample; with the Legendre
// recurrences and the dense sum in FP64 per sample, 256^3 samples of one
// component took 5.72 ms, now 0.215.
constexpr int kMaxSub = 8;

__device__ __forceinline__ void sub_table(int k, int sub, int (*tab)[2]) {
  for (int j = threadIdx.x; j < (k + 1) * kMaxSub; j += blockDim.x) {
    const int u = j / kMaxSub, s = j % kMaxSub;
    const Fx c = fx_split(s < sub ? fx_from(scaled_legendre(u, -1.0 + (2.0 * s + 1.0) / sub), 1025) : 0);
    tab[j][0] = c.h;
    tab[j][1] = c.l;
  }
  __syncthreads();
}

template <int K>
struct SubCell {
  static constexpr int N = nmodes(K), T = (K + 1) * (K + 2) / 2;
  Fx a1[T], a2[K + 1];
  int B;
  // the variable's coefficients (rows nc apart) contracted along z
  __device__ __forceinline__ void load(const double* __restrict__ y, size_t nc, const int (*tab)[2], int sz) {
    double w[N];
#pragma unroll
    for (int l = 0; l < N; ++l) w[l] = __ldg(y + (size_t)l * nc);
    B = fx_bound<K>(w);
#pragma unroll
    for (int u = 0, j = 0; u <= K; ++u)
#pragma unroll
      for (int v = 0; u + v <= K; ++v, ++j) {
        FxAcc s{0, 0};
#pragma unroll
        for (int ww = 1; u + v + ww <= K; ++ww)
          fx_mad(s, fx_split(fx_from(w[mode_index(u, v, ww)], B)), tab[ww * kMaxSub + sz][0], tab[ww * kMaxSub + sz][1]);
        a1[j] = fx_split(fx_val(s) + fx_from(w[mode_index(u, v, 0)], B));
      }
  }
  __device__ __forceinline__ void row(const int (*tab)[2], int sy) {
#pragma unroll
    for (int u = 0, j = 0; u <= K; ++u) {
      FxAcc s{0, 0};
      const long long x0 = fx_join(a1[j]);
      ++j;
#pragma unroll
      for (int v = 1; u + v <= K; ++v, ++j) fx_mad(s, a1[j], tab[v * kMaxSub + sy][0], tab[v * kMaxSub + sy][1]);
      a2[u] = fx_split(fx_val(s) + x0);
    }
  }
  __device__ __forceinline__ long long at(const int (*tab)[2], int sx) const {
    FxAcc s{0, 0};
#pragma unroll
    for (int u = 1; u <= K; ++u) fx_mad(s, a2[u], tab[u * kMaxSub + sx][0], tab[u * kMaxSub + sx][1]);
    return fx_val(s) + fx_join(a2[0]);
  }
  __device__ __forceinline__ double value(const int (*tab)[2], int sx) const {
    return B < kFxHuge ? fx_to_double(at(tab, sx), B) : __longlong_as_double(0x7ff8000000000000LL);
  }
};

// item e = ((iz n + iy) sub + sz) n + ix
__device__ __forceinline__ void sub_item(long long e, int n, int sub, int& ix, int& iy, int& iz, int& sz) {
  ix = (int)(e % n);
  const long long r = e / n;
  sz = (int)(r % sub);
  const int yz = (int)(r / sub);
  iy = yz % n;
  iz = yz / n;
}

template <int K>
__device__ __forceinline__ void sample_cells(const double* __restrict__ y, int n, int sub, int comp,
                                             double* __restrict__ out, const int (*tab)[2]) {
  const int M = n * sub;
  const long long total = (long long)n * n * n * sub, nc = (long long)n * n * n;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    int ix, iy, iz, sz;
    sub_item(e, n, sub, ix, iy, iz, sz);
    const long long cell = ((long long)iz * n + iy) * n + ix;
    SubCell<K> r, m;
    r.load(y + cell, nc, tab, sz);
    m.load(y + (size_t)((1 + comp) * SubCell<K>::N) * nc + cell, nc, tab, sz);
    double* o = out + ((size_t)(iz * sub + sz) * M + (size_t)iy * sub) * M + (size_t)ix * sub;
#pragma unroll 1
    for (int sy = 0; sy < sub; ++sy, o += M) {
      r.row(tab, sy);
      m.row(tab, sy);
#pragma unroll 2
      for (int sx = 0; sx < sub; ++sx) o[sx] = m.value(tab, sx) * rcp64(r.value(tab, sx));
    }
  }
}

// out[(Z * M + Y) * M + X] = m_comp / rho of the state polynomial at the
// centre of sub-cell (X % sub, Y % sub, Z % sub) of cell (X, Y, Z) / sub
__global__ void __launch_bounds__(256) sample_kernel(const double* __restrict__ y, int k, int n, int sub, int comp,
                                                     double* __restrict__ out) {
  __shared__ int tab[4 * kMaxSub][2];
  sub_table(k, sub, tab);
  if (k == 0) sample_cells<0>(y, n, sub, comp, out, tab);
  else if (k == 1) sample_cells<1>(y, n, sub, comp, out, tab);
  else if (k == 2) sample_cells<2>(y, n, sub, comp, out, tab);
  else sample_cells<3>(y, n, sub, comp, out, tab);
}

// shell round(sqrt(k2)) of an integer k2: the b with b^2 - b < k2 <= b^2 + b
__device__ __forceinline__ int shell_of(long long k2) {
  long long b = (long long)sqrtf((float)k2);
  while (b > 0 && b * b - b >= k2) --b;
  while (b * b + b < k2) ++b;
  return (int)b;
}

// shell sums of the half spectrum [M][M][M/2 + 1]: each element stands for
// itself and (unless its last index is 0 or M/2) its conjugate partner. A
// thread takes kRun consecutive elements of a row (one 128-byte line), along
// which the shell never falls, and adds one sum per shell to its warp's copy of
// the bins where there is room for one per warp (copies; shared memory holds nb
// doubles per copy): a double has no native shared-memory atomic, and with one
// addition per element on one copy 256^3 took 0.431 ms per component, now 0.137.
constexpr int kRun = 8;
__global__ void __launch_bounds__(256) bin_kernel(const double2* __restrict__ sp, int M, int nb,
                                                  double* __restrict__ bins, int copies = 1) {
  extern __shared__ double sh[];
  for (int b = threadIdx.x; b < nb * copies; b += blockDim.x) sh[b] = 0.0;
  __syncthreads();
  double* mine = sh + (size_t)((int)(threadIdx.x >> 5) % copies) * nb;
  const int H = M / 2 + 1, chunks = (H + kRun - 1) / kRun;
  const long long total = (long long)M * M * chunks;
  const double norm = 1.0 / ((double)M * M * M) / ((double)M * M * M);
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int first = (int)(e % chunks) * kRun, last = min(first + kRun, H);
    const long long row = e / chunks;
    const int b = (int)(row % M), a = (int)(row / M);
    const int ky = b <= M / 2 ? b : b - M, kz = a <= M / 2 ? a : a - M;
    const long long yz = (long long)ky * ky + (long long)kz * kz;
    const double2* z = sp + row * H;
    int run = -1;
    double p = 0.0;
    for (int c = first; c < last; ++c) {
      const int bin = shell_of(yz + (long long)c * c);
      if (bin != run) {
        if (run >= 0 && run < nb) atomicAdd(&mine[run], p);
        run = bin;
        p = 0.0;
      }
      const double w = (c == 0 || (M % 2 == 0 && c == M / 2)) ? norm : 2.0 * norm;
      p = fma(w, fma(z[c].x, z[c].x, z[c].y * z[c].y), p);
    }
    if (run >= 0 && run < nb) atomicAdd(&mine[run], p);
  }
  __syncthreads();
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    double s = 0.0;
    for (int j = 0; j < copies; ++j) s += sh[(size_t)j * nb + b];
    if (s != 0.0) atomicAdd(&bins[b], s);
  }
}

// cuFFT plan of an M^3 D2Z transform with a caller-owned work area
cufftResult make_plan(int M, cufftHandle* plan, size_t* ws) {
  cufftResult r = cufftCreate(plan);
  if (r != CUFFT_SUCCESS) return r;
  r = cufftSetAutoAllocation(*plan, 0);
  if (r == CUFFT_SUCCESS) r = cufftMakePlan3d(*plan, M, M, M, CUFFT_D2Z, ws);
  if (r != CUFFT_SUCCESS) cufftDestroy(*plan);
  return r;
}

// Histogram of ln(rho) of the state polynomial at the sub-cell centres:
// counts[0] below lo (and non-positive or non-finite densities),
// counts[1 + j] for floor((ln rho - lo) / (hi - lo) * nb) = j, counts[nb + 1]
// at or above hi; integer counts (order-independent). The bin comes from an
// FP32 logarithm; where its error could reach a bin's edge, from FP64 as the
// definition has it. A thread's samples mostly fall into one bin after the
// other: runs are counted before they go to the shared histogram. The FP64
// logarithm and the dense sum of every sample took 6.54 ms for 256^3 samples,
// now 0.133.
__device__ __forceinline__ int density_bin(long long r, int B, double lo, double hi, int nb, float flo, float scale,
                                           float slack) {
  if (B >= kFxHuge || r <= 0) return 0;
  // ln r from the significand in [1, 2) and the exponent
  const int lz = clz64((unsigned long long)r);
  const unsigned m = (unsigned)(((unsigned long long)r << lz) >> 32);
  const int ex = B - 1083 + 63 - lz;
  const float f = __uint_as_float(0x3f800000u | ((m >> 8) & 0x7fffffu));
  const float s = fmaf((float)ex, 0.69314718056f, logf(f));
  const float t = (s - flo) * scale, e = slack + fabsf(s) * scale * 1e-6f, j = floorf(t);
  if (t - j > e && j + 1.f - t > e && t > -1e6f && t < 1e6f) return t < 0.f ? 0 : (t >= (float)nb ? nb + 1 : 1 + (int)j);
  const double rho = fx_to_double(r, B);
  if (!(rho > 0.0)) return 0;
  const double sv = log(rho);
  if (sv >= hi) return nb + 1;
  if (!(sv >= lo)) return 0;
  const int k = (int)floor((sv - lo) / (hi - lo) * nb);
  return 1 + (k < nb ? k : nb - 1);
}

template <int K>
__device__ __forceinline__ void hist_cells(const double* __restrict__ y, int n, int sub, double lo, double hi, int nb,
                                           const int (*tab)[2], unsigned int* shc) {
  const long long total = (long long)n * n * n * sub, nc = (long long)n * n * n;
  // FP32 bin position (s - lo) scale; the rounding of s, lo and scale stays
  // below 1e-6 (|s| + |lo|) scale, to which `slack` adds that of the products
  const float flo = (float)lo, scale = (float)(nb / (hi - lo));
  const float slack = (fabsf(flo) + 1.f) * scale * 1e-6f + (float)nb * 1e-6f + 1e-6f;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    int ix, iy, iz, sz;
    sub_item(e, n, sub, ix, iy, iz, sz);
    SubCell<K> r;
    r.load(y + ((long long)iz * n + iy) * n + ix, nc, tab, sz);
    int run = -1;
    unsigned count = 0;
#pragma unroll 1
    for (int sy = 0; sy < sub; ++sy) {
      r.row(tab, sy);
#pragma unroll 2
      for (int sx = 0; sx < sub; ++sx) {
        const int b = density_bin(r.at(tab, sx), r.B, lo, hi, nb, flo, scale, slack);
        if (b != run) {
          if (count) atomicAdd(&shc[run], count);
          run = b;
          count = 0;
        }
        ++count;
      }
    }
    atomicAdd(&shc[run], count);
  }
}

__global__ void __launch_bounds__(256) density_hist_kernel(const double* __restrict__ y, int k, int n, int sub,
                                                           double lo, double hi, int nb,
                                                           unsigned long long* __restrict__ counts) {
  extern __shared__ unsigned int shc[];
  __shared__ int tab[4 * kMaxSub][2];
  for (int b = threadIdx.x; b < nb + 2; b += blockDim.x) shc[b] = 0u;
  sub_table(k, sub, tab);
  if (k == 0) hist_cells<0>(y, n, sub, lo, hi, nb, tab, shc);
  else if (k == 1) hist_cells<1>(y, n, sub, lo, hi, nb, tab, shc);
  else if (k == 2) hist_cells<2>(y, n, sub, lo, hi, nb, tab, shc);
  else hist_cells<3>(y, n, sub, lo, hi, nb, tab, shc);
  __syncthreads();
  for (int b = threadIdx.x; b < nb + 2; b += blockDim.x)
    if (shc[b]) atomicAdd(&counts[b], (unsigned long long)shc[b]);
}

}  // namespace

namespace {
// ------------------------------------ 3D real transform, M a power of two
// The velocity spectrum only needs |v_hat|^2 by shell, so for M = 32 .. 1024 a
// power of two the transform is three passes over M^3 / 2 complex numbers (rows
// along x two at a time as one complex row, lines along y, lines along z), the
// last of which adds the powers to the bins instead of storing them. The values
// along x at n_x = 0 and M/2 are real: they share the column n_x = 0 as real and
// imaginary part, so that every pass has M/2 columns. A pass is a radix-4
// Stockham transform of a block's 4096 numbers in shared memory in 64-bit fixed
// point, one exponent per line: values start at 60 bits and each pass divides by
// its radix, so that the error of a line stays near one unit of 2^-60 of its
// largest value times sqrt(M) (an FP64 transform rounds its sums at 53 bits). A
// butterfly is 64-bit additions and three fixed-point products. cuFFT's FP64 transform is
// bound by the FP64 pipe (256^3: 1.75 ms per component, all other sizes still
// take it); these passes take 0.8, the shell sums included.
struct Cx {
  long long x, y;
};
constexpr int kFftPoints = 4096;  // complex numbers per CTA

__host__ __device__ constexpr bool own_fft(int M) { return M >= 32 && M <= 1024 && (M & (M - 1)) == 0; }

// exp(-2 pi i j / M), j < M, in units of 2^-58
__global__ void twiddle_kernel(int M, longlong2* __restrict__ tw) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= M) return;
  double sn, cs;
  sincospi(-2.0 * j / M, &sn, &cs);
  tw[j] = longlong2{fx_from(cs, 1025), fx_from(sn, 1025)};
}

// z times w (limbs); exact products, one rounding per part
__device__ __forceinline__ Cx fx_rotate(Cx z, longlong2 w) {
  const Fx zx = fx_split(z.x), zy = fx_split(z.y), c = fx_split(w.x), s = fx_split(w.y);
  FxAcc re{0, 0}, im{0, 0};
  fx_mad(re, zx, c.h, c.l);
  fx_mad(re, zy, -s.h, -s.l);
  fx_mad(im, zx, s.h, s.l);
  fx_mad(im, zy, c.h, c.l);
  return {fx_val(re), fx_val(im)};
}

__device__ __forceinline__ long long quarter(long long x) { return (x + 2) >> 2; }

// one Stockham pass of length n, stride st over every line of the block: four
// (radix 4) or eight (radix 2) butterflies per thread, read, barrier, written
template <int LINE, int ELEM, int RADIX>
__device__ __forceinline__ void fft_pass(Cx* z, int lines, int M, int logm, int n, int logst,
                                         const longlong2* __restrict__ tw) {
  constexpr int NB = kFftPoints / 256 / RADIX;
  const int per = M / RADIX, st = 1 << logst;  // butterflies per line
  const int sl = LINE ? LINE : M + 1, se = ELEM ? ELEM : lines;
  Cx v[NB][RADIX];
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int id = threadIdx.x + 256 * b;
    const int line = LINE ? id & (lines - 1) : id / per, j = LINE ? id / lines : id & (per - 1);
#pragma unroll
    for (int r = 0; r < RADIX; ++r) v[b][r] = z[line * sl + (j + r * per) * se];
  }
  __syncthreads();
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int id = threadIdx.x + 256 * b;
    const int line = LINE ? id & (lines - 1) : id / per, j = LINE ? id / lines : id & (per - 1);
    const int q = j & (st - 1), p = j >> logst;
    Cx* o = z + line * sl + (q + (p * RADIX << logst)) * se;
    const int step = st * se;
    if constexpr (RADIX == 4) {
      const Cx a{v[b][0].x + v[b][2].x, v[b][0].y + v[b][2].y}, c{v[b][0].x - v[b][2].x, v[b][0].y - v[b][2].y};
      const Cx d{v[b][1].x + v[b][3].x, v[b][1].y + v[b][3].y}, e{v[b][1].x - v[b][3].x, v[b][1].y - v[b][3].y};
      Cx y1{quarter(c.x + e.y), quarter(c.y - e.x)}, y2{quarter(a.x - d.x), quarter(a.y - d.y)};
      Cx y3{quarter(c.x - e.y), quarter(c.y + e.x)};
      if (n > 4) {
        const int t = p * (M / n);
        y1 = fx_rotate(y1, tw[t]);
        y2 = fx_rotate(y2, tw[2 * t]);
        y3 = fx_rotate(y3, tw[3 * t]);
      }
      o[0] = {quarter(a.x + d.x), quarter(a.y + d.y)};
      o[step] = y1;
      o[2 * step] = y2;
      o[3 * step] = y3;
    } else {
      o[0] = {(v[b][0].x + v[b][1].x + 1) >> 1, (v[b][0].y + v[b][1].y + 1) >> 1};
      o[step] = {(v[b][0].x - v[b][1].x + 1) >> 1, (v[b][0].y - v[b][1].y + 1) >> 1};
    }
  }
  __syncthreads();
}
template <int LINE, int ELEM>
__device__ __forceinline__ void fft_lines(Cx* z, int lines, int M, int logm, const longlong2* __restrict__ tw) {
  int n = M, logst = 0;
  for (; n >= 4; n >>= 2, logst += 2) fft_pass<LINE, ELEM, 4>(z, lines, M, logm, n, logst, tw);
  if (n == 2) fft_pass<LINE, ELEM, 2>(z, lines, M, logm, n, logst, tw);
}

__device__ __forceinline__ unsigned mag_hi(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }
__device__ __forceinline__ double fft_out(long long r, int B) {
  return B < kFxHuge ? fx_to_double(r, B) : __longlong_as_double(0x7ff8000000000000LL);
}

// rows along x: real [M][M][M] -> [M][M][M/2], n_x = M/2 in the imaginary part
// of n_x = 0. Shared memory: lines of M + 1 numbers, a maximum per line.
__global__ void __launch_bounds__(256, 2) fft_rows_kernel(const double* __restrict__ real, double2* __restrict__ sp,
                                                          int M, int logm, const longlong2* __restrict__ tw) {
  extern __shared__ __align__(16) unsigned char fft_smem[];
  Cx* z = reinterpret_cast<Cx*>(fft_smem);
  const int lines = kFftPoints / M, H = M / 2;
  unsigned long long* top = reinterpret_cast<unsigned long long*>(z + lines * (M + 1));
  for (int l = threadIdx.x; l < lines; l += 256) top[l] = 0ull;
  __syncthreads();
  const double* in = real + (size_t)blockIdx.x * lines * 2 * M;  // two rows per line
  // the numbers as they come, 16 per thread
#pragma unroll
  for (int b = 0; b < kFftPoints / 256; ++b) {
    const int id = threadIdx.x + 256 * b, line = id >> logm, e = id & (M - 1);
    const double re = in[(size_t)line * 2 * M + e], im = in[(size_t)line * 2 * M + M + e];
    z[line * (M + 1) + e] = {__double_as_longlong(re), __double_as_longlong(im)};
    unsigned m = max(mag_hi(re), mag_hi(im));  // a warp's 32 numbers lie in one line
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&top[line], (unsigned long long)m);
  }
  __syncthreads();
#pragma unroll
  for (int b = 0; b < kFftPoints / 256; ++b) {
    const int id = threadIdx.x + 256 * b, line = id >> logm, e = id & (M - 1);
    const int B = max(kFxTiny, bexp((unsigned)top[line]) + 1);
    Cx& v = z[line * (M + 1) + e];
    v = {fx_from(__longlong_as_double(v.x), B), fx_from(__longlong_as_double(v.y), B)};
  }
  __syncthreads();
  fft_lines<0, 1>(z, lines, M, logm, tw);
  double2* out = sp + (size_t)blockIdx.x * lines * 2 * H;
  for (int id = threadIdx.x; id < lines * H; id += 256) {
    const int line = id / H, k = id & (H - 1);
    const int B = max(kFxTiny, bexp((unsigned)top[line]) + 1);
    const Cx a = z[line * (M + 1) + k], c = z[line * (M + 1) + (k ? M - k : H)];
    double2 u, w;
    if (k == 0) {
      u = {fft_out(a.x, B + logm), fft_out(c.x, B + logm)};
      w = {fft_out(a.y, B + logm), fft_out(c.y, B + logm)};
    } else {
      // (Z_k + conj Z_-k) / 2 and (Z_k - conj Z_-k) / 2i
      u = {fft_out(a.x + c.x, B + logm - 1), fft_out(a.y - c.y, B + logm - 1)};
      w = {fft_out(a.y + c.y, B + logm - 1), fft_out(c.x - a.x, B + logm - 1)};
    }
    out[(size_t)(2 * line) * H + k] = u;
    out[(size_t)(2 * line + 1) * H + k] = w;
  }
}

// lines along y (Z = false, in place) or along z (Z = true): the powers of the
// columns n_x >= 1 go to the bins, the packed column n_x = 0 is stored.
template <bool Z>
__global__ void __launch_bounds__(256, 2) fft_lines_kernel(double2* __restrict__ sp, int M, int logm,
                                                           const longlong2* __restrict__ tw, int nb, int copies,
                                                           double* __restrict__ bins) {
  extern __shared__ __align__(16) unsigned char fft_smem[];
  Cx* z = reinterpret_cast<Cx*>(fft_smem);
  unsigned long long* top = reinterpret_cast<unsigned long long*>(z + kFftPoints);
  const int lines = kFftPoints / M, H = M / 2;
  double* sh = reinterpret_cast<double*>(top + lines);
  if (Z)
    for (int b = threadIdx.x; b < nb * copies; b += 256) sh[b] = 0.0;
  double* mine = sh + (size_t)((int)(threadIdx.x >> 5) % copies) * nb;
  const double norm = 1.0 / ((double)M * M * M) / ((double)M * M * M);
  const int tiles = M * H / lines;
  const size_t stride = Z ? (size_t)M * H : (size_t)H;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    for (int l = threadIdx.x; l < lines; l += 256) top[l] = 0ull;
    __syncthreads();
    const int line0 = tile * lines;
    // line l: column l % H of row l / H (of y for Z, of z otherwise)
    const int line = threadIdx.x & (lines - 1), l = line0 + line;
    double2* base = sp + (Z ? (size_t)l : (size_t)(l / H) * M * H + (l & (H - 1)));
    unsigned m = 0;
#pragma unroll
    for (int b = 0; b < kFftPoints / 256; ++b) {
      const int e = (threadIdx.x + 256 * b) / lines;
      const double2 v = base[e * stride];
      z[e * lines + line] = {__double_as_longlong(v.x), __double_as_longlong(v.y)};
      m = max(m, max(mag_hi(v.x), mag_hi(v.y)));
    }
    atomicMax(&top[line], (unsigned long long)m);
    __syncthreads();
    const int B = max(kFxTiny, bexp((unsigned)top[line]) + 1);
#pragma unroll
    for (int b = 0; b < kFftPoints / 256; ++b) {
      Cx& v = z[(threadIdx.x + 256 * b) / lines * lines + line];
      v = {fx_from(__longlong_as_double(v.x), B), fx_from(__longlong_as_double(v.y), B)};
    }
    __syncthreads();
    fft_lines<1, 0>(z, lines, M, logm, tw);
    if (!Z) {
#pragma unroll
      for (int b = 0; b < kFftPoints / 256; ++b) {
        const int e = (threadIdx.x + 256 * b) / lines;
        const Cx v = z[e * lines + line];
        base[e * stride] = {fft_out(v.x, B + logm), fft_out(v.y, B + logm)};
      }
    } else {
      // 16 consecutive numbers per thread: the columns of a row, or of several
      int run = -1;
      double p = 0.0;
      for (int j = 0; j < kFftPoints / 256; ++j) {
        const int id = threadIdx.x * (kFftPoints / 256) + j, e = id / lines, ll = id & (lines - 1);
        const int kx = (line0 + ll) & (H - 1), y = (line0 + ll) / H;
        const int Bl = max(kFxTiny, bexp((unsigned)top[ll]) + 1);
        const Cx v = z[id];
        const double2 u = {fft_out(v.x, Bl + logm), fft_out(v.y, Bl + logm)};
        if (kx == 0) {
          sp[(size_t)(line0 + ll) + e * stride] = u;
          continue;
        }
        const int ky = y <= H ? y : y - M, kz = e <= H ? e : e - M;
        const int bin = shell_of((long long)kx * kx + (long long)ky * ky + (long long)kz * kz);
        if (bin != run) {
          if (run >= 0 && run < nb) atomicAdd(&mine[run], p);
          run = bin;
          p = 0.0;
        }
        p = fma(2.0 * norm, fma(u.x, u.x, u.y * u.y), p);
      }
      if (run >= 0 && run < nb) atomicAdd(&mine[run], p);
    }
    __syncthreads();
  }
  if (Z)
    for (int b = threadIdx.x; b < nb; b += 256) {
      double t = 0.0;
      for (int j = 0; j < copies; ++j) t += sh[(size_t)j * nb + b];
      if (t != 0.0) atomicAdd(&bins[b], t);
    }
}

// the packed column: P = F_0 + i F_{M/2} with F_0, F_{M/2} the transforms of real
// data, F_0(k) = (P(k) + conj P(-k)) / 2, F_{M/2}(k) = (P(k) - conj P(-k)) / 2i
__global__ void __launch_bounds__(256) fft_packed_bins_kernel(const double2* __restrict__ sp, int M, int nb,
                                                              double* __restrict__ bins) {
  const int H = M / 2;
  const double norm = 1.0 / ((double)M * M * M) / ((double)M * M * M);
  for (int id = blockIdx.x * 256 + threadIdx.x; id < M * M; id += gridDim.x * 256) {
    const int y = id & (M - 1), zz = id / M;
    const double2 a = sp[(size_t)id * H];
    const double2 c = sp[((size_t)((M - zz) & (M - 1)) * M + ((M - y) & (M - 1))) * H];
    const double f0 = 0.25 * ((a.x + c.x) * (a.x + c.x) + (a.y - c.y) * (a.y - c.y));
    const double fn = 0.25 * ((a.x - c.x) * (a.x - c.x) + (a.y + c.y) * (a.y + c.y));
    const int ky = y <= H ? y : y - M, kz = zz <= H ? zz : zz - M;
    const long long yz = (long long)ky * ky + (long long)kz * kz;
    const int b0 = shell_of(yz), bn = shell_of(yz + (long long)H * H);
    if (b0 < nb) atomicAdd(&bins[b0], norm * f0);
    if (bn < nb) atomicAdd(&bins[bn], norm * fn);
  }
}

}  // namespace

cudaError_t density_pdf(int k, const double* y, int n, int sub, double lo, double hi, int nb,
                        unsigned long long* counts_dev, long long* counts_host, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(counts_dev, 0, sizeof(unsigned long long) * (nb + 2), s);
  if (e != cudaSuccess) return e;
  const long long items = (long long)n * n * n * sub;
  const unsigned grid = (unsigned)((items + 255) / 256 < 152 * 16 ? (items + 255) / 256 : 152 * 16);
  density_hist_kernel<<<grid, 256, sizeof(unsigned int) * (nb + 2), s>>>(y, k, n, sub, lo, hi, nb, counts_dev);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  e = cudaMemcpyAsync(counts_host, counts_dev, sizeof(unsigned long long) * (nb + 2), cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) return e;
  return cudaStreamSynchronize(s);
}

int n_bins(int M) { return (int)std::floor(std::sqrt(3.0) * M / 2.0) + 2; }

void release(PlanCache* cache) {
  if (cache->M) cufftDestroy((cufftHandle)cache->handle);
  cache->M = 0;
  cache->ws = 0;
}

// the cached plan for M points per axis, made if the cache holds another
// size or none
static cufftResult cached_plan(int M, PlanCache* cache) {
  if (cache->M == M) return CUFFT_SUCCESS;
  release(cache);
  cufftHandle plan;
  size_t ws = 0;
  const cufftResult r = make_plan(M, &plan, &ws);
  if (r != CUFFT_SUCCESS) return r;
  cache->handle = (int)plan;
  cache->M = M;
  cache->ws = ws;
  return CUFFT_SUCCESS;
}

// work area: bins, twiddles, one real grid, one complex half spectrum and, for
// the sizes that take cuFFT, its work area
struct Work {
  size_t tw, real, cplx, area, end;
  Work(int M, size_t ws) {
    const size_t M3 = (size_t)M * M * M, half = (size_t)M * M * (M / 2 + 1);
    tw = align256(sizeof(double) * n_bins(M));
    real = tw + (own_fft(M) ? align256(sizeof(longlong2) * M) : 0);
    cplx = real + align256(sizeof(double) * M3);
    area = cplx + align256(sizeof(double2) * half);
    end = area + align256(ws);
  }
};

size_t work_bytes(int M, PlanCache* cache) {
  if (own_fft(M)) return Work(M, 0).end;
  if (cached_plan(M, cache) != CUFFT_SUCCESS) return 0;
  return Work(M, cache->ws).end;
}

namespace {
// shell sums of one component's samples by the fixed-point transform
cudaError_t own_spectrum(int M, const double* real, double2* cplx, const longlong2* tw, double* bins, cudaStream_t s) {
  const int nb = n_bins(M), lines = kFftPoints / M, copies = nb * 64 <= 48 * 1024 ? 8 : 1;
  int logm = 0;
  while ((1 << logm) < M) ++logm;
  const size_t rows = sizeof(Cx) * (size_t)lines * (M + 1) + 8 * (size_t)lines;
  const size_t cols = sizeof(Cx) * (size_t)kFftPoints + 8 * (size_t)lines;
  const size_t colz = cols + sizeof(double) * (size_t)nb * copies;
  cudaError_t e = cudaFuncSetAttribute(fft_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rows);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fft_lines_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cols);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fft_lines_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)colz);
  if (e != cudaSuccess) return e;
  const unsigned tiles = (unsigned)((long long)M * M / 2 / lines);
  fft_rows_kernel<<<tiles, 256, rows, s>>>(real, cplx, M, logm, tw);
  fft_lines_kernel<false><<<tiles, 256, cols, s>>>(cplx, M, logm, tw, nb, 1, nullptr);
  // persistent: a CTA's bins take many tiles before they go out
  fft_lines_kernel<true><<<tiles < 152u * 2 ? tiles : 152u * 2, 256, colz, s>>>(cplx, M, logm, tw, nb, copies, bins);
  fft_packed_bins_kernel<<<(unsigned)(((long long)M * M + 255) / 256), 256, 0, s>>>(cplx, M, nb, bins);
  return cudaGetLastError();
}
}  // namespace

cudaError_t velocity_spectrum(int k, const double* y, int n, int sub, void* work, size_t bytes, double* bins_out,
                              cudaStream_t s, int* cufft_status, PlanCache* cache) {
  *cufft_status = 0;
  const int M = n * sub, nb = n_bins(M);
  const bool own = own_fft(M);
  cufftResult r = own ? CUFFT_SUCCESS : cached_plan(M, cache);
  if (r != CUFFT_SUCCESS) {
    *cufft_status = (int)r;
    return cudaSuccess;
  }
  const Work w(M, own ? 0 : cache->ws);
  if ((own ? w.end : w.area + cache->ws) > bytes) {
    *cufft_status = -1;
    return cudaSuccess;
  }
  unsigned char* p = static_cast<unsigned char*>(work);
  double* bins = reinterpret_cast<double*>(p);
  longlong2* tw = reinterpret_cast<longlong2*>(p + w.tw);
  double* real = reinterpret_cast<double*>(p + w.real);
  double2* cplx = reinterpret_cast<double2*>(p + w.cplx);
  const cufftHandle plan = (cufftHandle)cache->handle;
  cudaError_t e = cudaSuccess;
  if (!own && (r = cufftSetWorkArea(plan, p + w.area)) == CUFFT_SUCCESS) r = cufftSetStream(plan, s);
  if (r == CUFFT_SUCCESS) e = cudaMemsetAsync(bins, 0, sizeof(double) * nb, s);
  if (own && e == cudaSuccess) {
    twiddle_kernel<<<(M + 255) / 256, 256, 0, s>>>(M, tw);
    e = cudaGetLastError();
  }
  // a copy of the bins per warp while the eight fit 48 KB
  const int copies = (size_t)nb * sizeof(double) * 8 <= 48 * 1024 ? 8 : 1;
  const long long items = (long long)n * n * n * sub;
  const unsigned grid = (unsigned)((items + 255) / 256 < 152 * 16 ? (items + 255) / 256 : 152 * 16);
  for (int comp = 0; comp < 3 && r == CUFFT_SUCCESS && e == cudaSuccess; ++comp) {
    sample_kernel<<<grid, 256, 0, s>>>(y, k, n, sub, comp, real);
    if ((e = cudaGetLastError()) != cudaSuccess) break;
    if (own) {
      e = own_spectrum(M, real, cplx, tw, bins, s);
      continue;
    }
    if ((r = cufftExecD2Z(plan, real, reinterpret_cast<cufftDoubleComplex*>(cplx))) != CUFFT_SUCCESS) break;
    bin_kernel<<<152 * 4, 256, sizeof(double) * nb * copies, s>>>(cplx, M, nb, bins, copies);
    e = cudaGetLastError();
  }
  if (r == CUFFT_SUCCESS && e == cudaSuccess)
    e = cudaMemcpyAsync(bins_out, bins, sizeof(double) * nb, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (r != CUFFT_SUCCESS) *cufft_status = (int)r;
  return e;
}

}  // namespace spec
}  // namespace dg
