// launch_driver.cpp -- runs the library's kernels under the host emulation on
// the routes and with the sizes that its launchers use now: driver.cpp's set-up
// with commands of its own (test infrastructure).
//
//   launch_driver queue nx ny nz gamma eps_rho eps_p lim_vol in.bin queued.bin plain.bin
//       every cell through the queued limiter's two kernels (queued.bin) and
//       through limit_cell (plain.bin), with the second pass's own shared memory
//   launch_driver limit nx ny nz gamma eps_rho eps_p lim_vol in.bin out.bin
//       limit_kernel (dg_limit), FP32 point screen included
//   launch_driver rhs nx ny nz prec gamma lx ly lz in.bin out.bin n_modes modes.bin seg
//       R(y) in a box of lengths lx, ly, lz: FP64 the fixed-point kernels from
//       degree 1 on, mixed the fused kernel from degree 1 on with seg planes per
//       segment
//   launch_driver step nx ny nz prec gamma eps_rho eps_p lim_vol in.bin out.bin dt n_modes modes.bin c_iso rho0 seg
//       one dg_step in the unit box, then (c_iso > 0) dg_energy_reset. The queue's
//       counter is as the kernels leave it; before the unfused stages, whose face
//       kernels clear it, it starts with another value
//
//   launch_driver fft M in.bin out.bin
//       shell sums of the M^3 real samples in in.bin by the library's own transform
//       (M = 32 .. 1024 a power of two)
//
// States in the state layout [5][N][n_cells], FP64. Prints "err=<device error
// word>" and what else a command says.
#include <type_traits>
#include "dg_kernels.cuh"
#include "dg_fused.cuh"
#define main driver_main
#include "driver.cpp"
#undef main
struct longlong2 {
  long long x, y;
};
inline void sincospi(double x, double* s, double* c) {
  *s = (double)sinl(3.14159265358979323846264338327950288L * x);
  *c = (double)cosl(3.14159265358979323846264338327950288L * x);
}
namespace dg {
namespace spec {
#include "fft_kernels.inc"
}  // namespace spec
}  // namespace dg

// the launcher's grid of a kernel over a queue (limit_grid)
static unsigned queue_grid(long long nc, int per, unsigned most) {
  return (unsigned)std::min<long long>((nc + per - 1) / per, most);
}

static bool write_file(const char* path, const double* p, size_t n) {
  FILE* f = std::fopen(path, "wb");
  if (!f) return false;
  const bool ok = std::fwrite(p, 8, n, f) == n;
  std::fclose(f);
  return ok;
}

// the queued limiter as limit_list launches it: n_deep is 0 on entry, the
// second pass gets its own, smaller shared memory
static void limit_launch(Setup& S, double* y, const int* list, int count_queued, float* yf, const double* y0,
                         float* dinc, std::vector<int>& deep) {
  using LL = ListLim<K>;
  emu::launch(queue_grid(S.nc, LL::THREADS, 152 * LL::MINB), LL::THREADS, LL::smem(), [&] {
    limit_screen_list_kernel<K>(y, list, &S.ctrl.n_flag, S.t64.data(), S.t32.data(), S.g, &S.ctrl, count_queued,
                                deep.data());
  });
  emu::launch(queue_grid(S.nc, LL::THREADS / 32, 152 * 4), LL::THREADS, LL::smem_deep(), [&] {
    limit_list_kernel<K>(y, deep.data(), &S.ctrl.n_deep, S.t64.data(), S.g, &S.ctrl, yf, y0, dinc);
  });
}

static int run_queue(int argc, char** argv) {
  if (argc != 12) return 2;
  Setup S;
  make_setup(S, std::atoi(argv[2]), std::atoi(argv[3]), std::atoi(argv[4]), std::atof(argv[5]), std::atoi(argv[8]));
  S.g.eps_rho = std::atof(argv[6]);
  S.g.eps_p = std::atof(argv[7]);
  std::vector<double> y((size_t)5 * TB::N * S.nc);
  if (!read_file(argv[9], y.data(), y.size())) return 3;
  std::vector<double> plain(y);
  std::vector<int> list(S.nc), deep(S.nc, -1);
  for (int c = 0; c < (int)S.nc; ++c) list[c] = c;
  S.ctrl.n_flag = (unsigned)S.nc;
  limit_launch(S, y.data(), list.data(), 1, nullptr, nullptr, nullptr, deep);
  unsigned err = 0;
  for (long long c = 0; c < S.nc; ++c)
    limit_cell<K>(plain.data() + c, S.nc, S.t64.data(), S.g.gamma, S.g.eps_rho, S.g.eps_p, &err, S.g.lim_vol);
  if (!write_file(argv[10], y.data(), y.size()) || !write_file(argv[11], plain.data(), plain.size())) return 3;
  std::printf("err=%u plain_err=%u deep=%u n_flag=%u\n", S.ctrl.err, err, S.ctrl.n_deep, S.ctrl.n_flag);
  return 0;
}

static int run_limit(int argc, char** argv) {
  if (argc != 11) return 2;
  Setup S;
  make_setup(S, std::atoi(argv[2]), std::atoi(argv[3]), std::atoi(argv[4]), std::atof(argv[5]), std::atoi(argv[8]));
  S.g.eps_rho = std::atof(argv[6]);
  S.g.eps_p = std::atof(argv[7]);
  std::vector<double> y((size_t)5 * TB::N * S.nc);
  if (!read_file(argv[9], y.data(), y.size())) return 3;
  emu::launch(grid1(S.nc, kThreads), kThreads, 0,
              [&] { limit_kernel<K>(y.data(), nullptr, S.t64.data(), S.g, &S.ctrl, S.t32.data()); });
  if (!write_file(argv[10], y.data(), y.size())) return 3;
  std::printf("err=%u n_limited=%llu\n", S.ctrl.err, (unsigned long long)S.ctrl.n_limited);
  return 0;
}

#if DG_K >= 1
// driver.cpp has these from degree 2 on
static void launch_fused_setup(const Setup& S) {
  using FT = FzTab<K>;
  constexpr int KQ = (K + 1) * (K + 1);
  for (int j = 0; j < KQ; ++j) {
    c_fz[FT::P + j] = (float)S.t64[TB::P1 + j];
    c_fz[FT::PW + j] = (float)S.t64[TB::P1W + j];
    c_fz[FT::DW + j] = (float)S.t64[TB::D1W + j];
  }
  for (int e = 0; e <= K; ++e) {
    c_fz[FT::EM + e] = (float)S.t64[TB::FEND + e];
    c_fz[FT::EP + e] = (float)S.t64[TB::FEND + K + 1 + e];
  }
  for (int l = 0; l < TB::N; ++l) {
    c_fz[FT::LM + l] = (float)S.t64[TB::LMAX + l];
    c_fz[FT::LMV + l] = (float)S.t64[TB::LMAXV + l];
  }
}

static void launch_fused(Setup& S, FusedArgs a, bool force, int seg) {
  using FC = FusedCfg<K>;
  a.nbx = (S.g.nx + FC::BX - 1) / FC::BX;
  a.nby = (S.g.ny + FC::BY - 1) / FC::BY;
  a.lz = seg;
  a.eps_r = (float)S.g.eps_rho;
  a.eps_p = (float)S.g.eps_p;
  a.ctrl = &S.ctrl;
  const unsigned grid = (unsigned)(a.nbx * a.nby * ((S.g.nz + seg - 1) / seg));
  if (force) emu::launch(grid, FC::THREADS, FC::smem(), [&] { fused_f32_kernel<K, true, 0>(S.g, a); });
  else emu::launch(grid, FC::THREADS, FC::smem(), [&] { fused_f32_kernel<K, false, 0>(S.g, a); });
}
#endif

template <typename T>
static void launch_faces(Setup& S, const double* ys, float* yf, T* fh) {
  if constexpr (sizeof(T) == 4) {
    emu::launch(grid1(S.nc, 32), 96, 0, [&] { face_flux_f32_kernel<K, 0>(yf, fh, S.g, &S.ctrl); });
  } else {
    const unsigned tiles = grid1(S.nc, 32);
    emu::launch2(tiles, tiles * 2 < 152u * FaceSF64<K>::MINB ? 3 : 1, FaceSF64<K>::THREADS, FaceSF64<K>::smem(),
                 [&] { face_sf64_kernel<K, 0, (K >= 1)>(ys, fh, S.g, &S.ctrl); });
  }
}

template <typename T, int MODE, bool FORCE>
static void launch_volume(Setup& S, const double* ys, float* yf, const T* fh, const T* field, StageArgs st, double* R) {
  if constexpr (sizeof(T) == 8 && K >= 1) {
    using CF = VolSF<K, double>;
    emu::launch(grid1(S.nc, CF::C), kThreads, CF::smem(), [&] {
      volume_sf_kernel<K, double, MODE, FORCE>(ys, nullptr, fh, field, S.t64.data(), S.t64.data(), S.g, st, R,
                                               &S.ctrl);
    });
  } else {
    volume<T, MODE, FORCE>(S, ys, yf, fh, field, st, R);
  }
}

template <typename T>
static std::vector<T> driving(Setup& S, const std::vector<double>& modes, int nm, const double* L) {
  std::vector<T> field(nm > 0 ? (size_t)3 * TB::Q3 * S.nc : 1, T(std::nan("")));
  if (nm > 0)
    emu::launch2(grid1(S.nc, kThreads), TB::Q3, kThreads, 0, [&] {
      forcing_field_kernel<K, T>(field.data(), modes.data(), nm, S.t64.data(), S.g, L[0], L[1], L[2]);
    });
  return field;
}

template <typename T>
static void rhs_launch(Setup& S, std::vector<double>& y, std::vector<double>& R, const std::vector<double>& modes,
                       int nm, const double* L, int seg) {
  std::vector<T> field = driving<T>(S, modes, nm, L);
#if DG_K >= 1
  if constexpr (sizeof(T) == 4) {
    launch_fused_setup(S);
    FusedArgs a{};
    a.ys = y.data();
    a.R = R.data();
    a.field = field.data();
    launch_fused(S, a, nm > 0, seg);
    return;
  }
#endif
  std::vector<float> yf(sizeof(T) == 4 ? y.size() : 1);
  if (sizeof(T) == 4)
    for (size_t i = 0; i < y.size(); ++i) yf[i] = (float)y[i];
  std::vector<T> fh((size_t)15 * TB::Q2 * S.nc, T(std::nan("")));
  launch_faces<T>(S, y.data(), yf.data(), fh.data());
  if (nm > 0) launch_volume<T, MODE_RHS, true>(S, y.data(), yf.data(), fh.data(), field.data(), StageArgs{}, R.data());
  else launch_volume<T, MODE_RHS, false>(S, y.data(), yf.data(), fh.data(), nullptr, StageArgs{}, R.data());
}

static int run_rhs_launch(int argc, char** argv) {
  if (argc != 15) return 2;
  Setup S;
  make_setup(S, std::atoi(argv[2]), std::atoi(argv[3]), std::atoi(argv[4]), std::atof(argv[6]), 0);
  const double L[3] = {std::atof(argv[7]), std::atof(argv[8]), std::atof(argv[9])};
  const int n3[3] = {S.g.nx, S.g.ny, S.g.nz}, nm = std::atoi(argv[12]), seg = std::atoi(argv[14]);
  for (int a = 0; a < 3; ++a) {
    S.g.dx[a] = L[a] / n3[a];
    S.g.inv_dx[a] = 1.0 / S.g.dx[a];
  }
  std::vector<double> y((size_t)5 * TB::N * S.nc), R(y.size(), std::nan("")), modes((size_t)9 * nm + 1);
  if (!read_file(argv[10], y.data(), y.size())) return 3;
  if (nm > 0 && !read_file(argv[13], modes.data(), (size_t)9 * nm)) return 3;
  if (std::atoi(argv[5])) rhs_launch<float>(S, y, R, modes, nm, L, seg);
  else rhs_launch<double>(S, y, R, modes, nm, L, seg);
  if (!write_file(argv[11], R.data(), R.size())) return 3;
  std::printf("err=%u\n", S.ctrl.err);
  return 0;
}

template <typename T>
static void step_launch(Setup& S, std::vector<double>& y, double dt, const std::vector<double>& modes, int nm,
                        double c_iso, double rho0, int seg) {
  const long long nc = S.nc;
  const double L[3] = {1.0, 1.0, 1.0};
  const bool force = nm > 0, shadow = sizeof(T) == 4;
  std::vector<T> field = driving<T>(S, modes, nm, L);
  emu::launch(grid1(nc, kThreads), kThreads, 0,
              [&] { limit_kernel<K>(y.data(), nullptr, S.t64.data(), S.g, &S.ctrl, S.t32.data()); });
  std::vector<float> yf(shadow ? y.size() : 1);
  if (shadow)
    for (size_t i = 0; i < y.size(); ++i) yf[i] = (float)y[i];
  float* yfp = shadow ? yf.data() : nullptr;
  std::vector<T> fh((size_t)15 * TB::Q2 * nc, T(std::nan("")));
  std::vector<double> ybuf(y.size(), std::nan("")), ybuf2(y.size(), std::nan(""));
  std::vector<float> dinc(y.size(), std::nanf(""));
  std::vector<int> list(nc, -1), deep(nc, -1);
  const double a0[3] = {0.0, 0.75, 1.0 / 3.0}, b0[3] = {1.0, 0.25, 2.0 / 3.0};
  const double* ys = y.data();
  S.ctrl.n_flag = sizeof(T) == 4 && K >= 1 ? 0 : 3;
  for (int s = 0; s < 3; ++s) {
#if DG_K >= 1
    if constexpr (sizeof(T) == 4) {
      launch_fused_setup(S);
      double* out = s == 0 ? ybuf.data() : (s == 1 ? ybuf2.data() : y.data());
      FusedArgs a{};
      a.ys = ys;
      a.out = out;
      a.d = dinc.data();
      a.yf = s == 2 ? yfp : nullptr;
      a.field = field.data();
      a.list = list.data();
      a.b0dt = (float)(b0[s] * dt);
      a.a0 = (float)a0[s];
      a.b0dt_d = b0[s] * dt;
      a.a0_d = a0[s];
      a.b0_d = b0[s];
      a.y0 = y.data();
      a.stage = s + 1;
      launch_fused(S, a, force, seg);
      limit_launch(S, out, list.data(), 1, s == 2 ? yfp : nullptr, s < 2 ? y.data() : nullptr,
                   s < 2 ? dinc.data() : nullptr, deep);
      ys = out;
      continue;
    }
#endif
    double* out = s < 2 ? ybuf.data() : y.data();
    launch_faces<T>(S, ys, yfp, fh.data());
    StageArgs st{ys, y.data(), out, a0[s], b0[s], dt, list.data(), yfp};
    if (force) launch_volume<T, MODE_STAGE, true>(S, ys, yfp, fh.data(), field.data(), st, nullptr);
    else launch_volume<T, MODE_STAGE, false>(S, ys, yfp, fh.data(), nullptr, st, nullptr);
    limit_launch(S, out, list.data(), 1, yfp, nullptr, nullptr, deep);
    ys = out;
  }
  double diss = 0.0;
  if (c_iso > 0.0) {
    const unsigned nbr = grid1(nc, 32);
    std::vector<double> part(nbr, 0.0);
    ResetConsts<T> rc;
    rc.c2g = (T)(c_iso * c_iso / (S.g.gamma - 1.0));
    rc.inv_rho0 = (T)(1.0 / rho0);
    rc.gm1 = (T)(S.g.gamma - 1.0);
    rc.two_thirds = std::fabs(S.g.gamma - 1.0 - 2.0 / 3.0) < 1e-15 ? 1 : 0;
    const T* tabT = sizeof(T) == 8 ? (const T*)(const void*)S.t64.data() : (const T*)(const void*)S.t32.data();
    emu::launch(nbr, ResetSF<K, T>::THREADS, ResetSF<K, T>::smem(), [&] {
      energy_reset_sf_kernel<K, T>(y.data(), tabT, S.g, rc, part.data(), list.data(), &S.ctrl, yfp);
    });
    limit_launch(S, y.data(), list.data(), 0, yfp, nullptr, nullptr, deep);
    for (unsigned b = 0; b < nbr; ++b) diss += part[b];
    diss *= S.g.dx[0] * S.g.dx[1] * S.g.dx[2];
  }
  std::printf("err=%u dissipated=%.17g n_flag=%u queued=%llu full=%llu\n", S.ctrl.err, diss, S.ctrl.n_flag,
              (unsigned long long)S.ctrl.n_queued_total, (unsigned long long)S.ctrl.n_full_total);
}

static int run_step_launch(int argc, char** argv) {
  if (argc != 18) return 2;
  Setup S;
  make_setup(S, std::atoi(argv[2]), std::atoi(argv[3]), std::atoi(argv[4]), std::atof(argv[6]), std::atoi(argv[9]));
  S.g.eps_rho = std::atof(argv[7]);
  S.g.eps_p = std::atof(argv[8]);
  const int nm = std::atoi(argv[13]), seg = std::atoi(argv[17]);
  std::vector<double> y((size_t)5 * TB::N * S.nc), modes((size_t)9 * nm + 1);
  if (!read_file(argv[10], y.data(), y.size())) return 3;
  if (nm > 0 && !read_file(argv[14], modes.data(), (size_t)9 * nm)) return 3;
  const double dt = std::atof(argv[12]), c_iso = std::atof(argv[15]), rho0 = std::atof(argv[16]);
  if (std::atoi(argv[5])) step_launch<float>(S, y, dt, modes, nm, c_iso, rho0, seg);
  else step_launch<double>(S, y, dt, modes, nm, c_iso, rho0, seg);
  return write_file(argv[11], y.data(), y.size()) ? 0 : 3;
}

static int run_fft(int argc, char** argv) {
  if (argc != 5) return 2;
  using namespace spec;
  const int M = std::atoi(argv[2]);
  if (!own_fft(M)) return 2;
  // sizes and launches of own_spectrum
  const int nb = (int)std::floor(std::sqrt(3.0) * M / 2.0) + 2, lines = kFftPoints / M;
  const int copies = nb * 64 <= 48 * 1024 ? 8 : 1;
  int logm = 0;
  while ((1 << logm) < M) ++logm;
  const size_t rows = sizeof(Cx) * (size_t)lines * (M + 1) + 8 * (size_t)lines;
  const size_t cols = sizeof(Cx) * (size_t)kFftPoints + 8 * (size_t)lines;
  const size_t colz = cols + sizeof(double) * (size_t)nb * copies;
  std::vector<double> real((size_t)M * M * M), bins(nb, 0.0);
  if (!read_file(argv[3], real.data(), real.size())) return 3;
  std::vector<double2> cplx((size_t)M * M * (M / 2), double2{std::nan(""), std::nan("")});
  std::vector<longlong2> tw(M);
  const unsigned tiles = (unsigned)((long long)M * M / 2 / lines);
  emu::launch((M + 255) / 256, 256, 0, [&] { twiddle_kernel(M, tw.data()); });
  emu::launch(tiles, 256, rows, [&] { fft_rows_kernel(real.data(), cplx.data(), M, logm, tw.data()); });
  emu::launch(tiles, 256, cols, [&] { fft_lines_kernel<false>(cplx.data(), M, logm, tw.data(), nb, 1, nullptr); });
  emu::launch(std::min(tiles, 152u * 2), 256, colz,
              [&] { fft_lines_kernel<true>(cplx.data(), M, logm, tw.data(), nb, copies, bins.data()); });
  emu::launch((unsigned)(((long long)M * M + 255) / 256), 256, 0,
              [&] { fft_packed_bins_kernel(cplx.data(), M, nb, bins.data()); });
  if (!write_file(argv[4], bins.data(), bins.size())) return 3;
  std::printf("bins=%d\n", nb);
  return 0;
}

int main(int argc, char** argv) {
  if (argc < 2) return 2;
  if (std::strcmp(argv[1], "fft") == 0) return run_fft(argc, argv);
  if (std::strcmp(argv[1], "queue") == 0) return run_queue(argc, argv);
  if (std::strcmp(argv[1], "limit") == 0) return run_limit(argc, argv);
  if (std::strcmp(argv[1], "rhs") == 0) return run_rhs_launch(argc, argv);
  if (std::strcmp(argv[1], "step") == 0) return run_step_launch(argc, argv);
  return 2;
}
