// launch_driver.cpp -- runs the library's kernels under the host emulation on
// the routes and with the sizes that its launchers use now: driver.cpp's set-up
// with commands of its own (test infrastructure).
//
//   launch_driver queue nx ny nz gamma eps_rho eps_p lim_vol in.bin queued.bin plain.bin
//       every cell through the queued limiter's two kernels (queued.bin) and
//       through limit_cell (plain.bin), with the second pass's own shared memory
//
// States in the state layout [5][N][n_cells], FP64. Prints "err=<device error
// word>" and what else a command says.
#include <type_traits>
#include "dg_kernels.cuh"
#include "dg_fused.cuh"
#define main driver_main
#include "driver.cpp"
#undef main

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

int main(int argc, char** argv) {
  if (argc >= 2 && std::strcmp(argv[1], "queue") == 0) return run_queue(argc, argv);
  return 2;
}
