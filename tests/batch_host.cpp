// The batched solver's host driver (paper_2311_12180_gb300/csrc/pdlp_batch.cu)
// on the stand-in of tests/cuda_runtime_host.cpp, used by
// tests/test_solver_host.py: argv = resident CTAs, small LPs, large LPs; prints
// what the calls returned and the grids launched.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "pdlp.h"
#include "pdlp_internal.cuh"
#include "pdlp_setup.cuh"

extern int resident_ctas, last_grid;

static int in_flight = 0, most_in_flight = 0;
namespace pdlp {
void count_in_flight(int, int by, bool) {
  in_flight += by;
  if (in_flight > most_in_flight) most_in_flight = in_flight;
}
cudaError_t setup_pow_table(double *, long long, cudaStream_t) { return cudaSuccess; }
int set_error(int code, const char *msg) {
  std::printf("error %d %s\n", code, msg);
  return code;
}
}  // namespace pdlp
extern "C" void pdlp_default_params(pdlp_params *p) {
  *p = pdlp_params{};
  p->check_period = 64;
  p->value_bits = 64;
}

int main(int argc, char **argv) {
  if (argc != 4) return 2;
  resident_ctas = std::atoi(argv[1]);
  const int small = std::atoi(argv[2]), large = std::atoi(argv[3]), rows = 256;
  // a row of one entry, or 256 rows of 256
  std::vector<int32_t> p1{0, 1}, p2(rows + 1), i1{0}, i2;
  for (int r = 0; r <= rows; ++r) p2[r] = r * rows;
  for (int k = 0; k < rows * rows; ++k) i2.push_back(k % rows);
  std::vector<double> ones(rows * rows, 1.0), zeros(rows, 0.0);
  std::vector<pdlp_lp> lps;
  for (int k = 0; k < small + large; ++k) {
    pdlp_lp l{};
    l.m = l.n = l.n_eq = k < small ? 1 : rows;
    l.row_ptr = k < small ? p1.data() : p2.data();
    l.col_idx = k < small ? i1.data() : i2.data();
    l.c = l.q = l.u = l.val = ones.data();
    l.l = zeros.data();
    lps.push_back(l);
  }
  pdlp_batch *b = nullptr;
  std::printf("create %d", pdlp_batch_create(&b, small + large, lps.data(), nullptr, nullptr));
  std::printf(" grid %d in_flight %d left %d\n", last_grid, most_in_flight, in_flight);
  most_in_flight = 0;
  std::printf("solve %d", pdlp_batch_solve(b, nullptr, nullptr, 1e-6, 100, nullptr, nullptr, nullptr, nullptr));
  std::printf(" grid %d in_flight %d left %d\n", last_grid, most_in_flight, in_flight);
  pdlp_batch_destroy(b);
  return 0;
}
