// The MLP's host code (paper_2311_12180_gb300/csrc/pdlp_mlp.cu) on the stand-in
// of tests/cuda_runtime_host.cpp, used by tests/test_solver_host.py: a network
// whose predictions can exceed 8 MB; prints each call's result, the page-locked
// allocations and streams made so far, and whether exactly the prediction was
// written.
#include <cstdio>
#include <sys/mman.h>

#include <cstdlib>
#include <cstring>
#include <vector>

#include "pdlp.h"

extern int n_pinned, n_streams, fail_pinned, device_fill;
extern const void *page_locked;

static int in_flight = 0, most_in_flight = 0;
namespace pdlp {
void count_in_flight(int, int by, bool) {
  in_flight += by;
  if (in_flight > most_in_flight) most_in_flight = in_flight;
}
int set_error(int code, const char *msg) {
  std::printf("error %d %s\n", code, msg);
  return code;
}
}  // namespace pdlp

int main(int argc, char **argv) {
  fail_pinned = argc > 1 && std::atoi(argv[1]);
  device_fill = 0x3c;
  const int in = 2, hid = 8, out = 40001, batch = 64;
  const size_t guard = 1000;  // 10.2 MB a batch
  pdlp_mlp *net = nullptr;
  int written = 1;
  auto show = [&](const char *what, int rc) {
    std::printf("%s %d pinned %d streams %d written %d in_flight %d left %d\n", what, rc, n_pinned, n_streams, written,
                most_in_flight, in_flight);
    most_in_flight = 0;
  };
  show("create", pdlp_mlp_create(&net, in, hid, out, batch, nullptr));
  std::vector<float> X(300 * in, 1.0f);
  // into memory whose pages are not there, are, or are page-locked
  enum Where { FRESH, WRITTEN, LOCKED };
  auto predict = [&](const char *what, int count, Where where) {
    const size_t n = (size_t)count * out, all = sizeof(float) * (guard + n + guard);
    float *Y = (float *)mmap(nullptr, all, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
    if (where != FRESH) std::memset(Y, 0, all);
    page_locked = where == LOCKED ? Y + guard : nullptr;
    const int rc = pdlp_mlp_predict(net, count, X.data(), Y + guard);
    written = 1;
    float want;  // no kernel runs: the prediction is what new device memory holds
    std::memset(&want, device_fill, sizeof(want));
    for (size_t i = 0; i < guard + n + guard; ++i)
      if (Y[i] != (i >= guard && i < guard + n ? want : 0.0f)) written = 0;
    munmap(Y, all);
    show(what, rc);
  };
  predict("small", 20, FRESH);
  predict("locked", 64, LOCKED);
  predict("written", 150, WRITTEN);
  predict("first", 64, FRESH);
  predict("second", 64, FRESH);
  predict("batches", 150, FRESH);  // two staged ones and a small rest
  pdlp_mlp_destroy(net);
  // 36.8 MB a prediction: the first one pays
  show("big", pdlp_mlp_create(&net, in, hid, out, 256, nullptr));
  predict("written", 230, WRITTEN);
  predict("once", 230, FRESH);
  pdlp_mlp_destroy(net);
  return 0;
}
