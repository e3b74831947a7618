// The MLP's host code (paper_2311_12180_gb300/csrc/pdlp_mlp.cu) on the stand-in
// of tests/cuda_runtime_host.cpp, used by tests/test_solver_host.py: a network
// whose predictions can exceed 8 MB; prints each call's result, the page-locked
// allocations and streams made so far, and whether exactly the prediction was
// written.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "pdlp.h"

extern int n_pinned, n_streams, fail_pinned;
extern const void *page_locked;

namespace pdlp {
int set_error(int code, const char *msg) {
  std::printf("error %d %s\n", code, msg);
  return code;
}
}  // namespace pdlp

int main(int argc, char **argv) {
  fail_pinned = argc > 1 && std::atoi(argv[1]);
  const int in = 2, hid = 8, out = 40001, batch = 64, guard = 1000;  // 10.2 MB a batch
  pdlp_mlp *net = nullptr;
  int written = 1;
  auto show = [&](const char *what, int rc) {
    std::printf("%s %d pinned %d streams %d written %d\n", what, rc, n_pinned, n_streams, written);
  };
  show("create", pdlp_mlp_create(&net, in, hid, out, batch, nullptr));
  std::vector<float> X(300 * in, 1.0f);
  auto predict = [&](const char *what, int count, bool locked) {
    std::vector<float> Y(guard + (size_t)count * out + guard, 7.0f);
    page_locked = locked ? Y.data() + guard : nullptr;
    const int rc = pdlp_mlp_predict(net, count, X.data(), Y.data() + guard);
    written = 1;
    for (size_t i = 0; i < Y.size(); ++i)  // no kernel runs: the prediction is zeros
      if ((Y[i] == 0.0f) != (i >= guard && i < guard + (size_t)count * out)) written = 0;
    show(what, rc);
  };
  predict("small", 20, false);
  predict("locked", 64, true);
  predict("first", 64, false);
  predict("second", 64, false);
  predict("batches", 150, false);  // two staged ones and a small rest
  pdlp_mlp_destroy(net);
  // 36.8 MB a prediction: the first one pays
  show("big", pdlp_mlp_create(&net, in, hid, out, 256, nullptr));
  predict("once", 230, false);
  pdlp_mlp_destroy(net);
  return 0;
}
