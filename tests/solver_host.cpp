// The solver's host driver (paper_2311_12180_gb300/csrc/pdlp_capi.cu) on a
// stand-in for the CUDA runtime (tests/cuda_runtime_host.cpp) and one for the
// kernels' launchers: launches are counted, and a chosen call returns a chosen
// error.  Used by tests/test_solver_host.py: argv[1] names a scenario, which prints what the
// calls returned.
#include <cuda_runtime.h>

#include <cstdio>
#include <string>

#include "pdlp.h"
#include "pdlp_internal.cuh"
#include "pdlp_setup.cuh"

extern int fail_capture, capturing, n_graph, stream_captured;     // of the runtime's stand-in
static int plan_ctas = 0;                        // what period_plan decides
static bool plan_cluster = false;
static cudaError_t period_error = cudaSuccess;   // of launch_period
static int n_period = 0, n_check = 0, n_step = 0;  // launches

namespace pdlp {
static cudaError_t counted(int &n) {
  n += !capturing;
  return cudaSuccess;
}
cudaError_t launch_primal(const SellMat &, const Vecs &, DevState *, int, cudaStream_t) { return counted(n_step); }
cudaError_t launch_dual(const SellMat &, const Vecs &, DevState *, int, cudaStream_t) { return counted(n_step); }
cudaError_t launch_check_primal(const SellMat &, const Vecs &, DevState *, int, cudaStream_t) { return counted(n_check); }
cudaError_t launch_check_dual(const SellMat &, const Vecs &, DevState *, int, cudaStream_t) { return counted(n_check); }
cudaError_t launch_restart(const Vecs &, DevState *, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_infeas(const Vecs &, DevState *, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_output(const Vecs &, DevState *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_time_limit(DevState *, cudaStream_t) { return cudaSuccess; }
const char *kernel_class_name(int) { return ""; }
int occupancy_grid(int, int sms) { return 4 * sms; }
cudaError_t kernels_init() { return cudaSuccess; }
cudaError_t period_init() { return cudaSuccess; }
void period_plan(PeriodPlan &p, int32_t, int32_t, const int4 *, int, const int4 *, int, int64_t, int, int, cudaStream_t) {
  p.ctas = plan_ctas;
  p.cluster = plan_cluster;
}
cudaError_t launch_period(const PeriodPlan &, const SellMat &, const SellMat &, const Vecs &, DevState *, int, cudaStream_t) {
  n_period += period_error == cudaSuccess;
  return period_error;
}
cudaError_t setup_pow_table(double *, long long, cudaStream_t) { return cudaSuccess; }
cudaError_t setup_col_starts(int32_t, int64_t, const int32_t *, int32_t *, int32_t *, cudaStream_t) { return cudaSuccess; }
size_t col_starts_work_ints(int32_t n) { return n + 16; }
cudaError_t setup_transpose(int32_t, int32_t, int64_t, const int32_t *, const int32_t *, const double *, const int32_t *,
                            int32_t *, double *, int32_t *, cudaStream_t) { return cudaSuccess; }
size_t transpose_work_ints(int32_t n, int64_t nnz) { return n + 4 * nnz; }
int transpose_max_segment() { return 4096; }
cudaError_t setup_scale(int32_t, int32_t, int64_t, int32_t *, int32_t *, double *, int32_t *, int32_t *, double *, double *,
                        double *, const ScaleWork &, int, double, cudaStream_t) { return cudaSuccess; }
cudaError_t setup_scale_perm(int32_t, int32_t, int64_t, const int32_t *, const int32_t *, double *, const int32_t *, double *,
                             const int32_t *, const int32_t *, double *, double *, double *, double *, double *, double *,
                             int32_t *, int32_t *, int, double, cudaStream_t) { return cudaSuccess; }
cudaError_t setup_vectors(int32_t, int32_t, const double *, const double *, const double *, const double *, const double *,
                          const double *, double *, double *, double *, double *, cudaStream_t) { return cudaSuccess; }
cudaError_t setup_f32(int64_t, const double *, float *, cudaStream_t) { return cudaSuccess; }
cudaError_t setup_recip(int32_t, const double *, double *, cudaStream_t) { return cudaSuccess; }
cudaError_t setup_scalars(int32_t, int32_t, int64_t, const double *, const double *, const double *, double *, double *,
                          cudaStream_t) { return cudaSuccess; }
size_t scalars_work_doubles() { return 16; }
cudaError_t setup_invert(int32_t, const int32_t *, int32_t *, cudaStream_t) { return cudaSuccess; }
cudaError_t setup_sell_fill(int32_t, int64_t, const int32_t *, const int32_t *, const uint8_t *, const int32_t *,
                            const int32_t *, const double *, const int32_t *, int32_t *, double *, cudaStream_t) { return cudaSuccess; }
cudaError_t setup_check_sell(int32_t, int32_t, int64_t, int32_t, const int4 *, const int32_t *, const double *, const float *,
                             unsigned int *c, cudaStream_t) { return c[0] = c[1] = c[2] = 0, cudaSuccess; }
cudaError_t setup_check_entries(int64_t, const int32_t *, const double *, int32_t, int64_t *, int *, cudaStream_t) { return cudaSuccess; }
cudaError_t setup_qp_diag(int32_t, const int32_t *, const double *, const double *, double *, cudaStream_t) { return cudaSuccess; }
cudaError_t setup_permute(int32_t, const int32_t *, const double *, double *, cudaStream_t) { return cudaSuccess; }
cudaError_t setup_warm_perm(int32_t, int32_t, const double *, const double *, const int32_t *, const int32_t *, const double *,
                            const double *, double *, double *, cudaStream_t) { return cudaSuccess; }
}  // namespace pdlp

static pdlp_solver *create() {
  const double c = 1.0, v = 1.0, q = 1.0, l = 0.0, u = 2.0;
  const int32_t rp[2] = {0, 1}, ci = 0;
  pdlp_solver *s = nullptr;
  if (pdlp_create(&s, 1, 1, 1, &c, rp, &ci, &v, &q, &l, &u) != PDLP_OK) std::printf("create: %s\n", pdlp_last_error());
  return s;
}
static void show(const char *what, int rc) {
  std::printf("%s %d graph %d period %d check %d\n", what, rc, n_graph, n_period, n_check);
}

int main(int argc, char **argv) {
  const std::string scenario = argc > 1 ? argv[1] : "";
  if (scenario == "capture") {  // the graph is rebuilt after pdlp_set_quadratic, and that fails
    pdlp_solver *s = create();
    show("quadratic", pdlp_set_quadratic(s, nullptr));
    fail_capture = 1;
    show("begin", pdlp_begin(s, nullptr, nullptr, 1e-6, 100));
    show("run", pdlp_run_periods(s, 2));
    fail_capture = 0;
    show("begin", pdlp_begin(s, nullptr, nullptr, 1e-6, 100));
    show("run", pdlp_run_periods(s, 2));
    pdlp_destroy(s);
    return 0;
  }
  if (scenario == "refused" || scenario == "refused later" || scenario == "broken") {
    // a small LP whose one-launch period does not fit the stream's SMs, from
    // the start or from some launch on; or fails for another reason
    plan_ctas = 152;
    pdlp_solver *s = create();
    if (scenario != "refused later") period_error = scenario == "broken" ? cudaErrorIllegalAddress : cudaErrorCooperativeLaunchTooLarge;
    show("begin", pdlp_begin(s, nullptr, nullptr, 1e-6, 100));
    if (scenario == "refused later") period_error = cudaErrorInvalidClusterSize;
    show("run", pdlp_run_periods(s, 2));
    int st;
    int64_t it;
    double x, y;
    show("finish", pdlp_finish(s, &x, &y, &st, &it));
    pdlp_layout_info info;
    show("layout", pdlp_get_layout(s, &info));
    show("ctas", info.period_ctas);
    pdlp_destroy(s);
    return 0;
  }
  if (scenario == "captured" || scenario == "captured graph") {  // the caller captures the solver's stream
    plan_ctas = scenario == "captured" ? 152 : 0;
    pdlp_solver *s = create();
    show("begin", pdlp_begin(s, nullptr, nullptr, 1e-6, 100));
    stream_captured = 1;
    show("run", pdlp_run_periods(s, 2));
    stream_captured = 0;
    show("run", pdlp_run_periods(s, 2));
    pdlp_destroy(s);
    return 0;
  }
  if (scenario == "several") {  // whole-GPU periods only while a solver is the only one with work in flight
    plan_ctas = 152;
    pdlp_solver *a = create(), *b = create();
    int st;
    int64_t it;
    double x, y;
    show("begin_a", pdlp_begin(a, nullptr, nullptr, 1e-6, 100));
    show("run_a", pdlp_run_periods(a, 1));
    show("begin_b", pdlp_begin(b, nullptr, nullptr, 1e-6, 100));
    show("run_b", pdlp_run_periods(b, 1));
    show("run_a", pdlp_run_periods(a, 1));
    show("finish_a", pdlp_finish(a, &x, &y, &st, &it));
    show("run_b", pdlp_run_periods(b, 1));
    show("poll_b", pdlp_poll(b, &st, &it));
    show("run_a", pdlp_run_periods(a, 1));
    show("run_b", pdlp_run_periods(b, 1));
    pdlp_destroy(a);
    show("run_b", pdlp_run_periods(b, 1));
    show("poll_b", pdlp_poll(b, &st, &it));
    {
      const pdlp::InFlight call(0);  // a network's call under way
      show("run_b", pdlp_run_periods(b, 1));
    }
    show("run_b", pdlp_run_periods(b, 1));
    plan_cluster = true;  // a cluster leaves room: always its own launch
    pdlp_solver *c = create();
    show("begin_c", pdlp_begin(c, nullptr, nullptr, 1e-6, 100));
    show("run_c", pdlp_run_periods(c, 1));
    {
      const pdlp::InFlight batch(0, true);  // but not beside a batch
      show("run_c", pdlp_run_periods(c, 1));
      show("begin_c", pdlp_begin(c, nullptr, nullptr, 1e-6, 100));
    }
    show("run_c", pdlp_run_periods(c, 1));
    pdlp_destroy(b);
    pdlp_destroy(c);
    return 0;
  }
  return 2;
}
