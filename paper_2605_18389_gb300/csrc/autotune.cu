// Autotuner for the launch shapes of one grid and field count.
//
// On the first solve with a given number of fields the tuner times, with CUDA events on
// the workspace, the candidates of the grid's tunable: the FP32 Legendre tile width, or the
// BF16x3 analysis pipeline depth.  Neither choice changes any summation order, so the tuned
// launches give bit-identical results; only their speed differs.  The winner is cached in the
// grid per field count.
#include <float.h>

#include <functional>

#include "shot_internal.cuh"

namespace shot {


namespace {

int time_ms(float* out, cudaStream_t st, cudaEvent_t e0, cudaEvent_t e1, const std::function<int()>& fn) {
  int rc = fn();  // warm-up (also sets any function attributes)
  if (rc) return rc;
  SHOT_CUDA(cudaEventRecord(e0, st));
  for (int r = 0; r < 3; ++r)
    if ((rc = fn())) return rc;
  SHOT_CUDA(cudaEventRecord(e1, st));
  SHOT_CUDA(cudaEventSynchronize(e1));
  SHOT_CUDA(cudaEventElapsedTime(out, e0, e1));
  return SHOT_OK;
}

}  // namespace

int autotune(Grid& g, int nf, cudaStream_t st) {
  for (const Tuning& t : g.tuning)
    if (t.nf == nf) {
      g.active = t;
      return SHOT_OK;
    }
  if (profiling_on()) {   // keep profiled runs free of tuning launches
    g.active = Tuning{};
    return SHOT_OK;
  }
  Workspace& w = g.ws;
  Tuning t;
  t.nf = nf;
  g.active = t;
  cudaEvent_t e0, e1;
  SHOT_CUDA(cudaEventCreate(&e0));
  SHOT_CUDA(cudaEventCreate(&e1));
  int rc = SHOT_OK;
  auto pick = [&](int* slot, std::initializer_list<int> cands, const std::function<int()>& fn) -> int {
    float best = FLT_MAX;
    int arg = 0;
    for (int c : cands) {
      *slot = c;
      g.active = t;
      float ms = 0.f;
      int r = time_ms(&ms, st, e0, e1, fn);
      if (r) return r;
      if (ms < best) {
        best = ms;
        arg = c;
      }
    }
    *slot = arg;
    g.active = t;
    return SHOT_OK;
  };
  auto run_leg = [&]() { return launch_legendre(g, nf, w.XY, w.C, w.XY, w.ldc, st); };
  if (g.mode == SHOT_TABLE && g.precision == SHOT_FP32) rc = pick(&t.simt_bn, {16, 32, 48, 64}, run_leg);
  if (!rc && g.mode == SHOT_TABLE && g.precision == SHOT_BF16X3) rc = pick(&t.tc_stages, {2, 3, 4}, run_leg);
  cudaStreamSynchronize(st);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc) {
    g.active = Tuning{};
    return rc;
  }
  g.tuning.push_back(t);
  g.active = t;
  return SHOT_OK;
}

}  // namespace shot

extern "C" int shot_grid_autotune(shot_grid gh, int nfields, int* choice, void* stream) {
  using namespace shot;
  Grid* g = reinterpret_cast<Grid*>(gh);
  if (!g || nfields < 1) {
    set_error("shot_grid_autotune: bad argument");
    return SHOT_ERR_INVALID_ARG;
  }
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  int rc = ensure_workspace(*g, nfields, st);
  if (rc) return rc;
  if ((rc = launch_heat_mult(*g, 0.0, st))) return rc;
  if ((rc = autotune(*g, nfields, st))) return rc;
  if (choice) {
    choice[0] = dft_fields_per_cta(*g, nfields, false);   // rules on sizes, not timed
    choice[1] = dft_fields_per_cta(*g, nfields, true);    // (the solver's half-steps)
    choice[2] = g->active.simt_bn;
    choice[3] = g->active.tc_stages;
  }
  return SHOT_OK;
}
