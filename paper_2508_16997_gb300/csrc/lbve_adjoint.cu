// lbve_adjoint.cu -- launchers of the adjoint passes (see lbve_adjoint.cuh).
#include <cuda_runtime.h>

#include "lbve_adjoint.cuh"
#include "lbve_internal.h"

namespace lbve {

template <typename R>
static AdjArgs<R> cast_args(const AdjArgsRaw& a) {
  AdjArgs<R> A;
  A.X = (const R*)a.X;
  A.init = a.init;
  A.force = (const R*)a.force;
  A.M = (R*)a.M;
  A.lam_next = (const R*)a.lam_next;
  A.lam_fields = a.lam_fields;
  A.lam_pulled = (R*)a.lam_pulled;
  A.lam_G = (R*)a.lam_G;
  A.lam_dir = (R*)a.lam_dir;
  A.lam_mh = (R*)a.lam_mh;
  A.lam_cur = (R*)a.lam_cur;
  A.dF = a.dF;
  A.mask = a.mask;
  A.widx = a.widx;
  A.walls = a.walls;
  A.dq = a.dq;
  A.drag_w[0] = a.drag_w[0];
  A.drag_w[1] = a.drag_w[1];
  A.final_pass = a.final_pass;
  return A;
}

template <typename R, typename K>
static void launch(K kernel, int blocks, int threads, bool overlap, const InstDev* d,
                   const AdjArgs<R>& A, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.stream = st;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = overlap ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, d, A);
}

// OPEN: the node passes' variant with an open channel's inlet and outlet
// columns (one-sided x-differences there in every mode, the column pass's
// completion in the step modes).
// Whether a pass launches with the programmatic dependency, i.e. starts while the
// one before it ends.  Float32: always.  Float64: CTAs that arrive early share an
// SM's float64 pipe and registers with running ones once they are more than the
// idle SMs hold, so each pass decides by its own CTAs: at most a third of the SMs
// of 256 threads; for the local pass, whose CTAs fill half an SM's registers, at
// most 0.4 per SM.  50 steps in ms, all passes plain / all early / by this rule:
// 64^2 3.53 / 3.20 / 3.25, 88^2 3.72 / 3.54 / 3.53, 92^2 3.88 / 4.00 / 3.70 (from
// here on the local pass is plain), 96^2 3.70 / 4.18 / 3.49, 112^2 4.25 / 4.04 /
// 4.03, 120^2 4.29 / 4.88 / 4.29 (from here on all are), 128^2 4.26 / 5.13 / 4.26.
template <typename R, int MODE, bool OPEN, bool PUSH>
static void run_pass(int pass, const InstDev* d, const AdjArgs<R>& A, int blocks, cudaStream_t st) {
  const int local = blocks * (256 / kAdjLocalThreads);
  const bool early = sizeof(R) == 4 || 3 * blocks <= kNumSMs;
  const bool early_local = sizeof(R) == 4 || 5 * local <= 2 * kNumSMs;
  switch (pass) {
    case 0: launch(adj_moments<R, MODE, OPEN>, blocks, 256, early, d, A, st); break;
    case 1:
      launch(adj_local<R, MODE, OPEN, PUSH>, local, kAdjLocalThreads, early_local, d, A, st);
      break;
    case 2: launch(adj_gather<R, MODE, OPEN, PUSH>, blocks, 256, early, d, A, st); break;
    case 4: launch(adj_column<R, MODE>, blocks, 256, early, d, A, st); break;
    default: launch(adj_pull<R>, blocks, 256, early, d, A, st); break;
  }
}

template <typename R, int MODE>
static void run_mode(int pass, const AdjArgsRaw& a, const InstDev* d, const AdjArgs<R>& A,
                     int blocks, cudaStream_t st) {
  if (a.open) run_pass<R, MODE, true, false>(pass, d, A, blocks, st);
  else if (a.push) run_pass<R, MODE, false, true>(pass, d, A, blocks, st);
  else run_pass<R, MODE, false, false>(pass, d, A, blocks, st);
}

template <typename R>
static void run(int mode, int pass, const AdjArgsRaw& a, const InstDev* d, int blocks,
                cudaStream_t st) {
  const AdjArgs<R> A = cast_args<R>(a);
  if (mode == kAdjStep) run_mode<R, kAdjStep>(pass, a, d, A, blocks, st);
  else if (mode == kAdjFields) run_mode<R, kAdjFields>(pass, a, d, A, blocks, st);
  else run_mode<R, kAdjInit>(pass, a, d, A, blocks, st);
}

int launch_adjoint(int prec, int mode, int pass, const InstDev* d_desc, const AdjArgsRaw& a,
                   int n_nodes, void* stream) {
  const int blocks = (n_nodes + 255) / 256;
  if (blocks <= 0) return 0;
  cudaStream_t st = (cudaStream_t)stream;
  if (prec == 0) run<double>(mode, pass, a, d_desc, blocks, st);
  else run<float>(mode, pass, a, d_desc, blocks, st);
  return cudaPeekAtLastError() == cudaSuccess ? 0 : -1;  // the caller reads and clears it
}

}  // namespace lbve
