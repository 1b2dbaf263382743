// Retrieval driver: the sampler loop of the paper (Sec. 3, Fig. 1: the
// sampler proposes parameters, the profile generator and transit produce a
// spectrum, the spectrum integrator gives band values compared with the data)
// run natively, one generation per CUDA-graph launch.
//
// A generation is two half-steps.  Each half-step is, on the context's stream:
//   propose -> [surrogate forward] -> surrogate log-likelihood and screen ->
//   exact forward model of the survivors only (inactive proposals' CTAs exit
//   at once) -> exact log-likelihood, accept, statistics and an increment of
//   the device half-step counter that the sampler kernels read,
// five launches, so the captured graph replays every generation unchanged.
// The first generation runs eagerly: it sizes the scratch buffers and uploads
// the constant tables, after which the captured calls launch kernels only.
#include <cmath>
#include <cstring>
#include <vector>

#include "demc.cuh"
#include "emission.cuh"

namespace {

__global__ void record_kernel(const float* __restrict__ x, int n, const int64_t* __restrict__ hs, int64_t first,
                              float* __restrict__ chain) {
  const int64_t gen = (*hs - first) / 2 - 1;    // generation just completed
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    chain[gen * n + i] = x[i];
}

}  // namespace

extern "C" bart_status bart_retrieval_run(bart_ctx* ctx, bart_demc* s, bart_mlp* surrogate,
                                          const bart_grid_desc* grid, const bart_fwd_cfg* cfg,
                                          const bart_filters* filters, const float* data, const float* sigma,
                                          int64_t first_half_step, int n_generations, int use_graph,
                                          float* chain, bart_retrieval_stats* stats) {
  if (!ctx) return BART_EINVAL;
  BART_REQUIRE(ctx, s && grid && cfg && filters && filters->weights && data && sigma,
               "NULL sampler, grid, cfg, filters, data or sigma");
  BART_REQUIRE(ctx, n_generations >= 1 && first_half_step >= 0 && (first_half_step % 2) == 0,
               "n_generations >= 1 and an even first_half_step are required");
  BART_REQUIRE(ctx, cfg->geometry == BART_EMISSION || cfg->geometry == BART_TRANSMISSION, "bad geometry");
  const int C = bart_demc_chains(s), d = bart_demc_params(s), nb = filters->n_bands;
  BART_REQUIRE(ctx, d == 5 + grid->n_species, "the sampler needs 5 + n_species parameters");
  BART_REQUIRE(ctx, cfg->geometry == BART_EMISSION, "the retrieval loop runs the emission geometry");
  BART_CUDA(ctx, cudaSetDevice(ctx->device));
  cudaStream_t st = ctx->stream;
  bart_status r;
  void *p_y, *p_inbox, *p_pass, *p_lsy, *p_be, *p_bs, *p_hs, *p_stats, *p_done;
  if ((r = bart_scratch(ctx, "rt_y", (size_t)C * d * 4, &p_y)) != BART_OK) return r;
  if ((r = bart_scratch(ctx, "rt_inbox", (size_t)C * 4, &p_inbox)) != BART_OK) return r;
  if ((r = bart_scratch(ctx, "rt_pass", (size_t)C * 4, &p_pass)) != BART_OK) return r;
  if ((r = bart_scratch(ctx, "rt_lsy", (size_t)C * 8, &p_lsy)) != BART_OK) return r;
  if ((r = bart_scratch(ctx, "rt_be", (size_t)C * nb * 4, &p_be)) != BART_OK) return r;
  if ((r = bart_scratch(ctx, "rt_bs", (size_t)C * nb * 4, &p_bs)) != BART_OK) return r;
  if ((r = bart_scratch(ctx, "rt_hs", sizeof(int64_t), &p_hs)) != BART_OK) return r;
  if ((r = bart_scratch(ctx, "rt_stats", sizeof(DemcStats), &p_stats)) != BART_OK) return r;
  if ((r = bart_scratch(ctx, "rt_done", sizeof(unsigned int), &p_done)) != BART_OK) return r;
  int64_t* hs = (int64_t*)p_hs;
  float *y = (float*)p_y, *be = (float*)p_be, *bs = (float*)p_bs;
  int32_t *inbox = (int32_t*)p_inbox, *pass = (int32_t*)p_pass;
  const DemcHalfStep half{y, inbox, pass, nb, surrogate ? bs : nullptr, be, (double*)p_lsy, data, sigma,
                          (DemcStats*)p_stats, (unsigned int*)p_done};
  // host staging copies live in the context's constant cache so the async
  // uploads read memory that outlives this call
  void* dummy;
  if ((r = bart_upload_const(ctx, "rt_hs_init", &first_half_step, sizeof(int64_t), &dummy)) != BART_OK) return r;
  BART_CUDA(ctx, cudaMemcpyAsync(hs, dummy, sizeof(int64_t), cudaMemcpyDeviceToDevice, st));
  BART_CUDA(ctx, cudaMemsetAsync(p_stats, 0, sizeof(DemcStats), st));
  bart_demc_use_counter(s, hs);

  bart_batch batch{};
  batch.n = C;
  batch.theta = y;
  batch.active = pass;

  auto half_step = [&]() -> bart_status {
    bart_status q;
    if ((q = bart_demc_propose(s, 0, y, inbox)) != BART_OK) return q;
    if (surrogate && (q = bart_mlp_forward(surrogate, y, C, bs)) != BART_OK) return q;
    if ((q = bart_demc_screen_bands(s, half)) != BART_OK) return q;
    if ((q = bart_forward_spectra_batch(ctx, grid, cfg, &batch, nullptr, filters, be)) != BART_OK) return q;
    return bart_demc_finish(s, half, hs);
  };
  auto generation = [&]() -> bart_status {
    bart_status q;
    if ((q = half_step()) != BART_OK) return q;
    if ((q = half_step()) != BART_OK) return q;
    if (chain) {
      record_kernel<<<(C * d + 255) / 256, 256, 0, ctx->stream>>>(bart_demc_states(s), C * d, hs, first_half_step,
                                                                  chain);
      if ((q = bart_check_launch(ctx, "record_kernel")) != BART_OK) return q;
    }
    return BART_OK;
  };

  // One check of the grid for all generations, which lets the emission columns
  // end early: some proposals are screened out, so from twice the proposals on
  // that a single call asks.  (What is not valid is left to the forward model.)
  struct Checked {
    bart_ctx* ctx;
    ~Checked() { ctx->grid_bad = nullptr; }
  } checked{ctx};
  if ((double)C * n_generations >= 32.0 * grid->n_temps &&
      bartem::check_forward_request(ctx, grid, cfg, &batch) == BART_OK && bartem::columns_may_end(ctx, grid, cfg, &batch))
    r = bartem::check_grid_values(ctx, grid, &ctx->grid_bad);
  if (r == BART_OK) r = generation();           // eager: sizes scratch, uploads constants
  if (r == BART_OK && n_generations > 1) {
    if (use_graph) {
      // Capture on a private non-blocking stream ordered after the caller's
      // (the legacy default stream cannot be captured), replay on the caller's.
      cudaStream_t cap = nullptr;
      cudaEvent_t ev = nullptr;
      BART_CUDA(ctx, cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
      if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess ||
          cudaEventRecord(ev, st) != cudaSuccess || cudaStreamWaitEvent(cap, ev, 0) != cudaSuccess) {
        cudaGetLastError();
        if (ev) cudaEventDestroy(ev);
        cudaStreamDestroy(cap);
        bart_demc_use_counter(s, nullptr);
        return bart_fail(ctx, BART_ECUDA, "could not order the capture stream");
      }
      cudaGraph_t graph = nullptr;
      cudaGraphExec_t exec = nullptr;
      cudaError_t ce = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
      bart_status rc = BART_OK;
      if (ce == cudaSuccess) {
        ctx->stream = cap;
        ctx->own_capture = true;
        rc = generation();
        ctx->own_capture = false;
        ctx->stream = st;
        ce = cudaStreamEndCapture(cap, &graph);   // always ends the capture
      }
      cudaEventDestroy(ev);
      cudaStreamDestroy(cap);
      if (rc != BART_OK || ce != cudaSuccess) {
        cudaGetLastError();
        if (graph) cudaGraphDestroy(graph);
        bart_demc_use_counter(s, nullptr);
        return rc != BART_OK ? rc : bart_fail(ctx, BART_ECUDA, "graph capture failed: %s", cudaGetErrorString(ce));
      }
      ce = cudaGraphInstantiate(&exec, graph, 0);
      cudaGraphDestroy(graph);
      if (ce != cudaSuccess) {
        bart_demc_use_counter(s, nullptr);
        return bart_fail(ctx, BART_ECUDA, "graph instantiation failed: %s", cudaGetErrorString(ce));
      }
      for (int gidx = 1; gidx < n_generations && ce == cudaSuccess; ++gidx) ce = cudaGraphLaunch(exec, st);
      cudaGraphExecDestroy(exec);
      if (ce != cudaSuccess) {
        bart_demc_use_counter(s, nullptr);
        return bart_fail(ctx, BART_ECUDA, "graph launch failed: %s", cudaGetErrorString(ce));
      }
    } else {
      for (int gidx = 1; gidx < n_generations && r == BART_OK; ++gidx) r = generation();
    }
  }
  bart_demc_use_counter(s, nullptr);
  if (r != BART_OK) return r;
  if (stats) {
    DemcStats h{};
    BART_CUDA(ctx, cudaMemcpyAsync(&h, p_stats, sizeof(DemcStats), cudaMemcpyDeviceToHost, st));
    BART_CUDA(ctx, cudaStreamSynchronize(st));
    stats->proposals = (int64_t)h.proposals;
    stats->screened_out = (int64_t)h.screened_out;
    stats->exact_evals = (int64_t)h.exact_evals;
    stats->accepted = (int64_t)h.accepted;
    stats->surrogate_err_sum = h.err_sum;
    float m;
    std::memcpy(&m, &h.err_max_bits, 4);
    stats->surrogate_err_max = m;
  }
  return BART_OK;
}
