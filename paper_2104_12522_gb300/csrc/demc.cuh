// What the retrieval loop (retrieval.cu) uses of the sampler (demc.cu).
#pragma once

#include "bart_internal.cuh"

// Counts of a retrieval, on the device.
struct DemcStats {
  unsigned long long proposals, screened_out, exact_evals, accepted;
  double err_sum;
  unsigned int err_max_bits;    // non-negative float, ordered as its bit pattern
};

// Device buffers of one half-step.
struct DemcHalfStep {
  float* y;                     // [C][d] proposals
  int32_t* inbox;               // [C]
  int32_t* pass;                // [C] proposals that reach the exact model
  int n_bands;
  const float* bands_s;         // [C][n_bands] surrogate band values, or NULL
  const float* bands;           // [C][n_bands] exact band values
  double* ls_y;                 // [C] surrogate log-likelihoods
  const float* data;            // [n_bands]
  const float* sigma;           // [n_bands]
  DemcStats* stats;
  unsigned int* done;           // CTAs finished, 0 between launches
};

// The sampler kernels read the half-step index at hs_dev (NULL: their argument).
void bart_demc_use_counter(bart_demc* s, const int64_t* hs_dev);
int bart_demc_chains(const bart_demc* s);
int bart_demc_params(const bart_demc* s);
const float* bart_demc_states(const bart_demc* s);
// Surrogate log-likelihoods (if any) and the screen; then, after the exact model,
// log-likelihoods, acceptance, statistics, archive, and *hs += 1.
bart_status bart_demc_screen_bands(bart_demc* s, const DemcHalfStep& h);
bart_status bart_demc_finish(bart_demc* s, const DemcHalfStep& h, int64_t* hs);
