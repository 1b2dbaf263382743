// The surrogate network's state, shared by the kernels for any width (mlp.cu)
// and those for networks of at most MF_WIDTH units a layer (mlp_fused.cu).
#pragma once

#include <cuda_bf16.h>

#include <vector>

#include "bart_internal.cuh"

struct bart_mlp {
  bart_ctx* ctx = nullptr;
  std::vector<int> widths;
  int n_layers = 0;
  int64_t n_params = 0;
  int bf16 = 1;
  int log_outputs = 0;
  int max_batch = 0;
  int64_t step = 0;
  std::vector<int64_t> w_off, b_off;   // offsets into the flat vector
  float* p = nullptr;                  // master FP32 params
  float* m = nullptr;                  // Adam moments
  float* v = nullptr;
  float* g = nullptr;                  // gradient
  __nv_bfloat16* wb = nullptr;         // BF16 weights (same offsets as p)
  float* act = nullptr;                // activations: per layer z and h, [max_batch][width]
  std::vector<int64_t> z_off, h_off;
  float* scale = nullptr;              // in_shift[in], in_scale[in], out_shift[out], out_scale[out]
  float* loss = nullptr;
  float* part = nullptr;               // K-slice partial sums of the tensor-core GEMMs
  int64_t part_elems = 0;
  float* xg = nullptr;                 // gathered batch inputs [max_batch][in] (bart_mlp_train_steps)
  float* tg = nullptr;                 // gathered batch targets [max_batch][out]
  // BF16 networks with no width above MF_WIDTH run on the kernels of
  // mlp_fused.cu; their buffers replace act's h slots, part, xg, tg and wb
  bool fused = false;
  unsigned char* pack = nullptr;       // weights as tensor-core operand images
  std::vector<int64_t> wp_off, wt_off; // byte offsets of W_l and of its transpose in pack
  int64_t pack_bytes = 0;
  unsigned char* tr = nullptr;         // activations and output gradients of a batch as operand images
  std::vector<int64_t> ht_off, dt_off; // byte offsets of layer l's input and of its dz in tr
  int64_t batch_pad = 0;               // max_batch rounded up to whole 64-row blocks
  float* gpart = nullptr;              // K-slice partial weight gradients [slices][n_params]
  float* bpart = nullptr;              // bias gradients per CTA
  double* lpart = nullptr;             // squared errors per CTA
};

constexpr int MF_WIDTH = 256;          // widest layer of the fused kernels
constexpr int MF_MAX_LAYERS = 15;
constexpr int MF_SLICES = 16;          // most K slices of a weight gradient

// Forward pass of B rows of x (physical inputs) into y (physical outputs).
bart_status mlp_fused_forward(bart_mlp* net, const float* x, int B, float* y);
// Gradient of the loss on a batch, into grad (or NULL), or with adam one Adam
// step with it; rows: row indices of the batch in x and t (n_rows rows), or
// NULL for rows 0 .. B-1.
struct MlpAdam {
  float lr, c1, c2;
};
bart_status mlp_fused_gradient(bart_mlp* net, const float* x, const float* t, int64_t n_rows, const int32_t* rows,
                               int B, float* grad, float* loss, const MlpAdam* adam);
// Operand images of the master weights.
bart_status mlp_fused_pack(bart_mlp* net);
// Sizes and allocations; false when memory is missing.
bool mlp_fused_create(bart_mlp* net);

// Shared-memory matrix descriptor of tcgen05: start address, leading- and
// stride-dimension byte offsets (all >> 4), the fixed version bits 46..48 =
// 0b001, no swizzle.
__device__ __forceinline__ unsigned long long um_desc(unsigned int addr, unsigned int lbo, unsigned int sbo) {
  return (unsigned long long)((addr & 0x3FFFFu) >> 4) | ((unsigned long long)(lbo >> 4) << 16) |
         ((unsigned long long)(sbo >> 4) << 32) | (1ull << 46);
}

// Instruction descriptor of tcgen05.mma kind::f16: FP32 accumulator, BF16 A
// and B, both K-major, N >> 3 at bits 17..22, M >> 4 at bits 24..28.
__host__ __device__ constexpr unsigned int um_idesc(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned int)(n >> 3) << 17) | ((unsigned int)(m >> 4) << 24);
}

// D (+)= A B^T for one 128 x N x 16 step: A and B from their descriptors, D
// in tensor memory; acc = 0 overwrites D
__device__ __forceinline__ void um_mma(unsigned int tmem, unsigned long long a, unsigned long long b,
                                       unsigned int idesc, unsigned int acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

// BF16 hi and lo parts of a value: v = hi + lo to about 16 bits.
__device__ __forceinline__ void split_bf16(float v, __nv_bfloat16& hi, __nv_bfloat16& lo) {
  hi = __float2bfloat16_rn(v);
  lo = __float2bfloat16_rn(v - __bfloat162float(hi));
}

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float x) {
  return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * 0.3989422804014327f * expf(-0.5f * x * x);
}
