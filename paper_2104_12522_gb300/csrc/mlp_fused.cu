// The surrogate network in a few launches, for BF16 networks with no layer
// wider than MF_WIDTH (the screening network is 9-256-256-256-10).
//
// Such a network is far too small to be bound by arithmetic (2,048 rows: 0.6
// GFLOP, 0.3 us of the tensor cores) and layer-by-layer GEMMs spent their time
// on launches, K-slice partials and operand conversions between them.  Here
//   mlp_rows_kernel    takes a tile of R rows through the whole network: for
//                      inference scaling, every layer and the physical outputs
//                      in one launch; for training also the loss, and the
//                      gradient back to every layer's pre-activation.
//   mlp_dw_kernel      all layers' weight gradients: units of (128 output rows,
//                      up to 128 input columns, K slice of the batch).
//   mlp_update_kernel  adds the K slices and the CTAs' bias sums in order, then
//                      the Adam step and the operand images of the weights.
// An inference is 1 launch (it was 10 to 12), a training step 3 (about 30).
//
// Layout.  Features run along M (the 128 lanes of an accumulator), batch rows
// along N: a CTA with few rows still fills the tensor core's M, the accumulator
// of a layer is 4 R columns, and a thread owns one feature of 8 rows (16 of 32), so
// bias, GELU and the split into BF16 hi + lo stay in its registers.  A layer's
// B operand holds the rows' hi parts and lo parts side by side (N = 2 R), so
// one MMA multiplies the weights with both and the epilogue adds them.  The
// weights are kept in global memory as the core-matrix images the tensor cores
// read (8 rows x 16 bytes, K-major, no swizzle), so a 64-deep K block is one
// contiguous bulk copy; a producer warp streams the blocks of all layers
// through a ring while the epilogue of the layer before still runs.  The
// training pass writes activations and gradients as images too, transposed
// (features by batch rows), which is what the weight gradients multiply.
//
// R is the smallest of 8, 16, 32 that gives every tile its own SM.
// Measured (9-256-256-256-10): 2,048 rows 71.7 us layer by layer, 18.4 us here
// (22.8 us with one thread to a feature of all rows and erff); a training step
// on 1,024 rows 250 us and 67 us.
#include <algorithm>
#include <cmath>

#include "mlp.cuh"

namespace {

// Epilogue threads: 256 per group of 8 rows (16 of 32), one per feature; then
// the producer warp and the MMA warp.
__host__ __device__ constexpr int mf_rows_per_thread(int R) { return R == 32 ? 16 : 8; }
__host__ __device__ constexpr int mf_groups(int R) { return R / mf_rows_per_thread(R); }
__host__ __device__ constexpr int mf_threads(int R) { return 256 * mf_groups(R) + 64; }
constexpr int MF_STAGES = 4;
constexpr unsigned int MF_BLOCK_BYTES = MF_WIDTH * 64 * 2;   // weights of one 64-deep K block
constexpr unsigned int MF_SPIN_LIMIT = 1u << 22;             // try_wait rounds before a wait is given up
constexpr int DW_THREADS = 160;                  // 4 epilogue warps + the issuing warp
constexpr unsigned int DW_TILE = 128 * 64 * 2;   // one 128-row image block (64 batch rows)

__host__ __device__ constexpr int pad_to(int v, int m) { return (v + m - 1) / m * m; }

// Kernel argument: shapes and places of a network.
struct MfNet {
  int L;                                         // layers
  int w[MF_MAX_LAYERS + 1];
  unsigned int wp[MF_MAX_LAYERS], wt[MF_MAX_LAYERS];   // byte offsets in pack: W_l, W_l transposed
  unsigned int w_off[MF_MAX_LAYERS], b_off[MF_MAX_LAYERS];
  int bias_at[MF_MAX_LAYERS];                    // first bias of layer l among all biases
  int n_bias;
  long long z[MF_MAX_LAYERS + 1];                // element offsets of the pre-activations
  long long ht[MF_MAX_LAYERS], dt[MF_MAX_LAYERS];   // byte offsets of the images of layer l's input and dz
  long long plane;                               // batch rows of an image (multiple of 64)
};

struct MfArgs {
  MfNet n;
  const unsigned char* pack;
  const float* p;
  const float* scale;          // in_shift, in_scale, out_shift, out_scale
  int log_outputs;
  const float* x;
  const float* t;
  const int32_t* rows;
  int64_t n_rows;
  int B, tiles;
  float inv;                   // 2 / (B n_out)
  float* y;
  float* z;
  unsigned char* tr;
  float* bpart;
  double* lpart;
  int* status;
};

// Byte offset of the core matrix (feature group f >> 3, batch group b >> 3) of
// an image with `rows` features, within its 64-row block.
__device__ __forceinline__ long long image_at(int f, long long b, int rows) {
  return (b >> 6) * ((long long)rows * 128) + ((f >> 3) * 8 + (int)((b & 63) >> 3)) * 128 + (f & 7) * 16;
}

__device__ __forceinline__ unsigned int sm_u32(const void* p) { return (unsigned int)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(unsigned long long* b, unsigned int n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sm_u32(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive(unsigned long long* b) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}" ::"r"(sm_u32(b)) : "memory");
}
__device__ __forceinline__ void bar_expect(unsigned long long* b, unsigned int bytes) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}" ::"r"(sm_u32(b)),
               "r"(bytes)
               : "memory");
}
// Bounded wait for the phase of the given parity; false once it, or another
// thread of the CTA, has given up.
__device__ __forceinline__ bool bar_wait(unsigned long long* b, unsigned int parity, volatile int* fail) {
  const unsigned int a = sm_u32(b);
  for (unsigned int it = 0; it < MF_SPIN_LIMIT; ++it) {
    unsigned int ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((it & 255u) == 255u && *fail) return false;
  }
  *fail = 1;
  return false;
}
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, unsigned int bytes, unsigned long long* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   sm_u32(dst)),
               "l"(src), "r"(bytes), "r"(sm_u32(bar))
               : "memory");
}
__device__ __forceinline__ void mma_commit(unsigned long long* b) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(sm_u32(b))
               : "memory");
}

// N consecutive accumulator columns of this thread's TMEM lane.
template <int N>
__device__ __forceinline__ void tmem_load(unsigned int addr, float (&v)[N]) {
  static_assert(N == 8 || N % 16 == 0, "");
  if constexpr (N == 8) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(addr)
                 : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = __uint_as_float(r[q]);
  } else {
#pragma unroll
    for (int c = 0; c < N; c += 16) {
      uint32_t r[16];
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
          "%15}, [%16];"
          : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
            "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
          : "r"(addr + c)
          : "memory");
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int q = 0; q < 16; ++q) v[c + q] = __uint_as_float(r[q]);
    }
  }
}

// The MMA steps of a pass in order: forward layers 0 .. L-1, then (training)
// the transposed weights of layers L-1 .. 1.
struct MfStep {
  unsigned int at;             // byte offset of the weights' image
  int m, k;                    // output features, input features
};
__device__ __forceinline__ MfStep mf_step(const MfNet& n, int s) {
  MfStep r;
  if (s < n.L) {
    r.at = n.wp[s];
    r.m = n.w[s + 1];
    r.k = n.w[s];
  } else {
    const int l = 2 * n.L - 1 - s;
    r.at = n.wt[l];
    r.m = n.w[l];
    r.k = n.w[l + 1];
  }
  return r;
}

// hi | lo << 16 of a value.
__device__ __forceinline__ unsigned int split_word(float v) {
  __nv_bfloat16 h, l;
  split_bf16(v, h, l);
  return (unsigned int)__bfloat16_as_ushort(h) | ((unsigned int)__bfloat16_as_ushort(l) << 16);
}

// The normal distribution function Phi(x) and, for the gradient, exp(-x^2 / 2):
// Phi(-|x|) = erfc(z) / 2, z = |x| / sqrt 2, with erfc(z) = exp(-z^2) t P(t),
// t = 1 / (1 + 0.3 z), P fitted by least squares (reweighted towards the largest
// error) to 2.1e-8 relative over z <= 12.  Relative error of x Phi(x) in FP32
// 1.4e-6 for |x| <= 5, absolute 3.8e-7 (erff: 4.5e-7, without the relative
// accuracy below zero); no branch, a third of erff's instructions.
__device__ __forceinline__ float normal_cdf(float x, float& e) {
  const float ax = fabsf(x);
  float t;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(t) : "f"(fmaf(ax, 0.3f * 0.70710678118654752f, 1.0f)));
  float p = -0.12925601f;
  p = fmaf(p, t, 0.484315053f);
  p = fmaf(p, t, -0.50979936f);
  p = fmaf(p, t, 0.544997127f);
  p = fmaf(p, t, -0.0928463923f);
  p = fmaf(p, t, 0.214189869f);
  p = fmaf(p, t, 0.148519151f);
  p = fmaf(p, t, 0.170691216f);
  p = fmaf(p, t, 0.169189338f);
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(ax * ax * -0.72134752044448170f));
  const float tail = 0.5f * t * p * e;
  return x >= 0.0f ? 1.0f - tail : tail;
}
__device__ __forceinline__ float mf_gelu(float x) {
  float e;
  return x * normal_cdf(x, e);
}
__device__ __forceinline__ float mf_gelu_grad(float x) {
  float e;
  const float c = normal_cdf(x, e);
  return fmaf(x * 0.3989422804014327f, e, c);
}

template <int R, bool TRAIN>
__global__ void __launch_bounds__(mf_threads(R), 1)
mlp_rows_kernel(const __grid_constant__ MfArgs a) {
  static_assert(R == 8 || R == 16 || R == 32, "");
  constexpr int N = 2 * R;                       // hi parts of the rows, then lo parts
  constexpr int RT = mf_rows_per_thread(R), EPI = 256 * mf_groups(R);   // rows a thread, epilogue threads
  constexpr unsigned int B_SBO = 128, B_LBO = (N / 8) * 128;
  constexpr unsigned int TMEM_COLS = 2 * N;      // two halves of 128 features; a power of two >= 32
  constexpr unsigned int IDESC = um_idesc(128, N);
  extern __shared__ __align__(1024) unsigned char mf_smem[];
  unsigned char* ring = mf_smem;                                     // [MF_STAGES][MF_BLOCK_BYTES]
  unsigned char* opnd = mf_smem + MF_STAGES * MF_BLOCK_BYTES;        // B operand: K up to 256 x N, BF16
  float* bacc = reinterpret_cast<float*>(opnd + (MF_WIDTH / 8) * B_LBO);   // [row group][n_bias] (training)
  __shared__ __align__(8) unsigned long long full[MF_STAGES], empty[MF_STAGES], acc_bar, in_bar;
  __shared__ unsigned int s_tmem;
  __shared__ volatile int s_fail;
  __shared__ double s_loss[EPI / 32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int L = a.n.L, steps = TRAIN ? 2 * L - 1 : L;

  if (warp == EPI / 32 + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sm_u32(&s_tmem)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int q = 0; q < MF_STAGES; ++q) {
      bar_init(&full[q], 1);
      bar_init(&empty[q], 1);
    }
    bar_init(&acc_bar, 1);
    bar_init(&in_bar, EPI);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_fail = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned int tmem = s_tmem;

  if (warp == EPI / 32) {
    // ---- producer: the K blocks of every step of every tile, in order
    if (lane == 0) {
      unsigned int q = 0;
      bool ok = true;
      for (int tile = blockIdx.x; ok && tile < a.tiles; tile += gridDim.x)
        for (int s = 0; ok && s < steps; ++s) {
          const MfStep st = mf_step(a.n, s);
          const int kp = pad_to(st.k, 16), mp = pad_to(st.m, 128);
          const unsigned char* src = a.pack + st.at;
          for (int k0 = 0; ok && k0 < kp; k0 += 64, ++q) {
            const unsigned int sg = q % MF_STAGES, bytes = (unsigned int)(mp * min(64, kp - k0) * 2);
            if (q >= MF_STAGES && !bar_wait(&empty[sg], (q / MF_STAGES - 1) & 1u, &s_fail)) {
              ok = false;
              break;
            }
            bar_expect(&full[sg], bytes);
            bulk_copy(ring + sg * MF_BLOCK_BYTES, src, bytes, &full[sg]);
            src += bytes;
          }
        }
      // after a failure: copies in flight land before the CTA leaves
      if (s_fail) {
        volatile int none = 0;
        for (unsigned int i = q > MF_STAGES ? q - MF_STAGES : 0; i < q; ++i)
          bar_wait(&full[i % MF_STAGES], (i / MF_STAGES) & 1u, &none);
      }
    }
  } else if (warp == EPI / 32 + 1) {
    // ---- MMA: one thread issues
    if (lane == 0) {
      unsigned int q = 0, done = 0;
      bool ok = true;
      for (int tile = blockIdx.x; ok && tile < a.tiles; tile += gridDim.x)
        for (int s = 0; ok && s < steps; ++s, ++done) {
          const MfStep st = mf_step(a.n, s);
          const int kp = pad_to(st.k, 16), halves = st.m > 128 ? 2 : 1;
          if (!bar_wait(&in_bar, done & 1u, &s_fail)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          for (int k0 = 0; k0 < kp; k0 += 64, ++q) {
            const unsigned int sg = q % MF_STAGES;
            const int kw = min(64, kp - k0);
            const unsigned int sbo = (unsigned int)(kw / 8) * 128;
            if (!bar_wait(&full[sg], (q / MF_STAGES) & 1u, &s_fail)) {
              ok = false;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const unsigned int wa = sm_u32(ring + sg * MF_BLOCK_BYTES), ba = sm_u32(opnd) + (unsigned int)(k0 / 8) * B_LBO;
            for (int ks = 0; ks < kw / 16; ++ks) {
              const unsigned long long bd = um_desc(ba + ks * 2 * B_LBO, B_LBO, B_SBO);
              for (int h = 0; h < halves; ++h)
                um_mma(tmem + h * N, um_desc(wa + h * 16 * sbo + ks * 256, 128, sbo), bd, IDESC,
                       (k0 == 0 && ks == 0) ? 0u : 1u);
            }
            mma_commit(&empty[sg]);
          }
          if (ok) mma_commit(&acc_bar);
        }
    }
  } else {
    // ---- epilogue: thread = feature, RT rows from r0 in registers (warp & 3 is
    // the quadrant of TMEM lanes that a warp can read)
    const int f = tid & 255, half = (warp >> 2) & 1, rg = tid >> 8, r0 = rg * RT;
    const unsigned int t_addr = tmem + ((unsigned int)((warp & 3) * 32) << 16) + (unsigned int)(half * N + r0);
    const int g = (lane >> 3) & 3;
    unsigned char* const my_opnd = opnd + (f >> 3) * B_LBO + (r0 / 8) * 128 + (f & 7) * 2;
    float* const my_bacc = bacc + rg * a.n.n_bias;
    unsigned int done = 0;
    double loss = 0.0;
    const int n_in = a.n.w[0], n_out = a.n.w[L];
    if (TRAIN)
      for (int l = 0; l < L; ++l)                // bias_at[l] + f of a row group belongs to one thread
        if (f < a.n.w[l + 1]) my_bacc[a.n.bias_at[l] + f] = 0.0f;
    // B operand of the next step, K = f: the rows' hi and lo parts.  The eight
    // rows of a core matrix are stored starting at a row that depends on the
    // lane's core matrix, so a warp's stores meet 32 different banks' words.
    auto put = [&](const unsigned int (&w)[RT]) {
#pragma unroll
      for (int q = 0; q < RT / 8; ++q) {
        unsigned int u[8], v[8];
#pragma unroll
        for (int s = 0; s < 8; ++s) u[s] = (g & 1) ? w[8 * q + ((s + 2) & 7)] : w[8 * q + s];
#pragma unroll
        for (int s = 0; s < 8; ++s) v[s] = (g & 2) ? u[(s + 4) & 7] : u[s];
#pragma unroll
        for (int s = 0; s < 8; ++s) {
          unsigned char* o = my_opnd + q * 128 + ((s + 2 * g) & 7) * 16;
          *reinterpret_cast<unsigned short*>(o) = (unsigned short)v[s];
          *reinterpret_cast<unsigned short*>(o + (R / 8) * 128) = (unsigned short)(v[s] >> 16);
        }
      }
    };
    // the same values as an image for the weight gradients, K = batch rows
    auto put_image = [&](long long at, int rows, long long b0, const unsigned int (&w)[RT]) {
#pragma unroll
      for (int q = 0; q < RT / 8; ++q) {
        unsigned int h[4], l[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          h[s] = __byte_perm(w[8 * q + 2 * s], w[8 * q + 2 * s + 1], 0x5410);
          l[s] = __byte_perm(w[8 * q + 2 * s], w[8 * q + 2 * s + 1], 0x7632);
        }
        unsigned char* o = a.tr + at + image_at(f, b0 + 8 * q, rows);
        *reinterpret_cast<uint4*>(o) = make_uint4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<uint4*>(o + a.n.plane * rows * 2) = make_uint4(l[0], l[1], l[2], l[3]);
      }
    };
    auto publish = [&]() {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      bar_arrive(&in_bar);
    };
    // waits for the step's accumulator; v = its hi and lo products added
    auto take = [&](int m, float (&v)[RT]) -> bool {
      if (!__all_sync(0xffffffffu, bar_wait(&acc_bar, done & 1u, &s_fail))) return false;
      ++done;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (half * 128 < m) {                      // uniform over the warp
        float d[RT];
        tmem_load<RT>(t_addr, v);
        tmem_load<RT>(t_addr + R, d);
#pragma unroll
        for (int r = 0; r < RT; ++r) v[r] += d[r];
      } else {
#pragma unroll
        for (int r = 0; r < RT; ++r) v[r] = 0.0f;
      }
      return true;
    };

    bool ok = true;
    for (int tile = blockIdx.x; ok && tile < a.tiles; tile += gridDim.x) {
      const int64_t b0 = (int64_t)tile * R + r0;   // the thread's first row
      unsigned int w[RT];
      if (f < pad_to(n_in, 16)) {
#pragma unroll
        for (int r = 0; r < RT; ++r) {
          float v = 0.0f;
          if (f < n_in && b0 + r < a.B) {
            int64_t row = b0 + r;
            if (a.rows) {
              row = a.rows[b0 + r];
              if (row < 0 || row >= a.n_rows) {
                atomicOr(a.status, BART_DEV_RANGE);
                row = 0;
              }
            }
            v = (a.x[row * n_in + f] - a.scale[f]) * a.scale[n_in + f];
          }
          w[r] = split_word(v);
        }
        put(w);
        if (TRAIN) put_image(a.n.ht[0], pad_to(n_in, 16), b0, w);
      }
      publish();
      float v[RT];
      for (int l = 0; ok && l < L; ++l) {
        const int m = a.n.w[l + 1];
        // what the epilogue reads from memory is requested before the wait
        const float bias = f < m ? a.p[a.n.b_off[l] + f] : 0.0f;
        float target[RT];
        if (TRAIN && l + 1 == L) {
#pragma unroll
          for (int r = 0; r < RT; ++r) {
            target[r] = 1.0f;
            if (f < m && b0 + r < a.B) {
              int64_t row = b0 + r;
              if (a.rows) {
                row = a.rows[b0 + r];
                if (row < 0 || row >= a.n_rows) row = 0;
              }
              target[r] = a.t[row * m + f];
            }
          }
        }
        if (!take(m, v)) {
          ok = false;
          break;
        }
        if (l + 1 < L) {
          if (f < pad_to(m, 16)) {
            float* z = TRAIN ? a.z + a.n.z[l + 1] + b0 * m + f : nullptr;
#pragma unroll
            for (int r = 0; r < RT; ++r) {
              const float zz = v[r] + bias;
              if (TRAIN && f < m) z[(int64_t)r * m] = zz;
              w[r] = f < m ? split_word(mf_gelu(zz)) : 0u;
            }
            put(w);
            if (TRAIN) put_image(a.n.ht[l + 1], pad_to(m, 16), b0, w);
          }
          publish();
        } else if (!TRAIN) {
          if (f < m) {
            const float osh = a.scale[2 * n_in + f], osc = a.scale[2 * n_in + n_out + f];
#pragma unroll
            for (int r = 0; r < RT; ++r)
              if (b0 + r < a.B) {
                const float s = (v[r] + bias) / osc + osh;
                a.y[(b0 + r) * m + f] = a.log_outputs ? exp10f(s) : s;
              }
          }
        } else if (f < pad_to(m, 16)) {
          // the gradient of the loss by the standardised output
          float db = 0.0f;
#pragma unroll
          for (int r = 0; r < RT; ++r) {
            float dy = 0.0f;
            if (f < m && b0 + r < a.B) {
              const float tv = target[r], ts = a.log_outputs ? log10f(tv) : tv;
              const float e = (v[r] + bias) - (ts - a.scale[2 * n_in + f]) * a.scale[2 * n_in + n_out + f];
              dy = a.inv * e;
              loss += (double)e * e;
            }
            db += dy;
            w[r] = split_word(dy);
          }
          put(w);
          put_image(a.n.dt[l], pad_to(m, 128), b0, w);
          if (f < m) my_bacc[a.n.bias_at[l] + f] += db;
        }
      }
      if (TRAIN && ok && L > 1) {
        publish();
        for (int l = L - 1; l >= 1; --l) {       // dz of layer l-1 from dz of layer l
          const int m = a.n.w[l];
          float z[RT];
#pragma unroll
          for (int r = 0; r < RT; ++r) z[r] = f < m ? a.z[a.n.z[l] + (b0 + r) * m + f] : 0.0f;   // this thread's own, from above
          if (!take(m, v)) {
            ok = false;
            break;
          }
          if (f < pad_to(m, 16)) {
            float db = 0.0f;
#pragma unroll
            for (int r = 0; r < RT; ++r) {
              // rows past the batch carry zeros
              const float dz = f < m ? v[r] * mf_gelu_grad(z[r]) : 0.0f;
              db += dz;
              w[r] = split_word(dz);
            }
            if (l > 1) put(w);
            put_image(a.n.dt[l - 1], pad_to(m, 128), b0, w);
            if (f < m) my_bacc[a.n.bias_at[l - 1] + f] += db;
          }
          if (l > 1) publish();
        }
      }
    }
    if (TRAIN && ok) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
      if (lane == 0) s_loss[warp] = loss;
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (tid == 0) {
    if (s_fail) {
      atomicOr(a.status, BART_DEV_TIMEOUT);
    } else if (TRAIN) {
      double s = 0.0;
      for (int q = 0; q < EPI / 32; ++q) s += s_loss[q];
      a.lpart[blockIdx.x] = s;
    }
  }
  if (TRAIN && !s_fail)
    for (int q = tid; q < a.n.n_bias; q += blockDim.x) {
      float s = bacc[q];
      for (int g = 1; g < mf_groups(R); ++g) s += bacc[g * a.n.n_bias + q];
      a.bpart[(int64_t)blockIdx.x * a.n.n_bias + q] = s;
    }
  if (warp == EPI / 32 + 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
}

// ---- weight gradients: dW_l[o][i] = sum_b dz_l[b][o] h_l[b][i]
struct DwArgs {
  MfNet n;
  const unsigned char* tr;
  float* part;                 // [slices][n_params]
  int64_t n_params;
  int slices, blocks, per;     // K slices, 64-row blocks of the batch, blocks per slice
  int* status;
};

__global__ void __launch_bounds__(DW_THREADS)
mlp_dw_kernel(const __grid_constant__ DwArgs a) {
  constexpr unsigned int STAGE = 4 * DW_TILE;    // dz hi, dz lo, h hi, h lo
  extern __shared__ __align__(1024) unsigned char mf_smem[];
  __shared__ __align__(8) unsigned long long full[2], empty[2], acc_bar;
  __shared__ unsigned int s_tmem;
  __shared__ volatile int s_fail;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // the unit: layer, 128 outputs from o0, up to 128 inputs from i0
  int u = blockIdx.x, l = 0, o0 = 0, i0 = 0;
  for (;; ++l) {
    const int mt = pad_to(a.n.w[l + 1], 128) / 128, nt = pad_to(a.n.w[l], 128) / 128;
    if (u < mt * nt) {
      o0 = u / nt * 128;
      i0 = u % nt * 128;
      break;
    }
    u -= mt * nt;
  }
  const int no = a.n.w[l + 1], ni = a.n.w[l];
  const int nb = min(128, pad_to(ni, 16) - i0);  // columns of the tile, a multiple of 16
  const int kb0 = blockIdx.y * a.per, nk = min(a.per, a.blocks - kb0);   // >= 1
  if (warp == 4) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sm_u32(&s_tmem)), "r"(128)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int q = 0; q < 2; ++q) {
      bar_init(&full[q], 1);
      bar_init(&empty[q], 1);
    }
    bar_init(&acc_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_fail = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned int tmem = s_tmem;
  if (warp == 4) {
    if (lane == 0) {
      const int rd = pad_to(no, 128), rh = pad_to(ni, 16);
      const unsigned char* dz = a.tr + a.n.dt[l] + (long long)o0 * 128;
      const unsigned char* hh = a.tr + a.n.ht[l] + (long long)i0 * 128;
      const long long dz_lo = a.n.plane * rd * 2, h_lo = a.n.plane * rh * 2;
      const unsigned int hb = (unsigned int)nb * 128;
      const unsigned int idesc = um_idesc(128, nb);
      int issued = 0;
      auto load = [&](int k) {
        unsigned char* s = mf_smem + (k & 1) * STAGE;
        unsigned long long* bar = &full[k & 1];
        const unsigned char* d = dz + (long long)(kb0 + k) * rd * 128;
        const unsigned char* h = hh + (long long)(kb0 + k) * rh * 128;
        bar_expect(bar, 2 * DW_TILE + 2 * hb);
        bulk_copy(s, d, DW_TILE, bar);
        bulk_copy(s + DW_TILE, d + dz_lo, DW_TILE, bar);
        bulk_copy(s + 2 * DW_TILE, h, hb, bar);
        bulk_copy(s + 3 * DW_TILE, h + h_lo, hb, bar);
        issued = k + 1;
      };
      load(0);
      if (nk > 1) load(1);
      bool ok = true;
      for (int k = 0; k < nk; ++k) {
        if (!bar_wait(&full[k & 1], (k >> 1) & 1u, &s_fail)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const unsigned int s = sm_u32(mf_smem + (k & 1) * STAGE);
        for (int ks = 0; ks < 4; ++ks) {
          const unsigned long long dh = um_desc(s + ks * 256, 128, 1024), dl = um_desc(s + DW_TILE + ks * 256, 128, 1024);
          const unsigned long long xh = um_desc(s + 2 * DW_TILE + ks * 256, 128, 1024);
          const unsigned long long xl = um_desc(s + 3 * DW_TILE + ks * 256, 128, 1024);
          um_mma(tmem, dh, xh, idesc, (k == 0 && ks == 0) ? 0u : 1u);
          um_mma(tmem, dl, xh, idesc, 1u);
          um_mma(tmem, dh, xl, idesc, 1u);
        }
        mma_commit(&empty[k & 1]);
        if (k + 2 < nk) {
          if (!bar_wait(&empty[k & 1], (k >> 1) & 1u, &s_fail)) {
            ok = false;
            break;
          }
          load(k + 2);
        }
      }
      if (ok) mma_commit(&acc_bar);
      if (s_fail) {
        volatile int none = 0;
        for (int k = max(0, issued - 2); k < issued; ++k) bar_wait(&full[k & 1], (k >> 1) & 1u, &none);
      }
    }
  } else if (__all_sync(0xffffffffu, bar_wait(&acc_bar, 0u, &s_fail))) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const int o = o0 + warp * 32 + lane;
    float* dst = a.part + (int64_t)blockIdx.y * a.n_params + a.n.w_off[l] + (int64_t)o * ni + i0;
    const bool vec = ((ni | (int)a.n.w_off[l] | (int)a.n_params) & 3) == 0;
    for (int c = 0; c < nb; c += 16) {
      float v[16];
      tmem_load<16>(tmem + ((unsigned int)(warp * 32) << 16) + (unsigned int)c, v);
      if (o < no) {
        if (vec && i0 + c + 16 <= ni) {
#pragma unroll
          for (int q = 0; q < 16; q += 4)
            *reinterpret_cast<float4*>(dst + c + q) = make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
        } else {
#pragma unroll
          for (int q = 0; q < 16; ++q)
            if (i0 + c + q < ni) dst[c + q] = v[q];
        }
      }
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (tid == 0 && s_fail) atomicOr(a.status, BART_DEV_TIMEOUT);
  if (warp == 4)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(128) : "memory");
}

// ---- gradient from its partial sums, the Adam step and the operand images
struct UpArgs {
  MfNet n;
  int64_t n_params;
  const float* part;
  const float* bpart;
  const double* lpart;
  int slices, ctas;
  double n_loss;               // B n_out
  float* grad;                 // or NULL
  float* loss;                 // or NULL
  float* p;
  float* m;
  float* v;
  unsigned char* pack;
  int mode;                    // 0 pack only, 1 gradient only, 2 Adam step
  MlpAdam adam;
};

// Byte offset of element (m, k) of an operand image with the given outputs and
// inputs: 64-deep K blocks of core matrices.
__device__ __forceinline__ unsigned int operand_at(int m, int k, int outs, int ins) {
  const int kp = pad_to(ins, 16), mp = pad_to(outs, 128), kb = k & ~63, kw = min(64, kp - kb);
  return (unsigned int)(mp * kb * 2 + ((m >> 3) * (kw / 8) + ((k - kb) >> 3)) * 128 + (m & 7) * 16 + (k & 7) * 2);
}

__global__ void __launch_bounds__(256)
mlp_update_kernel(const __grid_constant__ UpArgs a) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (a.mode && e == 0 && a.loss) {
    double s = 0.0;
    for (int q = 0; q < a.ctas; ++q) s += a.lpart[q];
    *a.loss = (float)(s / a.n_loss);
  }
  if (e >= a.n_params) return;
  int l = 0;
  while (l + 1 < a.n.L && e >= a.n.w_off[l + 1]) ++l;
  const bool weight = e < a.n.b_off[l];
  float p = a.p[e];
  if (a.mode) {
    float g = 0.0f;
    if (weight) {
      for (int z = 0; z < a.slices; ++z) g += a.part[(int64_t)z * a.n_params + e];
    } else {
      const float* b = a.bpart + a.n.bias_at[l] + (e - a.n.b_off[l]);
#pragma unroll 8
      for (int q = 0; q < a.ctas; ++q) g += b[(int64_t)q * a.n.n_bias];
    }
    if (a.grad) a.grad[e] = g;
    if (a.mode == 1) return;
    const float b1 = 0.9f, b2 = 0.999f;
    const float m = b1 * a.m[e] + (1.f - b1) * g;
    const float v = b2 * a.v[e] + (1.f - b2) * g * g;
    a.m[e] = m;
    a.v[e] = v;
    p -= a.adam.lr * (m / a.adam.c1) / (sqrtf(v / a.adam.c2) + 1e-8f);
    a.p[e] = p;
  }
  if (weight) {
    const int ni = a.n.w[l], no = a.n.w[l + 1], r = (int)(e - a.n.w_off[l]);
    const int o = r / ni, i = r % ni;
    const __nv_bfloat16 q = __float2bfloat16_rn(p);
    *reinterpret_cast<__nv_bfloat16*>(a.pack + a.n.wp[l] + operand_at(o, i, no, ni)) = q;
    if (l > 0) *reinterpret_cast<__nv_bfloat16*>(a.pack + a.n.wt[l] + operand_at(i, o, ni, no)) = q;
  }
}

MfNet net_args(const bart_mlp* net) {
  MfNet n{};
  n.L = net->n_layers;
  for (int l = 0; l <= n.L; ++l) {
    n.w[l] = net->widths[l];
    n.z[l] = net->z_off[l];
  }
  for (int l = 0; l < n.L; ++l) {
    n.wp[l] = (unsigned int)net->wp_off[l];
    n.wt[l] = (unsigned int)net->wt_off[l];
    n.w_off[l] = (unsigned int)net->w_off[l];
    n.b_off[l] = (unsigned int)net->b_off[l];
    n.ht[l] = net->ht_off[l];
    n.dt[l] = net->dt_off[l];
    n.bias_at[l] = n.n_bias;
    n.n_bias += n.w[l + 1];
  }
  n.plane = net->batch_pad;
  return n;
}

int max_ctas(const bart_mlp* net) { return net->ctx->sm_count; }   // one resident CTA per SM (shared memory)

// Launches the row kernel over `rows` batch rows (a multiple of 64 for
// training); returns the number of CTAs.
template <int R, bool TRAIN>
cudaError_t launch_rows(bart_mlp* net, MfArgs& a, int64_t rows, int* ctas) {
  const size_t smem = (size_t)MF_STAGES * MF_BLOCK_BYTES + (size_t)(MF_WIDTH / 8) * (2 * R / 8) * 128 +
                      (TRAIN ? (size_t)mf_groups(R) * a.n.n_bias * sizeof(float) : 0);
  cudaError_t e = cudaFuncSetAttribute(mlp_rows_kernel<R, TRAIN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  a.tiles = (int)((rows + R - 1) / R);
  *ctas = std::min(a.tiles, max_ctas(net));
  mlp_rows_kernel<R, TRAIN><<<*ctas, mf_threads(R), smem, net->ctx->stream>>>(a);
  return cudaGetLastError();
}

template <bool TRAIN>
cudaError_t run_rows(bart_mlp* net, MfArgs& a, int64_t rows, int* ctas) {
  const int64_t sms = max_ctas(net);
  if (rows <= 8 * sms) return launch_rows<8, TRAIN>(net, a, rows, ctas);
  if (rows <= 16 * sms) return launch_rows<16, TRAIN>(net, a, rows, ctas);
  return launch_rows<32, TRAIN>(net, a, rows, ctas);
}

MfArgs row_args(bart_mlp* net, const float* x, int B) {
  MfArgs a{};
  a.n = net_args(net);
  a.pack = net->pack;
  a.p = net->p;
  a.scale = net->scale;
  a.log_outputs = net->log_outputs;
  a.x = x;
  a.B = B;
  a.n_rows = B;
  a.z = net->act;
  a.tr = net->tr;
  a.bpart = net->bpart;
  a.lpart = net->lpart;
  a.status = net->ctx->d_status;
  return a;
}

}  // namespace

bool mlp_fused_create(bart_mlp* net) {
  const int L = net->n_layers;
  const auto& w = net->widths;
  int64_t at = 0;
  for (int l = 0; l < L; ++l) {
    net->wp_off.push_back(at);
    at += (int64_t)pad_to(w[l + 1], 128) * pad_to(w[l], 16) * 2;
    net->wt_off.push_back(at);
    if (l > 0) at += (int64_t)pad_to(w[l], 128) * pad_to(w[l + 1], 16) * 2;
  }
  net->pack_bytes = at;
  net->batch_pad = ((int64_t)net->max_batch + 63) / 64 * 64;
  int64_t z = 0, t = 0, biases = 0;
  net->z_off.assign(L + 1, 0);
  for (int l = 0; l < L; ++l) {
    if (l > 0) {                                // pre-activations of the hidden layers
      net->z_off[l] = z;
      z += net->batch_pad * w[l];
    }
    net->ht_off.push_back(t);                   // hi and lo planes
    t += net->batch_pad * pad_to(w[l], 16) * 4;
    net->dt_off.push_back(t);
    t += net->batch_pad * pad_to(w[l + 1], 128) * 4;
    biases += w[l + 1];
  }
  const int ctas = max_ctas(net);
  return cudaMalloc(&net->pack, (size_t)net->pack_bytes) == cudaSuccess &&
         cudaMalloc(&net->act, (size_t)std::max<int64_t>(z, 1) * 4) == cudaSuccess &&
         cudaMalloc(&net->tr, (size_t)t) == cudaSuccess &&
         cudaMalloc(&net->gpart, (size_t)MF_SLICES * net->n_params * 4) == cudaSuccess &&
         cudaMalloc(&net->bpart, (size_t)ctas * biases * 4) == cudaSuccess &&
         cudaMalloc(&net->lpart, (size_t)ctas * 8) == cudaSuccess;
}

static bart_status launch_update(bart_mlp* net, UpArgs& u) {
  u.n = net_args(net);
  u.n_params = net->n_params;
  u.p = net->p;
  u.m = net->m;
  u.v = net->v;
  u.pack = net->pack;
  mlp_update_kernel<<<(unsigned)((net->n_params + 255) / 256), 256, 0, net->ctx->stream>>>(u);
  return bart_check_launch(net->ctx, "mlp_update_kernel");
}

bart_status mlp_fused_pack(bart_mlp* net) {
  UpArgs u{};
  return launch_update(net, u);
}

bart_status mlp_fused_forward(bart_mlp* net, const float* x, int B, float* y) {
  MfArgs a = row_args(net, x, B);
  a.y = y;
  int ctas = 0;
  const cudaError_t e = run_rows<false>(net, a, B, &ctas);
  if (e != cudaSuccess)
    return bart_fail(net->ctx, BART_ECUDA, "launch of mlp_rows_kernel failed: %s", cudaGetErrorString(e));
  return BART_OK;
}

bart_status mlp_fused_gradient(bart_mlp* net, const float* x, const float* t, int64_t n_rows, const int32_t* rows,
                               int B, float* grad, float* loss, const MlpAdam* adam) {
  MfArgs a = row_args(net, x, B);
  a.t = t;
  a.rows = rows;
  a.n_rows = n_rows;
  const int n_out = net->widths[net->n_layers];
  a.inv = 2.0f / (float)((int64_t)B * n_out);
  int ctas = 0;
  // whole 64-row blocks: the rows past the batch write zeros into the images
  const int64_t blocks = ((int64_t)B + 63) / 64;
  cudaError_t e = run_rows<true>(net, a, blocks * 64, &ctas);
  if (e != cudaSuccess)
    return bart_fail(net->ctx, BART_ECUDA, "launch of mlp_rows_kernel failed: %s", cudaGetErrorString(e));
  DwArgs d{};
  d.n = a.n;
  d.tr = net->tr;
  d.part = net->gpart;
  d.n_params = net->n_params;
  int tiles = 0;
  for (int l = 0; l < net->n_layers; ++l)
    tiles += pad_to(net->widths[l + 1], 128) / 128 * (pad_to(net->widths[l], 128) / 128);
  // as many K slices as give every SM a unit
  d.blocks = (int)blocks;
  const int want = std::max(1, std::min({(int)blocks, MF_SLICES, net->ctx->sm_count / tiles}));
  d.per = (d.blocks + want - 1) / want;
  d.slices = (d.blocks + d.per - 1) / d.per;
  d.status = net->ctx->d_status;
  const int smem = 2 * 4 * DW_TILE;
  e = cudaFuncSetAttribute(mlp_dw_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess) {
    mlp_dw_kernel<<<dim3((unsigned)tiles, (unsigned)d.slices), DW_THREADS, smem, net->ctx->stream>>>(d);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess)
    return bart_fail(net->ctx, BART_ECUDA, "launch of mlp_dw_kernel failed: %s", cudaGetErrorString(e));
  UpArgs u{};
  u.part = net->gpart;
  u.bpart = net->bpart;
  u.lpart = net->lpart;
  u.slices = d.slices;
  u.ctas = ctas;
  u.n_loss = (double)B * n_out;
  u.grad = grad;
  u.loss = loss;
  u.mode = adam ? 2 : 1;
  if (adam) u.adam = *adam;
  return launch_update(net, u);
}
