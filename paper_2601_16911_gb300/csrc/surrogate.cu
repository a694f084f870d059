// The surrogate sensor network: its training on the GPU (forward, backward, deterministic
// gradient reduction and Adam, all hand-written: BF16-rounded inputs and weights, FP32
// arithmetic), the packing of its weights into tensor-core fragments, stand-alone
// inference (the same warp-level MMA routine the fused stage kernel runs), the features
// mode of the stage kernel that produces training data, and attaching a trained network
// to a mesh.  The paper has no learned component; the network estimates its sensor
// gamma_e (eq. gamma) from cell-vertex data, and the plain sensor decides wherever the
// network's confidence is low.
#include <math.h>
#include <string.h>

#include <new>
#include <vector>

#include "mlp_mma.cuh"
#include "stage_common.cuh"

using namespace cvw;

namespace {

inline cudaStream_t S(void* s) { return reinterpret_cast<cudaStream_t>(s); }
inline cvweno_status cuda_status(cudaError_t e) { return e == cudaSuccess ? CVWENO_OK : CVWENO_ERR_CUDA; }

constexpr int kGradThreads = 256;
constexpr int kSub = 32;            // samples per shared-memory sub-batch
constexpr int kMaxGradBlocks = 304; // 2 x 152 SMs
constexpr int kGradStride = (kMlpParams + 3) / 4 * 4;  // floats of one block's partial gradient
constexpr float kLam = 0.1f, kTau = 0.05f;

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// tanh-form GELU and its derivative with the accurate tanhf (training path)
__device__ __forceinline__ float gelu_acc(float x, float& dgelu) {
  const float c = 0.7978845608028654f;
  const float u = c * fmaf(0.044715f * x * x, x, x);
  const float t = tanhf(u);
  dgelu = 0.5f * (1.0f + t) + 0.5f * x * (1.0f - t * t) * c * fmaf(3.0f * 0.044715f, x * x, 1.0f);
  return 0.5f * x * (1.0f + t);
}

__device__ __forceinline__ float sigm(float x) { return 1.0f / (1.0f + expf(-x)); }
__device__ __forceinline__ float softplus(float x) { return fmaxf(x, 0.0f) + log1pf(expf(-fabsf(x))); }

// Shared-memory layout of the gradient kernel (floats).  Rows of 64 are padded to 68, so that
// 16-byte loads of eight consecutive rows cover all banks.
constexpr int kRow = 68;
struct GradLayout {
  static constexpr int W1 = 0;                     // [64][12], rounded to bf16
  static constexpr int W2 = W1 + 64 * kMlpIn;      // [j][k], rounded to bf16
  static constexpr int W2T = W2 + 64 * kRow;       // [k][j]
  static constexpr int W3 = W2T + 64 * kRow;       // [2][64]
  static constexpr int B = W3 + 128;               // b1 [64], b2 [64], b3 [2]
  static constexpr int X = B + 132;                // [kSub][12]
  static constexpr int G1 = X + kSub * kMlpIn;     // [kSub][kRow] GELU'(z1), then dz1
  static constexpr int A1 = G1 + kSub * kRow;
  static constexpr int G2 = A1 + kSub * kRow;      // GELU'(z2), then dz2
  static constexpr int A2 = G2 + kSub * kRow;
  static constexpr int DO = A2 + kSub * kRow;      // [kSub][2] gradient of the outputs
  static constexpr int FLOATS = DO + kSub * 2;
};

// acc[s][o] += sum over K of v[row s][k] w[row o][k], in pairs over k: two samples by four outputs
// (rows o, o + 16, ...) per thread, 16-byte loads of both.
template <int K>
__device__ __forceinline__ void dot_tile(const float* v, int vstride, const float* w, int wstride, f2 (&acc)[2][4]) {
#pragma unroll 4
  for (int k = 0; k < K; k += 4) {
    float4 x[2], y[4];
#pragma unroll
    for (int t = 0; t < 2; ++t) x[t] = *reinterpret_cast<const float4*>(v + t * vstride + k);
#pragma unroll
    for (int o = 0; o < 4; ++o) y[o] = *reinterpret_cast<const float4*>(w + 16 * o * wstride + k);
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        acc[t][o] = fma2(mk2(x[t].x, x[t].y), mk2(y[o].x, y[o].y), acc[t][o]);
        acc[t][o] = fma2(mk2(x[t].z, x[t].w), mk2(y[o].z, y[o].w), acc[t][o]);
      }
  }
}

// Forward and backward over samples [begin, end) of this block's share of the batch;
// writes the block's summed gradient (already divided by the batch size n) and loss.
// Sub-batches of 32 samples live in shared memory; every product is a register-tiled one on
// two-wide FMAs (2 samples x 4 outputs per thread forward and back, 4 x 4 of dW2 over the
// samples), so a shared-memory load feeds several FMAs.  32 samples rather than 64 give a
// minibatch of 4,096 128 blocks.  Bound by FP32 issue (tanhf and the products).
// Minibatch 4,096: 20 us (one output per thread and step, W2 rows 64 floats apart: every
// load of a warp hit one bank: 65 us).
// Plain pointers, here and in the reduction: a block may be resident before pdl_wait() while the
// kernel before it writes params (or gpart), so nothing may be read as unchanging data.
__global__ void __launch_bounds__(kGradThreads, 2)
    mlp_grad_kernel(const float* params, const float* X, const float* y, int64_t n, int64_t per_block, float* gpart,
                    float* lpart) {
  extern __shared__ __align__(16) float sm[];
  using L = GradLayout;
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  pdl_wait();
  pdl_launch_dependents();
  for (int i = tid; i < 64 * kMlpIn; i += kGradThreads) sm[L::W1 + i] = bf16r(params[kMlpOffW1 + i]);
  for (int i = tid; i < 64 * 64; i += kGradThreads) {
    const float w = bf16r(params[kMlpOffW2 + i]);
    sm[L::W2 + (i >> 6) * kRow + (i & 63)] = w;
    sm[L::W2T + (i & 63) * kRow + (i >> 6)] = w;
  }
  if (tid < 128) {
    sm[L::W3 + tid] = bf16r(params[kMlpOffW3 + tid]);
    sm[L::B + tid] = tid < 64 ? params[kMlpOffB1 + tid] : params[kMlpOffB2 + tid - 64];
  }
  if (tid < 2) sm[L::B + 128 + tid] = params[kMlpOffB3 + tid];
  float* xs = sm + L::X;
  float *g1 = sm + L::G1, *a1 = sm + L::A1, *g2 = sm + L::G2, *a2 = sm + L::A2, *dout = sm + L::DO;
  // this thread's sums: dW2 rows 4 ty .. + 3, columns 4 tx .. + 3; dW1 row tid / 4, columns
  // 3 (tid % 4) .. + 2; one of db1, db2, dW3; db3 on the first two
  f2 w2acc[4][2];
  float w1acc[3] = {0.0f, 0.0f, 0.0f}, bacc = 0.0f, b3acc = 0.0f, lsum = 0.0f;
#pragma unroll
  for (int o = 0; o < 4; ++o) w2acc[o][0] = w2acc[o][1] = mk2(0.0f, 0.0f);
  const int64_t begin = (int64_t)blockIdx.x * per_block;
  const int64_t end = begin + per_block < n ? begin + per_block : n;
  const float inv_n = 1.0f / (float)n;
  for (int64_t s0 = begin; s0 < end; s0 += kSub) {
    const int nb = (int)(end - s0 < kSub ? end - s0 : kSub);
    for (int i = tid; i < kSub * kMlpIn; i += kGradThreads)
      xs[i] = i / kMlpIn < nb ? bf16r(X[s0 * kMlpIn + i]) : 0.0f;
    __syncthreads();
    // layers 1 and 2: samples 2 ty, 2 ty + 1, outputs tx + 16 o
    auto layer = [&](const f2 (&acc)[2][4], const float* bias, float* a, float* g) {
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int o = 0; o < 4; ++o) {
          const int j = tx + 16 * o, at = (2 * ty + t) * kRow + j;
          float dg;
          a[at] = gelu_acc(bias[j] + (acc[t][o].x + acc[t][o].y), dg);
          g[at] = dg;  // kept for the backward pass
        }
    };
    f2 acc[2][4];
    auto zero = [&] {
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int o = 0; o < 4; ++o) acc[t][o] = mk2(0.0f, 0.0f);
    };
    zero();
    dot_tile<kMlpIn>(xs + 2 * ty * kMlpIn, kMlpIn, sm + L::W1 + tx * kMlpIn, kMlpIn, acc);
    layer(acc, sm + L::B, a1, g1);
    __syncthreads();
    zero();
    dot_tile<64>(a1 + 2 * ty * kRow, kRow, sm + L::W2 + tx * kRow, kRow, acc);
    layer(acc, sm + L::B + 64, a2, g2);
    __syncthreads();
    // outputs, loss (S5) and the output gradient: eight lanes per sample, eight inputs each
    {
      const int b = tid / 8, l = tid % 8;
      float o0 = 0.0f, o1 = 0.0f;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float v = a2[b * kRow + l + 8 * k];
        o0 = fmaf(sm[L::W3 + l + 8 * k], v, o0);
        o1 = fmaf(sm[L::W3 + 64 + l + 8 * k], v, o1);
      }
#pragma unroll
      for (int d = 1; d < 8; d *= 2) {
        o0 += __shfl_xor_sync(0xffffffffu, o0, d, 8);
        o1 += __shfl_xor_sync(0xffffffffu, o1, d, 8);
      }
      o0 += sm[L::B + 128];
      o1 += sm[L::B + 129];
      if (l == 0) {
        float d0 = 0.0f, d1 = 0.0f;
        if (b < nb) {
          const float yy = y[s0 + b];
          const float gh = sigm(o0);
          const float t = fabsf(gh - yy) < kTau ? 1.0f : 0.0f;
          lsum += (gh - yy) * (gh - yy) + kLam * (softplus(o1) - t * o1);
          d0 = 2.0f * (gh - yy) * gh * (1.0f - gh) * inv_n;
          d1 = kLam * (sigm(o1) - t) * inv_n;
        }
        dout[2 * b] = d0;
        dout[2 * b + 1] = d1;
      }
    }
    __syncthreads();
    // dz2 = (dout W3) * GELU'(z2), in place of GELU'(z2)
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        const int b = 2 * ty + t, j = tx + 16 * o;
        g2[b * kRow + j] *= fmaf(dout[2 * b], sm[L::W3 + j], dout[2 * b + 1] * sm[L::W3 + 64 + j]);
      }
    __syncthreads();
    // dz1 = (dz2 W2) * GELU'(z1), in place of GELU'(z1)
    zero();
    dot_tile<64>(g2 + 2 * ty * kRow, kRow, sm + L::W2T + tx * kRow, kRow, acc);
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int o = 0; o < 4; ++o) g1[(2 * ty + t) * kRow + tx + 16 * o] *= acc[t][o].x + acc[t][o].y;
    __syncthreads();
    // parameter gradients of this sub-batch, summed over its samples in order (samples past
    // nb have dout = 0, hence zero dz)
#pragma unroll 4
    for (int b = 0; b < kSub; ++b) {
      const float4 d = *reinterpret_cast<const float4*>(g2 + b * kRow + 4 * ty);
      const float4 v = *reinterpret_cast<const float4*>(a1 + b * kRow + 4 * tx);
      const f2 lo = mk2(v.x, v.y), hi = mk2(v.z, v.w);
      w2acc[0][0] = fma2(dup2(d.x), lo, w2acc[0][0]);
      w2acc[0][1] = fma2(dup2(d.x), hi, w2acc[0][1]);
      w2acc[1][0] = fma2(dup2(d.y), lo, w2acc[1][0]);
      w2acc[1][1] = fma2(dup2(d.y), hi, w2acc[1][1]);
      w2acc[2][0] = fma2(dup2(d.z), lo, w2acc[2][0]);
      w2acc[2][1] = fma2(dup2(d.z), hi, w2acc[2][1]);
      w2acc[3][0] = fma2(dup2(d.w), lo, w2acc[3][0]);
      w2acc[3][1] = fma2(dup2(d.w), hi, w2acc[3][1]);
      const float e = g1[b * kRow + tid / 4];
#pragma unroll
      for (int c = 0; c < 3; ++c) w1acc[c] = fmaf(e, xs[b * kMlpIn + 3 * (tid % 4) + c], w1acc[c]);
      if (tid < 64)
        bacc += g1[b * kRow + tid];
      else if (tid < 128)
        bacc += g2[b * kRow + tid - 64];
      else
        bacc = fmaf(dout[2 * b + (tid - 128) / 64], a2[b * kRow + tid % 64], bacc);
      if (tid < 2) b3acc += dout[2 * b + tid];
    }
    __syncthreads();
  }
  float* gp = gpart + (size_t)blockIdx.x * kGradStride;
#pragma unroll
  for (int o = 0; o < 4; ++o)
    *reinterpret_cast<float4*>(gp + kMlpOffW2 + (4 * ty + o) * 64 + 4 * tx) =
        make_float4(w2acc[o][0].x, w2acc[o][0].y, w2acc[o][1].x, w2acc[o][1].y);
#pragma unroll
  for (int c = 0; c < 3; ++c) gp[kMlpOffW1 + 3 * tid + c] = w1acc[c];
  gp[tid < 64 ? kMlpOffB1 + tid : tid < 128 ? kMlpOffB2 + tid - 64 : kMlpOffW3 + tid - 128] = bacc;
  if (tid < 2) gp[kMlpOffB3 + tid] = b3acc;
  // loss: the samples' lanes, in order
  if (tid % 8 == 0) dout[tid / 8] = lsum;
  __syncthreads();
  if (tid == 0) {
    float s = 0.0f;
    for (int b = 0; b < kSub; ++b) s += dout[b];
    lpart[blockIdx.x] = s * inv_n;
  }
}

// Moments and learning rate of one Adam step with bias correction (c1 = 1 - beta1^t,
// c2 = 1 - beta2^t from the host).
struct AdamArgs {
  float *params, *m, *v;
  float lr, b1, b2, c1, c2, eps;
};
__device__ __forceinline__ void adam_update(const AdamArgs& a, int p, float g) {
  const float mm = fmaf(a.b1, a.m[p], (1.0f - a.b1) * g);
  const float vv = fmaf(a.b2, a.v[p], (1.0f - a.b2) * g * g);
  a.m[p] = mm;
  a.v[p] = vv;
  a.params[p] -= a.lr * (mm / a.c1) / (sqrtf(vv / a.c2) + a.eps);
}

// grad[p] = sum over the blocks' partial gradients, and with ADAM the parameter's step: 32
// parameters per block, eight slices of the partials each summed in block order, then the
// slices in order.  loss likewise (block 0).
constexpr int kRedParams = 32, kRedSlices = 8;
template <bool ADAM>
__global__ void __launch_bounds__(kRedParams* kRedSlices)
    mlp_reduce_kernel(const float* gpart, const float* lpart, int nblk, float* grad, float* loss, AdamArgs a) {
  __shared__ float part[kRedSlices][kRedParams];
  const int c = threadIdx.x % kRedParams, sl = threadIdx.x / kRedParams, p = blockIdx.x * kRedParams + c;
  pdl_wait();
  pdl_launch_dependents();
  float s = 0.0f;
  if (p < kMlpParams) {
#pragma unroll 8
    for (int b = sl; b < nblk; b += kRedSlices) s += gpart[(size_t)b * kGradStride + p];
  }
  part[sl][c] = s;
  __syncthreads();
  if (sl == 0 && p < kMlpParams) {
    s = part[0][c];
#pragma unroll
    for (int k = 1; k < kRedSlices; ++k) s += part[k][c];
    grad[p] = s;
    if (ADAM) adam_update(a, p, s);
  }
  if (blockIdx.x == 0 && sl == 1) {
    float l = 0.0f;
    for (int b = c; b < nblk; b += 32) l += lpart[b];
#pragma unroll
    for (int d = 16; d > 0; d /= 2) l += __shfl_down_sync(0xffffffffu, l, d);
    if (c == 0) *loss = l;
  }
}

__global__ void mlp_adam_kernel(const float* __restrict__ grad, AdamArgs a) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < kMlpParams) adam_update(a, p, grad[p]);
}

}  // namespace

namespace {

// FP32 master parameters -> tensor-core fragments (bf16, round to nearest even) + biases.
// Thread = (lane, slot) of one fragment.
__global__ void mlp_pack_kernel(const float* __restrict__ params, MlpPacked* __restrict__ out) {
  const float* W1 = params + kMlpOffW1;
  const float* W2 = params + kMlpOffW2;
  const float* W3 = params + kMlpOffW3;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = i & 31, g = lane >> 2, t = lane & 3, f = i >> 5;
  auto w1 = [&](int n, int k) { return k < kMlpIn ? W1[n * kMlpIn + k] : 0.0f; };
  auto w3 = [&](int n, int k) { return n < kMlpOut ? W3[n * 64 + k] : 0.0f; };
  if (f < 8) {  // layer 1, N tile f: B[k][n] = W1[n][k]
    const int n = 8 * f + g;
    out->w1[f][lane] = make_uint2(pack_bf16x2(w1(n, 2 * t), w1(n, 2 * t + 1)),
                                  pack_bf16x2(w1(n, 2 * t + 8), w1(n, 2 * t + 9)));
  } else if (f < 8 + 32) {  // layer 2, (kk, nt)
    const int kk = (f - 8) >> 3, nt = (f - 8) & 7, n = 8 * nt + g, k0 = 16 * kk + 2 * t;
    out->w2[kk][nt][lane] = make_uint2(pack_bf16x2(W2[n * 64 + k0], W2[n * 64 + k0 + 1]),
                                       pack_bf16x2(W2[n * 64 + k0 + 8], W2[n * 64 + k0 + 9]));
  } else if (f < 8 + 32 + 4) {  // layer 3, K step kk
    const int kk = f - 40, n = g, k0 = 16 * kk + 2 * t;
    out->w3[kk][lane] = make_uint2(pack_bf16x2(w3(n, k0), w3(n, k0 + 1)), pack_bf16x2(w3(n, k0 + 8), w3(n, k0 + 9)));
  } else if (f == 44) {
    out->b1[lane] = params[kMlpOffB1 + lane];
    out->b1[lane + 32] = params[kMlpOffB1 + lane + 32];
    out->b2[lane] = params[kMlpOffB2 + lane];
    out->b2[lane + 32] = params[kMlpOffB2 + lane + 32];
    if (lane < 4) out->b3[lane] = lane < kMlpOut ? params[kMlpOffB3 + lane] : 0.0f;
  }
}
constexpr int kPackThreads = 45 * 32;

// Stand-alone inference: one warp per 32 samples through the tensor-core routine of the
// fused stage kernel.  out[i][0] = o0, out[i][1] = o1 (pre-sigmoid outputs).
constexpr int kInferThreads = 128;
__global__ void __launch_bounds__(kInferThreads)
    mlp_infer_kernel(const MlpPacked* __restrict__ W, const float* __restrict__ X, int64_t n, float* __restrict__ out) {
  __shared__ __align__(16) MlpPacked sw;
  __shared__ __align__(16) __nv_bfloat16 xs[kInferThreads / 32][32 * 16];
  {
    const uint4* src = reinterpret_cast<const uint4*>(W);
    uint4* dst = reinterpret_cast<uint4*>(&sw);
    for (int i = threadIdx.x; i < (int)(sizeof(MlpPacked) / 16); i += kInferThreads) dst[i] = src[i];
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5;
  for (int64_t base = ((int64_t)blockIdx.x * (kInferThreads / 32) + warp) * 32; base < n;
       base += (int64_t)gridDim.x * kInferThreads) {
    const int64_t i = base + (threadIdx.x & 31);
    float x[kMlpIn];
#pragma unroll
    for (int k = 0; k < kMlpIn; ++k) x[k] = i < n ? X[i * kMlpIn + k] : 0.0f;
    float o0, o1;
    mlp_warp(sw, x, xs[warp], o0, o1);  // warp-uniform loop: every lane takes part
    if (i < n) {
      out[2 * i] = o0;
      out[2 * i + 1] = o1;
    }
  }
}

}  // namespace

struct cvweno_mlp_s {
  int device = 0;
  float* d_params = nullptr;  // FP32 master
  float* d_m = nullptr;
  float* d_v = nullptr;
  float* d_grad = nullptr;
  float* d_loss = nullptr;
  float* d_gpart = nullptr;   // [kMaxGradBlocks][kGradStride]
  float* d_lpart = nullptr;
  MlpPacked* d_packed = nullptr;
  unsigned int* d_fallbacks = nullptr;
  float* h_loss = nullptr;    // pinned
  int64_t step = 0;
};

namespace {

void free_mlp(cvweno_mlp n) {
  cudaFree(n->d_params);
  cudaFree(n->d_m);
  cudaFree(n->d_v);
  cudaFree(n->d_grad);
  cudaFree(n->d_loss);
  cudaFree(n->d_gpart);
  cudaFree(n->d_lpart);
  cudaFree(n->d_packed);
  cudaFree(n->d_fallbacks);
  if (n->h_loss) cudaFreeHost(n->h_loss);
  delete n;
}

cudaError_t repack(cvweno_mlp n, cudaStream_t s) {
  mlp_pack_kernel<<<(kPackThreads + 127) / 128, 128, 0, s>>>(n->d_params, n->d_packed);
  return cudaGetLastError();
}

// Arguments of the network's next Adam step.
AdamArgs next_adam(cvweno_mlp n, float lr) {
  const double b1 = 0.9, b2 = 0.999;
  n->step += 1;
  return AdamArgs{n->d_params, n->d_m, n->d_v, lr, (float)b1, (float)b2, (float)(1.0 - pow(b1, (double)n->step)),
                  (float)(1.0 - pow(b2, (double)n->step)), 1e-8f};
}

// Gradient of the batch into d_grad, and with adam the step too.  Both kernels are launched
// with programmatic stream serialisation (they wait before they touch anything).
cudaError_t enqueue_grad(cvweno_mlp n, const float* X, const float* y, int64_t count, const AdamArgs* adam, cudaStream_t s) {
  int64_t nblk = (count + kSub - 1) / kSub;
  if (nblk > kMaxGradBlocks) nblk = kMaxGradBlocks;
  const int64_t per_block = ((count + nblk - 1) / nblk + kSub - 1) / kSub * kSub;
  nblk = (count + per_block - 1) / per_block;
  const size_t smem = sizeof(float) * GradLayout::FLOATS;
  cudaError_t e = launch_pdl(mlp_grad_kernel, dim3((unsigned)nblk), dim3(kGradThreads), smem, s, n->d_params, X, y, count,
                             per_block, n->d_gpart, n->d_lpart);
  if (e != cudaSuccess) return e;
  const dim3 grid((kMlpParams + kRedParams - 1) / kRedParams), block(kRedParams * kRedSlices);
  return launch_pdl(adam ? mlp_reduce_kernel<true> : mlp_reduce_kernel<false>, grid, block, 0, s, n->d_gpart, n->d_lpart,
                    (int)nblk, n->d_grad, n->d_loss, adam ? *adam : AdamArgs{});
}

cudaError_t enqueue_adam(cvweno_mlp n, float lr, cudaStream_t s) {
  mlp_adam_kernel<<<(kMlpParams + 255) / 256, 256, 0, s>>>(n->d_grad, next_adam(n, lr));
  return cudaGetLastError();
}

}  // namespace

extern "C" {

cvweno_status cvweno_mlp_create(const float* params, cvweno_mlp* out) {
  if (!out) return CVWENO_ERR_ARG;
  *out = nullptr;
  cvweno_mlp n = new (std::nothrow) cvweno_mlp_s;
  if (!n) return CVWENO_ERR_NOMEM;
  const size_t pb = sizeof(float) * kMlpParams;
  cudaError_t e = cudaGetDevice(&n->device);
  if (e == cudaSuccess) e = cudaMalloc(&n->d_params, pb);
  if (e == cudaSuccess) e = cudaMalloc(&n->d_m, pb);
  if (e == cudaSuccess) e = cudaMalloc(&n->d_v, pb);
  if (e == cudaSuccess) e = cudaMalloc(&n->d_grad, pb);
  if (e == cudaSuccess) e = cudaMalloc(&n->d_loss, sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&n->d_gpart, sizeof(float) * kGradStride * kMaxGradBlocks);
  if (e == cudaSuccess) e = cudaMalloc(&n->d_lpart, sizeof(float) * kMaxGradBlocks);
  if (e == cudaSuccess) e = cudaMalloc(&n->d_packed, sizeof(MlpPacked));
  if (e == cudaSuccess) e = cudaMalloc(&n->d_fallbacks, sizeof(unsigned int));
  if (e == cudaSuccess) e = cudaMallocHost(&n->h_loss, sizeof(float));
  if (e == cudaSuccess) e = cudaMemset(n->d_m, 0, pb);
  if (e == cudaSuccess) e = cudaMemset(n->d_v, 0, pb);
  if (e == cudaSuccess) e = cudaMemset(n->d_fallbacks, 0, sizeof(unsigned int));
  if (e == cudaSuccess)
    e = params ? cudaMemcpy(n->d_params, params, pb, cudaMemcpyHostToDevice) : cudaMemset(n->d_params, 0, pb);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(sizeof(float) * GradLayout::FLOATS));
  if (e == cudaSuccess) e = repack(n, 0);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    free_mlp(n);
    return CVWENO_ERR_CUDA;
  }
  *out = n;
  return CVWENO_OK;
}

cvweno_status cvweno_mlp_destroy(cvweno_mlp n) {
  if (!n) return CVWENO_ERR_ARG;
  cudaDeviceSynchronize();
  free_mlp(n);
  return CVWENO_OK;
}

cvweno_status cvweno_mlp_get_params(cvweno_mlp n, float* params) {
  if (!n || !params) return CVWENO_ERR_ARG;
  return cuda_status(cudaMemcpy(params, n->d_params, sizeof(float) * kMlpParams, cudaMemcpyDeviceToHost));
}

cvweno_status cvweno_mlp_loss_grad(cvweno_mlp n, const float* X, const float* y, int64_t count, float* loss,
                                   float* grad, void* stream) {
  if (!n || !X || !y || count < 1) return CVWENO_ERR_ARG;
  cudaStream_t s = S(stream);
  cudaError_t e = enqueue_grad(n, X, y, count, nullptr, s);
  if (e == cudaSuccess && loss) e = cudaMemcpyAsync(n->h_loss, n->d_loss, sizeof(float), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess && grad)
    e = cudaMemcpyAsync(grad, n->d_grad, sizeof(float) * kMlpParams, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess && (loss || grad)) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return CVWENO_ERR_CUDA;
  if (loss) *loss = *n->h_loss;
  return CVWENO_OK;
}

cvweno_status cvweno_mlp_adam_step(cvweno_mlp n, float lr, void* stream) {
  if (!n || !(lr > 0.0f)) return CVWENO_ERR_ARG;
  cudaStream_t s = S(stream);
  cudaError_t e = enqueue_adam(n, lr, s);
  if (e == cudaSuccess) e = repack(n, s);
  return cuda_status(e);
}

cvweno_status cvweno_mlp_train(cvweno_mlp n, const float* X, const float* y, int64_t count, int64_t batch,
                               int epochs, float lr, float* last_loss, void* stream) {
  if (!n || !X || !y || count < 1 || batch < 1 || epochs < 0 || !(lr > 0.0f)) return CVWENO_ERR_ARG;
  cudaStream_t s = S(stream);
  cudaError_t e = cudaSuccess;
  for (int ep = 0; ep < epochs && e == cudaSuccess; ++ep)
    for (int64_t b0 = 0; b0 < count && e == cudaSuccess; b0 += batch) {
      const int64_t nb = count - b0 < batch ? count - b0 : batch;
      const AdamArgs adam = next_adam(n, lr);
      e = enqueue_grad(n, X + b0 * kMlpIn, y + b0, nb, &adam, s);
    }
  if (e == cudaSuccess) e = repack(n, s);
  if (e == cudaSuccess && last_loss)
    e = cudaMemcpyAsync(n->h_loss, n->d_loss, sizeof(float), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess && last_loss) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return CVWENO_ERR_CUDA;
  if (last_loss) *last_loss = epochs > 0 ? *n->h_loss : 0.0f;
  return CVWENO_OK;
}

cvweno_status cvweno_mlp_infer(cvweno_mlp n, const float* X, int64_t count, float* out, void* stream) {
  if (!n || !X || !out || count < 1) return CVWENO_ERR_ARG;
  const int64_t warps = (count + 31) / 32;
  int64_t blocks = (warps + kInferThreads / 32 - 1) / (kInferThreads / 32);
  if (blocks > 4 * 152) blocks = 4 * 152;
  mlp_infer_kernel<<<(int)blocks, kInferThreads, 0, S(stream)>>>(n->d_packed, X, count, out);
  return cuda_status(cudaGetLastError());
}

cvweno_status cvweno_features(cvweno_mesh m, const float* u, float* feats, float* gamma, float* norm,
                              void* stream) {
  if (!m || !u || !feats) return CVWENO_ERR_ARG;
  if (m->dim != 2 || m->kind != CVWENO_DG || m->desc.system == CVWENO_EULER) return CVWENO_ERR_UNSUPPORTED;
  StageArgs a = stage_base_args(m);
  a.u_in = u;
  a.feat_out = feats;
  a.gamma_out = gamma;
  a.norm_out = norm;
  a.mlp = nullptr;
  a.mode = kModeFeatures;
  return cuda_status(launch_stage(m, a, S(stream)));
}

cvweno_status cvweno_mesh_set_surrogate(cvweno_mesh m, cvweno_mlp n, float conf_min) {
  if (!m || !(conf_min >= 0.0f && conf_min <= 1.0f)) return CVWENO_ERR_ARG;
  if (n && (m->dim != 2 || m->kind != CVWENO_DG || m->desc.system == CVWENO_EULER)) return CVWENO_ERR_UNSUPPORTED;
  m->surrogate = n ? n->d_packed : nullptr;
  m->surrogate_conf_min = conf_min;
  m->surrogate_fallbacks = n ? n->d_fallbacks : nullptr;
  return CVWENO_OK;
}

cvweno_status cvweno_mlp_fallbacks(cvweno_mlp n, uint64_t* count, int reset, void* stream) {
  if (!n || !count) return CVWENO_ERR_ARG;
  cudaStream_t s = S(stream);
  unsigned int h = 0;
  cudaError_t e = cudaMemcpyAsync(&h, n->d_fallbacks, sizeof(unsigned int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e == cudaSuccess && reset) e = cudaMemsetAsync(n->d_fallbacks, 0, sizeof(unsigned int), s);
  if (e == cudaSuccess && reset) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return CVWENO_ERR_CUDA;
  *count = h;
  return CVWENO_OK;
}

}  // extern "C"
