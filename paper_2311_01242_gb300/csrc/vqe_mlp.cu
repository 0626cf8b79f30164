// Warm-start network kernels: a 3-layer perceptron n_in -> H -> H -> n_out with
// SiLU, BF16 weights and GEMM operands, FP32 accumulation (tensor cores via
// mma.sync m16n8k16 BF16 -> FP32), Adam on FP32 master weights. The network is
// tiny (tens of MFLOP per pass) and latency-bound: every GEMM is 16x8 warp tiles, a
// forward layer is one launch (the last with the loss's gradient), a backward layer
// another (input gradient, weight gradient and bias gradient on blocks of their own).
// BF16 rounding happens exactly where the oracle rounds:
// x, h1, h2 (forward), dy, da2, da1 (backward); biases, pre-activations,
// bias gradients and the loss stay FP32.
#include <cstdint>
#include <string>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "../../include/vqe.h"
#include "vqe_internal.h"

namespace {

struct MlpDims {
  int B, Bp, I, Ip, H, O, Op;
};

MlpDims mlp_dims(int batch, int n_in, int n_hidden, int n_out) {
  MlpDims d;
  d.B = batch;
  d.Bp = (batch + 15) / 16 * 16;
  d.I = n_in;
  d.Ip = (n_in + 15) / 16 * 16;
  d.H = n_hidden;
  d.O = n_out;
  d.Op = (n_out + 15) / 16 * 16;
  return d;
}

struct ParamOffsets {
  int64_t W1, b1, W2, b2, W3, b3, total;
};

ParamOffsets param_offsets(const MlpDims& d) {
  ParamOffsets p;
  p.W1 = 0;
  p.b1 = p.W1 + int64_t(d.H) * d.Ip;
  p.W2 = p.b1 + d.H;
  p.b2 = p.W2 + int64_t(d.H) * d.H;
  p.W3 = p.b2 + d.H;
  p.b3 = p.W3 + int64_t(d.Op) * d.H;
  p.total = p.b3 + d.Op;
  return p;
}

struct MlpWs {
  __nv_bfloat16 *xb, *h1b, *h2b, *dyb, *da2b, *da1b;
  float *a1, *a2, *y, *dy, *da2, *da1;
  size_t total;
};

size_t al(size_t v) { return (v + 255) & ~size_t(255); }

MlpWs ws_layout(const MlpDims& d, void* base) {
  char* b = static_cast<char*>(base);
  size_t o = 0;
  MlpWs w;
  auto take = [&](size_t bytes) {
    char* p = b ? b + o : nullptr;
    o += al(bytes);
    return p;
  };
  w.xb = reinterpret_cast<__nv_bfloat16*>(take(size_t(d.Bp) * d.Ip * 2));
  w.a1 = reinterpret_cast<float*>(take(size_t(d.Bp) * d.H * 4));
  w.h1b = reinterpret_cast<__nv_bfloat16*>(take(size_t(d.Bp) * d.H * 2));
  w.a2 = reinterpret_cast<float*>(take(size_t(d.Bp) * d.H * 4));
  w.h2b = reinterpret_cast<__nv_bfloat16*>(take(size_t(d.Bp) * d.H * 2));
  w.y = reinterpret_cast<float*>(take(size_t(d.Bp) * d.Op * 4));
  w.dy = reinterpret_cast<float*>(take(size_t(d.Bp) * d.Op * 4));
  w.dyb = reinterpret_cast<__nv_bfloat16*>(take(size_t(d.Bp) * d.Op * 2));
  w.da2 = reinterpret_cast<float*>(take(size_t(d.Bp) * d.H * 4));
  w.da2b = reinterpret_cast<__nv_bfloat16*>(take(size_t(d.Bp) * d.H * 2));
  w.da1 = reinterpret_cast<float*>(take(size_t(d.Bp) * d.H * 4));
  w.da1b = reinterpret_cast<__nv_bfloat16*>(take(size_t(d.Bp) * d.H * 2));
  w.total = o;
  return w;
}

__device__ __forceinline__ uint32_t pack2(__nv_bfloat16 lo, __nv_bfloat16 hi) {
  return uint32_t(__bfloat16_as_ushort(lo)) | (uint32_t(__bfloat16_as_ushort(hi)) << 16);
}

__device__ __forceinline__ uint32_t ld2(const __nv_bfloat16* p) { return *reinterpret_cast<const uint32_t*>(p); }

__device__ __forceinline__ void mma_bf16(float c[4], const uint32_t a[4], const uint32_t b[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ float silu_f(float a) { return a / (1.0f + expf(-a)); }
__device__ __forceinline__ float dsilu_f(float a) {
  const float s = 1.0f / (1.0f + expf(-a));
  return s * (1.0f + a * (1.0f - s));
}

// Every kernel may start while the one before it on the stream ends (programmatic
// dependent launch): it first waits for that kernel, then lets the next one begin. A
// training step is a chain of launches of a microsecond or two each, so what it waits
// for between and inside them is its time (128 samples, 9 -> 256 -> 256 -> 360:
// 117.4 us as fifteen plain launches with one step's loads in flight per warp, 37.6 us as
// eight with eight steps' loads).
__device__ __forceinline__ void follow() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

constexpr int kSteps = 8;  // steps of 16 along the summed dimension whose loads are in flight together

// Sums over n (a multiple of 16) in steps of 16, in order: every load of kSteps steps,
// then their products.
template <typename LoadA, typename LoadB>
__device__ __forceinline__ void tile_sum(float c[4], int n, LoadA load_a, LoadB load_b) {
  for (int k0 = 0; k0 < n; k0 += 16 * kSteps) {
    uint32_t a[kSteps][4], b[kSteps][2];
#pragma unroll
    for (int u = 0; u < kSteps; ++u)
      if (k0 + 16 * u < n) {
        load_a(k0 + 16 * u, a[u]);
        load_b(k0 + 16 * u, b[u]);
      }
#pragma unroll
    for (int u = 0; u < kSteps; ++u)
      if (k0 + 16 * u < n) mma_bf16(c, a[u], b[u]);
  }
}

// C[b][n] = sum_k A[b][k] W[n][k] + bias[n] for a [Bp x K] BF16 A and [N x K] BF16 W.
// kFirst: A = bf16(x) with zero padding, also written to xb; kHidden: pre-activation to
// pre (FP32) and bf16(silu) to actb; kOut: C to out (row stride ld_out) for rows <
// B and cols < O; kLoss: dy = 2 (y - t) / (B O) on the valid block, 0 on padding, with
// a BF16 copy, and each block's sum of (y - t)^2 to part.
enum FwdKind { kFirst, kHidden, kOut, kLoss };
struct FwdArgs {
  const __nv_bfloat16* A;
  const __nv_bfloat16* W;
  const float* bias;
  int K, N, B, O, ld_out;
  float* pre;
  __nv_bfloat16* actb;
  float* out;            // kLoss: dy
  const float* x;        // kFirst: [B x I], I = O
  __nv_bfloat16* xb;
  const float* target;   // kLoss: [B x O]
  float* part;
};
template <int KIND>
__global__ void __launch_bounds__(128) k_gemm_fwd(const FwdArgs p) {
  __shared__ float red[4];
  follow();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, tg = lane & 3;
  const int r0 = blockIdx.y * 16, n0 = (blockIdx.x * 4 + warp) * 8, K = p.K, N = p.N;
  float sq = 0.0f;
  if (n0 < N) {
    float c[4] = {0.f, 0.f, 0.f, 0.f};
    auto load_b = [&](int k0, uint32_t* b) {
      b[0] = ld2(p.W + (n0 + g) * K + k0 + tg * 2);
      b[1] = ld2(p.W + (n0 + g) * K + k0 + 8 + tg * 2);
    };
    auto load_a = [&](int k0, uint32_t* a) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = r0 + g + 8 * (q & 1), col = k0 + 8 * (q >> 1) + tg * 2;
        if constexpr (KIND == kFirst) {
          const float* x = p.x + int64_t(r) * p.O + col;
          const float x0 = r < p.B && col < p.O ? x[0] : 0.0f, x1 = r < p.B && col + 1 < p.O ? x[1] : 0.0f;
          a[q] = pack2(__float2bfloat16_rn(x0), __float2bfloat16_rn(x1));
          if (n0 == 0) *reinterpret_cast<uint32_t*>(p.xb + r * K + col) = a[q];
        } else {
          a[q] = ld2(p.A + r * K + col);
        }
      }
    };
    tile_sum(c, K, load_a, load_b);
    const int col = n0 + tg * 2;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int row = r0 + g + 8 * h;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float v = c[2 * h + j] + p.bias[col + j];
        if constexpr (KIND == kFirst || KIND == kHidden) {
          p.pre[row * N + col + j] = v;
          p.actb[row * N + col + j] = __float2bfloat16_rn(silu_f(v));
        } else if constexpr (KIND == kOut) {
          if (row < p.B && col + j < p.O) p.out[row * p.ld_out + col + j] = v;
        } else {
          float d = 0.0f;
          if (row < p.B && col + j < p.O) {
            const float e = v - p.target[int64_t(row) * p.O + col + j];
            sq += e * e;
            d = 2.0f / float(p.B * p.O) * e;
          }
          p.out[row * N + col + j] = d;
          p.actb[row * N + col + j] = __float2bfloat16_rn(d);
        }
      }
    }
  }
  if constexpr (KIND == kLoss) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (lane == 0) red[warp] = sq;
    __syncthreads();
    if (threadIdx.x == 0) p.part[blockIdx.y * gridDim.x + blockIdx.x] = red[0] + red[1] + red[2] + red[3];
  }
}

// One layer's backward step, each part on its own blocks of one launch: first da_prev[b][k] =
// (sum_n dA[b][n] W[n][k]) silu'(a_prev[b][k]) (FP32 and BF16), then dW[n][k] = sum_b
// dA[b][n] X[b][k], then db[n] = sum over valid rows of d[b][n] in row order, and with
// the last layer one block for loss = sum(part) / (B O) in a fixed order.
struct BackArgs {
  const __nv_bfloat16* dA;   // [Bp x N]
  const __nv_bfloat16* W;    // [N x K]
  const __nv_bfloat16* X;    // [Bp x K]
  const float* d;            // [Bp x N]
  const float* a_prev;       // [Bp x K]
  float* da;
  __nv_bfloat16* dab;
  float* dW;
  float* db;
  int Bp, B, N, K;
  int dx_blocks, dw_blocks, db_blocks, across;  // across: blocks of 32 columns of K
  const float* part;
  int parts;
  float count;
  float* loss;
};
__global__ void __launch_bounds__(128) k_back(const BackArgs p) {
  __shared__ float red[128];
  follow();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, tg = lane & 3, N = p.N, K = p.K;
  int blk = blockIdx.x;
  if (blk < p.dx_blocks) {
    const int r0 = blk / p.across * 16, k0 = (blk % p.across * 4 + warp) * 8;
    if (k0 >= K) return;
    float c[4] = {0.f, 0.f, 0.f, 0.f};
    tile_sum(
        c, N,
        [&](int m0, uint32_t* a) {
          a[0] = ld2(p.dA + (r0 + g) * N + m0 + tg * 2);
          a[1] = ld2(p.dA + (r0 + g + 8) * N + m0 + tg * 2);
          a[2] = ld2(p.dA + (r0 + g) * N + m0 + 8 + tg * 2);
          a[3] = ld2(p.dA + (r0 + g + 8) * N + m0 + 8 + tg * 2);
        },
        [&](int m0, uint32_t* b) {
          const __nv_bfloat16* w = p.W + int64_t(m0 + tg * 2) * K + k0 + g;
          b[0] = pack2(w[0], w[K]);
          b[1] = pack2(w[8 * K], w[9 * K]);
        });
    const int col = k0 + tg * 2;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int idx = (r0 + g + 8 * h) * K + col + j;
        const float v = c[2 * h + j] * dsilu_f(p.a_prev[idx]);
        p.da[idx] = v;
        p.dab[idx] = __float2bfloat16_rn(v);
      }
    return;
  }
  blk -= p.dx_blocks;
  if (blk < p.dw_blocks) {
    const int n0 = blk / p.across * 16, k0 = (blk % p.across * 4 + warp) * 8;
    if (k0 >= K) return;
    float c[4] = {0.f, 0.f, 0.f, 0.f};
    tile_sum(
        c, p.Bp,
        [&](int b0, uint32_t* a) {
          const __nv_bfloat16* v = p.dA + int64_t(b0 + tg * 2) * N + n0 + g;
          a[0] = pack2(v[0], v[N]);
          a[1] = pack2(v[8], v[N + 8]);
          a[2] = pack2(v[8 * N], v[9 * N]);
          a[3] = pack2(v[8 * N + 8], v[9 * N + 8]);
        },
        [&](int b0, uint32_t* b) {
          const __nv_bfloat16* v = p.X + int64_t(b0 + tg * 2) * K + k0 + g;
          b[0] = pack2(v[0], v[K]);
          b[1] = pack2(v[8 * K], v[9 * K]);
        });
    const int col = k0 + tg * 2;
    p.dW[(n0 + g) * K + col] = c[0];
    p.dW[(n0 + g) * K + col + 1] = c[1];
    p.dW[(n0 + g + 8) * K + col] = c[2];
    p.dW[(n0 + g + 8) * K + col + 1] = c[3];
    return;
  }
  blk -= p.dw_blocks;
  if (blk < p.db_blocks) {
    const int n = blk * 128 + threadIdx.x;
    if (n >= N) return;
    float s = 0.0f;
    int b = 0;
    for (; b + 16 <= p.B; b += 16) {
      float v[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = p.d[int64_t(b + u) * N + n];
#pragma unroll
      for (int u = 0; u < 16; ++u) s += v[u];
    }
    for (; b < p.B; ++b) s += p.d[int64_t(b) * N + n];
    p.db[n] = s;
    return;
  }
  float s = 0.0f;
  for (int i = threadIdx.x; i < p.parts; i += 128) s += p.part[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = 64; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) p.loss[0] = red[0] / p.count;
}

template <typename... KArgs, typename... Args>
cudaError_t launch(void (*kernel)(KArgs...), dim3 grid, int threads, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(unsigned(threads));
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

__global__ void k_adam(int64_t n, float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, const int* __restrict__ step, float lr, float beta1, float beta2,
                       float eps, __nv_bfloat16* __restrict__ wb) {
  follow();
  const int t = *step;
  const float c1 = 1.0f / (1.0f - powf(beta1, float(t)));
  const float c2 = 1.0f / (1.0f - powf(beta2, float(t)));
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const float gi = g[i];
    const float mi = beta1 * m[i] + (1.0f - beta1) * gi;
    const float vi = beta2 * v[i] + (1.0f - beta2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi * c1) / (sqrtf(vi * c2) + eps);
    w[i] = wi;
    wb[i] = __float2bfloat16_rn(wi);
  }
}

__global__ void k_step_inc(int* step) {
  follow();
  *step += 1;
}

__global__ void k_to_bf16(int64_t n, const float* __restrict__ src, __nv_bfloat16* __restrict__ dst) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    dst[i] = __float2bfloat16_rn(src[i]);
}

int check_dims(int batch, int n_in, int n_hidden, int n_out) {
  if (batch < 1 || batch > (1 << 20) || n_in < 1 || n_in > 4096 || n_out < 1 || n_out > 65536 || n_hidden < 16 ||
      n_hidden > 8192 || n_hidden % 16 != 0)
    return vqe::set_error(VQE_ERR_INVALID_ARG,
                          "MLP dims: batch >= 1, 1 <= n_in <= 4096, n_hidden a multiple of 16 in [16, 8192]");
  return VQE_OK;
}

int cuda_check(const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return vqe::set_error(VQE_ERR_CUDA, (std::string(what) + ": " + cudaGetErrorString(e)).c_str());
  return VQE_OK;
}

// forward through the three layers into the workspace; the last layer writes
// to out (row stride ld_out) for the valid rows/cols, or with a target dy, its BF16
// copy and the loss's partial sums
void forward_layers(const MlpDims& d, const MlpWs& w, const float* x, const float* params, const __nv_bfloat16* pb,
                    float* out, const float* target, cudaStream_t s) {
  const ParamOffsets po = param_offsets(d);
  auto grid = [&](int n) { return dim3(unsigned(n / 8 + 3) / 4, unsigned(d.Bp / 16)); };
  FwdArgs a{};
  a.B = d.B;
  a.O = d.I;
  a.x = x;
  a.xb = w.xb;
  a.W = pb + po.W1;
  a.bias = params + po.b1;
  a.K = d.Ip;
  a.N = d.H;
  a.pre = w.a1;
  a.actb = w.h1b;
  launch(k_gemm_fwd<kFirst>, grid(d.H), 128, s, a);
  a.A = w.h1b;
  a.W = pb + po.W2;
  a.bias = params + po.b2;
  a.K = d.H;
  a.pre = w.a2;
  a.actb = w.h2b;
  launch(k_gemm_fwd<kHidden>, grid(d.H), 128, s, a);
  a.A = w.h2b;
  a.W = pb + po.W3;
  a.bias = params + po.b3;
  a.N = d.Op;
  a.O = d.O;
  if (!target) {
    a.out = out;
    a.ld_out = d.O;
    launch(k_gemm_fwd<kOut>, grid(d.Op), 128, s, a);
  } else {
    a.out = w.dy;
    a.actb = w.dyb;
    a.target = target;
    a.part = w.y;
    launch(k_gemm_fwd<kLoss>, grid(d.Op), 128, s, a);
  }
}

}  // namespace

extern "C" {

int64_t vqe_mlp_param_count(int n_in, int n_hidden, int n_out) {
  if (check_dims(1, n_in, n_hidden, n_out)) return 0;
  return param_offsets(mlp_dims(1, n_in, n_hidden, n_out)).total;
}

size_t vqe_mlp_workspace_bytes(int batch, int n_in, int n_hidden, int n_out) {
  if (check_dims(batch, n_in, n_hidden, n_out)) return 0;
  return ws_layout(mlp_dims(batch, n_in, n_hidden, n_out), nullptr).total;
}

int vqe_mlp_to_bf16(int64_t n, const float* src, uint16_t* dst, vqe_stream_t stream) {
  if (n < 0 || (n > 0 && (!src || !dst))) return vqe::set_error(VQE_ERR_INVALID_ARG, "bad bf16 conversion arguments");
  if (n == 0) return VQE_OK;
  k_to_bf16<<<int((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      n, src, reinterpret_cast<__nv_bfloat16*>(dst));
  return cuda_check("k_to_bf16");
}

int vqe_mlp_forward(int batch, int n_in, int n_hidden, int n_out, const float* x, const float* params,
                    const uint16_t* params_bf16, float* y, void* workspace, size_t workspace_bytes,
                    vqe_stream_t stream_) {
  int rc = check_dims(batch, n_in, n_hidden, n_out);
  if (rc) return rc;
  if (!x || !params || !params_bf16 || !y || !workspace) return vqe::set_error(VQE_ERR_INVALID_ARG, "NULL pointer");
  const MlpDims d = mlp_dims(batch, n_in, n_hidden, n_out);
  const MlpWs w = ws_layout(d, workspace);
  if (workspace_bytes < w.total) return vqe::set_error(VQE_ERR_WORKSPACE, "MLP workspace too small");
  cudaStream_t s = static_cast<cudaStream_t>(stream_);
  forward_layers(d, w, x, params, reinterpret_cast<const __nv_bfloat16*>(params_bf16), y, nullptr, s);
  return cuda_check("mlp forward");
}

int vqe_mlp_loss_grad(int batch, int n_in, int n_hidden, int n_out, const float* x, const float* target,
                      const float* params, const uint16_t* params_bf16, float* grads, float* loss,
                      void* workspace, size_t workspace_bytes, vqe_stream_t stream_) {
  int rc = check_dims(batch, n_in, n_hidden, n_out);
  if (rc) return rc;
  if (!x || !target || !params || !params_bf16 || !grads || !loss || !workspace)
    return vqe::set_error(VQE_ERR_INVALID_ARG, "NULL pointer");
  const MlpDims d = mlp_dims(batch, n_in, n_hidden, n_out);
  const MlpWs w = ws_layout(d, workspace);
  if (workspace_bytes < w.total) return vqe::set_error(VQE_ERR_WORKSPACE, "MLP workspace too small");
  cudaStream_t s = static_cast<cudaStream_t>(stream_);
  const ParamOffsets po = param_offsets(d);
  const __nv_bfloat16* pb = reinterpret_cast<const __nv_bfloat16*>(params_bf16);
  forward_layers(d, w, x, params, pb, nullptr, target, s);
  auto back = [&](const __nv_bfloat16* dA, const float* dd, int N, const __nv_bfloat16* X, int K, int64_t W, int64_t b,
                  const float* a_prev, float* da, __nv_bfloat16* dab, bool last) {
    BackArgs a{};
    a.dA = dA;
    a.W = pb + W;
    a.X = X;
    a.d = dd;
    a.a_prev = a_prev;
    a.da = da;
    a.dab = dab;
    a.dW = grads + W;
    a.db = grads + b;
    a.Bp = d.Bp;
    a.B = d.B;
    a.N = N;
    a.K = K;
    a.across = (K / 8 + 3) / 4;
    a.dx_blocks = a_prev ? a.across * (d.Bp / 16) : 0;
    a.dw_blocks = a.across * (N / 16);
    a.db_blocks = (N + 127) / 128;
    a.part = w.y;
    a.parts = (d.Op / 8 + 3) / 4 * (d.Bp / 16);
    a.count = float(d.B * d.O);
    a.loss = loss;
    launch(k_back, dim3(unsigned(a.dx_blocks + a.dw_blocks + a.db_blocks + (last ? 1 : 0))), 128, s, a);
  };
  back(w.dyb, w.dy, d.Op, w.h2b, d.H, po.W3, po.b3, w.a2, w.da2, w.da2b, true);
  back(w.da2b, w.da2, d.H, w.h1b, d.H, po.W2, po.b2, w.a1, w.da1, w.da1b, false);
  back(w.da1b, w.da1, d.H, w.xb, d.Ip, po.W1, po.b1, nullptr, nullptr, nullptr, false);
  return cuda_check("mlp loss_grad");
}

int vqe_mlp_adam(int64_t n, float* params, const float* grads, float* m, float* v, int* step_dev, float lr,
                 float beta1, float beta2, float eps, uint16_t* params_bf16, vqe_stream_t stream) {
  if (n < 1 || !params || !grads || !m || !v || !params_bf16 || !step_dev)
    return vqe::set_error(VQE_ERR_INVALID_ARG, "bad Adam arguments");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int blocks = int((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
  launch(k_adam, dim3(unsigned(blocks)), 256, s, n, params, grads, m, v, static_cast<const int*>(step_dev), lr, beta1,
         beta2, eps, reinterpret_cast<__nv_bfloat16*>(params_bf16));
  launch(k_step_inc, dim3(1), 1, s, step_dev);
  return cuda_check("k_adam");
}

}  // extern "C"
