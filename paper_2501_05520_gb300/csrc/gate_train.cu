// Training kernels of the learned gate: mean binary cross-entropy of sigmoid(score)
// against 0/1 labels, its gradient with respect to the 5057 float32 parameters, and an
// Adam update.  Layout of the parameter vector: W1 [64,12], b1 [64], W2 [64,64], b2 [64],
// w3 [64], b3 [1] (row-major), the same as pt_set_gate takes.
//
// k_gate_grad: one 256-thread CTA per 32 samples (grid-stride), the weights and a tile's
// activations in shared memory, every product as a register tile: a thread holds 2 samples
// x 4 units of the forward and backward products and 4 x 4 of dW2, so that 32 multiply-adds
// share six 16-byte shared loads.  Rows are padded to 68 floats (and the 4 units of a
// forward tile are 16 apart), which keeps those loads free of bank conflicts.  A sample's
// score is reduced over the 16 lanes that hold its units, so loss and output gradient need
// no shared memory; the gradients of the biases and of the last layer stay in registers.
// The gradient sums of all of a CTA's tiles go to global memory once, four at a time where
// the caller's array is 16-byte aligned.  32 samples, because the training minibatch of
// 4096 then spreads over 128 SMs.
//
// Bound by its latency (weights in, five dependent products, sums out) at the minibatch.
// 4096 samples, loss, gradient and Adam step together: 15 us, against 173 when 32 CTAs of 128
// samples each took the products one scalar at a time (rows without padding, so that the 32
// lanes of a load met in one bank).
#include "ptca_internal.cuh"

namespace ptca {

namespace {

constexpr int kS = 32;                  // samples per tile
constexpr int kH = kGateHidden;         // 64
constexpr int kF = kGateFeat;           // 12
constexpr int kOW1 = 0, kOB1 = kOW1 + kH * kF, kOW2 = kOB1 + kH, kOB2 = kOW2 + kH * kH;
constexpr int kOW3 = kOB2 + kH, kOB3 = kOW3 + kH;
constexpr int kRow = kH + 4;            // padded row
constexpr int kGradThreads = 256;       // 16 unit groups x 16 sample groups
constexpr int kGradBlocksPerSm = 2;
static_assert(sizeof(float) * (kH * kF + 3 * kS * kRow + kH * kRow + 3 * kH + kS * kF + 4) <=
                  48 * 1024, "static shared memory");
static_assert(kS == 32 && kGradThreads == 256, "tile shapes");
static_assert(kOW1 % 4 == 0 && kOB1 % 4 == 0 && kOW2 % 4 == 0 && kOB2 % 4 == 0 && kOW3 % 4 == 0,
              "four gradients at a time");

struct alignas(16) GradSmem {
  float w1[kH * kF];
  float w2[kH][kRow];
  float b1[kH], b2[kH], w3[kH];
  float x[kS][kF];
  float h1[kS][kRow];
  float d2[kS][kRow];
  float d1[kS][kRow];
  float b3;
};

__device__ __forceinline__ float4 ld4(const float* p) { return *(const float4*)p; }
__device__ __forceinline__ void fma4(float& a, float4 u, float4 v) {
  a = fmaf(u.x, v.x, a);
  a = fmaf(u.y, v.y, a);
  a = fmaf(u.z, v.z, a);
  a = fmaf(u.w, v.w, a);
}
__device__ __forceinline__ void fma4(float (&a)[4], float u, float4 v) {
  a[0] = fmaf(u, v.x, a[0]);
  a[1] = fmaf(u, v.y, a[1]);
  a[2] = fmaf(u, v.z, a[2]);
  a[3] = fmaf(u, v.w, a[3]);
}
__device__ __forceinline__ void add4(float* g, const float (&v)[4], bool vec) {
  if (vec) {
    atomicAdd((float4*)g, make_float4(v[0], v[1], v[2], v[3]));
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) atomicAdd(g + i, v[i]);
  }
}

__global__ void k_gate_zero(float* grad, float* loss) {
  pdl_sync();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < kGateParams) grad[i] = 0.0f;
  if (i == kGateParams) *loss = 0.0f;
}

__global__ void __launch_bounds__(kGradThreads)
    k_gate_grad(const float* __restrict__ w, const float* __restrict__ X,
                const float* __restrict__ y, int64_t n, float* grad, float* loss) {
  pdl_sync();
  __shared__ GradSmem S;
  const int tid = threadIdx.x;
  const int ug = tid & 15, sg = tid >> 4;  // unit group, sample group
  for (int i = tid; i < kH * kF; i += kGradThreads) S.w1[i] = w[kOW1 + i];
#pragma unroll
  for (int i = 0; i < kH * kH / kGradThreads; ++i) {
    const int e = tid + i * kGradThreads;
    S.w2[e / kH][e % kH] = w[kOW2 + e];
  }
  if (tid < kH) {
    S.b1[tid] = w[kOB1 + tid];
    S.b2[tid] = w[kOB2 + tid];
    S.w3[tid] = w[kOW3 + tid];
  }
  if (tid == 0) S.b3 = w[kOB3];
  const float inv_n = 1.0f / (float)n;
  float g2[4][4] = {};                                     // dW2: units 4 sg.., inputs 4 ug..
  float g1[3] = {};                                        // dW1: unit tid / 4, inputs 3 (tid % 4)..
  float gb2[4] = {}, gw3[4] = {}, gb1[4] = {}, gb3 = 0.0f;  // over this thread's samples
  float lsum = 0.0f;
  for (int64_t base = (int64_t)blockIdx.x * kS; base < n; base += (int64_t)gridDim.x * kS) {
    __syncthreads();
    for (int i = tid; i < kS * kF; i += kGradThreads)
      S.x[i / kF][i % kF] = base + i / kF < n ? X[base * kF + i] : 0.0f;
    float yv[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int64_t g = base + sg + 16 * r;
      yv[r] = g < n ? y[g] : 0.0f;
    }
    __syncthreads();
    // layer 1: samples sg + 16 r, units ug + 16 c
    float z[2][4];
#pragma unroll
    for (int c = 0; c < 4; ++c) z[0][c] = z[1][c] = S.b1[ug + 16 * c];
#pragma unroll
    for (int k = 0; k < kF; k += 4) {
      const float4 x0 = ld4(&S.x[sg][k]), x1 = ld4(&S.x[sg + 16][k]);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float4 wv = ld4(&S.w1[(ug + 16 * c) * kF + k]);
        fma4(z[0][c], wv, x0);
        fma4(z[1][c], wv, x1);
      }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) S.h1[sg + 16 * r][ug + 16 * c] = fmaxf(z[r][c], 0.0f);
    __syncthreads();
    // layer 2, the same tile
#pragma unroll
    for (int c = 0; c < 4; ++c) z[0][c] = z[1][c] = S.b2[ug + 16 * c];
#pragma unroll 4
    for (int k = 0; k < kH; k += 4) {
      const float4 x0 = ld4(&S.h1[sg][k]), x1 = ld4(&S.h1[sg + 16][k]);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float4 wv = ld4(&S.w2[ug + 16 * c][k]);
        fma4(z[0][c], wv, x0);
        fma4(z[1][c], wv, x1);
      }
    }
    // output, loss, d loss / d score (the 16 lanes of a sample alike), gradient at z2
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      float sc = 0.0f;
#pragma unroll
      for (int c = 0; c < 4; ++c) sc = fmaf(S.w3[ug + 16 * c], fmaxf(z[r][c], 0.0f), sc);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) sc += __shfl_xor_sync(kFull, sc, o);
      sc += S.b3;
      float ds = 0.0f;
      if (base + sg + 16 * r < n) {
        if (ug == 0) lsum += (fmaxf(sc, 0.0f) - yv[r] * sc + log1pf(expf(-fabsf(sc)))) * inv_n;
        ds = (1.0f / (1.0f + expf(-sc)) - yv[r]) * inv_n;
      }
      gb3 += ds;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float d = z[r][c] > 0.0f ? ds * S.w3[ug + 16 * c] : 0.0f;
        gw3[c] = fmaf(ds, fmaxf(z[r][c], 0.0f), gw3[c]);
        gb2[c] += d;
        S.d2[sg + 16 * r][ug + 16 * c] = d;
      }
    }
    __syncthreads();
    // gradient at z1: samples sg + 16 r, units 4 ug..
    float d1[2][4] = {};
#pragma unroll 4
    for (int j = 0; j < kH; j += 4) {
      const float4 a0 = ld4(&S.d2[sg][j]), a1 = ld4(&S.d2[sg + 16][j]);
      const float4 w0 = ld4(&S.w2[j][4 * ug]), w1 = ld4(&S.w2[j + 1][4 * ug]);
      const float4 w2 = ld4(&S.w2[j + 2][4 * ug]), w3 = ld4(&S.w2[j + 3][4 * ug]);
      fma4(d1[0], a0.x, w0), fma4(d1[0], a0.y, w1), fma4(d1[0], a0.z, w2), fma4(d1[0], a0.w, w3);
      fma4(d1[1], a1.x, w0), fma4(d1[1], a1.y, w1), fma4(d1[1], a1.z, w2), fma4(d1[1], a1.w, w3);
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const float4 h = ld4(&S.h1[sg + 16 * r][4 * ug]);
      const float4 d = make_float4(h.x > 0.0f ? d1[r][0] : 0.0f, h.y > 0.0f ? d1[r][1] : 0.0f,
                                   h.z > 0.0f ? d1[r][2] : 0.0f, h.w > 0.0f ? d1[r][3] : 0.0f);
      *(float4*)&S.d1[sg + 16 * r][4 * ug] = d;
      gb1[0] += d.x, gb1[1] += d.y, gb1[2] += d.z, gb1[3] += d.w;
    }
    // dW2: units 4 sg.., inputs 4 ug..
#pragma unroll 4
    for (int t = 0; t < kS; ++t) {
      const float4 a = ld4(&S.d2[t][4 * sg]), h = ld4(&S.h1[t][4 * ug]);
      fma4(g2[0], a.x, h), fma4(g2[1], a.y, h), fma4(g2[2], a.z, h), fma4(g2[3], a.w, h);
    }
    __syncthreads();
    // dW1: unit tid / 4, inputs 3 (tid % 4)..
#pragma unroll 8
    for (int t = 0; t < kS; ++t) {
      const float a = S.d1[t][tid >> 2];
#pragma unroll
      for (int k = 0; k < 3; ++k) g1[k] = fmaf(a, S.x[t][3 * (tid & 3) + k], g1[k]);
    }
  }
  // sums to global memory; those over the sample groups are added up in shared memory first
  const bool vec = ((uintptr_t)grad & 15u) == 0;
#pragma unroll
  for (int c = 0; c < 4; ++c) add4(&grad[kOW2 + (4 * sg + c) * kH + 4 * ug], g2[c], vec);
#pragma unroll
  for (int k = 0; k < 3; ++k) atomicAdd(&grad[kOW1 + 3 * tid + k], g1[k]);
  __syncthreads();
  float* red = &S.h1[0][0];  // [4][16][68]: gb2, gw3 at units ug + 16 c, gb1 at 4 ug + c; h1, d2, d1
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    red[sg * kRow + ug + 16 * c] = gb2[c];
    red[(16 + sg) * kRow + ug + 16 * c] = gw3[c];
    red[(32 + sg) * kRow + 4 * ug + c] = gb1[c];
  }
  if (ug == 0) {
    red[(48 + sg) * kRow] = gb3;
    red[(48 + sg) * kRow + 1] = lsum;
  }
  __syncthreads();
  if (tid < 3 * kH) {
    const int which = tid / kH, u = tid % kH;
    float a = 0.0f;
    for (int q = 0; q < 16; ++q) a += red[(16 * which + q) * kRow + u];
    atomicAdd(&grad[(which == 0 ? kOB2 : which == 1 ? kOW3 : kOB1) + u], a);
  } else if (tid < 3 * kH + 2) {
    const int which = tid - 3 * kH;
    float a = 0.0f;
    for (int q = 0; q < 16; ++q) a += red[(48 + q) * kRow + which];
    atomicAdd(which == 0 ? &grad[kOB3] : loss, a);
  }
}

__global__ void k_gate_adam(float* w, float* m, float* v, const float* g, int64_t n, float lr,
                            float b1, float b2, float eps, float c1, float c2) {
  pdl_sync();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

}  // namespace

cudaError_t launch_gate_grad(const float* w, const float* X, const float* y, int64_t n,
                             float* grad, float* loss, int sms, cudaStream_t s) {
  launch_pdl(k_gate_zero, (kGateParams + 1 + 255) / 256, 256, 0, s, grad, loss);
  const int64_t tiles = (n + kS - 1) / kS;
  const int64_t most = (int64_t)kGradBlocksPerSm * sms;
  const int grid = (int)(tiles < most ? tiles : most);
  if (grid > 0) launch_pdl(k_gate_grad, grid, kGradThreads, 0, s, w, X, y, n, grad, loss);
  return cudaGetLastError();
}

cudaError_t launch_gate_adam(float* w, float* m, float* v, const float* g, int64_t n, float lr,
                             float b1, float b2, float eps, int step, cudaStream_t s) {
  const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
  launch_pdl(k_gate_adam, (int)((n + 255) / 256), 256, 0, s, w, m, v, g, n, lr, b1, b2, eps, c1,
             c2);
  return cudaGetLastError();
}

}  // namespace ptca
