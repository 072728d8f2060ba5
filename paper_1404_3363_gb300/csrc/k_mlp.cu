// Learned initial guess for the inverse geometry map (not in the paper): per
// block, a 3-64-64-3 perceptron with ReLU hidden layers maps a world point
// normalised to the block's control-point box, g_hat = (g - c) / h per axis, to a
// parameter-space guess p_hat.  It is trained on samples of the forward map
// the method itself evaluates (p uniform in [0,1]^3, g = phi(p)).
//
//   K7a mlp_samples  -- counter-based uniform p per (block, index), g = phi(p)
//   K7b mlp_fwd_bwd  -- forward, squared-error loss and backward for one
//                       mini-batch, 32 samples per CTA and tile; the weight
//                       gradients of a CTA's samples are summed in registers
//                       into one partial gradient per CTA (no atomics, so
//                       training is deterministic)
//   K7c mlp_reduce   -- sums the partial gradients; in training also applies
//                       Adam and refreshes the FP16 copy used for inference
// The inference (K6) is in k_mlp_tc.cu.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "ivv_device.cuh"
#include "mlp.cuh"

namespace ivv {

namespace {

// ----------------------------------------------------------- sampling
__device__ __forceinline__ unsigned hash32(unsigned x) {
  x ^= x >> 16;
  x *= 0x7feb352du;
  x ^= x >> 15;
  x *= 0x846ca68bu;
  x ^= x >> 16;
  return x;
}

__device__ __forceinline__ float unit_float(unsigned long long seed, unsigned a, unsigned b, unsigned c) {
  unsigned h = hash32((unsigned)seed ^ hash32(a * 0x9e3779b9u ^ hash32(b + 0x632be5abu * c + (unsigned)(seed >> 32))));
  return ((h >> 8) + 0.5f) * (1.0f / 16777216.0f);
}

template <int P>
__global__ void k_mlp_samples(DevVolume V, MlpNorm norm, int block, int S, unsigned long long seed,
                              float4* __restrict__ x_out, float4* __restrict__ p_out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= S) return;
  float p[3] = {unit_float(seed, block, i, 0), unit_float(seed, block, i, 1), unit_float(seed, block, i, 2)};
  const BlockInfo B = V.blocks[block];
  float phi[3], J[3][3], rho;
  eval_block<P, float, false>(V, B, p, phi, J, rho);
  x_out[i] = make_float4((phi[0] - norm.c[0]) * norm.inv_h[0], (phi[1] - norm.c[1]) * norm.inv_h[1],
                         (phi[2] - norm.c[2]) * norm.inv_h[2], 0.f);
  p_out[i] = make_float4(p[0], p[1], p[2], 0.f);
}

// ----------------------------------------------------------- training
// A step is a chain of two short kernels, so its time is their latency: 32
// samples per tile put the default batch of 4096 on 128 SMs (one tile of 128
// samples per CTA and one thread per sample held 32 SMs, with two shared
// memory reads per multiply-add).  The three 64 x 64 products of a tile are
// register tiles fed by 128-bit shared memory reads (six reads for 32
// multiply-adds in the two passes over W2, two for 16 in its gradient), rows
// padded so that they meet no bank conflict.  The second kernel sums the
// partial gradients and takes the Adam step.
// 128 steps of batch 4096 on the bar: 7.51 ms before, 1.65 now (kernels: 46 + 3.6 + 4 us a step, then 11 + 4).
constexpr int kTrainThreads = 256;
constexpr int kTile = 32;               // samples per tile
constexpr int kLd = kMlpH + 4;          // padded row stride (16-byte aligned rows, shifted by 4 banks)
constexpr int kPartial = kMlpParams + 1;   // a partial gradient and its loss
constexpr int kTrainCtas = 1024;        // at most (beyond, a CTA takes several tiles)

static_assert(kTrainThreads == 4 * kMlpH && kOffW2 % 4 == 0 && kMlpStride % 4 == 0, "weight loads of the training kernel");

struct TrainSmem {
  float w2[kMlpH][kLd];
  float h1[kTile][kLd], h2[kTile][kLd], d1[kTile][kLd], d2[kTile][kLd];   // activations and their gradients
  float w1[kMlpH * 3], b1[kMlpH], b2[kMlpH], w3[3 * kMlpH], b3[4];
  float4 x[kTile], dy[kTile];           // dy.w: the sample's loss
};

__device__ __forceinline__ float4 lds4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void fma4(float& acc, const float4& a, const float4& b) {
  acc = fmaf(a.x, b.x, acc);
  acc = fmaf(a.y, b.y, acc);
  acc = fmaf(a.z, b.z, acc);
  acc = fmaf(a.w, b.w, acc);
}

// Forward and backward of samples [first, first + n) (indices mod S), tile
// after tile; each CTA's gradient and loss sums to partial[cta][kPartial].
// scale is the 1/N of the mean over the whole batch.  GRAD = false: the loss
// alone.
template <bool GRAD>
__global__ void __launch_bounds__(kTrainThreads) k_mlp_fwd_bwd(const float* __restrict__ theta,
                                                               const float4* __restrict__ xs,
                                                               const float4* __restrict__ ps, int S, int first,
                                                               int n, float scale, float* __restrict__ partial) {
  extern __shared__ float4 smem_raw[];
  TrainSmem& sm = *reinterpret_cast<TrainSmem*>(smem_raw);
  const int tid = threadIdx.x;
  pdl_wait();
  // every load of the weights in flight at once (parameter vectors start on
  // 16-byte boundaries)
  {
    const float4* w2 = reinterpret_cast<const float4*>(theta + kOffW2);
    float4 w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = w2[tid + kTrainThreads * q];
    const float wa = tid < 3 * kMlpH ? theta[kOffW1 + tid] : theta[kOffB1 + tid - 3 * kMlpH];
    const float wb = tid < 3 * kMlpH ? theta[kOffW3 + tid] : theta[kOffB2 + tid - 3 * kMlpH];
    if (tid < 3) sm.b3[tid] = theta[kOffB3 + tid];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = 4 * (tid + kTrainThreads * q);
      *reinterpret_cast<float4*>(&sm.w2[i / kMlpH][i % kMlpH]) = w[q];
    }
    (tid < 3 * kMlpH ? sm.w1[tid] : sm.b1[tid - 3 * kMlpH]) = wa;
    (tid < 3 * kMlpH ? sm.w3[tid] : sm.b2[tid - 3 * kMlpH]) = wb;
  }
  // thread tiles: (2 samples) x (4 outputs ig + 16 q, or 4 kg ..), and the
  // 4 x 4 block of W2's gradient at (4 rg, 4 kg)
  const int kg = tid & 15, rg = tid >> 4, s0 = 2 * rg;
  const int sp = tid >> 3, kp = 8 * (tid & 7);        // layer 3: eight threads per sample
  float g2[4][4] = {}, g_b = 0.f, g_a = 0.f, g_3 = 0.f, loss = 0.f;
  const unsigned tiles = ((unsigned)n + kTile - 1) / kTile;
  for (unsigned tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    __syncthreads();                                  // weights loaded; the last tile's rows are free
    if (tid < kTile) {
      const unsigned local = tile * kTile + tid;
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f), t = x;
      if (local < (unsigned)n) {
        const unsigned idx = ((unsigned)first + local) % (unsigned)S;
        x = xs[idx];
        t = ps[idx];
        x.w = 1.f;
      } else {
        x.w = 0.f;
      }
      sm.x[tid] = x;
      sm.dy[tid] = t;                                 // the target until layer 3 replaces it
    }
    __syncthreads();
    // layer 1
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = kg + 16 * q;
      const float wa = sm.w1[3 * i], wb = sm.w1[3 * i + 1], wc = sm.w1[3 * i + 2], bb = sm.b1[i];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const float4 x = sm.x[s0 + r];
        const float z = bb + wa * x.x + wb * x.y + wc * x.z;
        sm.h1[s0 + r][i] = z > 0.f ? z : 0.f;
      }
    }
    __syncthreads();
    // layer 2: rows i = kg + 16 q of W2
    {
      float z[2][4];
#pragma unroll
      for (int q = 0; q < 4; ++q) z[0][q] = z[1][q] = sm.b2[kg + 16 * q];
#pragma unroll 4
      for (int k = 0; k < kMlpH; k += 4) {
        const float4 ha = lds4(&sm.h1[s0][k]), hb = lds4(&sm.h1[s0 + 1][k]);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 w = lds4(&sm.w2[kg + 16 * q][k]);
          fma4(z[0][q], w, ha);
          fma4(z[1][q], w, hb);
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int r = 0; r < 2; ++r) sm.h2[s0 + r][kg + 16 * q] = z[r][q] > 0.f ? z[r][q] : 0.f;
    }
    __syncthreads();
    // layer 3, the error, and the gradient of the second hidden layer
    {
      const float4 ha = lds4(&sm.h2[sp][kp]), hb = lds4(&sm.h2[sp][kp + 4]);
      const float4 t = sm.dy[sp];
      float y[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        float z = 0.f;
        fma4(z, lds4(&sm.w3[c * kMlpH + kp]), ha);
        fma4(z, lds4(&sm.w3[c * kMlpH + kp + 4]), hb);
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
        y[c] = z + sm.b3[c];
      }
      const bool in = sm.x[sp].w != 0.f;
      const float ex = in ? y[0] - t.x : 0.f, ey = in ? y[1] - t.y : 0.f, ez = in ? y[2] - t.z : 0.f;
      const float dx = 2.f * ex * scale, dy = 2.f * ey * scale, dz = 2.f * ez * scale;
      __syncwarp();                                   // every lane has read its sample's target
      if (kp == 0) sm.dy[sp] = make_float4(dx, dy, dz, (ex * ex + ey * ey + ez * ez) * scale);
      if (GRAD) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const float h = k < 4 ? (&ha.x)[k] : (&hb.x)[k - 4];
          const float g = sm.w3[kp + k] * dx + sm.w3[kMlpH + kp + k] * dy + sm.w3[2 * kMlpH + kp + k] * dz;
          sm.d2[sp][kp + k] = h > 0.f ? g : 0.f;
        }
      }
    }
    __syncthreads();
    if (tid == kTrainThreads - 1) {
#pragma unroll 8
      for (int r = 0; r < kTile; ++r) loss += sm.dy[r].w;
    }
    if (!GRAD) continue;
    // gradient of the first hidden layer: columns 4 kg .. of W2
    {
      float z[2][4] = {};
#pragma unroll 4
      for (int i = 0; i < kMlpH; i += 4) {
        const float4 ga = lds4(&sm.d2[s0][i]), gb = lds4(&sm.d2[s0 + 1][i]);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float4 w = lds4(&sm.w2[i + u][4 * kg]);
          const float a = (&ga.x)[u], b = (&gb.x)[u];
          z[0][0] = fmaf(w.x, a, z[0][0]); z[0][1] = fmaf(w.y, a, z[0][1]);
          z[0][2] = fmaf(w.z, a, z[0][2]); z[0][3] = fmaf(w.w, a, z[0][3]);
          z[1][0] = fmaf(w.x, b, z[1][0]); z[1][1] = fmaf(w.y, b, z[1][1]);
          z[1][2] = fmaf(w.z, b, z[1][2]); z[1][3] = fmaf(w.w, b, z[1][3]);
        }
      }
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const float4 h = lds4(&sm.h1[s0 + r][4 * kg]);
        float4 d;
        d.x = h.x > 0.f ? z[r][0] : 0.f;
        d.y = h.y > 0.f ? z[r][1] : 0.f;
        d.z = h.z > 0.f ? z[r][2] : 0.f;
        d.w = h.w > 0.f ? z[r][3] : 0.f;
        *reinterpret_cast<float4*>(&sm.d1[s0 + r][4 * kg]) = d;
      }
    }
    // dW2[i][k] = sum_s d2[s][i] h1[s][k]
#pragma unroll 8
    for (int r = 0; r < kTile; ++r) {
      const float4 gi = lds4(&sm.d2[r][4 * rg]), hk = lds4(&sm.h1[r][4 * kg]);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float a = (&gi.x)[u];
        g2[u][0] = fmaf(a, hk.x, g2[u][0]); g2[u][1] = fmaf(a, hk.y, g2[u][1]);
        g2[u][2] = fmaf(a, hk.z, g2[u][2]); g2[u][3] = fmaf(a, hk.w, g2[u][3]);
      }
    }
    // dW3 (threads 0..191), db2 (192..255), db3 (0..2)
    if (tid < 3 * kMlpH) {
      const int c = tid / kMlpH, k = tid % kMlpH;
#pragma unroll 8
      for (int r = 0; r < kTile; ++r) g_a = fmaf((&sm.dy[r].x)[c], sm.h2[r][k], g_a);
    } else {
#pragma unroll 8
      for (int r = 0; r < kTile; ++r) g_a += sm.d2[r][tid - 3 * kMlpH];
    }
    if (tid < 3) {
#pragma unroll 8
      for (int r = 0; r < kTile; ++r) g_3 += (&sm.dy[r].x)[tid];
    }
    __syncthreads();
    // dW1 (threads 0..191), db1 (192..255)
    if (tid < 3 * kMlpH) {
      const int i = tid / 3, c = tid % 3;
#pragma unroll 8
      for (int r = 0; r < kTile; ++r) g_b = fmaf(sm.d1[r][i], (&sm.x[r].x)[c], g_b);
    } else {
#pragma unroll 8
      for (int r = 0; r < kTile; ++r) g_b += sm.d1[r][tid - 3 * kMlpH];
    }
  }
  float* out = partial + (size_t)blockIdx.x * kPartial;
  if (tid == kTrainThreads - 1) out[kMlpParams] = loss;
  if (!GRAD) return;
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int k = 0; k < 4; ++k) out[kOffW2 + (4 * rg + u) * kMlpH + 4 * kg + k] = g2[u][k];
  out[tid < 3 * kMlpH ? kOffW3 + tid : kOffB2 + tid - 3 * kMlpH] = g_a;
  out[tid < 3 * kMlpH ? kOffW1 + tid : kOffB1 + tid - 3 * kMlpH] = g_b;
  if (tid < 3) out[kOffB3 + tid] = g_3;
}

// Sums the per-CTA partial gradients (fixed order, so training is
// deterministic): a lane per parameter, the partials split over eight warps.
// ADAM: then Adam (Kingma & Ba) on the parameter and its FP16 inference copy;
// else the gradient.  `from`: the first parameter (kMlpParams: the loss only).
template <bool ADAM>
__global__ void __launch_bounds__(256) k_mlp_reduce(const float* __restrict__ partial, int nparts, int from,
                                                    float* __restrict__ grad, float* __restrict__ loss,
                                                    float* __restrict__ theta, float* __restrict__ m,
                                                    float* __restrict__ v, float lr, float b1, float b2, float eps,
                                                    float bc1, float bc2, __half* __restrict__ theta16) {
  __shared__ float s_part[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i = from + blockIdx.x * 32 + lane;
  pdl_wait();
  float m0 = 0.f, v0 = 0.f, t0 = 0.f;
  if (ADAM && w == 0 && i < kMlpParams) {
    m0 = m[i];
    v0 = v[i];
    t0 = theta[i];
  }
  float acc = 0.f;
  if (i <= kMlpParams) {
#pragma unroll 16
    for (int c = w; c < nparts; c += 8) acc += partial[(size_t)c * kPartial + i];
  }
  s_part[w][lane] = acc;
  __syncthreads();
  if (w != 0 || i > kMlpParams) return;
  float g = 0.f;
#pragma unroll
  for (int k = 0; k < 8; ++k) g += s_part[k][lane];
  if (i == kMlpParams) {
    *loss = g;
    return;
  }
  if constexpr (ADAM) {
    const float mi = b1 * m0 + (1.f - b1) * g;
    const float vi = b2 * v0 + (1.f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    const float t = t0 - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
    theta[i] = t;
    theta16[i] = __float2half_rn(t);
  } else {
    grad[i] = g;
  }
}

__global__ void k_mlp_to_half(const float* __restrict__ theta, __half* __restrict__ theta16, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) theta16[i] = __float2half_rn(theta[i]);
}

}  // namespace

void launch_mlp_samples(const DevVolume& V, const MlpNorm& norm, int block, int S, unsigned long long seed,
                        float4* x_out, float4* p_out, cudaStream_t s) {
  if (V.P == 2)
    k_mlp_samples<2><<<(S + 255) / 256, 256, 0, s>>>(V, norm, block, S, seed, x_out, p_out);
  else
    k_mlp_samples<3><<<(S + 255) / 256, 256, 0, s>>>(V, norm, block, S, seed, x_out, p_out);
}

int mlp_train_ctas(int n) {
  const int tiles = n / kTile + (n % kTile != 0);
  return tiles < kTrainCtas ? tiles : kTrainCtas;
}

size_t mlp_partial_floats(int n) { return (size_t)mlp_train_ctas(n) * kPartial; }

cudaError_t launch_mlp_fwd_bwd(const float* theta, const float4* xs, const float4* ps, int S, int first, int n,
                               float scale, bool want_grad, float* partial, cudaStream_t s) {
  // per device and cheap: set on every call rather than remembered per process
  auto kern = want_grad ? k_mlp_fwd_bwd<true> : k_mlp_fwd_bwd<false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem));
  if (e != cudaSuccess) return e;
  launch_pdl_smem(kern, dim3(mlp_train_ctas(n)), dim3(kTrainThreads), sizeof(TrainSmem), s, theta, xs, ps, S, first, n,
                  scale, partial);
  return cudaGetLastError();
}

void launch_mlp_reduce(const float* partial, int nparts, bool want_grad, float* grad, float* loss, cudaStream_t s) {
  const int from = want_grad ? 0 : kMlpParams;
  launch_pdl(k_mlp_reduce<false>, dim3((kMlpParams + 1 - from + 31) / 32), dim3(256), s, partial, nparts, from, grad,
             loss, (float*)nullptr, (float*)nullptr, (float*)nullptr, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, (__half*)nullptr);
}

void launch_mlp_adam(const float* partial, int nparts, float* theta, float* m, float* v, float* loss, float lr,
                     int step, __half* theta16, cudaStream_t s) {
  const float b1 = 0.9f, b2 = 0.999f;
  const float bc1 = 1.f - powf(b1, (float)step), bc2 = 1.f - powf(b2, (float)step);
  launch_pdl(k_mlp_reduce<true>, dim3((kMlpParams + 1 + 31) / 32), dim3(256), s, partial, nparts, 0, (float*)nullptr,
             loss, theta, m, v, lr, b1, b2, 1e-8f, bc1, bc2, theta16);
}

void launch_mlp_to_half(const float* theta, __half* theta16, int n, cudaStream_t s) {
  k_mlp_to_half<<<(n + 255) / 256, 256, 0, s>>>(theta, theta16, n);
}


}  // namespace ivv
