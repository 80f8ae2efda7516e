// Training of the chemistry network: targets, loss, the element-wise parts of the backward
// pass and the Adam update. The GEMMs of the backward pass (weight gradients dZ^T H and input
// gradients dZ W, the latter scaled by GELU'(z) in its epilogue) run on the same tcgen05
// kernels as the forward pass (mlp_tc.cu, mlp_split.cu).
#include "dfgb_internal.cuh"
#include "planes.cuh"

#include <cuda_bf16.h>

#include <algorithm>

namespace dfgb {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxBlocks = kTrainScratchFloats;   // element-wise grids, one loss partial each

// BC(yt) - BC(y) for the Box-Cox transform BC(x) = (x^l - 1) / l. When both are positive
// it is formed as y^l expm1(l ln(yt / y)) / l: the difference yt - y in FP64 (no cancellation
// of two nearly equal values), its ratio to y as a correctly rounded FP32 division, the rest in
// FP32. That keeps the difference itself to ~2e-7 relative; GB300's FP64 division would cost
// more than the rest of the kernel.
__device__ __forceinline__ float dboxcox(double y, double yt, float lam) {
  if (y > 0.0 && yt > 0.0) {
    const float yf = (float)y;
    const float q = __fdiv_rn((float)(yt - y), yf);
    const float lr = (q > -0.5f && q < 1.0f) ? log1pf(q) : logf(__fdiv_rn((float)yt, yf));
    return powf(yf, lam) * expm1f(lam * lr) / lam;
  }
  const float a = yt > 0.0 ? powf((float)yt, lam) : 0.0f;
  const float b = y > 0.0 ? powf((float)y, lam) : 0.0f;
  return (a - b) / lam;
}

// Ohat[b][k] = (BC(Yt) - BC(Y) - out_mean_k) / out_std_k, FP32 [B x ldh], zero pad. A thread
// per state and group of four species (block y): the FP64 reads of Y and Yt are coalesced across the
// batch, and each thread writes 16 bytes of its row (ldh a multiple of 4). With all of a state's groups
// in one thread too few reads were in flight: 65,536 states of 30 species 39 -> 28 us.
__global__ void targets_kernel(EosParams P, int64_t B, const double* __restrict__ Y,
                               const double* __restrict__ Yt, int64_t ldY,
                               const double* __restrict__ norm, float* __restrict__ Oh,
                               int64_t ldh) {
  const int n = P.n, K0 = P.K0;
  const float lam = (float)P.lambda;
  __shared__ float mean_f[64], std_f[64];
  for (int k = threadIdx.x; k < n && k < 64; k += blockDim.x) {
    mean_f[k] = (float)norm[2 * K0 + k];
    std_f[k] = (float)norm[2 * K0 + n + k];
  }
  __syncthreads();
  const int k0 = 4 * blockIdx.y;
  for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < B;
       b += (int64_t)gridDim.x * blockDim.x) {
    float v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int k = k0 + j;
      v[j] = 0.0f;
      if (k < n) {
        const float du = dboxcox(Y[k * ldY + b], Yt[k * ldY + b], lam);
        v[j] = (du - mean_f[k]) / std_f[k];
      }
    }
    *reinterpret_cast<float4*>(Oh + b * ldh + k0) = make_float4(v[0], v[1], v[2], v[3]);
  }
}

// dO = 2 (O - Ohat) / B (columns >= n zero); part[block] = this block's share of
// sum (O - Ohat)^2 / B (summed in a fixed order by sum_parts_warp_kernel, so the loss is
// reproducible run to run).
template <typename GT>
__global__ void loss_grad_kernel(int64_t B, int n, const float* __restrict__ O, int64_t ldo,
                                 const float* __restrict__ Oh, int64_t ldh, GT* __restrict__ dO,
                                 int64_t ldd, float invB, float* __restrict__ part) {
  __shared__ float red[kThreads / 32];
  float acc = 0.0f;
  const int64_t total = B * ldd;
  const bool narrow = total < (int64_t)1 << 32;   // 32-bit divisions (65,536 x 32: 14.5 -> 11.7 us)
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = narrow ? (int64_t)((uint32_t)e / (uint32_t)ldd) : e / ldd;
    const int k = (int)(e - b * ldd);
    float g = 0.0f;
    if (k < n) {
      const float r = O[b * ldo + k] - Oh[b * ldh + k];
      acc = fmaf(r * r, invB, acc);
      g = 2.0f * r * invB;
    }
    dO[e] = (GT)g;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.0f;
    for (int w = 0; w < kThreads / 32; ++w) s += red[w];
    part[blockIdx.x] = s;
  }
}

// part[y * C + c] = sum over the rows y, y + gridDim.y, ... of column c of a matrix of NP BF16 planes
// (value = sum of the planes), FP32, in a fixed order: the bias gradient. Block x takes 256 columns, a
// warp one row at a time (512 contiguous bytes a plane), eight columns a lane.
// Bound by the reads of the gradients: eight rows in flight a warp, up to eight blocks an SM, of which the
// scratch for the partial sums leaves 64 a strip: under three for 1600 columns (65,536 rows of 1600 columns
// 61 -> 43 us, 4.8 TB/s, of 800 columns 32 -> 26 us, with four rows in flight and at most four blocks before).
template <int NP>
__global__ void __launch_bounds__(256) colsum_kernel(int64_t R, int64_t C,
                                                     const __nv_bfloat16* __restrict__ in, int64_t ld,
                                                     int64_t plane, float* __restrict__ part) {
  __shared__ float red[8][256];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t c = (int64_t)blockIdx.x * 256 + 8 * lane;
  float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  if (c < ld) {   // ld is a multiple of 8: whole 16-byte groups inside the row
    const int64_t step = (int64_t)gridDim.y * 8;
    constexpr int U = NP == 1 ? 8 : 4;   // rows in flight
    for (int64_t r0 = blockIdx.y * 8 + w; r0 < R; r0 += U * step) {
      uint4 q[U][NP];
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int p = 0; p < NP; ++p)
          q[u][p] = r0 + u * step < R
                        ? *reinterpret_cast<const uint4*>(in + p * plane + (r0 + u * step) * ld + c)
                        : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int p = NP - 1; p >= 0; --p) {
          const uint32_t x[4] = {q[u][p].x, q[u][p].y, q[u][p].z, q[u][p].w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {   // BF16 is the upper half of FP32
            v[2 * e] += __uint_as_float(x[e] << 16);
            v[2 * e + 1] += __uint_as_float(x[e] & 0xFFFF0000u);
          }
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) s[e] += v[e];
      }
    }
  }
#pragma unroll
  for (int e = 0; e < 8; ++e) red[w][8 * lane + e] = s[e];
  __syncthreads();
  const int64_t col = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (col < C) {
    float t = 0.0f;
    for (int k = 0; k < 8; ++k) t += red[k][threadIdx.x];
    part[(int64_t)blockIdx.y * C + col] = t;
  }
}

// out[i] = sum_{s < splits} part[s * stride + i], in order of s.
__global__ void split_sum_kernel(int splits, int64_t count, int64_t stride,
                                 const float* __restrict__ part, float* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x) {
    float s = 0.0f;
    for (int k = 0; k < splits; ++k) s += part[k * stride + i];
    out[i] = s;
  }
}

// out[c] = sum_{j < parts} part[j * C + c] with one warp per c: lane l sums parts l, l + 32, ...
// in order, then the lanes combine in a fixed butterfly, so the result is the same every run.
__global__ void sum_parts_warp_kernel(int parts, int C, const float* __restrict__ part,
                                      float* __restrict__ out) {
  const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (c >= C) return;
  float s = 0.0f;
  for (int j = lane; j < parts; j += 32) s += part[(int64_t)j * C + c];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) out[c] = s;
}

// Adam (Kingma & Ba 2015) on one parameter: m, v moving averages of g and g^2, bias corrections
// c1 = 1 - b1^t, c2 = 1 - b2^t, w -= lr (m / c1) / (sqrt(v / c2) + eps).
struct AdamStep {
  float lr, b1, b2, eps, c1, c2;
  __device__ __forceinline__ void operator()(float& w, float& m, float& v, float g) const {
    m = fmaf(b1, m, (1.0f - b1) * g);
    v = fmaf(b2, v, (1.0f - b2) * g * g);
    w -= lr * (m / c1) / (sqrtf(v / c2) + eps);
  }
};

// Every layer's update and its working copies in one launch (they were an update and a bias update per
// layer, then a copy kernel per layer: twelve launches, 66 us of a step on the four-layer network). A work
// item is four weights of a row (16-byte accesses) or four biases.
__global__ void __launch_bounds__(kThreads) adam_kernel(const __grid_constant__ AdamArgs a, AdamStep step) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < a.items;
       t += (int64_t)gridDim.x * blockDim.x) {
    int l = 0;
    while (l + 1 < a.L && t >= a.layer[l + 1].first) ++l;
    const AdamLayer& y = a.layer[l];
    int64_t i = t - y.first;
    const int64_t quads = y.N * y.ld / 4;
    if (i >= quads) {   // biases
      const int64_t c0 = 4 * (i - quads);
      for (int64_t c = c0; c < c0 + 4 && c < y.N; ++c) step(y.b[c], y.mb[c], y.vb[c], y.gb[c]);
      continue;
    }
    float4 w = reinterpret_cast<const float4*>(y.W)[i], m = reinterpret_cast<const float4*>(y.m)[i];
    float4 v = reinterpret_cast<const float4*>(y.v)[i];
    float4 g = reinterpret_cast<const float4*>(y.g)[i];
    const int64_t per_row = y.ld / 4, r = i / per_row, c = 4 * (i - r * per_row);
    if (c + 3 >= y.K) {   // pad columns hold another layer's sums
      if (c >= y.K) g.x = 0.0f;
      if (c + 1 >= y.K) g.y = 0.0f;
      if (c + 2 >= y.K) g.z = 0.0f;
      g.w = 0.0f;
    }
    step(w.x, m.x, v.x, g.x);
    step(w.y, m.y, v.y, g.y);
    step(w.z, m.z, v.z, g.z);
    step(w.w, m.w, v.w, g.w);
    reinterpret_cast<float4*>(y.W)[i] = w;
    reinterpret_cast<float4*>(y.m)[i] = m;
    reinterpret_cast<float4*>(y.v)[i] = v;
    if (y.Wb) {
      __align__(8) __nv_bfloat16 h[4] = {__float2bfloat16_rn(w.x), __float2bfloat16_rn(w.y),
                                         __float2bfloat16_rn(w.z), __float2bfloat16_rn(w.w)};
      *reinterpret_cast<uint2*>((__nv_bfloat16*)y.Wb + r * y.ldb + c) = *reinterpret_cast<const uint2*>(h);
    }
    if (y.W32) reinterpret_cast<float4*>(y.W32)[i] = w;
    if (y.Wp) {
      __align__(8) __nv_bfloat16 h[3][4];
      split_one(w.x, h[0][0], h[1][0], h[2][0]);
      split_one(w.y, h[0][1], h[1][1], h[2][1]);
      split_one(w.z, h[0][2], h[1][2], h[2][2]);
      split_one(w.w, h[0][3], h[1][3], h[2][3]);
#pragma unroll
      for (int p = 0; p < 3; ++p)
        *reinterpret_cast<uint2*>((__nv_bfloat16*)y.Wp + (p * (int64_t)y.N + r) * y.ldp + c) =
            *reinterpret_cast<const uint2*>(h[p]);
    }
  }
}

int blocks_for(int64_t work) {
  int64_t b = (work + kThreads - 1) / kThreads;
  if (b < 1) b = 1;
  return (int)(b < kMaxBlocks ? b : kMaxBlocks);
}

}  // namespace

cudaError_t launch_train_targets(const EosParams& P, int64_t B, const double* Y, const double* Yt,
                                 int64_t ldY, float* Oh, int64_t ldh, cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  if ((ldh & 3) || P.n > 64) return cudaErrorInvalidValue;
  targets_kernel<<<dim3(blocks_for(B), (unsigned)(ldh / 4)), kThreads, 0, st>>>(P, B, Y, Yt, ldY, P.norm, Oh, ldh);
  return cudaGetLastError();
}

cudaError_t launch_loss_grad(int64_t B, int n, const float* O, int64_t ldo, const float* Oh,
                             int64_t ldh, void* dO, int64_t ldd, bool bf16, float* loss,
                             float* scratch, cudaStream_t st) {
  if (B <= 0) return cudaMemsetAsync(loss, 0, sizeof(float), st);
  const float invB = 1.0f / (float)B;
  // few enough partial sums for the one warp that adds them (4096 took it 10 us)
  const int g = std::min(blocks_for(B * ldd), 640);
  if (bf16)
    loss_grad_kernel<__nv_bfloat16><<<g, kThreads, 0, st>>>(B, n, O, ldo, Oh, ldh,
                                                            (__nv_bfloat16*)dO, ldd, invB, scratch);
  else
    loss_grad_kernel<float><<<g, kThreads, 0, st>>>(B, n, O, ldo, Oh, ldh, (float*)dO, ldd, invB,
                                                    scratch);
  sum_parts_warp_kernel<<<1, 32, 0, st>>>(g, 1, scratch, loss);
  return cudaGetLastError();
}

cudaError_t launch_colsum(int64_t R, int64_t C, const void* in, int64_t ld, int planes, int64_t plane,
                          float* out, int num_sms, float* scratch, int64_t scratch_floats,
                          cudaStream_t st) {
  if (C <= 0) return cudaSuccess;
  if ((ld & 7) || scratch_floats < C) return cudaErrorInvalidValue;
  const int64_t strips = (C + 255) / 256;
  int64_t groups = std::max<int64_t>(1, std::min<int64_t>((R + 63) / 64, (8LL * std::max(num_sms, 1) + strips - 1) / strips));
  groups = std::min<int64_t>(groups, scratch_floats / C);
  const dim3 grid((unsigned)strips, (unsigned)groups);
  if (planes == 1) colsum_kernel<1><<<grid, 256, 0, st>>>(R, C, (const __nv_bfloat16*)in, ld, plane, scratch);
  else colsum_kernel<3><<<grid, 256, 0, st>>>(R, C, (const __nv_bfloat16*)in, ld, plane, scratch);
  sum_parts_warp_kernel<<<(unsigned)((C + 7) / 8), 256, 0, st>>>((int)groups, (int)C, scratch, out);
  return cudaGetLastError();
}

cudaError_t launch_sum_splits(int splits, int64_t count, int64_t stride, const float* part,
                              float* out, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  split_sum_kernel<<<blocks_for(count), kThreads, 0, st>>>(splits, count, stride, part, out);
  return cudaGetLastError();
}

cudaError_t launch_adam(AdamArgs a, float lr, float b1, float b2, float eps, float c1, float c2,
                        int num_sms, cudaStream_t st) {
  int64_t t = 0;
  for (int l = 0; l < a.L; ++l) {
    a.layer[l].first = t;
    t += a.layer[l].N * a.layer[l].ld / 4 + (a.layer[l].N + 3) / 4;
  }
  a.items = t;
  const int64_t g = std::max<int64_t>(1, std::min<int64_t>((t + kThreads - 1) / kThreads, 8LL * num_sms));
  adam_kernel<<<(unsigned)g, kThreads, 0, st>>>(a, AdamStep{lr, b1, b2, eps, c1, c2});
  return cudaGetLastError();
}

}  // namespace dfgb
