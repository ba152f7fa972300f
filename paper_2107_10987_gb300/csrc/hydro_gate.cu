// hydro_gate.cu -- the learned smoothness indicator: training data from the
// method itself (features and limiter-activity labels per cell), and the
// forward, backward and Adam kernels that train the network on the GPU.
//
// Network: 54 -> 32 (ReLU) -> 32 (ReLU) -> 1 (sigmoid).  The master
// parameters are FP32; every forward and backward pass uses them rounded to
// BF16 (the storage precision of the deployed indicator) and accumulates in
// FP32.  Loss: class-weighted binary cross-entropy, mean over the samples.
#include <cuda_bf16.h>

#include <cstdint>

#include "hydro.h"
#include "hydro_ctx.h"
#include "hydro_mixed.cuh"

namespace hyd {

// Significant limiter activity on one line of one field: the limited pair
// differs from the central-slope pair (Delta_j = (delta_{j-1}+delta_j)/2, no
// fix-ups) by more than 1e-4 of the field's scale at the cell.
constexpr float kLabelTol = 1e-4f;

__device__ __forceinline__ bool ppm32_significant(float s0, float s1, float s2, float s3, float s4, float scale) {
  float qp, qm;
  ppm32(s0, s1, s2, s3, s4, qp, qm);
  const float sixth = 1.f / 6.f;
  const float d0 = s1 - s0, d1 = s2 - s1, d2 = s3 - s2, d3 = s4 - s3;
  const float C0 = 0.5f * (d0 + d1), C1 = 0.5f * (d1 + d2), C2 = 0.5f * (d2 + d3);
  const float pu = 0.5f * (s2 + s3) - (C2 - C1) * sixth;
  const float mu = 0.5f * (s1 + s2) - (C1 - C0) * sixth;
  return fmaxf(fabsf(qp - pu), fabsf(qm - mu)) > kLabelTol * scale;
}

struct GateDataArgs {
  const double* U;
  float* X;       // [n_sub*N3][54] or null
  uint8_t* y;     // [n_sub*N3] or null
  int n_sub;
  double eta1;
  float gamma, gm1;
};

// The seven fields that features and labels read (rho, v, eps, tau, species),
// as slots of the shared primitive array.
constexpr int kLabelF = 7;
constexpr int kLabelThreads = 512;

// One CTA of 512 threads per 8^3 sub-grid (77 KB, 2 resident CTAs).  The
// features are written as the contiguous [512][54] block they form, so that a
// warp's stores fill whole 128-byte lines (a thread per cell wrote one value
// to each of 32 rows of 216 bytes per store); the labels, a thread per cell,
// are bound by FP32 issue: 13 lines x 7 fields x the limited and the central
// pair.  A sub-grid whose padded block is one uniform state needs neither:
// every difference is zero, so its features are 0 and its labels 0 (most of a
// blast's mesh; the indicator's step phase skips it likewise).
__global__ void __launch_bounds__(kLabelThreads, 2) hydro_gate_data_kernel(GateDataArgs A) {
  extern __shared__ __align__(128) float Qf[];  // [kLabelF][S3]
  __shared__ int off[kGateIn];                  // feature j's neighbour relative to the cell (field included)
  for (int j = threadIdx.x; j < kGateIn; j += kLabelThreads) off[j] = c_gate_off.off[j];
  for (int s = blockIdx.x; s < A.n_sub; s += gridDim.x) {
    const double* Us = A.U + (size_t)s * F * S3;
    for (int c = threadIdx.x; c < S3; c += kLabelThreads) {
      double u[F];
#pragma unroll
      for (int k = 0; k < F; ++k) u[k] = (k == ZX || k == ZY || k == ZZ) ? 0.0 : __ldg(Us + (size_t)k * S3 + c);
      float q[F];
      prims_mixed(u, A.eta1, A.gamma, q);
#pragma unroll
      for (int k = 0; k < kLabelF; ++k) Qf[k * S3 + c] = q[k < ZX ? k : SP0];
    }
    __syncthreads();
    bool same = Qf[RHO * S3] > 1e-30f && A.gm1 * Qf[EGAS * S3] > 1e-30f;  // 0 / subnormal is left to the division
    for (int c = threadIdx.x; c < S3; c += kLabelThreads)
#pragma unroll
      for (int k = 0; k < kLabelF; ++k) {
        const float d = Qf[k * S3 + c] - Qf[k * S3];  // NaN for infinities
        same &= d == 0.f;
      }
    const bool uniform = __syncthreads_and(same);
    if (A.X) {
      float* X = A.X + (size_t)s * N3 * kGateIn;
      if (uniform && ((uintptr_t)X & 15u) == 0) {
        for (int e = threadIdx.x; e < N3 * kGateIn / 4; e += kLabelThreads)
          reinterpret_cast<float4*>(X)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
      } else
      for (int e = threadIdx.x; e < N3 * kGateIn; e += kLabelThreads) {
        float v = 0.f;
        if (!uniform) {
          const int i = e / kGateIn, j = e - i * kGateIn;
          const int c = (((i >> 6) + G) * S + (((i >> 3) & (N - 1)) + G)) * S + ((i & (N - 1)) + G);
          const float q0 = Qf[(j < 27 ? RHO : EGAS) * S3 + c], q1 = Qf[c + off[j]];
          const float qc = j < 27 ? q0 : A.gm1 * q0, qk = j < 27 ? q1 : A.gm1 * q1;
          v = __fdividef(qk - qc, fabsf(qk) + fabsf(qc));
        }
        X[e] = v;
      }
    }
    if (A.y) {
      const int i = threadIdx.x;
      static_assert(kLabelThreads == N3, "a thread per cell");
      const int c = (((i >> 6) + G) * S + (((i >> 3) & (N - 1)) + G)) * S + ((i & (N - 1)) + G);
      bool fired = false;
      if (!uniform) {
        // scales: |q0| for density, eps, tau, species; |v| + c for velocity
        const float rho0 = Qf[RHO * S3 + c], eps0 = Qf[EGAS * S3 + c];
        const float vs = fabsf(Qf[SX * S3 + c]) + fabsf(Qf[SY * S3 + c]) + fabsf(Qf[SZ * S3 + c]) +
                         sqrtf(A.gamma * A.gm1 * eps0 / rho0);
        // the 13 lines through the cell: d with first non-zero component > 0
#pragma unroll 1
        for (int dz = 0; dz <= 1; ++dz)
#pragma unroll 1
          for (int dy = -1; dy <= 1; ++dy)
#pragma unroll 1
            for (int dx = -1; dx <= 1; ++dx) {
              if (dz == 0 && (dy < 0 || (dy == 0 && dx <= 0))) continue;
              const int st = (dz * S + dy) * S + dx;
#pragma unroll
              for (int k = 0; k < kLabelF; ++k) {  // the spin: always limited, never labelled
                const float* q = Qf + k * S3 + c;
                const float scale = (k >= SX && k <= SZ) ? vs : fabsf(q[0]);
                fired |= ppm32_significant(q[-2 * st], q[-st], q[0], q[st], q[2 * st], scale);
              }
            }
      }
      A.y[(size_t)s * N3 + i] = fired ? 1 : 0;
    }
    __syncthreads();
  }
}

// ---- MLP forward and training ------------------------------------------------
// The training step is FP32 contractions of 64-sample tiles against 54 x 32 and
// 32 x 32 weights, bound by shared-memory reads and the FP32 pipe (its
// parameters are BF16 values, but its activations are not, so the tensor
// cores would need them rounded or split).  A CTA of 128 threads keeps the
// weights and the tile's activations in shared memory and gives each thread
// a 4 x 4 block of a product: 8 float4 reads feed 64 multiply-adds, where a
// thread per sample read two operands per multiply-add.  Rows are padded to
// 60 and 36 floats (28 and 4 banks apart), so that the eight rows a quarter
// of a warp reads as float4 lie on distinct banks.  Measured: a training step
// (gradient, reduction, optimiser) at 65,536 samples 216 -> 47 us.
constexpr int kTile = 128;        // samples per partial of hydro_mlp_work_bytes
constexpr int kMt = 64;           // samples per tile
constexpr int kMThreads = 128;
constexpr int kMStrX = 60, kMStrH = 36;
constexpr int kGradPerSm = 3;     // resident CTAs of the gradient (70 KB each)
constexpr int kFwdPerSm = 4;      // and of the predictions

// Network weights in shared memory, rows padded with zeros: W1 [32][kMStrX],
// W2 [32][kMStrH], then b1, b2, w3 [32] each and b3.
struct MlpSmem {
  static constexpr int w1 = 0, w2 = w1 + kGateH * kMStrX, b1 = w2 + kGateH * kMStrH, b2 = b1 + kGateH,
                       w3 = b2 + kGateH, b3 = w3 + kGateH, end = b3 + 4;
};

__device__ __forceinline__ void mlp_load_weights(const float* __restrict__ params, float* sm) {
  for (int i = threadIdx.x; i < kGateH * kMStrX; i += kMThreads) {
    const int j = i / kMStrX, k = i % kMStrX;
    sm[MlpSmem::w1 + i] = k < kGateIn ? bf16r(params[j * kGateIn + k]) : 0.f;
  }
  for (int i = threadIdx.x; i < kGateH * kMStrH; i += kMThreads) {
    const int j = i / kMStrH, k = i % kMStrH;
    sm[MlpSmem::w2 + i] = k < kGateH ? bf16r(params[kGateW2 + j * kGateH + k]) : 0.f;
  }
  for (int i = threadIdx.x; i < kGateH; i += kMThreads) {
    sm[MlpSmem::b1 + i] = bf16r(params[kGateB1 + i]);
    sm[MlpSmem::b2 + i] = bf16r(params[kGateB2 + i]);
    sm[MlpSmem::w3 + i] = bf16r(params[kGateW3 + i]);
  }
  if (threadIdx.x == 0) sm[MlpSmem::b3] = bf16r(params[kGateB3]);
}

// The tile's features into xs [kMt][kMStrX] (columns 54 .. 59 zero; samples
// past n zero).  vec: X is 8-byte aligned (a tile
// starts at a multiple of 13,824 bytes, a row at a multiple of 216).
__device__ __forceinline__ void mlp_load_tile(const float* __restrict__ X, int tile, int n, bool vec, float* xs) {
  const int live = min(kMt, n - tile * kMt);
  const float* src = X + (size_t)tile * kMt * kGateIn;
  if (vec) {
    const float2* s2 = reinterpret_cast<const float2*>(src);
    for (int i = threadIdx.x; i < kMt * (kMStrX / 2); i += kMThreads) {
      const int s = i / (kMStrX / 2), k = i % (kMStrX / 2);
      float2 v = make_float2(0.f, 0.f);
      if (k < kGateIn / 2 && s < live) v = __ldg(s2 + s * (kGateIn / 2) + k);
      *reinterpret_cast<float2*>(xs + s * kMStrX + 2 * k) = v;
    }
  } else {
    for (int i = threadIdx.x; i < kMt * kMStrX; i += kMThreads) {
      const int s = i / kMStrX, k = i % kMStrX;
      xs[i] = (k < kGateIn && s < live) ? __ldg(src + s * kGateIn + k) : 0.f;
    }
  }
}

// acc[m][o] = sum over k < kK (kK a multiple of 4) of a[row m][k] b[row o][k],
// rows (threadIdx.x / 8) + 16 m of a and (threadIdx.x % 8) + 8 o of b: the
// even and the odd k in the two lanes of packed multiply-adds, added at the
// end.  The first operand of each chain is init[o] (lane 0).
template <int kK, int kSa, int kSb>
__device__ __forceinline__ void mlp_block(const float* __restrict__ a, const float* __restrict__ b,
                                          const float init[4], float acc[4][4]) {
  const float* pa = a + (threadIdx.x >> 3) * kSa;
  const float* pb = b + (threadIdx.x & 7) * kSb;
  float2 s[4][4];
#pragma unroll
  for (int m = 0; m < 4; ++m)
#pragma unroll
    for (int o = 0; o < 4; ++o) s[m][o] = f2(init[o], 0.f);
#pragma unroll
  for (int k = 0; k < kK; k += 4) {
    float4 va[4], vb[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) va[m] = *reinterpret_cast<const float4*>(pa + 16 * m * kSa + k);
#pragma unroll
    for (int o = 0; o < 4; ++o) vb[o] = *reinterpret_cast<const float4*>(pb + 8 * o * kSb + k);
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        s[m][o] = fma2(f2(va[m].x, va[m].y), f2(vb[o].x, vb[o].y), s[m][o]);
        s[m][o] = fma2(f2(va[m].z, va[m].w), f2(vb[o].z, vb[o].w), s[m][o]);
      }
  }
#pragma unroll
  for (int m = 0; m < 4; ++m)
#pragma unroll
    for (int o = 0; o < 4; ++o) acc[m][o] = s[m][o].x + s[m][o].y;
}

// Store the thread's block (rows as mlp_block's) to out [kMt][kMStrH].
__device__ __forceinline__ void mlp_store(float* out, const float v[4][4]) {
  const int r = threadIdx.x >> 3, c = threadIdx.x & 7;
#pragma unroll
  for (int m = 0; m < 4; ++m)
#pragma unroll
    for (int o = 0; o < 4; ++o) out[(r + 16 * m) * kMStrH + c + 8 * o] = v[m][o];
}

// w3 . h2 + b3 of sample s.
__device__ __forceinline__ float mlp_head(const float* sm, const float* h2, int s) {
  float z = sm[MlpSmem::b3];
#pragma unroll
  for (int j = 0; j < kGateH; j += 4) {
    const float4 h = *reinterpret_cast<const float4*>(h2 + s * kMStrH + j);
    const float4 w = *reinterpret_cast<const float4*>(sm + MlpSmem::w3 + j);
    z = fmaf(w.x, h.x, z);
    z = fmaf(w.y, h.y, z);
    z = fmaf(w.z, h.z, z);
    z = fmaf(w.w, h.w, z);
  }
  return z;
}

// Forward only, in the deployed form (BF16 inputs and first hidden layer,
// FP32 accumulation): out[i] = sigmoid(logit(x_i)).  The operands are BF16
// values, so the products are the tensor cores' own: a warp takes 16 samples
// (rows g and g + 8 of the fragments, see gate_tile_mma) and keeps the weights'
// fragments in registers over its tiles.  Each 16-column step starts from zero
// and is added in FP32, so that the sums round no worse than a chain of fused
// multiply-adds: relative error against FP64 of 65,536 predictions on four
// seeds 4.2e-7, 1.2e-6, 2.9e-7, 4.0e-7, with multiply-adds 1.1e-6, 1.3e-6,
// 7.7e-7, 3.8e-7 (it is the BF16 rounding of the hidden layer flipping).  Bound
// by reading X: features, labels and predictions of 512 sub-grids take 89 us,
// with tiled FP32 multiply-adds 161, with a sample per thread 936.
constexpr int kFwdThreads = 128;
__global__ void __launch_bounds__(kFwdThreads, kFwdPerSm) hydro_mlp_forward_kernel(
    const float* __restrict__ params, const float* __restrict__ X, int n, bool vec, float* __restrict__ out) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  GateFrags f;
  gate_load_frags(params, lane, f);
#pragma unroll
  for (int nt = 0; nt < 4; ++nt)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      f.b1[nt][e] = bf16r(f.b1[nt][e]);
      f.b2[nt][e] = bf16r(f.b2[nt][e]);
      f.w3[nt][e] = bf16r(f.w3[nt][e]);
    }
  f.b3 = bf16r(f.b3);
  const int tiles = (n - 1) / 16 + 1, stride = gridDim.x * (kFwdThreads / 32);
  for (int tile = blockIdx.x * (kFwdThreads / 32) + (threadIdx.x >> 5); tile < tiles; tile += stride) {
    const long long r0 = (long long)tile * 16 + g, r1 = r0 + 8;
    const float* x0 = X + min(r0, (long long)n - 1) * kGateIn;
    const float* x1 = X + min(r1, (long long)n - 1) * kGateIn;
    uint32_t a[4][4];
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = 16 * ks + 2 * t + 8 * h;  // columns c, c + 1 (54 is even)
        float2 v0 = f2(0.f), v1 = f2(0.f);
        if (c < kGateIn) {
          if (vec) {
            v0 = __ldg(reinterpret_cast<const float2*>(x0 + c));
            v1 = __ldg(reinterpret_cast<const float2*>(x1 + c));
          } else {
            v0 = f2(__ldg(x0 + c), __ldg(x0 + c + 1));
            v1 = f2(__ldg(x1 + c), __ldg(x1 + c + 1));
          }
        }
        a[ks][2 * h] = pack_bf16x2(v0.x, v0.y);
        a[ks][2 * h + 1] = pack_bf16x2(v1.x, v1.y);
      }
    }
    __syncwarp();  // the matrix instructions are the whole warp's, the loads above each lane's
    float acc[4][4];
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
      acc[nt][0] = acc[nt][2] = f.b1[nt][0];
      acc[nt][1] = acc[nt][3] = f.b1[nt][1];
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) {
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        mma_bf16_16816(d, a[ks], f.w1[ks][nt][0], f.w1[ks][nt][1]);
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[nt][e] += d[e];
      }
    }
    uint32_t h[2][4];
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) {
      h[ks][0] = pack_bf16x2(fmaxf(acc[2 * ks][0], 0.f), fmaxf(acc[2 * ks][1], 0.f));
      h[ks][1] = pack_bf16x2(fmaxf(acc[2 * ks][2], 0.f), fmaxf(acc[2 * ks][3], 0.f));
      h[ks][2] = pack_bf16x2(fmaxf(acc[2 * ks + 1][0], 0.f), fmaxf(acc[2 * ks + 1][1], 0.f));
      h[ks][3] = pack_bf16x2(fmaxf(acc[2 * ks + 1][2], 0.f), fmaxf(acc[2 * ks + 1][3], 0.f));
    }
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
      float z[4] = {f.b2[nt][0], f.b2[nt][1], f.b2[nt][0], f.b2[nt][1]};
#pragma unroll
      for (int ks = 0; ks < 2; ++ks) {
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        mma_bf16_16816(d, h[ks], f.w2[ks][nt][0], f.w2[ks][nt][1]);
#pragma unroll
        for (int e = 0; e < 4; ++e) z[e] += d[e];
      }
      s0 = fmaf(f.w3[nt][0], fmaxf(z[0], 0.f), s0);
      s0 = fmaf(f.w3[nt][1], fmaxf(z[1], 0.f), s0);
      s1 = fmaf(f.w3[nt][0], fmaxf(z[2], 0.f), s1);
      s1 = fmaf(f.w3[nt][1], fmaxf(z[3], 0.f), s1);
    }
    // the group's four lanes hold eight columns each: fixed-order sum
    s0 += __shfl_xor_sync(0xffffffffu, s0, 1);
    s0 += __shfl_xor_sync(0xffffffffu, s0, 2);
    s1 += __shfl_xor_sync(0xffffffffu, s1, 1);
    s1 += __shfl_xor_sync(0xffffffffu, s1, 2);
    if (t == 0 && r0 < n) out[r0] = 1.f / (1.f + __expf(-(s0 + f.b3)));
    if (t == 0 && r1 < n) out[r1] = 1.f / (1.f + __expf(-(s1 + f.b3)));
  }
}

// Loss and gradient: persistent CTAs over the 64-sample tiles.  Each thread
// keeps its block of the weight gradients in registers over all the CTA's
// tiles (8 x 4 of dW1 or dW2 on warps 0-2: 56 + 32 blocks; one column of db1,
// db2 and dw3 per lane of warp 3), so a CTA writes one partial
// (kGateParams gradient entries, then the loss) at its end.
constexpr int kGradSmem = MlpSmem::end + kGateH * kMStrH + kMt * kMStrX + 4 * kMt * kMStrH + 2 * kMt;  // floats
__global__ void __launch_bounds__(kMThreads, kGradPerSm) hydro_mlp_grad_kernel(const float* __restrict__ params,
                                                                      const float* __restrict__ X,
                                                                      const float* __restrict__ y, int n, bool vec,
                                                                      float w1, float w0, float inv_n,
                                                                      float* __restrict__ partial) {
  extern __shared__ __align__(16) float sm[];
  float* w2t = sm + MlpSmem::end;            // W2 transposed [i][j]
  float* xs = w2t + kGateH * kMStrH;         // [kMt][kMStrX]
  float* h1s = xs + kMt * kMStrX;            // [kMt][kMStrH] each
  float* h2s = h1s + kMt * kMStrH;
  float* g1s = h2s + kMt * kMStrH;           // dL/dz1
  float* g2s = g1s + kMt * kMStrH;           // dL/dz2
  float* g3s = g2s + kMt * kMStrH;           // dL/dz3 [kMt]
  float* ls = g3s + kMt;                     // loss terms [kMt]
  mlp_load_weights(params, sm);
  for (int i = threadIdx.x; i < kGateH * kMStrH; i += kMThreads) {
    const int r = i / kMStrH, k = i % kMStrH;
    w2t[i] = k < kGateH ? bf16r(params[kGateW2 + k * kGateH + r]) : 0.f;
  }
  const int tid = threadIdx.x, c = tid & 7;
  // this thread's gradient block: rows j0 .. j0 + 7 of g against columns
  // i0 .. i0 + 3 of v (dW1: g1, x; dW2: g2, h1)
  const bool in1 = tid < 56, in2 = tid >= 56 && tid < 88;
  const int t2 = tid - 56;
  const int j0 = 8 * (in1 ? tid / 14 : t2 / 8), i0 = 4 * (in1 ? tid % 14 : t2 % 8);
  float2 acc[4][4];  // [pair of j][i]
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[p][i] = f2(0.f);
  float sb1 = 0.f, sb2 = 0.f, sw3 = 0.f, sb3 = 0.f, sl = 0.f;

  const int tiles = (n + kMt - 1) / kMt;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    mlp_load_tile(X, tile, n, vec, xs);
    __syncthreads();
    float init[4], h1[4][4], v[4][4];
#pragma unroll
    for (int o = 0; o < 4; ++o) init[o] = sm[MlpSmem::b1 + c + 8 * o];
    mlp_block<56, kMStrX, kMStrX>(xs, sm + MlpSmem::w1, init, h1);
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int o = 0; o < 4; ++o) h1[m][o] = fmaxf(h1[m][o], 0.f);
    mlp_store(h1s, h1);
    __syncthreads();
#pragma unroll
    for (int o = 0; o < 4; ++o) init[o] = sm[MlpSmem::b2 + c + 8 * o];
    mlp_block<kGateH, kMStrH, kMStrH>(h1s, sm + MlpSmem::w2, init, v);
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int o = 0; o < 4; ++o) v[m][o] = fmaxf(v[m][o], 0.f);
    mlp_store(h2s, v);
    __syncthreads();
    if (tid < kMt) {
      const int i = tile * kMt + tid;
      const bool live = i < n;
      const float z3 = mlp_head(sm, h2s, tid);
      const float out = 1.f / (1.f + __expf(-z3));
      const float yy = live ? y[i] : 0.f;
      // -[w1 y log(out) + w0 (1-y) log(1-out)] with log(out) = -softplus(-z3)
      const float sp_neg = fmaxf(-z3, 0.f) + log1pf(__expf(-fabsf(z3)));  // softplus(-z3)
      const float sp_pos = sp_neg + z3;                                   // softplus(z3)
      ls[tid] = live ? (w1 * yy * sp_neg + w0 * (1.f - yy) * sp_pos) * inv_n : 0.f;
      g3s[tid] = live ? (w1 * yy * (out - 1.f) + w0 * (1.f - yy) * out) * inv_n : 0.f;
    }
    __syncthreads();
    // dL/dz2 of the thread's block (v holds its h2: positive where z2 is)
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const float g3 = g3s[(tid >> 3) + 16 * m];
#pragma unroll
      for (int o = 0; o < 4; ++o) v[m][o] = v[m][o] > 0.f ? g3 * sm[MlpSmem::w3 + c + 8 * o] : 0.f;
    }
    mlp_store(g2s, v);
    __syncthreads();
    const float zero[4] = {0.f, 0.f, 0.f, 0.f};
    mlp_block<kGateH, kMStrH, kMStrH>(g2s, w2t, zero, v);
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int o = 0; o < 4; ++o) v[m][o] = h1[m][o] > 0.f ? v[m][o] : 0.f;
    mlp_store(g1s, v);
    __syncthreads();
    // weight gradients: sums over the samples in index order
    if (in1 || in2) {
      const float* gp = (in1 ? g1s : g2s) + j0;
      const float* vp = (in1 ? xs : h1s) + i0;
      const int sv = in1 ? kMStrX : kMStrH;
#pragma unroll 4
      for (int s = 0; s < kMt; ++s) {
        const float4 ga = *reinterpret_cast<const float4*>(gp + s * kMStrH);
        const float4 gb = *reinterpret_cast<const float4*>(gp + s * kMStrH + 4);
        const float4 xv = *reinterpret_cast<const float4*>(vp + s * sv);
        const float2 g[4] = {f2(ga.x, ga.y), f2(ga.z, ga.w), f2(gb.x, gb.y), f2(gb.z, gb.w)};
        const float2 x[4] = {f2(xv.x), f2(xv.y), f2(xv.z), f2(xv.w)};
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[p][i] = fma2(g[p], x[i], acc[p][i]);
      }
    } else if (tid >= 96) {
      const int j = tid - 96;
#pragma unroll 4
      for (int s = 0; s < kMt; ++s) {
        sb1 += g1s[s * kMStrH + j];
        sb2 += g2s[s * kMStrH + j];
        sw3 = fmaf(g3s[s], h2s[s * kMStrH + j], sw3);
      }
      sb3 += g3s[j] + g3s[j + 32];
      sl += ls[j] + ls[j + 32];
    }
    __syncthreads();  // the next tile overwrites the activations
  }
  float* out = partial + (size_t)blockIdx.x * (kGateParams + 1);
  if (in1 || in2) {
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int j = j0 + 2 * p, k = i0 + i;
        if (in1 && k < kGateIn) {
          out[j * kGateIn + k] = acc[p][i].x;
          out[(j + 1) * kGateIn + k] = acc[p][i].y;
        } else if (in2) {
          out[kGateW2 + j * kGateH + k] = acc[p][i].x;
          out[kGateW2 + (j + 1) * kGateH + k] = acc[p][i].y;
        }
      }
  } else if (tid >= 96) {
    const int j = tid - 96;
    out[kGateB1 + j] = sb1;
    out[kGateB2 + j] = sb2;
    out[kGateW3 + j] = sw3;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      sb3 += __shfl_xor_sync(0xffffffffu, sb3, o);
      sl += __shfl_xor_sync(0xffffffffu, sl, o);
    }
    if (j == 0) {
      out[kGateB3] = sb3;
      out[kGateParams] = sl;
    }
  }
}

// The sum of the partials, 32 parameters per CTA: row r of the block adds
// partials r, r + kRedRows, ... (one 128-byte line per warp and partial), then
// the rows are added in order.
constexpr int kRedRows = 16;
__global__ void __launch_bounds__(32 * kRedRows) hydro_mlp_reduce_kernel(const float* __restrict__ partial, int parts,
                                                                         float* __restrict__ grad,
                                                                         float* __restrict__ loss) {
  __shared__ float rows[kRedRows][33];
  const int p = blockIdx.x * 32 + threadIdx.x, r = threadIdx.y;
  float acc = 0.f;
  if (p <= kGateParams) {
#pragma unroll 8
    for (int b = r; b < parts; b += kRedRows) acc += __ldg(partial + (size_t)b * (kGateParams + 1) + p);
  }
  rows[r][threadIdx.x] = acc;
  __syncthreads();
  if (r != 0 || p > kGateParams) return;
  float sum = rows[0][threadIdx.x];
#pragma unroll
  for (int k = 1; k < kRedRows; ++k) sum += rows[k][threadIdx.x];
  if (p < kGateParams)
    grad[p] = sum;
  else if (loss)
    *loss = sum;
}

__global__ void hydro_mlp_adam_kernel(float* params, float* m, float* v, const float* grad, float lr, float bc1,
                                      float bc2) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= kGateParams) return;
  const float g = grad[p];
  const float mm = 0.9f * m[p] + 0.1f * g, vv = 0.999f * v[p] + 0.001f * g * g;
  m[p] = mm;
  v[p] = vv;
  params[p] -= lr * (mm / bc1) / (sqrtf(vv / bc2) + 1e-8f);
}

struct SmemW {
  const float* w;
  __device__ float operator()(int i) const { return w[i]; }
};

// Logit of the network at all-zero features (parameters already rounded).
__global__ void hydro_gate_zero_kernel(const float* w, float* out) {
  float x[54];
#pragma unroll
  for (int k = 0; k < 54; ++k) x[k] = 0.f;
  out[0] = gate_logit_infer(SmemW{w}, x);
}

__global__ void hydro_bf16_round_kernel(const float* in, float* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = bf16r(in[i]);
}

size_t mlp_grad_smem() { return sizeof(float) * kGradSmem; }

// SMs of the current device, at least 1 (the network's entry points have no context).
static int device_sms() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 1;
  return n;
}

}  // namespace hyd

extern "C" {

int hydro_gate_data(hydro_ctx_t* c, const hydro_batch_t* B, float* X, uint8_t* y, void* stream) {
  if (!c || !B || B->n_sub < 0 || (!X && !y)) return HYDRO_EINVAL;
  if (c->N != hyd::N) return HYDRO_EUNSUP;
  if (B->n_sub == 0) return HYDRO_OK;
  if (!B->U) return HYDRO_EINVAL;
  const size_t smem = (size_t)hyd::kLabelF * hyd::S3 * sizeof(float);
  static unsigned long long attr = 0;
  if (hyd::once_per_device(&attr, [smem] {
        return cudaFuncSetAttribute(hyd::hydro_gate_data_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)smem);
      }) != cudaSuccess)
    return HYDRO_ECUDA;
  hyd::GateDataArgs A{B->U, X, y, B->n_sub, c->mode.de_eta1, (float)c->gamma, (float)(c->gamma - 1.0)};
  const int grid = B->n_sub < 2 * c->num_sms ? B->n_sub : 2 * c->num_sms;
  hyd::hydro_gate_data_kernel<<<grid, hyd::kLabelThreads, smem, (cudaStream_t)stream>>>(A);
  return cudaGetLastError() == cudaSuccess ? HYDRO_OK : HYDRO_ECUDA;
}

int hydro_mlp_forward(const float* params, const float* X, int n, float* out, void* stream) {
  if (!params || n < 0 || (n > 0 && (!X || !out))) return HYDRO_EINVAL;
  if (n == 0) return HYDRO_OK;
  int blocks = (n - 1) / (16 * hyd::kFwdThreads / 32) + 1;
  const int most = hyd::kFwdPerSm * hyd::device_sms();
  if (blocks > most) blocks = most;
  hyd::hydro_mlp_forward_kernel<<<blocks, hyd::kFwdThreads, 0, (cudaStream_t)stream>>>(
      params, X, n, ((uintptr_t)X & 7u) == 0, out);
  return cudaGetLastError() == cudaSuccess ? HYDRO_OK : HYDRO_ECUDA;
}

size_t hydro_mlp_work_bytes(int n) {
  const size_t tiles = (size_t)((n > 0 ? n : 0) + hyd::kTile - 1) / hyd::kTile;
  return tiles * (hyd::kGateParams + 1) * sizeof(float);
}

int hydro_mlp_loss_grad(const float* params, const float* X, const float* y, int n, float w1, float w0, float* grad,
                        float* loss, void* work_v, size_t work_bytes, void* stream) {
  float* work = static_cast<float*>(work_v);
  if (!params || !X || !y || !grad || !work || n <= 0) return HYDRO_EINVAL;
  if (work_bytes < hydro_mlp_work_bytes(n)) return HYDRO_EINVAL;
  static unsigned long long attr = 0;
  if (hyd::once_per_device(&attr, [] {
        return cudaFuncSetAttribute(hyd::hydro_mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)hyd::mlp_grad_smem());
      }) != cudaSuccess)
    return HYDRO_ECUDA;
  // one partial per CTA; the work buffer holds one per kTile samples
  int parts = (n - 1) / hyd::kTile + 1;
  const int most = hyd::kGradPerSm * hyd::device_sms();
  if (parts > most) parts = most;
  cudaStream_t st = (cudaStream_t)stream;
  hyd::hydro_mlp_grad_kernel<<<parts, hyd::kMThreads, hyd::mlp_grad_smem(), st>>>(
      params, X, y, n, ((uintptr_t)X & 7u) == 0, w1, w0, 1.f / n, work);
  hyd::hydro_mlp_reduce_kernel<<<(hyd::kGateParams + 1 + 31) / 32, dim3(32, hyd::kRedRows), 0, st>>>(work, parts,
                                                                                                     grad, loss);
  return cudaGetLastError() == cudaSuccess ? HYDRO_OK : HYDRO_ECUDA;
}

int hydro_mlp_adam(float* params, float* m, float* v, const float* grad, int t, float lr, void* stream) {
  if (!params || !m || !v || !grad || t < 1 || !(lr > 0.f)) return HYDRO_EINVAL;
  const float bc1 = 1.f - powf(0.9f, (float)t), bc2 = 1.f - powf(0.999f, (float)t);
  hyd::hydro_mlp_adam_kernel<<<(hyd::kGateParams + 255) / 256, 256, 0, (cudaStream_t)stream>>>(params, m, v, grad, lr,
                                                                                               bc1, bc2);
  return cudaGetLastError() == cudaSuccess ? HYDRO_OK : HYDRO_ECUDA;
}

int hydro_set_indicator(hydro_ctx_t* c, const float* params, double threshold, void* stream) {
  if (!c) return HYDRO_EINVAL;
  if (!params) {
    c->gate_on = 0;
    return HYDRO_OK;
  }
  if (!(threshold > 0.0 && threshold < 1.0)) return HYDRO_EINVAL;
  int rc = HYDRO_OK;
  if (!c->gate_w) {
    if (cudaMalloc(&c->gate_w, hyd::kGateParams * sizeof(float)) != cudaSuccess) return HYDRO_ENOMEM;
  }
  cudaStream_t st = (cudaStream_t)stream;
  hyd::hydro_bf16_round_kernel<<<(hyd::kGateParams + 255) / 256, 256, 0, st>>>(params, c->gate_w, hyd::kGateParams);
  if (cudaGetLastError() != cudaSuccess) rc = HYDRO_ECUDA;
  if (rc == HYDRO_OK) {
    // the network's decision at all-zero features (a uniform neighbourhood),
    // evaluated once with the same rounded parameters and arithmetic
    float* d_zero = nullptr;
    float h_zero = 1.f;
    if (cudaMalloc(&d_zero, 2 * sizeof(float)) != cudaSuccess) return HYDRO_ENOMEM;
    hyd::hydro_gate_zero_kernel<<<1, 1, 0, st>>>(c->gate_w, d_zero);
    if (cudaMemcpyAsync(&h_zero, d_zero, sizeof(float), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      rc = HYDRO_ECUDA;
    cudaFree(d_zero);
    if (rc != HYDRO_OK) return rc;
    c->gate_logit_thr = log(threshold / (1.0 - threshold));
    c->gate_zero_smooth = (h_zero < (float)c->gate_logit_thr) ? 1 : 0;
    c->gate_on = 1;
  }
  return rc;
}

}  // extern "C"
