// policy_train.cuh -- kernels of the learned-branching policy outside the
// search: feature extraction for training data, batched scoring, and one
// training step (forward, listwise softmax cross-entropy, backward, Adam).
// Every matrix product runs on the tensor cores through warp-level
// mma.sync m16n8k16 with BF16 operands and FP32 accumulation; the forward
// pass computes exactly what the search kernels compute (BF16 features,
// weights and first hidden layer, FP32 second layer and output).
#pragma once

#include <cuda_bf16.h>

#include "policy.cuh"

namespace pccp {

constexpr int kPolicyParams = 128 * 16 + 128 + 128 * 128 + 128 + 128 + 1;
// flat parameter layout (FP32 masters, gradients and Adam moments)
constexpr int kOffW1 = 0;                    // [128][16], inputs 12..15 stay 0
constexpr int kOffB1 = kOffW1 + 128 * 16;    // [128]
constexpr int kOffW2 = kOffB1 + 128;         // [128][128] (out, in)
constexpr int kOffB2 = kOffW2 + 128 * 128;   // [128]
constexpr int kOffW3 = kOffB2 + 128;         // [128]
constexpr int kOffB3 = kOffW3 + 128;         // [1]

// ------------------------------------------------------------ training step
//
// Four kernels: forward; softmax; backward through the layers; gradients with
// Adam and the policy's images.  A step's arithmetic is small (256 groups of about 16
// rows: 0.45 GFLOP), so what it cost was launches, intermediates written and read
// again, and above all the two weight-gradient products, whose warps walked
// all the rows with transposed two-byte loads: 20 launches, 520 us a step of
// 256 groups, 455 us of it the products.  Gradients and scores
// are summed in a fixed order (a product's rows one after the other on one
// accumulator, a score's units in order), so a trained policy's values do not
// depend on how the work is split; the loss is a tree over lanes and groups.  Now 4 launches,
// and 140 us with the weights and gradients read back by the host.

constexpr int kTrainRows = 64;     // rows of a tile
constexpr int kTrainPitch = 136;   // bf16 of a shared-memory row (272 B: ldmatrix without conflicts)

__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], uint32_t p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(p)
               : "memory");
}

__device__ __forceinline__ void ldsm_x4_trans(uint32_t (&r)[4], uint32_t p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(p)
               : "memory");
}

// 16 bytes from global to shared memory, of which the group is committed and
// waited for by the caller.
__device__ __forceinline__ void cp_async16(uint32_t to, const void* from) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to), "l"(from) : "memory");
}

// The A fragment (16 rows x 16 inputs) of feature rows r0 and r0 + 8 (BF16).
__device__ __forceinline__ void feature_fragment(uint32_t (&a)[4], const float* __restrict__ f, int n,
                                                 int r0, int t) {
  a[0] = a[1] = a[2] = a[3] = 0u;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int r = r0 + 8 * h;
    if (r >= n) continue;
    const float* row = f + static_cast<size_t>(r) * kPolicyFeatures;
    a[h] = pack_bf16x2(row[2 * t], row[2 * t + 1]);
    if (t < 2) a[2 + h] = pack_bf16x2(row[8 + 2 * t], row[9 + 2 * t]);
  }
}

// First hidden layer of a 16-row chunk as the second layer's A fragments; w1: the
// first layer's fragments.
__device__ __forceinline__ void layer1_fragments(const PolicyDev* __restrict__ pol, const uint2* w1,
                                                 const uint32_t (&a1)[4], int lane,
                                                 uint32_t (&a2)[8][4]) {
  const int t = lane & 3;
#pragma unroll
  for (int kk = 0; kk < 8; ++kk) {
    float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f};
    mma_16816(d0, a1, w1[64 * kk + lane]);
    mma_16816(d1, a1, w1[64 * kk + 32 + lane]);
    const float2 b0 = __ldg(reinterpret_cast<const float2*>(&pol->b1[16 * kk + 2 * t]));
    const float2 b1 = __ldg(reinterpret_cast<const float2*>(&pol->b1[16 * kk + 2 * t + 8]));
    a2[kk][0] = pack_bf16x2(fmaxf(d0[0] + b0.x, 0.f), fmaxf(d0[1] + b0.y, 0.f));
    a2[kk][1] = pack_bf16x2(fmaxf(d0[2] + b0.x, 0.f), fmaxf(d0[3] + b0.y, 0.f));
    a2[kk][2] = pack_bf16x2(fmaxf(d1[0] + b1.x, 0.f), fmaxf(d1[1] + b1.y, 0.f));
    a2[kk][3] = pack_bf16x2(fmaxf(d1[2] + b1.x, 0.f), fmaxf(d1[3] + b1.y, 0.f));
  }
}

// Forward pass of a 64-row tile (8 warps: four 16-row chunks, two halves of the
// second layer's units): X [R][16] and H1 [R][128] in BF16, H2 [R][128] in
// FP32, scores s, and ds cleared.  rows n .. R - 1 are computed as zero rows.
__global__ void __launch_bounds__(256) k_train_forward(const PolicyDev* __restrict__ pol, int n,
                                                       const float* __restrict__ f,
                                                       __nv_bfloat16* __restrict__ X,
                                                       __nv_bfloat16* __restrict__ H1,
                                                       float* __restrict__ H2, float* __restrict__ s,
                                                       float* __restrict__ ds) {
  __shared__ float sh[kTrainRows][129];
  __shared__ float sw3[128];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int chunk = warp & 3, half = warp >> 2;
  const int r0 = blockIdx.x * kTrainRows + 16 * chunk + g;
  uint32_t a1[4], a2[8][4];
  uint2 w[8];  // the second layer's fragments of the next tile of units
  feature_fragment(a1, f, n, r0, t);
#pragma unroll
  for (int kk = 0; kk < 8; ++kk) w[kk] = __ldg(&pol->w2[kk][8 * half][lane]);
  layer1_fragments(pol, &pol->w1[0][0], a1, lane, a2);
  if (threadIdx.x < 128) sw3[threadIdx.x] = __ldg(&pol->w3[threadIdx.x]);
  if (half == 0) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t* x = reinterpret_cast<uint32_t*>(X + static_cast<size_t>(r0 + 8 * h) * 16);
      x[t] = a1[h];
      x[4 + t] = a1[2 + h];
      uint32_t* o = reinterpret_cast<uint32_t*>(H1 + static_cast<size_t>(r0 + 8 * h) * 128);
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) {
        o[8 * kk + t] = a2[kk][h];
        o[8 * kk + 4 + t] = a2[kk][2 + h];
      }
    }
  }
#pragma unroll
  for (int jj = 0; jj < 8; ++jj) {
    const int j = 8 * half + jj;
    const int c = 8 * j + 2 * t;
    const float2 b = __ldg(reinterpret_cast<const float2*>(&pol->b2[c]));
    uint2 next[8] = {};
    if (jj < 7)
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) next[kk] = __ldg(&pol->w2[kk][j + 1][lane]);
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int kk = 0; kk < 8; ++kk) {
      mma_16816(acc, a2[kk], w[kk]);
      w[kk] = next[kk];
    }
    const float2 u = make_float2(fmaxf(acc[0] + b.x, 0.f), fmaxf(acc[1] + b.y, 0.f));
    const float2 v = make_float2(fmaxf(acc[2] + b.x, 0.f), fmaxf(acc[3] + b.y, 0.f));
    *reinterpret_cast<float2*>(H2 + static_cast<size_t>(r0) * 128 + c) = u;
    *reinterpret_cast<float2*>(H2 + static_cast<size_t>(r0 + 8) * 128 + c) = v;
    sh[16 * chunk + g][c] = u.x;
    sh[16 * chunk + g][c + 1] = u.y;
    sh[16 * chunk + g + 8][c] = v.x;
    sh[16 * chunk + g + 8][c + 1] = v.y;
  }
  __syncthreads();
  if (threadIdx.x < kTrainRows) {
    const size_t r = static_cast<size_t>(blockIdx.x) * kTrainRows + threadIdx.x;
    float acc = 0.f;
#pragma unroll 16
    for (int c = 0; c < 128; ++c) acc = fmaf(sh[threadIdx.x][c], sw3[c], acc);
    s[r] = acc + __ldg(&pol->b3);
    ds[r] = 0.f;
  }
}

// Listwise softmax cross-entropy, a warp per group of rows (a search node's
// candidates): ds = (softmax(s) - target) * scale; loss[group] =
// -sum target * log softmax.
__global__ void k_group_softmax(int n_groups, const int* __restrict__ off,
                                const float* __restrict__ s, const float* __restrict__ target,
                                float* __restrict__ ds, float* __restrict__ loss, float scale) {
  const int gi = static_cast<int>((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (gi >= n_groups) return;  // whole warps leave together
  const int a = off[gi], b = off[gi + 1];
  float mx = -3.4e38f;
  for (int r = a + lane; r < b; r += 32) mx = fmaxf(mx, s[r]);
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  float z = 0.f;  // in the order of the rows
  for (int r0 = a; r0 < b; r0 += 32) {
    const float e = r0 + lane < b ? __expf(s[r0 + lane] - mx) : 0.f;
    const int k = min(32, b - r0);
    for (int i = 0; i < k; ++i) z += __shfl_sync(0xffffffffu, e, i);
  }
  const float lz = __logf(z) + mx;
  float l = 0.f;
  for (int r = a + lane; r < b; r += 32) {
    const float p = __expf(s[r] - lz);
    ds[r] = (p - target[r]) * scale;  // gradient of the mean over groups
    l -= target[r] * (s[r] - lz);
  }
  for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  if (lane == 0) loss[gi] = l;
}

constexpr size_t kTrainBackSmem =
    2 * (2 * static_cast<size_t>(kTrainRows) * kTrainPitch + 128 * static_cast<size_t>(kTrainPitch));

// Backward through the layers, a CTA per 64-row tile: dZ2 = ds w3 where H2 > 0
// (BF16), dZ1 = dZ2 W2 where H1 > 0 (FP32 and BF16).
__global__ void __launch_bounds__(256) k_train_backward(const float* __restrict__ params,
                                                        const __nv_bfloat16* __restrict__ w2b,
                                                        const __nv_bfloat16* __restrict__ H1,
                                                        const float* __restrict__ H2,
                                                        const float* __restrict__ ds,
                                                        __nv_bfloat16* __restrict__ dZ2b,
                                                        float* __restrict__ dZ1,
                                                        __nv_bfloat16* __restrict__ dZ1b) {
  extern __shared__ __align__(16) __nv_bfloat16 tsm[];
  __nv_bfloat16* sZ2 = tsm;                             // [64][136]
  __nv_bfloat16* sH1 = sZ2 + kTrainRows * kTrainPitch;  // [64][136]
  __nv_bfloat16* sW2 = sH1 + kTrainRows * kTrainPitch;  // [128][136]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const size_t row0 = static_cast<size_t>(blockIdx.x) * kTrainRows;
  for (int i = tid; i < 128 * 16; i += 256)  // 16-byte pieces
    cp_async16(smem_u32(sW2 + (i >> 4) * kTrainPitch + 8 * (i & 15)), w2b + 128 * (i >> 4) + 8 * (i & 15));
  for (int i = tid; i < kTrainRows * 16; i += 256)
    cp_async16(smem_u32(sH1 + (i >> 4) * kTrainPitch + 8 * (i & 15)),
               H1 + (row0 + (i >> 4)) * 128 + 8 * (i & 15));
  const int c2 = 2 * (tid & 63), rr = tid >> 6;  // two columns of every fourth row
  const float wa = params[kOffW3 + c2], wb = params[kOffW3 + c2 + 1];
#pragma unroll 8
  for (int k = 0; k < kTrainRows / 4; ++k) {
    const int r = 4 * k + rr;
    const float2 h = *reinterpret_cast<const float2*>(H2 + (row0 + r) * 128 + c2);
    const float d = ds[row0 + r];
    const uint32_t z = pack_bf16x2(h.x > 0.f ? d * wa : 0.f, h.y > 0.f ? d * wb : 0.f);
    *reinterpret_cast<uint32_t*>(sZ2 + r * kTrainPitch + c2) = z;
    *reinterpret_cast<uint32_t*>(dZ2b + (row0 + r) * 128 + c2) = z;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  // 16 rows x 64 columns a warp; mrow, mhi, mlast: this lane's row of the four
  // 8 x 8 matrices of an ldmatrix
  const int chunk = warp & 3, half = warp >> 2;
  const int mrow = lane & 7, mhi = (lane >> 3) & 1, mlast = lane >> 4;
  float acc[8][4];
#pragma unroll
  for (int j = 0; j < 8; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
#pragma unroll
  for (int kk = 0; kk < 8; ++kk) {
    uint32_t a[4];
    ldsm_x4(a, smem_u32(sZ2 + (16 * chunk + mrow + 8 * mhi) * kTrainPitch + 16 * kk + 8 * mlast));
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
      uint32_t b[4];
      ldsm_x4_trans(b, smem_u32(sW2 + (16 * kk + mrow + 8 * mhi) * kTrainPitch + 64 * half +
                                8 * (j + mlast)));
      mma_16816(acc[j], a, make_uint2(b[0], b[1]));
      mma_16816(acc[j + 1], a, make_uint2(b[2], b[3]));
    }
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int c = 64 * half + 8 * j + 2 * t;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = 16 * chunk + g + 8 * h;
      const __nv_bfloat162 on = *reinterpret_cast<const __nv_bfloat162*>(sH1 + r * kTrainPitch + c);
      const float z0 = __low2float(on) > 0.f ? acc[j][2 * h] : 0.f;
      const float z1 = __high2float(on) > 0.f ? acc[j][2 * h + 1] : 0.f;
      *reinterpret_cast<float2*>(dZ1 + (row0 + r) * 128 + c) = make_float2(z0, z1);
      *reinterpret_cast<uint32_t*>(dZ1b + (row0 + r) * 128 + c) = pack_bf16x2(z0, z1);
    }
  }
}

// Parameter i of the flat layout into the images the kernels read: BF16 W2
// and the fragment image.
__device__ __forceinline__ void put_param(int i, float v, __nv_bfloat16* __restrict__ w2b,
                                          PolicyDev* __restrict__ d) {
  const __nv_bfloat16 h = __float2bfloat16_rn(v);
  if (i < kOffB1) {  // W1 [128][16]: fragments of tile o / 8
    const int o = i >> 4, c = i & 15, l = 4 * (o & 7) + ((c & 7) >> 1);
    reinterpret_cast<__nv_bfloat16*>(&d->w1[o >> 3][l])[2 * (c >> 3) + (c & 1)] = h;
  } else if (i < kOffW2) {
    d->b1[i - kOffB1] = v;
  } else if (i < kOffB2) {  // W2 [128][128]: k-step c / 16, tile o / 8
    const int k = i - kOffW2, o = k >> 7, c = k & 127, l = 4 * (o & 7) + ((c & 7) >> 1);
    w2b[k] = h;
    reinterpret_cast<__nv_bfloat16*>(&d->w2[c >> 4][o >> 3][l])[2 * ((c >> 3) & 1) + (c & 1)] = h;
  } else if (i < kOffW3) {
    d->b2[i - kOffB2] = v;
  } else if (i < kOffB3) {
    d->w3[i - kOffW3] = v;
  } else {
    d->b3 = v;
  }
}

struct TrainUpdate {
  float* p;  // parameters, gradients, Adam moments (flat layout)
  float* g;
  float* m;
  float* v;
  __nv_bfloat16* w2b;
  PolicyDev* d;
  float lr, b1, b2, eps, c1, c2;
};

// Parameter i and its moments.
__device__ __forceinline__ float3 train_state(const TrainUpdate& u, int i) {
  return make_float3(u.p[i], u.m[i], u.v[i]);
}

// Gradient gi of parameter i, Adam's step on it (inputs 12..15 of W1 stay zero),
// and the parameter's places in the images; old: its train_state.
__device__ __forceinline__ void train_update(const TrainUpdate& u, int i, float gi, float3 old) {
  u.g[i] = gi;
  if (i < kOffB1 && (i & 15) >= kPolicyFeatures) {
    u.p[i] = 0.f;
    put_param(i, 0.f, u.w2b, u.d);
    return;
  }
  const float mi = u.b1 * old.y + (1.f - u.b1) * gi;
  const float vi = u.b2 * old.z + (1.f - u.b2) * gi * gi;
  u.m[i] = mi;
  u.v[i] = vi;
  const float np = old.x - u.lr * (mi / u.c1) / (sqrtf(vi / u.c2) + u.eps);
  u.p[i] = np;
  put_param(i, np, u.w2b, u.d);
}

constexpr int kGradRows = 256;   // rows of a stage
constexpr int kGradStages = 4;
constexpr int kGradPitch = 24;   // bf16 of a staged row of 16 (48 B: ldmatrix without conflicts)
constexpr size_t kTrainGradSmem = 2 * 2 * static_cast<size_t>(kGradStages) * kGradRows * kGradPitch;
constexpr int kGradW2 = 64, kGradW1 = 8, kGradCols = 16;   // CTAs of each kind
constexpr int kGradBlocks = kGradW2 + kGradW1 + 2 * kGradCols + 1;

// Gradients over rows 0 .. R-1 (R a multiple of 16), each by one CTA, which then
// takes Adam's step on its parameters; one wave of CTAs:
//   dW2 = dZ2^T H1 (64 CTAs) and dW1 = dZ1^T X (8), 16 x 16 values each.  One warp's
//     two accumulators go through all the rows in order, a chain of R / 16
//     tensor-core products (4096 rows: about 5 us); the others' part is to
//     keep three 16 KB stages of rows on their way.
//   db2 and dw3 = H2^T ds (16 CTAs), db1 (16): 8 columns each, 256 partial sums
//     a column, summed as a tree of 32 and then in order.
//   db3, and the loss from the groups' (1).
// w3 is read and written by the same CTA (its columns); nothing here reads other
// CTAs' parameters.  4096 rows: 18.4 us (25.0 with the parameters and moments read
// one by one at the end and a lane for each staged row, whose 32 rows an
// instruction took 32 cycles of L1).
__global__ void __launch_bounds__(256, 1) k_train_gradients(int R, const __nv_bfloat16* __restrict__ X,
                                                            const __nv_bfloat16* __restrict__ H1,
                                                            const float* __restrict__ H2,
                                                            const float* __restrict__ ds,
                                                            const __nv_bfloat16* __restrict__ dZ2b,
                                                            const float* __restrict__ dZ1,
                                                            const __nv_bfloat16* __restrict__ dZ1b,
                                                            int n_groups,
                                                            const float* __restrict__ group_loss,
                                                            float* __restrict__ loss, TrainUpdate u) {
  extern __shared__ __align__(16) __nv_bfloat16 tsm[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int job = blockIdx.x;
  if (job < kGradW2 + kGradW1) {
    const bool second = job < kGradW2;
    const int m0 = 16 * (second ? job >> 3 : job - kGradW2), n0 = second ? 16 * (job & 7) : 0;
    const __nv_bfloat16* A = (second ? dZ2b : dZ1b) + m0;  // [R][128], 16 columns of it
    const __nv_bfloat16* B = (second ? H1 : X) + n0;       // [R][128 or 16]
    const int ldb = second ? 128 : 16, n_stages = (R + kGradRows - 1) / kGradRows;
    auto load = [&](int k) {  // stage k: two rows a thread, half of each; two lanes share a row's sector
      const uint32_t to = smem_u32(tsm) + 2u * 2u * kGradPitch * kGradRows * static_cast<uint32_t>(k % kGradStages);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int q = (tid >> 1) + 128 * h, r = k * kGradRows + q, e = 8 * (tid & 1);
        if (k < n_stages && r < R) {
          const uint32_t ta = to + 2u * static_cast<uint32_t>(kGradPitch * q + e), tb = ta + 2u * kGradPitch * kGradRows;
          cp_async16(ta, A + static_cast<size_t>(r) * 128 + e);
          cp_async16(tb, B + static_cast<size_t>(r) * ldb + e);
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int k = 0; k < kGradStages - 1; ++k) load(k);
    // warp 0's eight parameters and their moments, read before the products: read
    // one after another between the updates' stores, they were eight round trips
    const int g = lane >> 2, t = lane & 3;
    auto param = [&](int j, int e) {
      const int o = m0 + g + 8 * (e >> 1), c = n0 + 8 * j + 2 * t + (e & 1);
      return second ? kOffW2 + 128 * o + c : kOffW1 + 16 * o + c;
    };
    float3 old[2][4];
    if (warp == 0) {
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) old[j][e] = train_state(u, param(j, e));
    }
    float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    const int mrow = lane & 7, mhi = (lane >> 3) & 1, mlast = lane >> 4;
    for (int k = 0; k < n_stages; ++k) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kGradStages - 2) : "memory");
      __syncthreads();  // stage k is here, stage k - 1 is free
      load(k + kGradStages - 1);
      if (warp == 0) {
        const uint32_t at = smem_u32(tsm) + 2u * 2u * kGradPitch * kGradRows * static_cast<uint32_t>(k % kGradStages);
        const uint32_t pa = at + 2u * static_cast<uint32_t>((mrow + 8 * mlast) * kGradPitch + 8 * mhi);
        const uint32_t pb = at + 2u * static_cast<uint32_t>((kGradRows + mrow + 8 * mhi) * kGradPitch + 8 * mlast);
        const int steps = min(kGradRows, R - k * kGradRows) / 16;
#pragma unroll 4
        for (int i = 0; i < steps; ++i) {
          uint32_t a[4], b[4];
          ldsm_x4_trans(a, pa + 2u * 16u * kGradPitch * static_cast<uint32_t>(i));
          ldsm_x4_trans(b, pb + 2u * 16u * kGradPitch * static_cast<uint32_t>(i));
          mma_16816(acc[0], a, make_uint2(b[0], b[1]));
          mma_16816(acc[1], a, make_uint2(b[2], b[3]));
        }
      }
    }
    if (warp == 0) {
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) train_update(u, param(j, e), acc[j][e], old[j][e]);
    }
    return;
  }
  job -= kGradW2 + kGradW1;
  float* part = reinterpret_cast<float*>(tsm);  // [2][8][256]
  // partial sums of a column -> their sum on every lane of a warp
  auto column_sum = [&](const float* q) {
    float s = 0.f;
    for (int w = 0; w < 8; ++w) {
      float x = q[32 * w + lane];
      for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      s += x;
    }
    return s;
  };
  if (job < 2 * kGradCols) {
    const bool second = job < kGradCols;
    const int c0 = 8 * (job % kGradCols), q = tid & 1, c = c0 + 4 * q;
    const float* M = (second ? H2 : dZ1) + c;
    float w3[4] = {0.f, 0.f, 0.f, 0.f};
    if (second)
#pragma unroll
      for (int e = 0; e < 4; ++e) w3[e] = u.p[kOffW3 + c + e];
    float s1[2][4] = {}, s2[2][4] = {};  // db, dw3 of four columns, rows tid/2 and tid/2 + 128 modulo 256
#pragma unroll 4
    for (int r0 = tid >> 1; r0 < R; r0 += 256) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = r0 + 128 * h;
        if (r >= R) continue;
        const float4 x4 = *reinterpret_cast<const float4*>(M + static_cast<size_t>(r) * 128);
        const float x[4] = {x4.x, x4.y, x4.z, x4.w};
        if (second) {
          const float d = ds[r];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            s1[h][e] += x[e] > 0.f ? __fmul_rn(d, w3[e]) : 0.f;
            s2[h][e] = fmaf(x[e], d, s2[h][e]);
          }
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) s1[h][e] += x[e];
        }
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        part[256 * (4 * q + e) + (tid >> 1) + 128 * h] = s1[h][e];
        if (second) part[256 * (8 + 4 * q + e) + (tid >> 1) + 128 * h] = s2[h][e];
      }
    __syncthreads();
    const float db = column_sum(part + 256 * warp);
    const int ib = (second ? kOffB2 : kOffB1) + c0 + warp;
    if (lane == 0) train_update(u, ib, db, train_state(u, ib));
    if (second) {
      const float dw = column_sum(part + 256 * (8 + warp));
      if (lane == 0) train_update(u, kOffW3 + c0 + warp, dw, train_state(u, kOffW3 + c0 + warp));
    }
    return;
  }
  float sb = 0.f, sl = 0.f;
  for (int r = tid; r < R; r += 256) sb += ds[r];
  for (int k = tid; k < n_groups; k += 256) sl += group_loss[k];
  part[tid] = sb;
  part[256 + tid] = sl;
  __syncthreads();
  if (warp >= 2) return;
  const float s = column_sum(part + 256 * warp);
  if (lane == 0) {
    if (warp == 0)
      train_update(u, kOffB3, s, train_state(u, kOffB3));
    else
      *loss = s;
  }
}

// The images of the FP32 parameters.
__global__ void k_build_policy(int n, const float* __restrict__ p, __nv_bfloat16* __restrict__ w2b,
                               PolicyDev* __restrict__ d) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) put_param(i, p[i], w2b, d);
}

// Features of every branch variable of every store (the search kernels'
// write_features, rounded to BF16 as the network sees them); out is
// [n_stores][n_branch][12].  Stores are joined with the root first.  A thread a
// row; its 48 bytes go out in three 16-byte stores when `out` allows it.
template <bool kVec>
__global__ void k_policy_features(const uint8_t* __restrict__ image, const int2* __restrict__ root,
                                  int n_stores, int n_vars, const int32_t* __restrict__ lb,
                                  const int32_t* __restrict__ ub, const int32_t* __restrict__ depth,
                                  float* __restrict__ out) {
  const TableHeader* h = reinterpret_cast<const TableHeader*>(image);
  const BranchStatic* bs = reinterpret_cast<const BranchStatic*>(image + h->off_bstat);
  const int32_t* branch = reinterpret_cast<const int32_t*>(image + h->off_branch);
  const int nb = h->n_branch, objective = h->objective;
  const long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= static_cast<long long>(n_stores) * nb) return;
  const int s = i <= 0x7fffffffll ? static_cast<int>(i) / nb : static_cast<int>(i / nb);
  const int k = static_cast<int>(i - static_cast<long long>(s) * nb);
  // stores are in the caller's variable order; the table and root in the
  // library's (user_of: the caller's index of each variable, after the root)
  const int32_t* user_of = reinterpret_cast<const int32_t*>(root + n_vars) + n_vars;
  const int v = branch[k];
  const int32_t* l = lb + static_cast<size_t>(s) * n_vars;
  const int32_t* u = ub + static_cast<size_t>(s) * n_vars;
  const int2 R = root[v];
  const int vu = user_of[v];
  const int2 D = make_int2(max(l[vu], R.x), min(u[vu], R.y));
  float prog = 0.f;
  if (objective >= 0) {
    const int2 RO = root[objective];
    prog = static_cast<float>(max(l[user_of[objective]], RO.x) - RO.x) /
           (static_cast<float>(RO.y - RO.x) + 1.f);
  }
  uint32_t row[8];
  write_features(row, k, D, R, bs[k], nb, depth ? depth[s] : 0, prog);
  float* o = out + (static_cast<size_t>(s) * nb + k) * kPolicyFeatures;
  float x[kPolicyFeatures];
#pragma unroll
  for (int c = 0; c < kPolicyFeatures; ++c) {
    const uint32_t w = row[c >> 1];
    x[c] = __uint_as_float((c & 1) ? (w & 0xffff0000u) : (w << 16));
  }
#pragma unroll
  for (int c = 0; c < kPolicyFeatures; c += 4) {
    if (kVec) {
      *reinterpret_cast<float4*>(o + c) = make_float4(x[c], x[c + 1], x[c + 2], x[c + 3]);
    } else {
      o[c] = x[c];
      o[c + 1] = x[c + 1];
      o[c + 2] = x[c + 2];
      o[c + 3] = x[c + 3];
    }
  }
}

// Scores of n feature rows (FP32 [n][12]) by the search kernels' network, with
// the search's sums (mlp_score_tiles, mlp_row_score).  A warp takes 32 rows at a
// time, so every weight fragment read from shared memory (36 KB, staged once per
// CTA) feeds two products; with a 16-row chunk a warp and fragments from L2 each
// chunk moved 36 KB (120,000 rows: 22.9 us, 18.1 us with this kernel).
__global__ void __launch_bounds__(256, 2) k_policy_score(const PolicyDev* __restrict__ pol, int n,
                                                      const float* __restrict__ f,
                                                      float* __restrict__ s) {
  __shared__ __align__(16) uint2 sw[16 * 32 + 8 * 16 * 32];  // w1, then w2
  __shared__ float4 bw[16][4];  // b2, w3 of a lane's two units of a tile
  for (int i = threadIdx.x; i < (16 * 32 + 8 * 16 * 32) / 2; i += blockDim.x)
    reinterpret_cast<uint4*>(sw)[i] = __ldg(reinterpret_cast<const uint4*>(&pol->w1[0][0]) + i);
  if (threadIdx.x < 64) {
    const int c = 2 * static_cast<int>(threadIdx.x);
    bw[threadIdx.x >> 2][threadIdx.x & 3] = make_float4(__ldg(&pol->b2[c]), __ldg(&pol->b2[c + 1]),
                                                        __ldg(&pol->w3[c]), __ldg(&pol->w3[c + 1]));
  }
  __syncthreads();
  const uint2* w2 = sw + 16 * 32;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int n_warps = static_cast<int>(gridDim.x * (blockDim.x >> 5));
  const float b3 = __ldg(&pol->b3);
  for (int c = static_cast<int>(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)); 32ll * c < n;
       c += n_warps) {
    uint32_t a[2][8][4];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      uint32_t a1[4];
      feature_fragment(a1, f, n, 32 * c + 16 * q + g, t);
      layer1_fragments(pol, sw, a1, lane, a[q]);
    }
    float sum = 0.f;  // of row 32 c + 16 (t & 1) + 8 (t >> 1) + g
#pragma unroll 2
    for (int j = 0; j < 16; ++j) {
      float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) {
        const uint2 w = w2[(16 * kk + j) * 32 + lane];
        mma_16816(acc[0], a[0][kk], w);
        mma_16816(acc[1], a[1][kk], w);
      }
      const float4 B = bw[j][t];
      float part[2][2];  // [16-row half][8-row half]
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        part[q][0] = fmaxf(acc[q][0] + B.x, 0.f) * B.z + fmaxf(acc[q][1] + B.y, 0.f) * B.w;
        part[q][1] = fmaxf(acc[q][2] + B.x, 0.f) * B.z + fmaxf(acc[q][3] + B.y, 0.f) * B.w;
      }
      // the four lanes of a row, each ending with the sum of one of the four rows
      const bool odd = t & 1, high = t & 2;
      float x = odd ? part[1][0] : part[0][0], y = odd ? part[1][1] : part[0][1];
      x += __shfl_xor_sync(0xffffffffu, odd ? part[0][0] : part[1][0], 1);
      y += __shfl_xor_sync(0xffffffffu, odd ? part[0][1] : part[1][1], 1);
      sum += (high ? y : x) + __shfl_xor_sync(0xffffffffu, high ? x : y, 2);
    }
    const int r = 32 * c + 16 * (t & 1) + 8 * (t >> 1) + g;
    if (r < n) s[r] = sum + b3;
  }
}

}  // namespace pccp
