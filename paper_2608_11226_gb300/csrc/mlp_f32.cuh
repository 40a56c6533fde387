// fp32 building blocks of the policy/value MLPs (FFMA register tiles over
// activations held feature-major in shared memory: xT[feature][row]).
#pragma once

#include "common.cuh"

namespace pe {

// canonical flat parameter layout (row-major W[out][in]):
//   policy W1[H][D] b1[H] W2[H][H] b2[H] W3[A][H] b3[A]
//   value  V1[H][D] c1[H] V2[H][H] c2[H] V3[1][H] c3[1]
struct MlpLayout {
  int64_t w1, b1, w2, b2, w3, b3, v1, c1, v2, c2, v3, c3, total;
};

__host__ __device__ __forceinline__ MlpLayout mlp_layout(int D, int H, int A) {
  MlpLayout L;
  int64_t o = 0;
  L.w1 = o; o += (int64_t)H * D;
  L.b1 = o; o += H;
  L.w2 = o; o += (int64_t)H * H;
  L.b2 = o; o += H;
  L.w3 = o; o += (int64_t)A * H;
  L.b3 = o; o += A;
  L.v1 = o; o += (int64_t)H * D;
  L.c1 = o; o += H;
  L.v2 = o; o += (int64_t)H * H;
  L.c2 = o; o += H;
  L.v3 = o; o += H;
  L.c3 = o; o += 1;
  L.total = o;
  return L;
}

// dst[k][n] = W[n][k] for W[rows=N][cols=K] in global memory (N a multiple of
// 8, K of 4).  A warp takes 8 rows x 4 columns at a time: 8 runs of 16 bytes
// of global memory and a 4-way bank conflict on the stores.  (Rows across the
// lanes alone touch 32 lines per load: 128 x 128 weights took 8 us; columns
// alone put a warp's stores into one bank.)
__device__ __forceinline__ void load_transposed(const float* __restrict__ W, float* dst, int N, int K) {
  const int lane = threadIdx.x & 31, nt = N / 8;
#pragma unroll 8
  for (int t = threadIdx.x >> 5; t < nt * (K / 4); t += blockDim.x >> 5) {
    const int n = (t % nt) * 8 + (lane & 7), k = (t / nt) * 4 + (lane >> 3);
    dst[k * N + n] = __ldg(W + (int64_t)n * K + k);
  }
}

__device__ __forceinline__ void load_copy(const float* __restrict__ src, float* dst, int n) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = __ldg(src + i);
}

// RT = 2, 4 or 8 consecutive floats of shared memory as pairs
template <int RT>
__device__ __forceinline__ void load_pairs(const float* p, float2 (&v)[RT / 2]) {
  if constexpr (RT == 2) {
    v[0] = *reinterpret_cast<const float2*>(p);
  } else {
#pragma unroll
    for (int q = 0; q < RT / 4; ++q) {
      const float4 x = *reinterpret_cast<const float4*>(p + 4 * q);
      v[2 * q] = make_float2(x.x, x.y);
      v[2 * q + 1] = make_float2(x.z, x.w);
    }
  }
}

template <int RT>
__device__ __forceinline__ void store_pairs(float* p, const float2 (&v)[RT / 2]) {
  if constexpr (RT == 2) {
    *reinterpret_cast<float2*>(p) = v[0];
  } else {
#pragma unroll
    for (int q = 0; q < RT / 4; ++q)
      *reinterpret_cast<float4*>(p + 4 * q) = make_float4(v[2 * q].x, v[2 * q].y, v[2 * q + 1].x, v[2 * q + 1].y);
  }
}

// acc[r][c] = sum_k in[k][rows 2r, 2r + 1] * W[k][c] over k < K, in the order of
// k: an RT-row x CT-neuron register tile, row pairs in the two lanes of the
// packed FMA (__ffma2_rn: two round-to-nearest fused multiply-adds, the same
// results as fmaf, in one instruction; the weight is moved to both lanes once
// per RT / 2 FMAs).  in points at the tile's first row (rows of k LD floats
// apart), W at its first neuron.  The operands of the next two k are in flight
// while the current two are used; the compiler's own unrolled loops left the
// FMA pipe waiting for shared memory (128 x 128 layer, 32 rows, 4 warps: 5,700
// cycles against 7,000 to 8,400; 112 rows, 14 warps: 20,900 against 22,100).
template <int RT, int CT, int K, int LD, int LDW>
__device__ __forceinline__ void dense_tile(const float* __restrict__ in, const float* __restrict__ W,
                                           float2 (&acc)[RT / 2][CT]) {
  static_assert(K % 4 == 0 && CT % 4 == 0, "two buffers of two k each");
  float2 x[2][2][RT / 2];
  float w[2][2][CT];
  auto load = [&](int b, int k0) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      load_pairs<RT>(in + (k0 + u) * LD, x[b][u]);
#pragma unroll
      for (int q = 0; q < CT / 4; ++q) {
        const float4 v = *reinterpret_cast<const float4*>(W + (k0 + u) * LDW + 4 * q);
        w[b][u][4 * q] = v.x, w[b][u][4 * q + 1] = v.y, w[b][u][4 * q + 2] = v.z, w[b][u][4 * q + 3] = v.w;
      }
    }
  };
  auto use = [&](int b) {
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int c = 0; c < CT; ++c) {
        const float2 ww = make_float2(w[b][u][c], w[b][u][c]);
#pragma unroll
        for (int r = 0; r < RT / 2; ++r) acc[r][c] = __ffma2_rn(x[b][u][r], ww, acc[r][c]);
      }
  };
#pragma unroll
  for (int r = 0; r < RT / 2; ++r)
#pragma unroll
    for (int c = 0; c < CT; ++c) acc[r][c] = make_float2(0.0f, 0.0f);
  load(0, 0);
#pragma unroll 1
  for (int k = 0; k < K; k += 4) {
    load(1, k + 2);
    use(0);
    if (k + 4 < K) load(0, k + 4);
    use(1);
  }
}

// out[c][rows] = tanh(acc + bias[c]); out points at the tile's first row and neuron
template <int RT, int CT, int LD>
__device__ __forceinline__ void tanh_store(const float2 (&acc)[RT / 2][CT], const float* __restrict__ bias,
                                           float* __restrict__ out) {
#pragma unroll
  for (int c = 0; c < CT; ++c) {
    const float bb = bias[c];
    float2 o[RT / 2];
#pragma unroll
    for (int r = 0; r < RT / 2; ++r) o[r] = make_float2(tanhf(acc[r][c].x + bb), tanhf(acc[r][c].y + bb));
    store_pairs<RT>(out + c * LD, o);
  }
}

// out[e][a] = b[a] + sum_k W[a][k] * hT[k][e], summed in the order of k
template <int TE, int K, int NA, int LD = TE>
__device__ __forceinline__ void head_t(const float* __restrict__ hT, const float* __restrict__ W,
                                       const float* __restrict__ bias, float* __restrict__ out) {
  for (int j = threadIdx.x; j < TE * NA; j += blockDim.x) {
    const int e = j % TE, a = j / TE;
    float acc = 0.0f;
#pragma unroll 8
    for (int k = 0; k < K; k += 4) {
      const float4 w = *reinterpret_cast<const float4*>(W + a * K + k);
      acc = fmaf(w.x, hT[k * LD + e], acc);
      acc = fmaf(w.y, hT[(k + 1) * LD + e], acc);
      acc = fmaf(w.z, hT[(k + 2) * LD + e], acc);
      acc = fmaf(w.w, hT[(k + 3) * LD + e], acc);
    }
    out[e * NA + a] = acc + bias[a];
  }
}

}  // namespace pe
