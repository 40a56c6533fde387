// Fused rollout for fp32 policy networks (Tiny: 8-64-64x3, 7B: 16-128-128x5).
//
// One CTA owns a tile of TE envs for the whole horizon (the loop over t is
// sequential, envs are independent).  The policy weights and the tile's env
// state stay in shared memory; per step the CTA computes the observation
// features, the two tanh layers and the logits with FFMA register tiles,
// samples with Philox, steps the envs and writes one row of the time-major
// rollout buffer.  The value network does not steer the rollout, so it runs
// afterwards over all T*E observations as a separate, fully parallel kernel.
#include "env.cuh"
#include "mlp_f32.cuh"

namespace pe {

template <int D, int H, int A, int TE, int C, int OBS>
struct RolloutF32Smem {
  alignas(16) float w1t[D * H];
  float w2t[H * H], w3[A * H], b1[H], b2[H], b3[(A + 3) / 4 * 4];
  static constexpr int LD = TE + 4;  // row stride: columns are written, and x's read back, across the rows
  alignas(16) float xt[D * LD];
  float ht[H * LD], logits[TE * A];  // h1, then h2 in place
  uint32_t draw[TE];               // the step's action draws ...
  float next_x[C][TE];             // ... and the samples it consumes
  int32_t next_ph[TE];
  EnvTab<C> tab;
  EnvTile<TE, C> env;
};

// Threads and register tile of a CTA's layers: a quarter or half of the
// threads' registers hold more of the tile where the layer is large enough.
template <int TE, int H>
struct RolloutTile {
  static constexpr int NT = TE == 32 && H == 128 ? 256 : 128;
  static constexpr int RT = TE * H / 16 >= NT ? 4 : 2;           // rows per thread
  static constexpr int CT2 = TE == 32 && H == 128 ? 8 : 4;       // neurons per thread, layer 2
  static constexpr int EG = TE / RT, J1 = EG * H / 4, J2 = EG * H / CT2;  // row groups; tiles per layer
  static_assert(EG % 4 == 0 && J1 <= NT && J2 <= NT && J2 % 32 == 0, "tiles of a layer");
};

// A step is a chain of dependent phases, so their latencies set the time.
// Features are computed with the feature index uniform in a
// warp (one env per lane): with the features across the lanes every warp ran
// every feature's code in turn, 5,400 of the step's 19,300 cycles.  The
// action draw and the step's trace sample depend on nothing that the network
// computes and are fetched by a warp that the head leaves idle.  With the
// register tiles of dense_tile a 7B rollout (4,096 envs x 512 steps) went from
// 4.57 to 3.33 ms, 13,100 cycles per step: 6,600 in the 128 x 128 layer.  ONE:
// no cadence table.
template <int D, int H, int A, int TE, int C, int OBS, bool ONE>
__global__ void __launch_bounds__(RolloutTile<TE, H>::NT, 1)
    rollout_f32_kernel(EnvDev env, const float* __restrict__ params, int T, uint32_t it,
                       float lambda, int det, pe_rollout_buf buf) {
  using Smem = RolloutF32Smem<D, H, A, TE, C, OBS>;
  using Tl = RolloutTile<TE, H>;
  static_assert(TE <= 32, "one env per lane");
  constexpr int NT = Tl::NT, LD = Smem::LD, RT = Tl::RT, CT2 = Tl::CT2;
  constexpr int kAhead = NT - 32;  // first thread of the last warp
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem& s = *reinterpret_cast<Smem*>(smem_raw);
  const int e0 = blockIdx.x * TE;
  const int ne = min(TE, env.E - e0);
  const MlpLayout Lp = mlp_layout(D, H, A);
  load_transposed(params + Lp.w1, s.w1t, H, D);
  load_transposed(params + Lp.w2, s.w2t, H, H);
  load_copy(params + Lp.b1, s.b1, H);
  load_copy(params + Lp.b2, s.b2, H);
  load_copy(params + Lp.w3, s.w3, A * H);
  load_copy(params + Lp.b3, s.b3, A);
  load_tab<C>(env, s.tab);
  __syncthreads();
  load_tile<TE, C>(env, s.env, s.tab, e0, ne);
  __syncthreads();

  float* obs_out = reinterpret_cast<float*>(buf.obs);
  int32_t v1 = 0, v60 = 0;
  int64_t energy = 0, smp = 0;
  float tok = 0.0f, exc = 0.0f;
  const int tid = threadIdx.x;
  // a warp's tiles cover 4 row groups x 8 neuron groups
  const int eg = (tid >> 5) % (Tl::EG / 4) * 4 + (tid & 3), ng = (tid >> 5) / (Tl::EG / 4) * 8 + ((tid & 31) >> 2);

  for (int t = 0; t <= T; ++t) {
    // (1) observation features, one env per lane
    for (int idx = tid; idx < TE * D; idx += blockDim.x) {
      const int e = idx % TE, f = idx / TE;
      float v = 0.0f;
      if (e < ne) {
        TileAcc<TE, C> acc{s.env, s.tab, e};
        v = feature<C, OBS>(env, acc, f);
      }
      s.xt[f * LD + e] = v;
    }
    __syncthreads();
    // the buffer row, while the network starts (the obs rows of a tile are
    // consecutive; their address is a multiple of 4 floats from the buffer's)
    float* dst = t < T ? obs_out + ((int64_t)t * env.E + e0) * D
                       : reinterpret_cast<float*>(buf.obs_last) + (int64_t)e0 * D;
    for (int idx = tid; idx < ne * D; idx += blockDim.x) dst[idx] = s.xt[(idx % D) * LD + idx / D];
    if (t == T) break;
    // (2)-(4) policy network
    if (tid < Tl::J1) {
      float2 acc[RT / 2][4];
      dense_tile<RT, 4, D, LD, H>(s.xt + eg * RT, s.w1t + ng * 4, acc);
      tanh_store<RT, 4, LD>(acc, s.b1 + ng * 4, s.ht + ng * 4 * LD + eg * RT);
    }
    __syncthreads();
    {
      float2 acc[RT / 2][CT2];
      if (tid < Tl::J2) dense_tile<RT, CT2, H, LD, H>(s.ht + eg * RT, s.w2t + ng * CT2, acc);
      __syncthreads();  // h2 takes h1's place
      if (tid < Tl::J2) tanh_store<RT, CT2, LD>(acc, s.b2 + ng * CT2, s.ht + ng * CT2 * LD + eg * RT);
    }
    __syncthreads();
    if (tid >= kAhead && tid - kAhead < ne) {
      const int e = tid - kAhead;
      s.draw[e] = det ? 0u : draw32(env.seed, (uint32_t)(e0 + e), (uint32_t)t, it, kDrawAction);
      if (ONE) {
        const Samp<C> n = load_samp<C>(env, fam_of(env, s.env.fam[e]), s.env.pos[e]);
#pragma unroll
        for (int c = 0; c < C; ++c) s.next_x[c][e] = n.x[c];
        s.next_ph[e] = n.ph;
      }
    }
    head_t<TE, H, A, LD>(s.ht, s.w3, s.b3, s.logits);
    __syncthreads();
    // (5) sample, actuate, consume one sample, reward
    if (tid < ne) {
      const int e = tid;
      const uint32_t eg = (uint32_t)(e0 + e);
      float lp;
      const int a = sample_action<A>(s.logits + e * A, s.draw[e], det != 0, &lp);
      TileAcc<TE, C> acc{s.env, s.tab, e};
      Samp<C> next;
      if (ONE) {
#pragma unroll
        for (int c = 0; c < C; ++c) next.x[c] = s.next_x[c][e];
        next.ph = s.next_ph[e];
        next.act = (env.phase_mask >> next.ph) & 1;
      }
      const StepOut so = env_step<C, ONE>(env, acc, a, lambda, &next);
      const int64_t row = (int64_t)t * env.E + eg;
      buf.act[row] = (uint8_t)a;
      buf.logp[row] = lp;
      buf.reward[row] = so.reward;
      buf.done[row] = (uint8_t)so.done;
      if (buf.q) buf.q[row] = so.q;
      v1 += so.v1;
      v60 += so.v60;
      energy += so.q;
      smp += so.samples;
      tok += so.tokens;
      exc += so.excess;
      if (so.done) env_reset<C>(env, acc, eg, (uint32_t)t, it, kDrawReset);
    }
    __syncthreads();
  }
  if (tid < ne) {
    const int g = e0 + tid;
    buf.viol[2 * g] = v1;
    buf.viol[2 * g + 1] = v60;
    buf.tokens[g] = tok;
    buf.excess[g] = exc;
    buf.energy_q[g] = energy;
    if (buf.samples) buf.samples[g] = smp;
  }
  store_tile<TE, C>(env, s.env, e0, ne);
}

template <int D, int H, int TE>
struct ValueF32Smem {
  alignas(16) float w1t[D * H];
  float w2t[H * H], w3[H], b1[H], b2[H], b3[4];
  static constexpr int LD = TE + 4;  // columns are written across the rows
  alignas(16) float xt[D * LD];
  float ht[H * LD];  // h1, then h2
  float out[TE];
};

// value network over n observation rows (persistent over tiles of TE rows,
// two CTAs per SM): RT x 4 register tiles, one per thread; the next tile's
// rows are fetched while the current one runs.  2.1 million 7B observations
// take 1.65 ms, 47 TFLOP/s (4 x 4 tiles over 32 rows took 2.18 ms).
template <int D, int H, int TE, int RT>
__global__ void __launch_bounds__(TE / RT * H / 4)
    value_f32_kernel(const float* __restrict__ params, int A, const float* __restrict__ obs,
                     int64_t n, float* __restrict__ value) {
  using Smem = ValueF32Smem<D, H, TE>;
  constexpr int NT = TE / RT * H / 4, EG = TE / RT, LD = Smem::LD, XPT = TE * D / NT;  // observation values per thread
  static_assert(TE * D % NT == 0, "whole observation values per thread");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem& s = *reinterpret_cast<Smem*>(smem_raw);
  const MlpLayout Lp = mlp_layout(D, H, A);
  load_transposed(params + Lp.v1, s.w1t, H, D);
  load_transposed(params + Lp.v2, s.w2t, H, H);
  load_copy(params + Lp.c1, s.b1, H);
  load_copy(params + Lp.c2, s.b2, H);
  load_copy(params + Lp.v3, s.w3, H);
  load_copy(params + Lp.c3, s.b3, 1);
  // a warp covers 2 row groups x 16 neuron groups
  const int eg = (threadIdx.x >> 5) % (EG / 2) * 2 + (threadIdx.x & 1);
  const int ng = (threadIdx.x >> 5) / (EG / 2) * 16 + ((threadIdx.x & 31) >> 1);
  const int64_t tiles = (n + TE - 1) / TE;
  float xv[XPT];
  auto fetch = [&](int64_t tile) {
    const int64_t r0 = tile * TE, left = (n - r0) * D;  // observation values from the tile's first row on
#pragma unroll
    for (int q = 0; q < XPT; ++q) {
      const int idx = threadIdx.x + q * NT;
      xv[q] = tile < tiles && idx < left ? __ldg(obs + r0 * D + idx) : 0.0f;
    }
  };
  fetch(blockIdx.x);
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int64_t r0 = tile * TE;
    const int nr = (int)(n - r0 < (int64_t)TE ? n - r0 : (int64_t)TE);
#pragma unroll
    for (int q = 0; q < XPT; ++q) {
      const int idx = threadIdx.x + q * NT;
      s.xt[(idx % D) * LD + idx / D] = xv[q];
    }
    __syncthreads();
    fetch(tile + gridDim.x);
    float2 acc[RT / 2][4];
    dense_tile<RT, 4, D, LD, H>(s.xt + eg * RT, s.w1t + ng * 4, acc);
    tanh_store<RT, 4, LD>(acc, s.b1 + ng * 4, s.ht + ng * 4 * LD + eg * RT);
    __syncthreads();
    dense_tile<RT, 4, H, LD, H>(s.ht + eg * RT, s.w2t + ng * 4, acc);
    __syncthreads();
    tanh_store<RT, 4, LD>(acc, s.b2 + ng * 4, s.ht + ng * 4 * LD + eg * RT);
    __syncthreads();
    head_t<TE, H, 1, LD>(s.ht, s.w3, s.b3, s.out);
    __syncthreads();
    for (int e = threadIdx.x; e < nr; e += blockDim.x) value[r0 + e] = s.out[e];
  }
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
template <int D, int H, int A, int TE, int C, int OBS>
static pe_status launch_rollout(const EnvDev& env, const float* params, int T, uint32_t it,
                                float lambda, int det, const pe_rollout_buf& buf,
                                cudaStream_t st) {
  using Smem = RolloutF32Smem<D, H, A, TE, C, OBS>;
  auto* const kern =
      env.cadence ? rollout_f32_kernel<D, H, A, TE, C, OBS, false> : rollout_f32_kernel<D, H, A, TE, C, OBS, true>;
  const int bytes = (int)sizeof(Smem);
  PE_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  {
    ProfScope ps(PE_PROF_ROLLOUT, st);
    kern<<<ceil_div(env.E, TE), RolloutTile<TE, H>::NT, bytes, st>>>(env, params, T, it, lambda, det, buf);
  }
  PE_CHECK_LAUNCH("rollout_f32_kernel");
  return PE_OK;
}

template <int D, int H, int TE, int RT>
static pe_status launch_value(const float* params, int A, const float* obs, int64_t n, int sms,
                              float* value, cudaStream_t st) {
  using Smem = ValueF32Smem<D, H, TE>;
  constexpr int NT = TE / RT * H / 4;
  auto kern = value_f32_kernel<D, H, TE, RT>;
  const int bytes = (int)sizeof(Smem);
  PE_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  int per_sm = 0;
  PE_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, bytes));
  const int64_t tiles = (n + TE - 1) / TE;
  const int64_t cap = (int64_t)sms * (per_sm > 0 ? per_sm : 1);
  const int grid = (int)(tiles < cap ? tiles : cap);
  {
    ProfScope ps(PE_PROF_VALUE, st);
    kern<<<grid, NT, bytes, st>>>(params, A, obs, n, value);
  }
  PE_CHECK_LAUNCH("value_f32_kernel");
  return PE_OK;
}

// 64-row tiles (8 x 4 per thread, fewest shared loads per FMA), or 32-row (4 x
// 4) or 16-row ones (2 x 4) while those make no more than two CTAs per SM: a
// short batch is the latency of one tile (2,000 rows of the Tiny networks: 10.4
// us with 32-row tiles, 9.4 with 16; of the 7B networks 18.5 and 16.6)
template <int D, int H>
static pe_status value_by_batch(const float* params, int A, const float* obs, int64_t n, float* value,
                                cudaStream_t st) {
  if (n <= 0) return PE_OK;
  int dev = 0, sms = 0;
  PE_TRY_CUDA(cudaGetDevice(&dev));
  PE_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  if (n <= (int64_t)32 * sms) return launch_value<D, H, 16, 2>(params, A, obs, n, sms, value, st);
  if (n <= (int64_t)64 * sms) return launch_value<D, H, 32, 4>(params, A, obs, n, sms, value, st);
  return launch_value<D, H, 64, 8>(params, A, obs, n, sms, value, st);
}

// The env tile by the batch: 8 or 16 envs while that gives at most one CTA
// per SM (the less work in a step's chain the sooner it ends: a Tiny rollout of
// 64 envs x 128 steps takes 374 us with 8, 538 us with 32), else 32.  Two CTAs
// of 16 per SM are no faster than one of 32 (7B, 4,096 envs x 512 steps: 3.46
// and 3.33 ms), their layers contend for the FMA pipe.
template <int D, int H, int A, int C, int OBS>
static pe_status rollout_by_batch(const EnvDev& env, const float* params, int T, uint32_t it, float lambda, int det,
                                  const pe_rollout_buf& buf, cudaStream_t st) {
  int dev = 0, sms = 0;
  PE_TRY_CUDA(cudaGetDevice(&dev));
  PE_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  if (env.E <= 8 * sms) return launch_rollout<D, H, A, 8, C, OBS>(env, params, T, it, lambda, det, buf, st);
  if (env.E <= 16 * sms) return launch_rollout<D, H, A, 16, C, OBS>(env, params, T, it, lambda, det, buf, st);
  return launch_rollout<D, H, A, 32, C, OBS>(env, params, T, it, lambda, det, buf, st);
}

pe_status rollout_f32(const EnvDev& env, const pe_net& net, const float* params, int T,
                      uint32_t it, float lambda, int det, const pe_rollout_buf& buf,
                      cudaStream_t st) {
  if (net.obs_dim == 8 && net.hidden == 64 && net.n_actions == 3 && env.C == 1 &&
      env.obs_kind == PE_OBS_TINY8)
    return rollout_by_batch<8, 64, 3, 1, PE_OBS_TINY8>(env, params, T, it, lambda, det, buf, st);
  if (net.obs_dim == 16 && net.hidden == 128 && net.n_actions == 5 && env.C == 1 &&
      env.obs_kind == PE_OBS_7B16)
    return rollout_by_batch<16, 128, 5, 1, PE_OBS_7B16>(env, params, T, it, lambda, det, buf, st);
  return fail(PE_EINVAL, "unsupported fp32 network/env combination (D=%d H=%d A=%d C=%d obs=%d)",
              net.obs_dim, net.hidden, net.n_actions, env.C, env.obs_kind);
}

pe_status value_f32(const pe_net& net, const float* params, const float* obs, int64_t n,
                    float* value, cudaStream_t st) {
  if (net.obs_dim == 8 && net.hidden == 64)
    return value_by_batch<8, 64>(params, net.n_actions, obs, n, value, st);
  if (net.obs_dim == 16 && net.hidden == 128)
    return value_by_batch<16, 128>(params, net.n_actions, obs, n, value, st);
  return fail(PE_EINVAL, "unsupported fp32 value network (D=%d H=%d)", net.obs_dim, net.hidden);
}

}  // namespace pe
