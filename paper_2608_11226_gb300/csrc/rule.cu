// Baseline rule policies of the evaluation (Sec. 4.4 random policy and
// threshold heuristic, Sec. 4.5 hysteresis rule) and explicit episode starts
// for the full-trace replay.
//
// A rule rollout needs no network, so one thread (or, where a step consumes a
// batch of samples, a group of eight) runs one env through the whole horizon:
// decide from the state before the step, step (actuator, Eqs. 1-3, reward),
// record the action, reward and done flag, and the per-call counters.
#include <cuda_bf16.h>

#include <algorithm>

#include "env.cuh"

namespace pe {

// host-side twin declared in api.cu
struct RuleArgs {
  int32_t kind, hi_q, lo_q, drop30_q, climb30_q, climb10_q;
  int32_t T, obs_bf16;
  uint32_t it;
  float lambda;
  const uint8_t* forced;  // [T][E] actions of a replay (kind kRuleReplay)
};

// a replay (teacher-forced rollout): env e takes action forced[t][e] at step t
constexpr int32_t kRuleReplay = 4;

// lower / raise move one level: G for the inc/dec actuator (actions 1 and 2;
// the env keeps G in [g_min, g_max]), the level index otherwise (clamped).
// latest(): the latest actuated cluster sample; sums(s10, s30): the cluster's
// window sums.
template <class Latest, class Sums>
__device__ __forceinline__ int rule_action(const EnvDev& env, const RuleArgs& r, int lvl, uint32_t e, uint32_t t,
                                           Latest latest, Sums sums) {
  if (r.kind == kRuleReplay) return r.forced[(int64_t)t * env.E + e];
  const bool incdec = env.act_kind == PE_ACT_INCDEC;
  const int hold = incdec ? 0 : lvl;
  const int lower = incdec ? 1 : (lvl > 0 ? lvl - 1 : 0);
  const int raise = incdec ? 2 : (lvl < env.n_levels - 1 ? lvl + 1 : env.n_levels - 1);
  if (r.kind == PE_RULE_RANDOM) return (int)__umulhi(draw32(env.seed, e, t, r.it, kDrawAction), (uint32_t)env.A);
  if (r.kind == PE_RULE_THRESHOLD) {
    const int32_t q = latest();
    return q > r.hi_q ? lower : (q < r.lo_q ? raise : hold);
  }
  int64_t s10 = 0, s30 = 0;
  sums(s10, s30);
  if (s30 > (int64_t)kWLong * r.drop30_q) return lower;
  return (s30 < (int64_t)kWLong * r.climb30_q && s10 < (int64_t)kWShort * r.climb10_q) ? raise : hold;
}

// blocks of two warps, so that a few thousand envs reach every SM
constexpr int kRuleThreads = 64;

template <int C, int OBS, int D>
__device__ __forceinline__ void write_obs(const EnvDev& env, RegAcc<C>& a, void* dst, int bf16) {
  const Fam fm = fam_of(env, a.fam());
  if constexpr (OBS == PE_OBS_OCC32 || OBS == PE_OBS_OCC64) {
    float v[D];
    Recent<C, OBS> h;
    load_recent<C, OBS>(env, a, fm, a.pos() - 1, h);
    features_eq5<C, OBS, D>(env, a, fm, h, v);
    if (bf16) {
      __nv_bfloat16* o = reinterpret_cast<__nv_bfloat16*>(dst);
#pragma unroll
      for (int f = 0; f < D; ++f) o[f] = __float2bfloat16_rn(v[f]);
    } else {
      float* o = reinterpret_cast<float*>(dst);
#pragma unroll
      for (int f = 0; f < D; ++f) o[f] = v[f];
    }
    return;
  }
  if (bf16) {
    __nv_bfloat16* o = reinterpret_cast<__nv_bfloat16*>(dst);
#pragma unroll 1
    for (int f = 0; f < D; ++f) o[f] = __float2bfloat16_rn(feature<C, OBS>(env, a, fm, f));
  } else {
    float* o = reinterpret_cast<float*>(dst);
#pragma unroll 1
    for (int f = 0; f < D; ++f) o[f] = feature<C, OBS>(env, a, fm, f);
  }
}

template <int C, int OBS, int D, bool ONE>
__global__ void __launch_bounds__(kRuleThreads) rule_rollout_kernel(EnvDev env, RuleArgs r, pe_rollout_buf buf) {
  __shared__ EnvTab<C> tab;
  load_tab<C>(env, tab);
  __syncthreads();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= env.E) return;
  RegAcc<C> acc = load_reg<C>(env, tab, e);
  const size_t ob = r.obs_bf16 ? 2 : 4;
  int32_t v1 = 0, v60 = 0;
  float tok = 0.0f, exc = 0.0f;
  int64_t en = 0, smp = 0;
  for (int t = 0; t < r.T; ++t) {
    const int64_t row = (int64_t)t * env.E + e;
    if (buf.obs) write_obs<C, OBS, D>(env, acc, reinterpret_cast<char*>(buf.obs) + row * D * ob, r.obs_bf16);
    const int act = rule_action(
        env, r, acc.level(), (uint32_t)e, (uint32_t)t, [&] { return Qcl<C>(env, acc, fam_of(env, acc.fam()), 0); },
        [&](int64_t& s10, int64_t& s30) {
#pragma unroll
          for (int c = 0; c < C; ++c) {
            s10 += acc.ss(c);
            s30 += acc.sl(c);
          }
        });
    const StepOut so = env_step<C, ONE>(env, acc, act, r.lambda);
    buf.act[row] = (uint8_t)act;
    buf.reward[row] = so.reward;
    buf.done[row] = (uint8_t)so.done;
    if (buf.q) buf.q[row] = so.q;
    v1 += so.v1;
    v60 += so.v60;
    tok += so.tokens;
    exc += so.excess;
    en += so.q;
    smp += so.samples;
    if (so.done) env_reset<C>(env, acc, (uint32_t)e, (uint32_t)t, r.it, kDrawReset);
  }
  if (buf.obs_last) write_obs<C, OBS, D>(env, acc, reinterpret_cast<char*>(buf.obs_last) + (int64_t)e * D * ob, r.obs_bf16);
  buf.viol[2 * e] = v1;
  buf.viol[2 * e + 1] = v60;
  buf.tokens[e] = tok;
  buf.excess[e] = exc;
  buf.energy_q[e] = en;
  if (buf.samples) buf.samples[e] = smp;
  store_reg<C>(env, e, acc);
}

// ---------------------------------------------------------------------------
// A step that consumes a batch of samples (cadence table), without
// observations: eight lanes run one env, lane u taking samples u, u + 8, ..
// of each batch, with the last 64 actuated samples of every channel in shared
// memory.  A batch's windows are a running sum over its samples (Eq. 1's
// cluster totals, scanned across the lanes; whole numbers, so in any order);
// per-channel sums stay as each lane's own part until they are wanted.  The
// floating sums of a step are added in sample order, as by one thread.
//
// One thread per env was bound by the latency of a serial chain with two warps
// per SM, and by the L1: each sample's three 16-byte loads of the trace were
// 32 lines per warp.  Here a warp has four times as many in flight, its loads
// are 128 bytes per env, and the samples 20 and 60 back are not recomputed.
// Replaying 64 steps of 24 to 42 samples in 10,007 envs: 845 to 298 us.
// Below eight samples per step lanes idle, and the observations' features need
// the whole history per lane: those stay with one thread per env.
constexpr int kGroup = 8;
constexpr int kGroupThreads = 128;
constexpr int kGroupEnvs = kGroupThreads / kGroup;

template <int C>
struct GroupEnv {
  struct alignas(4 * C) Q {
    int32_t v[C];
  };
  Q q[kRing];                          // actuated samples, position p in slot p & 63
  alignas(16) uint8_t level[kRing];  // and the level of each
};

// the state env_step changes, as the accessors of apply_action see it
struct GroupAcc {
  int32_t pos_, k_, level_, prev_, b_, til_, fam_;
  __device__ int32_t& level() { return level_; }
  __device__ int32_t& prev() { return prev_; }
  __device__ int32_t& b() { return b_; }
  __device__ int32_t& til() { return til_; }
};

// the group's 60 samples before pos at the recorded levels into its ring; each
// lane's part of the window sums; returns the lane's part of the cluster's
// 30 s sum
template <int C>
__device__ __forceinline__ int32_t group_history(const EnvDev& env, const EnvTab<C>& tab, const Fam& fm, int pos,
                                                 int u, GroupEnv<C>& ge, int32_t (&ss)[C], int32_t (&sl)[C]) {
  int32_t s60 = 0;
#pragma unroll
  for (int c = 0; c < C; ++c) ss[c] = sl[c] = 0;
#pragma unroll 4
  for (int i = u + 1; i <= kWLong; i += kGroup) {
    const int pp = pos - i;
    typename GroupEnv<C>::Q q;
    sample_q<C>(tab, load_samp<C>(env, fm, pp), ge.level[pp & (kRing - 1)], q.v);
    ge.q[pp & (kRing - 1)] = q;
#pragma unroll
    for (int c = 0; c < C; ++c) {
      sl[c] += q.v[c];
      if (i <= kWShort) ss[c] += q.v[c];
      s60 += q.v[c];
    }
  }
  return s60;
}

template <int C, int OBS, int D>
__global__ void __launch_bounds__(kGroupThreads) rule_group_kernel(EnvDev env, RuleArgs r, pe_rollout_buf buf) {
  __shared__ EnvTab<C> tab;
  __shared__ GroupEnv<C> envs[kGroupEnvs];
  load_tab<C>(env, tab);
  const int lane = threadIdx.x & 31, u = lane & (kGroup - 1);
  const int g = blockIdx.x * kGroupEnvs + threadIdx.x / kGroup;
  // groups past the last env repeat it and write nothing
  const bool live = g < env.E;
  const int e = live ? g : env.E - 1;
  const uint32_t gmask = 0xFFu << (lane & 24);
  GroupEnv<C>& ge = envs[threadIdx.x / kGroup];
  GroupAcc a;
  a.pos_ = env.st[kStPos * env.E + e];
  a.k_ = env.st[kStK * env.E + e];
  a.level_ = env.st[kStLevel * env.E + e];
  a.prev_ = env.st[kStPrev * env.E + e];
  a.b_ = env.st[kStB * env.E + e];
  a.til_ = env.st[kStTil * env.E + e];
  a.fam_ = env.st[kStFam * env.E + e];
  reinterpret_cast<uint2*>(ge.level)[u] = reinterpret_cast<const uint2*>(env.ring + (int64_t)e * kRing)[u];
  __syncthreads();  // tables and rings written; a repeated env's state read before its owner stores it
  Fam fm = fam_of(env, a.fam_);
  int32_t ss[C], sl[C];  // this lane's part of the window sums
  auto group_sum = [&](int32_t v) {
#pragma unroll
    for (int o = 1; o < kGroup; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  int32_t S60 = group_sum(group_history<C>(env, tab, fm, a.pos_, u, ge, ss, sl));  // the cluster's 30 s sum
  __syncwarp();
  // the sample at position p for this lane; lanes past a batch's end may stand
  // past the trace's
  auto fetch = [&](int p) { return load_samp<C>(env, fm, min(p, fm.L - 1)); };
  Samp<C> s = fetch(a.pos_ + u);
  int32_t v1 = 0, v60 = 0;
  float tok = 0.0f, exc = 0.0f;
  int64_t en = 0, smp = 0;
  for (int t = 0; t < r.T; ++t) {
    const int64_t row = (int64_t)t * env.E + e;
    const int act = rule_action(
        env, r, a.level_, (uint32_t)e, (uint32_t)t,
        [&] {
          const typename GroupEnv<C>::Q q = ge.q[(a.pos_ - 1) & (kRing - 1)];
          int32_t v = 0;
#pragma unroll
          for (int c = 0; c < C; ++c) v += q.v[c];
          return v;
        },
        [&](int64_t& s10, int64_t& s30) {
          int32_t v = 0;
#pragma unroll
          for (int c = 0; c < C; ++c) v += ss[c];
          s10 = group_sum(v);
          s30 = S60;
        });
    const int nl = apply_action(env, a, act);
    const float rate = token_rate(env, a, tab.tokens[nl]);
    const int64_t B60 = (int64_t)kWLong * fm.B;
    const int n = tab.ns[nl];
    StepOut o;
    o.tokens = 0.0f;
    o.excess = 0.0f;
    float peak_w = 0.0f, fixed = 0.0f;
    int32_t oq = 0, o1 = 0, o60 = 0;
    for (int i = 0; __any_sync(0xffffffffu, i < n); i += kGroup) {
      const bool in = i + u < n;
      const int p = a.pos_ + i + u;
      const Samp<C> cur = s;
      // the next batch's sample, or the next step's first
      if (i < n) s = fetch(i + kGroup < n ? p + kGroup : a.pos_ + n + u);
      typename GroupEnv<C>::Q q;
      int32_t dq = 0, Q = 0;
      if (in) {
        const typename GroupEnv<C>::Q q20 = ge.q[(p - kWShort) & (kRing - 1)], q60 = ge.q[(p - kWLong) & (kRing - 1)];
        sample_q<C>(tab, cur, nl, q.v);
#pragma unroll
        for (int c = 0; c < C; ++c) {
          ss[c] += q.v[c] - q20.v[c];
          sl[c] += q.v[c] - q60.v[c];
          dq += q.v[c] - q60.v[c];
          Q += q.v[c];
        }
      }
#pragma unroll
      for (int k = 1; k < kGroup; k <<= 1) {
        const int32_t x = __shfl_up_sync(0xffffffffu, dq, k, kGroup);
        if (u >= k) dq += x;
      }
      const int64_t S = (int64_t)S60 + dq;
      S60 += __shfl_sync(0xffffffffu, dq, kGroup - 1, kGroup);
      __syncwarp();  // every lane has read the history of 60 back: slots p - 60 and p + 4 are one
      if (in) {
        ge.q[p & (kRing - 1)] = q;
        ge.level[p & (kRing - 1)] = (uint8_t)nl;
      }
      const bool w60 = in && S > B60;
      const float exc_w = w60 ? __fdiv_rn(__ll2float_rn(S - B60), 3840.0f) : 0.0f;  // watts over B
      const uint32_t m1 = __ballot_sync(0xffffffffu, in && Q > fm.B) >> (lane & 24) & 0xFFu;
      const uint32_t all60 = __ballot_sync(0xffffffffu, w60), m60 = all60 >> (lane & 24) & 0xFFu;
      const uint32_t m0 = __ballot_sync(0xffffffffu, in && cur.ph == 0) >> (lane & 24) & 0xFFu;
      oq += Q;
      o1 += __popc(m1);
      o60 += __popc(m60);
      peak_w = fmaxf(peak_w, exc_w);
      if (all60) {
#pragma unroll
        for (int k = 0; k < kGroup; ++k) o.excess += __shfl_sync(0xffffffffu, exc_w * 0.5f, k, kGroup);
      }
      const int n0 = __popc(m0);
#pragma unroll
      for (int k = 0; k < kGroup; ++k) o.tokens += k < n0 ? rate : 0.0f;
      if (env.reward_kind != PE_REWARD_LAGRANGE) {
        const uint32_t mv = env.reward_window == 1 ? m1 : m60;
#pragma unroll
        for (int k = 0; k < kGroup; ++k)
          if (i + k < n) fixed += ((mv >> k & 1) ? env.r_viol : env.r_ok) + env.bonus_coef * rate * env.inv_rate_max;
      }
      __syncwarp();
    }
#pragma unroll
    for (int k = 1; k < kGroup; k <<= 1) peak_w = fmaxf(peak_w, __shfl_xor_sync(0xffffffffu, peak_w, k));
    oq = group_sum(oq);
    const float reward = step_reward(env, o, r.lambda, peak_w, fixed);
    a.pos_ += n;
    a.k_ += 1;
    const bool done = a.k_ == env.ep_len;
    if (u == 0 && live) {
      buf.act[row] = (uint8_t)act;
      buf.reward[row] = reward;
      buf.done[row] = (uint8_t)done;
      if (buf.q) buf.q[row] = oq;
    }
    v1 += o1;
    v60 += o60;
    tok += o.tokens;
    exc += o.excess;
    en += oq;
    smp += n;
    if (done) {
      // a new episode (env_reset), its history shared out between the lanes
      const u32x4 w = philox10(u32x4{(uint32_t)e, (uint32_t)t, r.it, kDrawReset}, (uint32_t)env.seed,
                               (uint32_t)(env.seed >> 32));
      int fam;
      a.pos_ = reset_offset(env, w, fam);
      a.fam_ = fam;
      fm = fam_of(env, fam);
      a.k_ = 0;
      a.level_ = a.prev_ = env.level_init;
      a.b_ = env.b_init;
      a.til_ = 0;
      const uint32_t lw = 0x01010101u * (uint32_t)env.level_init;
      reinterpret_cast<uint2*>(ge.level)[u] = make_uint2(lw, lw);
      __syncwarp(gmask);
      S60 = (int32_t)__reduce_add_sync(gmask, group_history<C>(env, tab, fm, a.pos_, u, ge, ss, sl));
      s = fetch(a.pos_ + u);
    }
    __syncwarp();
  }
  int32_t s8[8];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    s8[c] = c < C ? group_sum(ss[c < C ? c : 0]) : 0;
    s8[4 + c] = c < C ? group_sum(sl[c < C ? c : 0]) : 0;
  }
  if (!live) return;
  reinterpret_cast<uint2*>(env.ring + (int64_t)e * kRing)[u] = reinterpret_cast<const uint2*>(ge.level)[u];
  if (u != 0) return;
  RegAcc<C> acc(tab);
  acc.pos_ = a.pos_;
  acc.k_ = a.k_;
  acc.level_ = a.level_;
  acc.prev_ = a.prev_;
  acc.b_ = a.b_;
  acc.til_ = a.til_;
  acc.fam_ = a.fam_;
  acc.ring = ge.level;
#pragma unroll
  for (int c = 0; c < C; ++c) {
    acc.ss_[c] = s8[c];
    acc.sl_[c] = s8[4 + c];
  }
  store_reg<C>(env, e, acc);
  if (buf.obs_last)
    write_obs<C, OBS, D>(env, acc, reinterpret_cast<char*>(buf.obs_last) + (int64_t)e * D * (r.obs_bf16 ? 2 : 4),
                         r.obs_bf16);
  buf.viol[2 * e] = v1;
  buf.viol[2 * e + 1] = v60;
  buf.tokens[e] = tok;
  buf.excess[e] = exc;
  buf.energy_q[e] = en;
  if (buf.samples) buf.samples[e] = smp;
}

// every env starts a new episode at offsets[e]; offsets outside
// [60, L - episode_len] set *flag and leave that env unchanged
template <int C>
__global__ void env_offsets_kernel(EnvDev env, const int32_t* __restrict__ offsets, int32_t* __restrict__ flag) {
  __shared__ EnvTab<C> tab;
  load_tab<C>(env, tab);
  __syncthreads();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= env.E) return;
  const int o = offsets[e];
  const int fam = env.st[kStFam * env.E + e];
  if (o < kWLong || o > fam_of(env, fam).L - env.span) {
    atomicOr(flag, 1);
    return;
  }
  RegAcc<C> a(tab);
  a.ring = env.ring + (int64_t)e * kRing;
  a.fam() = fam;  // the env keeps its episode's trace family
  env_reset_at<C>(env, a, o);
  store_reg<C>(env, e, a);
}

// a replay's actions must lie in [0, A)
__global__ void replay_check_kernel(const uint8_t* __restrict__ act, int64_t n, int A, int32_t* __restrict__ flag) {
  int bad = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    bad |= act[i] >= A;
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, 1);
}

pe_status replay_check(const uint8_t* act, int64_t n, int A, int32_t* flag, cudaStream_t st) {
  PE_TRY_CUDA(cudaMemsetAsync(flag, 0, sizeof(int32_t), st));
  replay_check_kernel<<<(int)std::min<int64_t>(ceil_div(n, 256), 4096), 256, 0, st>>>(act, n, A, flag);
  PE_CHECK_LAUNCH("replay_check_kernel");
  int32_t host = 0;
  PE_TRY_CUDA(cudaMemcpyAsync(&host, flag, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  PE_TRY_CUDA(cudaStreamSynchronize(st));
  if (host) return fail(PE_EINVAL, "replay action outside [0, A)");
  return PE_OK;
}

template <int C, int OBS, int D>
static void launch_rule(const EnvDev& env, const RuleArgs& r, const pe_rollout_buf& buf, cudaStream_t st) {
  int least = env.ns[0];
  for (int l = 1; l < env.n_levels; ++l) least = std::min(least, env.ns[l]);
  if (env.cadence && !buf.obs && least >= kGroup) {
    rule_group_kernel<C, OBS, D><<<ceil_div(env.E, kGroupEnvs), kGroupThreads, 0, st>>>(env, r, buf);
    return;
  }
  auto* const kern = env.cadence ? rule_rollout_kernel<C, OBS, D, false> : rule_rollout_kernel<C, OBS, D, true>;
  kern<<<ceil_div(env.E, kRuleThreads), kRuleThreads, 0, st>>>(env, r, buf);
}

pe_status rule_rollout(const EnvDev& env, const RuleArgs& r, const pe_rollout_buf& buf, cudaStream_t st) {
  ProfScope ps(PE_PROF_ROLLOUT, st);
  if (env.C == 1 && env.obs_kind == PE_OBS_TINY8) launch_rule<1, PE_OBS_TINY8, 8>(env, r, buf, st);
  else if (env.C == 1 && env.obs_kind == PE_OBS_7B16) launch_rule<1, PE_OBS_7B16, 16>(env, r, buf, st);
  else if (env.C == 4 && env.obs_kind == PE_OBS_OCC32) launch_rule<4, PE_OBS_OCC32, 32>(env, r, buf, st);
  else if (env.C == 4 && env.obs_kind == PE_OBS_OCC64) launch_rule<4, PE_OBS_OCC64, 64>(env, r, buf, st);
  else
    return fail(PE_EINVAL, "rule rollout: unsupported env (C=%d, obs kind %d)", env.C, env.obs_kind);
  PE_CHECK_LAUNCH("rule_rollout_kernel");
  return PE_OK;
}

pe_status env_set_offsets(const EnvDev& env, const int32_t* offsets, int32_t* flag, cudaStream_t st) {
  const int grid = ceil_div(env.E, 128);
  PE_TRY_CUDA(cudaMemsetAsync(flag, 0, sizeof(int32_t), st));
  switch (env.C) {
    case 1: env_offsets_kernel<1><<<grid, 128, 0, st>>>(env, offsets, flag); break;
    case 2: env_offsets_kernel<2><<<grid, 128, 0, st>>>(env, offsets, flag); break;
    case 3: env_offsets_kernel<3><<<grid, 128, 0, st>>>(env, offsets, flag); break;
    default: env_offsets_kernel<4><<<grid, 128, 0, st>>>(env, offsets, flag); break;
  }
  PE_CHECK_LAUNCH("env_offsets_kernel");
  int32_t h = 0;
  PE_TRY_CUDA(cudaMemcpyAsync(&h, flag, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  PE_TRY_CUDA(cudaStreamSynchronize(st));
  if (h) return fail(PE_EINVAL, "episode offset outside [60, L - episode_len x max(level_samples)]");
  return PE_OK;
}

// Dual ascent on the Eq. 6 multiplier (Eq. 7; the additive G3 form with the
// same relative gap): one block sums the rollout's violation counts exactly
// (int64), then one thread updates lambda in place.  The scalar update runs
// in fp64 (a handful of operations).
__global__ void __launch_bounds__(1024) dual_ascent_kernel(const int32_t* __restrict__ viol, int E, int64_t steps,
                                                           int col, int additive, float target, float eta, float lo,
                                                           float hi, float* __restrict__ lambda,
                                                           float* __restrict__ rate) {
  __shared__ long long red[32];
  long long n = 0;
  for (int e = threadIdx.x; e < E; e += blockDim.x) n += viol[2 * e + col];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = n;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long t = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    const double v = (double)t / ((double)E * (double)steps);
    const double gap = (v - (double)target) / (double)target;
    double l = additive ? (double)*lambda + (double)eta * gap : (double)*lambda * exp((double)eta * gap);
    l = l < (double)lo ? (double)lo : (l > (double)hi ? (double)hi : l);
    *lambda = (float)l;
    if (rate) *rate = (float)v;
  }
}

pe_status dual_ascent(const int32_t* viol, int E, int64_t steps, int window, int additive, float target,
                      float eta, float lo, float hi, float* lambda, float* rate, cudaStream_t st) {
  {
    ProfScope ps(PE_PROF_PPO_OTHER, st);
    dual_ascent_kernel<<<1, 1024, 0, st>>>(viol, E, steps, window == 1 ? 0 : 1, additive, target, eta, lo, hi,
                                           lambda, rate);
  }
  PE_CHECK_LAUNCH("dual_ascent_kernel");
  return PE_OK;
}

}  // namespace pe
