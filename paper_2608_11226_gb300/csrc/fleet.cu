// Fleet window accounting (Sec. 7 window analysis, Sec. 8 composed fleet).
//
// q_g = rint(64 x_g) per GPU (1/64 W) is summed per job (a job's GPUs share a
// start offset); composition n adds the J job rows at its offsets, and every
// window count and peak comes from differences of a running prefix of that
// sum, exact in 32 bits because the true window sums are below 2^31 (checked
// on the host from the per-job maxima).  What bounds the count is moving the
// job rows from L2 to the SMs, so the rows are kept as narrow as the traces
// allow, which the call learns from the per-job ranges that it reads back
// with the validation flag:
//   - J <= 8, ranges within 16 bits: 16-bit samples above the job's minimum,
//     in eight shifted copies (fleet_windows_h16_kernel, 2 bytes per job and
//     sample; the warp rebuilds the prefix with a scan);
//   - J <= 8, wider ranges: per-job prefix sums over the period unrolled once,
//       PREX[j][i] = sum_{k < i} sum_{g in j} q_g(k mod L),  i in [0, L + H],
//     modulo 2^32, in four shifted copies (fleet_windows_v4_kernel, 4 bytes);
//   - J <= 8 with a workspace of one copy only (fleet_windows_j8_kernel) and
//     J > 8 (fleet_windows_kernel): the same prefixes through 4-byte loads.
// One warp per composition walks t (per part of the horizon when there are
// few compositions), keeps the running prefix in a 1024-slot shared-memory
// ring, and reads pre(t - w) back for every window w <= 992 at once.
#include <algorithm>
#include <climits>
#include <type_traits>

#include "common.cuh"

namespace pe {

constexpr int kFleetRing = 1024;
constexpr int kFleetWarps = 8;
constexpr int kFleetChunk = 8192;   // prefix-scan chunk per block
constexpr float kFleetMaxWatts = 65536.0f;

struct FleetWs {
  uint32_t* prex;    // [J][Lp]
  uint32_t* totals;  // [J][nchunk] chunk sums, then exclusive chunk offsets
  int32_t* maxq;     // [32]: largest job sample, then [32]: INT_MAX less the smallest
  int32_t* flag;     // [1]: bit 0 bad sample, bit 1 bad job map, bit 2 bad offset
  int64_t Lp;        // row stride of prex
  int nchunk;
};

// the GPUs of job j, listed in shared memory by the block's first warp
struct JobGpus {
  int n;
  uint8_t g[64];
};

__device__ __forceinline__ void list_gpus(const int32_t* __restrict__ job_of_gpu, int G, int J, int j, JobGpus& s,
                                          int32_t* flag) {
  if (threadIdx.x < 32) {
    int n = 0;
    for (int g0 = 0; g0 < G; g0 += 32) {
      const int g = g0 + (int)threadIdx.x;
      const int jj = g < G ? job_of_gpu[g] : j;
      if (jj < 0 || jj >= J) atomicOr(flag, 2);
      const bool mine = g < G && jj == j;
      const uint32_t m = __ballot_sync(0xffffffffu, mine);
      if (mine) s.g[n + __popc(m & ((1u << threadIdx.x) - 1u))] = (uint8_t)g;
      n += __popc(m);
    }
    if (threadIdx.x == 0) s.n = n;
  }
  __syncthreads();
}

// sample i of a job's unrolled row (i < L + H <= INT32_MAX)
__device__ __forceinline__ int32_t job_sample(const float* __restrict__ traces, const JobGpus& s, int L, int i,
                                              int& bad) {
  const int src = i < L ? i : (int)((uint32_t)i % (uint32_t)L);
  int32_t q = 0;
  for (int k = 0; k < s.n; ++k) {
    const float x = __ldg(traces + (int64_t)s.g[k] * L + src);
    if (!(x >= 0.0f && x <= kFleetMaxWatts)) {
      bad = 1;
      continue;
    }
    q += __float2int_rn(x * 64.0f);
  }
  return q;
}

// per-job range of the samples (atomic maxima of q and of INT_MAX - q) and
// validation of the samples and the job map
constexpr int kRangeChunk = 2048;
__global__ void __launch_bounds__(256) fleet_range_kernel(const float* __restrict__ traces, int G, int L,
                                                          const int32_t* __restrict__ job_of_gpu, int J, FleetWs ws) {
  __shared__ JobGpus gpus;
  const int j = blockIdx.y;
  list_gpus(job_of_gpu, G, J, j, gpus, ws.flag);
  const int64_t i0 = (int64_t)blockIdx.x * kRangeChunk;
  int32_t hi = 0, lo = 0;
  int bad = 0;
#pragma unroll
  for (int k = 0; k < kRangeChunk / 256; ++k) {
    const int64_t i = i0 + k * 256 + threadIdx.x;
    if (i < L) {
      const int32_t q = job_sample(traces, gpus, L, (int)i, bad);
      hi = max(hi, q);
      lo = max(lo, INT_MAX - q);
    }
  }
  hi = __reduce_max_sync(0xffffffffu, hi);
  lo = __reduce_max_sync(0xffffffffu, lo);
  bad = __any_sync(0xffffffffu, bad);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(ws.maxq + j, hi);
    atomicMax(ws.maxq + 32 + j, lo);
    if (bad) atomicOr(ws.flag, 1);
  }
}

// prefix pass 1: per (job, chunk) sum
__global__ void __launch_bounds__(256) fleet_chunk_sums_kernel(const float* __restrict__ traces, int G, int L, int H,
                                                               const int32_t* __restrict__ job_of_gpu,
                                                               int J, FleetWs ws) {
  __shared__ JobGpus gpus;
  __shared__ uint32_t ss[8];
  const int j = blockIdx.y, c = blockIdx.x;
  list_gpus(job_of_gpu, G, J, j, gpus, ws.flag);
  const int64_t Lx = (int64_t)L + H;
  const int64_t i0 = (int64_t)c * kFleetChunk;
  uint32_t s = 0;
  int bad = 0;  // reported by fleet_range_kernel
  for (int64_t i = i0 + threadIdx.x; i < min(i0 + kFleetChunk, Lx); i += blockDim.x)
    s += (uint32_t)job_sample(traces, gpus, L, (int)i, bad);
  s = __reduce_add_sync(0xffffffffu, s);
  if ((threadIdx.x & 31) == 0) ss[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < 8; ++k) s += ss[k];
    ws.totals[(int64_t)j * ws.nchunk + c] = s;
  }
}

// prefix pass 2: exclusive scan of each job's chunk sums (one warp per job)
__global__ void fleet_chunk_scan_kernel(FleetWs ws) {
  const int j = blockIdx.x, lane = threadIdx.x;
  uint32_t carry = 0;
  for (int c0 = 0; c0 < ws.nchunk; c0 += 32) {
    const int c = c0 + lane;
    const uint32_t v = c < ws.nchunk ? ws.totals[(int64_t)j * ws.nchunk + c] : 0u;
    uint32_t x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
      if (lane >= d) x += y;
    }
    if (c < ws.nchunk) ws.totals[(int64_t)j * ws.nchunk + c] = carry + x - v;
    carry += __shfl_sync(0xffffffffu, x, 31);
  }
}

// prefix pass 3: prefix within each chunk, offset by the chunk's exclusive sum
__global__ void __launch_bounds__(256) fleet_prefix_kernel(const float* __restrict__ traces, int G, int L, int H,
                                                           const int32_t* __restrict__ job_of_gpu,
                                                           int J, FleetWs ws) {
  __shared__ JobGpus gpus;
  __shared__ uint32_t wsum[8];
  const int j = blockIdx.y, c = blockIdx.x;
  list_gpus(job_of_gpu, G, J, j, gpus, ws.flag);
  const int64_t Lx = (int64_t)L + H;
  const int64_t i0 = (int64_t)c * kFleetChunk;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t carry = ws.totals[(int64_t)j * ws.nchunk + c];
  uint32_t* row = ws.prex + (int64_t)j * ws.Lp;
  if (c == 0 && threadIdx.x == 0) row[0] = 0u;
  int bad = 0;
  for (int64_t b = i0; b < min(i0 + kFleetChunk, Lx); b += blockDim.x) {
    const int64_t i = b + threadIdx.x;
    const uint32_t q = i < Lx ? (uint32_t)job_sample(traces, gpus, L, (int)i, bad) : 0u;
    uint32_t x = q;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
      if (lane >= d) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    uint32_t before = 0, total = 0;
    for (int k = 0; k < 8; ++k) {
      if (k < w) before += wsum[k];
      total += wsum[k];
    }
    if (i < Lx) row[i + 1] = carry + before + x;
    carry += total;
    __syncthreads();
  }
}

__global__ void fleet_check_offsets_kernel(const int32_t* __restrict__ off, int64_t n, int L,
                                           int32_t* flag) {
  int bad = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t o = __ldg(off + i);
    bad |= (o < 0 || o >= L);
  }
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, 4);
}

struct FleetWindows {
  int32_t w[4];
  int32_t bw[4];  // budget_q * w
};

template <int NW>
__global__ void __launch_bounds__(32 * kFleetWarps)
    fleet_windows_kernel(const uint32_t* __restrict__ prex, int J, int64_t Lp,
                         const int32_t* __restrict__ offsets, int64_t N, int H, FleetWindows win,
                         int32_t* __restrict__ counts, int32_t* __restrict__ peaks) {
  __shared__ uint32_t ring_all[kFleetWarps][kFleetRing];
  __shared__ const uint32_t* base_all[kFleetWarps][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t n = (int64_t)blockIdx.x * kFleetWarps + wid;
  if (n >= N) return;  // the whole warp leaves together; no block-wide barrier follows
  uint32_t* ring = ring_all[wid];
  const uint32_t** base = base_all[wid];
  uint32_t pre_m1 = 0;  // pre(-1) = sum_j PREX[j][o_j]
  if (lane < J) {
    const int32_t o = __ldg(offsets + n * J + lane);
    const uint32_t* b = prex + (int64_t)lane * Lp + o;
    base[lane] = b + 1;
    pre_m1 = __ldg(b);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) pre_m1 += __shfl_xor_sync(0xffffffffu, pre_m1, o);
  if (lane == 0) ring[kFleetRing - 1] = pre_m1;
  __syncwarp();
  const uint32_t* b0 = base[0];
  int32_t cnt[NW], pk[NW];
#pragma unroll
  for (int k = 0; k < NW; ++k) cnt[k] = pk[k] = 0;
  for (int t0 = 0; t0 < H; t0 += 32) {
    const int t = t0 + lane;
    uint32_t pre = 0;
    if (t < H) {
      pre = __ldg(b0 + t);
      for (int j = 1; j < J; ++j) pre += __ldg(base[j] + t);
    }
    ring[t & (kFleetRing - 1)] = pre;
    __syncwarp();
    if (t < H) {
#pragma unroll
      for (int k = 0; k < NW; ++k) {
        const int w = win.w[k];
        if (t >= w - 1) {
          const int32_t S = (int32_t)(pre - ring[(t - w) & (kFleetRing - 1)]);
          cnt[k] += S > win.bw[k];
          pk[k] = max(pk[k], S);
        }
      }
    }
    __syncwarp();
  }
#pragma unroll
  for (int k = 0; k < NW; ++k) {
    int32_t c = cnt[k], p = pk[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      c += __shfl_xor_sync(0xffffffffu, c, o);
      p = max(p, __shfl_xor_sync(0xffffffffu, p, o));
    }
    if (lane == 0) {
      counts[n * NW + k] = c;
      peaks[n * NW + k] = p;
    }
  }
}

// The same walk for fleets of at most 8 jobs: the J stream pointers live
// in registers (no shared-memory pointer reloads), and each iteration
// issues the loads of two 32-sample blocks before using either.
constexpr int kFleetJMax = 8;

template <int NW>
__global__ void __launch_bounds__(32 * kFleetWarps)
    fleet_windows_j8_kernel(const uint32_t* __restrict__ prex, int J, int64_t Lp,
                            const int32_t* __restrict__ offsets, int64_t N, int H, FleetWindows win,
                            int32_t* __restrict__ counts, int32_t* __restrict__ peaks) {
  __shared__ uint32_t ring_all[kFleetWarps][kFleetRing];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t n = (int64_t)blockIdx.x * kFleetWarps + wid;
  if (n >= N) return;  // the whole warp leaves together; no block-wide barrier follows
  uint32_t* ring = ring_all[wid];
  // every lane holds all J stream bases (t = 0 at index 1 + o_j); lane j also
  // loads pre(-1)'s term PREX[j][o_j]
  const uint32_t* bp[kFleetJMax];
  uint32_t pre_m1 = 0;
#pragma unroll
  for (int j = 0; j < kFleetJMax; ++j) {
    bp[j] = prex;
    if (j < J) {
      const int32_t o = __ldg(offsets + n * J + j);
      bp[j] = prex + (int64_t)j * Lp + o + 1;
      if (lane == j) pre_m1 = __ldg(bp[j] - 1);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) pre_m1 += __shfl_xor_sync(0xffffffffu, pre_m1, o);
  if (lane == 0) ring[kFleetRing - 1] = pre_m1;
  __syncwarp();
  int32_t cnt[NW], pk[NW];
#pragma unroll
  for (int k = 0; k < NW; ++k) cnt[k] = pk[k] = 0;
  for (int t0 = 0; t0 < H; t0 += 64) {
    const int ta = t0 + lane, tb = t0 + 32 + lane;
    uint32_t pa = 0, pb = 0;
#pragma unroll
    for (int j = 0; j < kFleetJMax; ++j) {
      if (j < J) {
        if (ta < H) pa += __ldg(bp[j] + ta);
        if (tb < H) pb += __ldg(bp[j] + tb);
      }
    }
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int t = half ? tb : ta;
      const uint32_t pre = half ? pb : pa;
      ring[t & (kFleetRing - 1)] = pre;
      __syncwarp();
      if (t < H) {
#pragma unroll
        for (int k = 0; k < NW; ++k) {
          const int w = win.w[k];
          if (t >= w - 1) {
            const int32_t S = (int32_t)(pre - ring[(t - w) & (kFleetRing - 1)]);
            cnt[k] += S > win.bw[k];
            pk[k] = max(pk[k], S);
          }
        }
      }
      __syncwarp();
    }
  }
#pragma unroll
  for (int k = 0; k < NW; ++k) {
    int32_t c = cnt[k], p = pk[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      c += __shfl_xor_sync(0xffffffffu, c, o);
      p = max(p, __shfl_xor_sync(0xffffffffu, p, o));
    }
    if (lane == 0) {
      counts[n * NW + k] = c;
      peaks[n * NW + k] = p;
    }
  }
}

// Fleets of at most 8 jobs with 16-byte loads.  The workspace holds four
// copies of the prefix array, copy c shifted left by c samples
// (X_c[j][x] = PREX[j][x + c], zero past the end), so that for any offset the
// stream of job j starts 16-byte aligned in copy (o_j + 1) & 3.  Each lane
// composes 4 consecutive samples per load; one warp iteration covers 128.
// The 1024-slot ring keeps its size: windows of 128 samples or more read it
// before the block's prefixes are written (their starts all precede the
// block), shorter windows after (their starts lie at most 127 back).
template <bool EDGE, int NW>
__device__ __forceinline__ void fleet_block4(const uint32_t* ring, int T, int H, const uint4& pre,
                                             const FleetWindows& win, bool long_windows,
                                             int32_t (&cnt)[NW], int32_t (&pk)[NW]) {
  const uint32_t pv[4] = {pre.x, pre.y, pre.z, pre.w};
#pragma unroll
  for (int k = 0; k < NW; ++k) {
    const int w = win.w[k];
    if ((w >= 128) != long_windows) continue;
    uint32_t old[4];
    if ((w & 3) == 0) {
      const uint4 o4 = *reinterpret_cast<const uint4*>(ring + ((T - w) & (kFleetRing - 1)));
      old[0] = o4.x; old[1] = o4.y; old[2] = o4.z; old[3] = o4.w;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) old[i] = ring[(T + i - w) & (kFleetRing - 1)];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int32_t S = (int32_t)(pv[i] - old[i]);
      const bool in = !EDGE || (T + i < H && T + i >= w - 1);
      cnt[k] += (in && S > win.bw[k]);
      if (in) pk[k] = max(pk[k], S);
    }
  }
}

template <int NW>
__global__ void __launch_bounds__(32 * kFleetWarps)
    fleet_windows_v4_kernel(const uint32_t* __restrict__ prex4, int J, int64_t Lp, int64_t cs,
                            const int32_t* __restrict__ offsets, int64_t N, int H, FleetWindows win,
                            int wmax, int32_t* __restrict__ counts, int32_t* __restrict__ peaks) {
  __shared__ __align__(16) uint32_t ring_all[kFleetWarps][kFleetRing];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t n = (int64_t)blockIdx.x * kFleetWarps + wid;
  if (n >= N) return;  // the whole warp leaves together; no block-wide barrier follows
  uint32_t* ring = ring_all[wid];
  const uint4* bp[kFleetJMax];
  uint32_t pre_m1 = 0;
#pragma unroll
  for (int j = 0; j < kFleetJMax; ++j) {
    bp[j] = reinterpret_cast<const uint4*>(prex4);
    if (j < J) {
      const int32_t o = __ldg(offsets + n * J + j);
      const int s = o + 1, c = s & 3;
      bp[j] = reinterpret_cast<const uint4*>(prex4 + c * cs + (int64_t)j * Lp + (s - c));
      if (lane == j) pre_m1 = __ldg(prex4 + (int64_t)j * Lp + o);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) pre_m1 += __shfl_xor_sync(0xffffffffu, pre_m1, o);
  if (lane == 0) ring[kFleetRing - 1] = pre_m1;
  __syncwarp();
  int32_t cnt[NW], pk[NW];
#pragma unroll
  for (int k = 0; k < NW; ++k) cnt[k] = pk[k] = 0;
  for (int t0 = 0; t0 < H; t0 += 128) {
    const int T = t0 + 4 * lane;
    uint4 pre = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int j = 0; j < kFleetJMax; ++j) {
      if (j < J) {
        const uint4 v = __ldg(bp[j] + (t0 >> 2) + lane);
        pre.x += v.x; pre.y += v.y; pre.z += v.z; pre.w += v.w;
      }
    }
    const bool edge = t0 < wmax - 1 || t0 + 128 > H;
    if (edge) fleet_block4<true, NW>(ring, T, H, pre, win, true, cnt, pk);
    else fleet_block4<false, NW>(ring, T, H, pre, win, true, cnt, pk);
    __syncwarp();
    *reinterpret_cast<uint4*>(ring + (T & (kFleetRing - 1))) = pre;
    __syncwarp();
    if (edge) fleet_block4<true, NW>(ring, T, H, pre, win, false, cnt, pk);
    else fleet_block4<false, NW>(ring, T, H, pre, win, false, cnt, pk);
  }
#pragma unroll
  for (int k = 0; k < NW; ++k) {
    int32_t c = cnt[k], p = pk[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      c += __shfl_xor_sync(0xffffffffu, c, o);
      p = max(p, __shfl_xor_sync(0xffffffffu, p, o));
    }
    if (lane == 0) {
      counts[n * NW + k] = c;
      peaks[n * NW + k] = p;
    }
  }
}

// ---------------------------------------------------------------------------
// Fleets of at most 8 jobs whose samples span at most 16 bits (job samples
// above the job's minimum).  Eight copies of the rows, copy c shifted left by
// c samples, make every stream start 16-byte aligned: a load brings 8
// samples of a job, half the bytes per sample of the 32-bit prefixes.  Jobs
// are ordered into groups of GRP whose ranges add up to at most 65,535, so
// the samples of a group add as packed pairs without a carry; the groups then
// widen to 32 bits.  Each lane holds 8 consecutive composed samples, a warp
// scan turns them into the running prefix, and the windows difference it
// against the ring.  Powers below the jobs' minima (base) drop out of every
// difference: thresholds are lowered by w * base and peaks raised by it.
// Ring layout: 16-byte chunks, the even and the odd ones apart, so that the
// lanes' chunks (8 samples apart) are consecutive.  Measured on 100,000
// compositions of 380,000 samples, windows 1/60/600: 74.1 ms with the 32-bit
// prefixes (fleet_windows_v4_kernel), 47.3 ms with these.
// ---------------------------------------------------------------------------
struct FleetDelta {
  int8_t job[kFleetJMax];  // job of stream k (-1: none), grouped
  int32_t w[4];
  int32_t bw[4];           // budget_q * w less w * base: the threshold of a window sum above base
  int32_t bq[4];           // budget_q * w
  int32_t part;            // samples per part of the horizon (a multiple of 256)
  int32_t parts;           // > 1: several warps share a composition and combine with atomics
  int32_t warm;            // samples a part walks ahead of its start: the largest window, rounded up to 256
};

template <int NW, int GRP>
__global__ void __launch_bounds__(32 * kFleetWarps, 4)
    fleet_windows_h16_kernel(const uint4* __restrict__ rows, int J, int64_t rowq, int64_t copyq,
                             const int32_t* __restrict__ offsets, int64_t N, int H, FleetDelta f,
                             int32_t* __restrict__ counts, int32_t* __restrict__ peaks) {
  __shared__ uint4 ring_all[kFleetWarps][2][kFleetRing / 8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t id = (int64_t)blockIdx.x * kFleetWarps + wid;
  const int64_t n = f.parts > 1 ? id / f.parts : id;
  if (n >= N) return;  // the whole warp leaves together; no block-wide barrier follows
  const int lo = f.parts > 1 ? (int)(id % f.parts) * f.part : 0;  // this warp counts windows that end in [lo, hi)
  const int hi = f.parts > 1 ? min(H, lo + f.part) : H;
  const int ts = max(0, lo - f.warm);
  uint4* const ring0 = ring_all[wid][0];
  uint4* const ring1 = ring_all[wid][1];
  uint32_t at[kFleetJMax];  // 16-byte chunk of stream k at ts + 8 * lane (rows below 64 GB)
#pragma unroll
  for (int k = 0; k < kFleetJMax; ++k) {
    at[k] = 0;
    if (f.job[k] >= 0) {
      const int32_t o = __ldg(offsets + n * J + f.job[k]);
      at[k] = (uint32_t)((o & 7) * copyq + f.job[k] * rowq + (o >> 3) + (ts >> 3) + lane);
    }
  }
  if (lane == 0) reinterpret_cast<uint32_t*>(ring1 + (((ts - 8) >> 3) & (kFleetRing / 8 - 1)))[3] = 0u;  // pre(ts - 1)
  uint32_t carry = 0;
  int32_t cnt[NW], least[NW];  // windows over the threshold; least of threshold - sum
#pragma unroll
  for (int k = 0; k < NW; ++k) {
    cnt[k] = 0;
    least[k] = f.bw[k];
  }
  auto block = [&](int t0, auto edge_tag) {
    constexpr bool EDGE = decltype(edge_tag)::value;
    const int T = t0 + 8 * lane;
    uint32_t s[8], p[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) s[i] = 0;
    {
      uint4 v[kFleetJMax];
#pragma unroll
      for (int k = 0; k < kFleetJMax; ++k) {
        v[k] = make_uint4(0u, 0u, 0u, 0u);
        if (f.job[k] >= 0 && (!EDGE || T < H)) v[k] = __ldg(rows + at[k]);
        at[k] += 32;
      }
#pragma unroll
      for (int g = 0; g < kFleetJMax; g += GRP) {
        uint4 a = v[g];
#pragma unroll
        for (int k = 1; k < GRP; ++k) a.x += v[g + k].x, a.y += v[g + k].y, a.z += v[g + k].z, a.w += v[g + k].w;
        s[0] += a.x & 0xFFFFu, s[1] += a.x >> 16, s[2] += a.y & 0xFFFFu, s[3] += a.y >> 16;
        s[4] += a.z & 0xFFFFu, s[5] += a.z >> 16, s[6] += a.w & 0xFFFFu, s[7] += a.w >> 16;
      }
    }
    const uint32_t sum = ((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]));
    uint32_t inc = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
      if (lane >= d) inc += y;
    }
    p[0] = carry + (inc - sum) + s[0];
#pragma unroll
    for (int i = 1; i < 8; ++i) p[i] = p[i - 1] + s[i];
    carry += __shfl_sync(0xffffffffu, inc, 31);
    auto windows = [&](bool long_windows) {
#pragma unroll
      for (int k = 0; k < NW; ++k) {
        const int w = f.w[k];
        if ((w >= 256) != long_windows) continue;
        auto take = [&](int i, int32_t d) {  // d = threshold - window sum
          const bool in = !EDGE || (T + i < hi && T + i >= lo && T + i >= w - 1);
          if (in) {
            cnt[k] += (int32_t)((uint32_t)d >> 31);
            least[k] = min(least[k], d);
          }
        };
        if (w == 1) {
#pragma unroll
          for (int i = 0; i < 8; ++i) take(i, f.bw[k] - (int32_t)s[i]);
          continue;
        }
        const int x = T - w, q = x >> 2;  // arithmetic shift: slots before t = 0 wrap around the ring
        uint32_t o[12];
        auto get = [&](int c) {
          const uint4 r = (((q + c) & 1) ? ring1 : ring0)[((q + c) >> 1) & (kFleetRing / 8 - 1)];
          o[4 * c] = r.x, o[4 * c + 1] = r.y, o[4 * c + 2] = r.z, o[4 * c + 3] = r.w;
        };
        get(0);
        get(1);
        const int m = x & 3;  // the same for every lane
        if (m == 0) {
#pragma unroll
          for (int i = 0; i < 8; ++i) take(i, f.bw[k] + (int32_t)(o[i] - p[i]));
        } else {
          get(2);
#pragma unroll
          for (int i = 0; i < 8; ++i)
            take(i, f.bw[k] + (int32_t)((m == 1 ? o[i + 1] : m == 2 ? o[i + 2] : o[i + 3]) - p[i]));
        }
      }
    };
    windows(true);  // their starts precede the block: read before it overwrites the ring
    __syncwarp();
    ring0[(T >> 3) & (kFleetRing / 8 - 1)] = make_uint4(p[0], p[1], p[2], p[3]);
    ring1[(T >> 3) & (kFleetRing / 8 - 1)] = make_uint4(p[4], p[5], p[6], p[7]);
    __syncwarp();
    windows(false);
  };
  for (int t0 = ts; t0 < hi; t0 += 256) {
    if (t0 < max(lo, f.warm) || t0 + 256 > hi) block(t0, std::true_type());
    else block(t0, std::false_type());
  }
#pragma unroll
  for (int k = 0; k < NW; ++k) {
    const int32_t c = __reduce_add_sync(0xffffffffu, cnt[k]);
    const int32_t d = __reduce_min_sync(0xffffffffu, least[k]);
    if (lane == 0) {
      // no window in the horizon: the peak is 0
      const int32_t pk = H >= f.w[k] ? f.bq[k] - d : 0;
      if (f.parts > 1) {
        if (c) atomicAdd(counts + n * NW + k, c);
        atomicMax(peaks + n * NW + k, pk);
      } else {
        counts[n * NW + k] = c;
        peaks[n * NW + k] = pk;
      }
    }
  }
}

// the eight shifted 16-bit copies: a block takes 2,048 samples of a job's
// unrolled row (zero from L + H on), a thread the chunks of 8 samples c
// samples past its own 8, c = 0 .. 7
constexpr int kH16Tile = 2048;
__global__ void __launch_bounds__(256) fleet_h16_rows_kernel(const float* __restrict__ traces, int G, int L, int H,
                                                             const int32_t* __restrict__ job_of_gpu, int J,
                                                             FleetWs ws, uint4* __restrict__ rows, int64_t rowq,
                                                             int64_t copyq) {
  __shared__ JobGpus gpus;
  __shared__ __align__(16) uint16_t v[kH16Tile + 8];
  const int j = blockIdx.y;
  list_gpus(job_of_gpu, G, J, j, gpus, ws.flag);
  const int32_t base = INT_MAX - ws.maxq[32 + j];
  const int64_t i0 = (int64_t)blockIdx.x * kH16Tile, Lx = (int64_t)L + H;
  int bad = 0;  // reported by fleet_range_kernel
  for (int k = threadIdx.x; k < kH16Tile + 8; k += 256) {
    const int64_t i = i0 + k;
    v[k] = i < Lx ? (uint16_t)(job_sample(traces, gpus, L, (int)i, bad) - base) : (uint16_t)0;
  }
  __syncthreads();
  const int64_t q = (int64_t)blockIdx.x * (kH16Tile / 8) + threadIdx.x;
  if (q >= rowq) return;
  const uint4 lo = reinterpret_cast<const uint4*>(v)[threadIdx.x], hi = reinterpret_cast<const uint4*>(v)[threadIdx.x + 1];
  const uint32_t x[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    uint32_t y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      y[i] = (c & 1) ? __funnelshift_r(x[c / 2 + i], x[c / 2 + i + 1], 16) : x[c / 2 + i];
    rows[c * copyq + j * rowq + q] = make_uint4(y[0], y[1], y[2], y[3]);
  }
}

// 16-byte chunks per row of the 16-bit copies: a stream reads up to 7 samples
// past its last one
static int64_t fleet_rowq(int L, int H) { return ((int64_t)L + H + 8 + 7) / 8; }

// Groups of 4 (or of 2) streams whose ranges add up to at most 65,535, the
// widest jobs first and each into the group with the most room; 0: none.
static int fleet_groups(const int64_t* range, int J, int8_t (&job)[kFleetJMax]) {
  int order[kFleetJMax];
  for (int k = 0; k < J; ++k) order[k] = k;
  std::sort(order, order + J, [&](int a, int b) { return range[a] > range[b] || (range[a] == range[b] && a < b); });
  for (int grp = 4; grp >= 2; grp /= 2) {
    const int ng = kFleetJMax / grp;
    int64_t sum[kFleetJMax] = {0};
    int cnt[kFleetJMax] = {0};
    for (int k = 0; k < kFleetJMax; ++k) job[k] = -1;
    bool fits = true;
    for (int k = 0; k < J && fits; ++k) {
      int best = -1;
      for (int g = 0; g < ng; ++g)
        if (cnt[g] < grp && (best < 0 || sum[g] < sum[best])) best = g;
      sum[best] += range[order[k]];
      fits = sum[best] <= 65535;
      job[best * grp + cnt[best]++] = (int8_t)order[k];
    }
    if (fits) return grp;
  }
  return 0;
}

// copies 1..3 of nrows prefix rows for the 16-byte path (copy 0 is the rows
// themselves, copy c starts cs words after copy c - 1); entries past a row's
// last index are zero in every copy
__global__ void fleet_shift_copies_kernel(uint32_t* __restrict__ rows0, int nrows, int64_t Lp, int64_t cs,
                                          int64_t last) {
  const int64_t total = (int64_t)nrows * Lp;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t x = i % Lp;
    const uint32_t* row = rows0 + (i - x);
    if (x > last) rows0[i] = 0u;
#pragma unroll
    for (int c = 1; c < 4; ++c) rows0[c * cs + i] = x + c <= last ? row[x + c] : 0u;
  }
}

// row stride: PREX[j][0 .. L + H] plus the 127 words a 128-sample block of
// the 16-byte path may read past a stream's end, rounded to 16 bytes
static int64_t fleet_lp(int L, int H) { return (((int64_t)L + H + 1 + 127) + 3) / 4 * 4; }
static int fleet_ncopy(int J, int64_t workspace_bytes, int L, int H);
static int fleet_nchunk(int L, int H) { return (int)((((int64_t)L + H) + kFleetChunk - 1) / kFleetChunk); }

// rows = J job rows plus `extra` working rows, in each of ncopy copies
static int64_t fleet_bytes(int J, int L, int H, int ncopy, int extra = 0) {
  const int64_t prex = ((int64_t)ncopy * (J + extra) * fleet_lp(L, H) * 4 + 255) / 256 * 256;
  const int64_t tot = ((int64_t)J * fleet_nchunk(L, H) * 4 + 255) / 256 * 256;
  return prex + tot + 256 + 256;
}

// the least workspace (one prefix copy, 4-byte loads) and the workspace of
// the 16-byte path (four shifted copies; fleets of at most 8 jobs)
int64_t fleet_ws_min_bytes(int J, int L, int H) { return fleet_bytes(J, L, H, 1); }
int64_t fleet_ws_bytes(int J, int L, int H) { return fleet_bytes(J, L, H, J <= kFleetJMax ? 4 : 1); }
static int fleet_ncopy(int J, int64_t workspace_bytes, int L, int H) {
  return J <= kFleetJMax && workspace_bytes >= fleet_bytes(J, L, H, 4) ? 4 : 1;
}

// Validation of the traces, job map and offsets, and the per-job ranges; the
// call waits for them.  `extra`: working rows besides the J job rows.
static pe_status fleet_check(const float* traces, int G, int L, const int32_t* job_of_gpu, int J,
                             const int32_t* offsets, int64_t N, int H, void* workspace, int ncopy, int extra,
                             FleetWs& ws, int64_t& sum_max, int64_t* least, int64_t* range, cudaStream_t st) {
  char* base = reinterpret_cast<char*>(workspace);
  ws.Lp = fleet_lp(L, H);
  ws.nchunk = fleet_nchunk(L, H);
  const int64_t prex_bytes = ((int64_t)ncopy * (J + extra) * ws.Lp * 4 + 255) / 256 * 256;
  const int64_t tot_bytes = ((int64_t)J * ws.nchunk * 4 + 255) / 256 * 256;
  ws.prex = reinterpret_cast<uint32_t*>(base);
  ws.totals = reinterpret_cast<uint32_t*>(base + prex_bytes);
  ws.maxq = reinterpret_cast<int32_t*>(base + prex_bytes + tot_bytes);
  ws.flag = reinterpret_cast<int32_t*>(base + prex_bytes + tot_bytes + 256);
  PE_TRY_CUDA(cudaMemsetAsync(ws.maxq, 0, 256 + 4, st));
  {
    ProfScope ps(PE_PROF_FLEET_PREP, st);
    fleet_range_kernel<<<dim3(ceil_div(L, kRangeChunk), J), 256, 0, st>>>(traces, G, L, job_of_gpu, J, ws);
    if (N > 0)
      fleet_check_offsets_kernel<<<(int)std::min<int64_t>(ceil_div(N * J, 256), 4096), 256, 0, st>>>(
          offsets, N * J, L, ws.flag);
  }
  PE_CHECK_LAUNCH("fleet check kernels");
  int32_t host[64 + 1];
  PE_TRY_CUDA(cudaMemcpyAsync(host, ws.maxq, sizeof(host), cudaMemcpyDeviceToHost, st));
  PE_TRY_CUDA(cudaStreamSynchronize(st));
  const int32_t flag = host[64];
  if (flag & 1) return fail(PE_EOVERFLOW, "fleet trace holds a sample that is not finite or outside [0, %g] W", (double)kFleetMaxWatts);
  if (flag & 2) return fail(PE_EINVAL, "job_of_gpu entry outside [0, J)");
  if (flag & 4) return fail(PE_EINVAL, "fleet offset outside [0, L)");
  sum_max = 0;
  for (int j = 0; j < J; ++j) {
    sum_max += host[j];
    least[j] = (int64_t)INT_MAX - host[32 + j];
    range[j] = host[j] - least[j];
  }
  return PE_OK;
}

// per-job prefix sums (PREX), in ncopy shifted copies
static pe_status fleet_prefixes(const float* traces, int G, int L, const int32_t* job_of_gpu, int J, int H, int ncopy,
                                int extra, const FleetWs& ws, cudaStream_t st) {
  {
    ProfScope ps(PE_PROF_FLEET_PREP, st);
    const dim3 grid(ws.nchunk, J);
    fleet_chunk_sums_kernel<<<grid, 256, 0, st>>>(traces, G, L, H, job_of_gpu, J, ws);
    fleet_chunk_scan_kernel<<<J, 32, 0, st>>>(ws);
    fleet_prefix_kernel<<<grid, 256, 0, st>>>(traces, G, L, H, job_of_gpu, J, ws);
    if (ncopy == 4)
      fleet_shift_copies_kernel<<<(int)std::min<int64_t>(ceil_div((int64_t)J * ws.Lp, 256), 4096), 256, 0, st>>>(
          ws.prex, J, ws.Lp, (int64_t)(J + extra) * ws.Lp, (int64_t)L + H);
  }
  PE_CHECK_LAUNCH("fleet prefix kernels");
  return PE_OK;
}

// the 16-bit path (see fleet_windows_h16_kernel); grp: streams per group
static pe_status fleet_launch_h16(const float* traces, int G, int L, const int32_t* job_of_gpu, int J,
                                  const int32_t* offsets, int64_t N, int H, int W, int grp, FleetDelta& f, int wmax,
                                  const FleetWs& ws, int32_t* counts, int32_t* peaks, cudaStream_t st) {
  int dev = 0, sms = 0;
  PE_TRY_CUDA(cudaGetDevice(&dev));
  PE_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int64_t rowq = fleet_rowq(L, H), copyq = J * rowq;
  uint4* rows = reinterpret_cast<uint4*>(ws.prex);
  {
    ProfScope ps(PE_PROF_FLEET_PREP, st);
    fleet_h16_rows_kernel<<<dim3(ceil_div(rowq, kH16Tile / 8), J), 256, 0, st>>>(traces, G, L, H, job_of_gpu, J, ws,
                                                                               rows, rowq, copyq);
  }
  // few compositions: parts of the horizon, each at least four times the
  // history it walks first, until every SM has its 32 warps
  f.warm = (wmax + 255) / 256 * 256;
  const int64_t most = H / std::max(4 * f.warm, 2048), want = (int64_t)sms * 32 / N;
  f.parts = (int)std::max<int64_t>(1, std::min(most, want));
  if (f.parts > 1) {
    f.part = (H / f.parts + 256) / 256 * 256;  // at least H / parts
    f.parts = (int)(((int64_t)H + f.part - 1) / f.part);
    PE_TRY_CUDA(cudaMemsetAsync(counts, 0, N * W * 4, st));
    PE_TRY_CUDA(cudaMemsetAsync(peaks, 0, N * W * 4, st));
  }
  const int grid = ceil_div(N * f.parts, kFleetWarps);
  ProfScope ps(PE_PROF_FLEET_WINDOWS, st);
  auto go = [&](auto nw, auto gr) {
    fleet_windows_h16_kernel<decltype(nw)::value, decltype(gr)::value>
        <<<grid, 32 * kFleetWarps, 0, st>>>(rows, J, rowq, copyq, offsets, N, H, f, counts, peaks);
  };
  auto by_windows = [&](auto gr) {
    switch (W) {
      case 1: go(std::integral_constant<int, 1>(), gr); break;
      case 2: go(std::integral_constant<int, 2>(), gr); break;
      case 3: go(std::integral_constant<int, 3>(), gr); break;
      default: go(std::integral_constant<int, 4>(), gr); break;
    }
  };
  if (grp == 4) by_windows(std::integral_constant<int, 4>());
  else by_windows(std::integral_constant<int, 2>());
  PE_CHECK_LAUNCH("fleet_windows_h16_kernel");
  return PE_OK;
}

pe_status fleet_launch(const float* traces, int G, int L, const int32_t* job_of_gpu, int J,
                       const int32_t* offsets, int64_t N, int H, const int32_t* windows, int W,
                       int64_t budget_q, int32_t* counts, int32_t* peaks, void* workspace,
                       int64_t workspace_bytes, cudaStream_t st) {
  FleetWs ws;
  int64_t sum_max = 0;
  const int ncopy = fleet_ncopy(J, workspace_bytes, L, H);
  int64_t least[32], range[32], base = 0;
  pe_status s = fleet_check(traces, G, L, job_of_gpu, J, offsets, N, H, workspace, ncopy, 0, ws, sum_max, least,
                            range, st);
  if (s != PE_OK) return s;
  for (int j = 0; j < J; ++j) base += least[j];
  FleetWindows win{};
  FleetDelta delta{};
  int wmax = 0;
  for (int k = 0; k < W; ++k) {
    const int64_t w = windows[k];
    if (sum_max * w >= (int64_t)INT_MAX || budget_q * w >= (int64_t)INT_MAX)
      return fail(PE_EOVERFLOW, "window %d: composed window sum may exceed int32", (int)w);
    win.w[k] = (int32_t)w;
    win.bw[k] = (int32_t)(budget_q * w);
    wmax = std::max(wmax, (int)w);
    delta.w[k] = win.w[k];
    delta.bq[k] = win.bw[k];
    delta.bw[k] = (int32_t)(budget_q * w - base * w);
  }
  if (N == 0) return PE_OK;
  // Four prefix copies' room holds the eight 16-bit copies: two bytes instead
  // of four per job and sample, taken whenever the traces' ranges allow.
  const bool narrow = ncopy == 4 && 8 * (int64_t)J * fleet_rowq(L, H) <= (int64_t)UINT32_MAX;  // 32-bit chunk indices
  const int grp = narrow ? fleet_groups(range, J, delta.job) : 0;
  if (grp)
    return fleet_launch_h16(traces, G, L, job_of_gpu, J, offsets, N, H, W, grp, delta, wmax, ws, counts, peaks, st);
  s = fleet_prefixes(traces, G, L, job_of_gpu, J, H, ncopy, 0, ws, st);
  if (s != PE_OK) return s;
  const int grid_n = (int)((N + kFleetWarps - 1) / kFleetWarps);
  const int64_t Lx = ws.Lp;
  ProfScope ps(PE_PROF_FLEET_WINDOWS, st);
  const int64_t cs = (int64_t)J * Lx;
  if (ncopy == 4) {
    switch (W) {
      case 1: fleet_windows_v4_kernel<1><<<grid_n, 32 * kFleetWarps, 0, st>>>(ws.prex, J, Lx, cs, offsets, N, H, win, wmax, counts, peaks); break;
      case 2: fleet_windows_v4_kernel<2><<<grid_n, 32 * kFleetWarps, 0, st>>>(ws.prex, J, Lx, cs, offsets, N, H, win, wmax, counts, peaks); break;
      case 3: fleet_windows_v4_kernel<3><<<grid_n, 32 * kFleetWarps, 0, st>>>(ws.prex, J, Lx, cs, offsets, N, H, win, wmax, counts, peaks); break;
      default: fleet_windows_v4_kernel<4><<<grid_n, 32 * kFleetWarps, 0, st>>>(ws.prex, J, Lx, cs, offsets, N, H, win, wmax, counts, peaks); break;
    }
  } else if (J <= kFleetJMax) {
    switch (W) {
      case 1: fleet_windows_j8_kernel<1><<<grid_n, 32 * kFleetWarps, 0, st>>>(ws.prex, J, Lx, offsets, N, H, win, counts, peaks); break;
      case 2: fleet_windows_j8_kernel<2><<<grid_n, 32 * kFleetWarps, 0, st>>>(ws.prex, J, Lx, offsets, N, H, win, counts, peaks); break;
      case 3: fleet_windows_j8_kernel<3><<<grid_n, 32 * kFleetWarps, 0, st>>>(ws.prex, J, Lx, offsets, N, H, win, counts, peaks); break;
      default: fleet_windows_j8_kernel<4><<<grid_n, 32 * kFleetWarps, 0, st>>>(ws.prex, J, Lx, offsets, N, H, win, counts, peaks); break;
    }
  } else {
    switch (W) {
      case 1: fleet_windows_kernel<1><<<grid_n, 32 * kFleetWarps, 0, st>>>(ws.prex, J, Lx, offsets, N, H, win, counts, peaks); break;
      case 2: fleet_windows_kernel<2><<<grid_n, 32 * kFleetWarps, 0, st>>>(ws.prex, J, Lx, offsets, N, H, win, counts, peaks); break;
      case 3: fleet_windows_kernel<3><<<grid_n, 32 * kFleetWarps, 0, st>>>(ws.prex, J, Lx, offsets, N, H, win, counts, peaks); break;
      default: fleet_windows_kernel<4><<<grid_n, 32 * kFleetWarps, 0, st>>>(ws.prex, J, Lx, offsets, N, H, win, counts, peaks); break;
    }
  }
  PE_CHECK_LAUNCH("fleet_windows_kernel");
  return PE_OK;
}

// ---------------------------------------------------------------------------
// Phase-staggered schedule (Sec. 8): jobs placed greedily in index order.
// With A[i] the w-sample window sums of the jobs placed so far and B[x] those
// of the next job's unrolled stream (i, x: the window's first sample), the
// peak of candidate offset o is max_i (A[i] + B[i + o]): a correlation of two
// rows in which the sum of products is a maximum of sums.  A peaks kernel
// evaluates it for every candidate, a one-block argmin keeps the lowest
// candidate among equal peaks, and the job's prefix row at that offset is
// added to the partial fleet's.  The chosen offsets never leave the device
// between stages.
// ---------------------------------------------------------------------------
// partial-fleet prefix row R[y] = sum over the placed jobs k of PREX[k][o_k + y]
// for y in [0, H]: adds job j at its chosen offset (job 0 starts the row)
__global__ void stagger_compose_kernel(uint32_t* __restrict__ R, const uint32_t* __restrict__ prex, int64_t Lp, int j,
                                       const int32_t* __restrict__ chosen, int H) {
  const uint32_t* src = prex + (int64_t)j * Lp + chosen[j];
  for (int64_t y = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; y <= H; y += (int64_t)gridDim.x * blockDim.x)
    R[y] = (j > 0 ? R[y] : 0u) + src[y];
}

// Candidate peaks, stride s: with i = s u + r and o = s c the correlation
// splits into one per residue r, peak(c) = max_r max_u A_r[u] + B_r[u + c],
// A_r[u] = A[s u + r] and B_r[v] = B[s v + r].  A block takes kStTile
// candidates and a list of items (a residue and a chunk of u), stages both
// rows in shared memory (window sums from the prefix rows), and each thread
// slides a register window of B under its 8 consecutive candidates: 64
// add-and-maximum instructions (__viaddmax_s32) per 4 16-byte shared loads,
// two of them broadcasts.  B is kept as the even and the odd 16-byte chunks,
// so that threads 8 samples apart read consecutive chunks.  What bounds it is
// the rate of that one instruction per candidate and sample; a warp per
// candidate over the 16-byte window-count kernel, which this replaced, spent
// about 15 on the same pair.  Measured with every offset of 60,000 samples a
// candidate (8 jobs, 2.9e10 pairs): 23.1 ms before, 1.90 ms now, 1.5e13 pairs
// per second.
constexpr int kStThreads = 128;
constexpr int kStTile = kStThreads * 8;  // candidates per block
constexpr int kStChunk = 2048;           // most u per item

__global__ void __launch_bounds__(kStThreads)
    stagger_peaks_kernel(const uint32_t* __restrict__ R, const uint32_t* __restrict__ job, int64_t M, int64_t xmax,
                         int w, int stride, int64_t nc, int chunk, int64_t nchunk, int64_t items,
                         int32_t* __restrict__ peaks) {
  __shared__ int4 sa[kStChunk / 4];
  __shared__ int4 se[(kStTile + kStChunk) / 8], so[(kStTile + kStChunk) / 8];
  const int tid = threadIdx.x;
  const int64_t c0 = (int64_t)blockIdx.x * kStTile;
  int m[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) m[k] = 0;  // sums of powers: no peak is below 0
  for (int64_t it = blockIdx.y; it < items; it += gridDim.y) {
    const int64_t r = it / nchunk, u0 = (it % nchunk) * chunk;
    __syncthreads();  // the previous item has been read
    for (int y = tid; y < chunk; y += kStThreads) {
      const int64_t i = (u0 + y) * stride + r;
      int v = INT_MIN;  // past the last window: below every peak with any B >= 0
      if (i < M) v = R ? (int)(__ldg(R + i + w) - __ldg(R + i)) : 0;
      reinterpret_cast<int*>(sa)[y] = v;
    }
    for (int y = tid; y < kStTile + chunk; y += kStThreads) {
      const int64_t x = (c0 + u0 + y) * stride + r;
      const int v = x <= xmax ? (int)(__ldg(job + x + w) - __ldg(job + x)) : 0;
      reinterpret_cast<int*>((y & 4) ? so : se)[(y >> 3) * 4 + (y & 3)] = v;
    }
    __syncthreads();
    int b[16];
    auto load8 = [&](int n, int (&dst)[16], int at) {
      const int4 e = se[n], o = so[n];
      dst[at] = e.x, dst[at + 1] = e.y, dst[at + 2] = e.z, dst[at + 3] = e.w;
      dst[at + 4] = o.x, dst[at + 5] = o.y, dst[at + 6] = o.z, dst[at + 7] = o.w;
    };
    auto step = [&](int k, int lo) {  // 8 samples; the window's older half is at b[lo ..]
      load8(tid + k + 1, b, lo ^ 8);
      const int4 a0 = sa[2 * k], a1 = sa[2 * k + 1];
      const int a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
      for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int c = 0; c < 8; ++c) m[c] = __viaddmax_s32(a[u], b[(lo + u + c) & 15], m[c]);
    };
    load8(tid, b, 0);
    for (int k = 0; k < chunk / 8; k += 2) {  // chunk is a multiple of 16
      step(k, 0);
      step(k + 1, 8);
    }
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int64_t c = c0 + 8 * tid + k;
    if (c < nc) atomicMax(peaks + c, m[k]);
  }
}

// the lowest candidate of least peak; the peaks are zeroed for the next stage
__global__ void __launch_bounds__(1024) stagger_argmin_kernel(int32_t* __restrict__ peaks, int64_t ncand, int stride,
                                                              int j, int32_t* __restrict__ chosen,
                                                              int32_t* __restrict__ chosen_peak) {
  __shared__ int32_t sp[32];
  __shared__ int64_t sc[32];
  int32_t bp = INT_MAX;
  int64_t bc = ncand;
  // ascending scan: the first (lowest) candidate of a tie stays
  auto take = [&](int32_t p, int64_t c) {
    if (p < bp) {
      bp = p;
      bc = c;
    }
  };
  int4* p4 = reinterpret_cast<int4*>(peaks);
#pragma unroll 4
  for (int64_t q = threadIdx.x; q < ncand / 4; q += blockDim.x) {
    const int4 v = p4[q];
    p4[q] = make_int4(0, 0, 0, 0);
    take(v.x, 4 * q);
    take(v.y, 4 * q + 1);
    take(v.z, 4 * q + 2);
    take(v.w, 4 * q + 3);
  }
  for (int64_t c = ncand / 4 * 4 + threadIdx.x; c < ncand; c += blockDim.x) {
    take(peaks[c], c);
    peaks[c] = 0;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const int32_t op = __shfl_xor_sync(0xffffffffu, bp, o);
    const int64_t oc = __shfl_xor_sync(0xffffffffu, bc, o);
    if (op < bp || (op == bp && oc < bc)) {
      bp = op;
      bc = oc;
    }
  }
  if ((threadIdx.x & 31) == 0) {
    sp[threadIdx.x >> 5] = bp;
    sc[threadIdx.x >> 5] = bc;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
      if (sp[w] < bp || (sp[w] == bp && sc[w] < bc)) {
        bp = sp[w];
        bc = sc[w];
      }
    chosen[j] = (int32_t)(bc * stride);
    chosen_peak[j] = bp;
  }
}

static int64_t stagger_ncand(int L, int stride) { return ((int64_t)L + stride - 1) / stride; }

// The size asked of callers: four prefix copies of the J job rows and a
// partial-fleet row, then four words per candidate.  (The stages use one copy
// and one word per candidate; programs hold workspaces of this size.)
int64_t fleet_stagger_ws_bytes(int J, int L, int H, int stride) {
  const int64_t nc = stagger_ncand(L, stride);
  const int64_t cand = (nc * 2 * 4 + 255) / 256 * 256;
  const int64_t outs = (nc * 4 + 255) / 256 * 256;
  return fleet_bytes(J, L, H, 4, 1) + cand + 2 * outs;
}

pe_status fleet_stagger_launch(const float* traces, int G, int L, const int32_t* job_of_gpu, int J, int H,
                               int w, int stride, int32_t* offsets_out, int32_t* peaks_out, void* workspace,
                               cudaStream_t st) {
  FleetWs ws;
  int64_t sum_max = 0;
  // job rows 0..J-1 and the partial-fleet row J
  int64_t least[32], range[32];
  pe_status s = fleet_check(traces, G, L, job_of_gpu, J, nullptr, 0, H, workspace, 1, 1, ws, sum_max, least, range, st);
  if (s != PE_OK) return s;
  if (sum_max * w >= (int64_t)INT_MAX) return fail(PE_EOVERFLOW, "window %d: composed window sum may exceed int32", w);
  s = fleet_prefixes(traces, G, L, job_of_gpu, J, H, 1, 1, ws, st);
  if (s != PE_OK) return s;
  const int64_t nc = stagger_ncand(L, stride);
  int32_t* pk = reinterpret_cast<int32_t*>(reinterpret_cast<char*>(workspace) + fleet_bytes(J, L, H, 1, 1));
  uint32_t* R = ws.prex + (int64_t)J * ws.Lp;
  const int64_t M = std::max<int64_t>((int64_t)H - w + 1, 0);  // windows of the horizon (none: every peak is 0)
  const int64_t xmax = (int64_t)L + H - w;                     // last window of an unrolled job
  const int64_t per = (M + stride - 1) / stride, residues = std::min<int64_t>(stride, M);
  const int64_t tiles = (nc + kStTile - 1) / kStTile;
  // items short enough to give every SM eight blocks (64 samples at least: an
  // item stages 1,024 of B whatever its length)
  int dev = 0, sms = 0;
  PE_TRY_CUDA(cudaGetDevice(&dev));
  PE_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int64_t want = (per * residues * tiles + 8 * sms - 1) / (8 * sms);
  const int chunk = (int)std::min<int64_t>(kStChunk, (std::max<int64_t>(std::min(want, per), 64) + 15) / 16 * 16);
  const int64_t nchunk = (per + chunk - 1) / chunk, items = nchunk * residues;
  const dim3 grid((unsigned)tiles, (unsigned)std::max<int64_t>(1, std::min<int64_t>(items, 4096)));
  PE_TRY_CUDA(cudaMemsetAsync(pk, 0, nc * 4, st));
  for (int j = 0; j < J; ++j) {
    {
      ProfScope ps(PE_PROF_FLEET_WINDOWS, st);
      stagger_peaks_kernel<<<grid, kStThreads, 0, st>>>(j ? R : nullptr, ws.prex + (int64_t)j * ws.Lp, M, xmax, w,
                                                        stride, nc, chunk, nchunk, items, pk);
    }
    ProfScope ps(PE_PROF_FLEET_PREP, st);
    stagger_argmin_kernel<<<1, 1024, 0, st>>>(pk, nc, stride, j, offsets_out, peaks_out);
    if (j + 1 < J)
      stagger_compose_kernel<<<(int)std::min<int64_t>(ceil_div((int64_t)H + 1, 256), 4096), 256, 0, st>>>(
          R, ws.prex, ws.Lp, j, offsets_out, H);
    PE_CHECK_LAUNCH("fleet stagger kernels");
  }
  return PE_OK;
}

}  // namespace pe
