// Reverse-time generalised advantage estimation over a time-major [T][E]
// buffer (Sec. 4.2: gamma 0.99, lambda 0.95):
//   delta_t = r_t + gamma (1 - d_t) V_{t+1} - V_t,  A_t = delta_t + gamma lambda (1 - d_t) A_{t+1}.
//
// HBM-bound: 9 bytes in and 8 bytes out per env-step.  A thread owns V = 1 or 2
// consecutive envs (vector loads/stores; a warp covers 32*V envs of one row)
// and one time chunk of CL steps held in registers; the NW warps of a CTA
// cover NW consecutive chunks.  Each thread first reduces its chunk to the
// affine map A_start = alpha + beta * A_end, warp 0 chains the chunk maps
// through shared memory, and each thread then re-runs its chunk with the
// right carry-in and streams A and R out.  Longer horizons loop over
// super-chunks of CL*NW steps from the end.  That time-parallel form serves
// narrow batches; wider ones (the rule is in gae_launch) take the barrier-free
// per-column kernel below.
#include <type_traits>

#include "common.cuh"

namespace pe {

template <int CL, int NW, int V>
__global__ void __launch_bounds__(32 * NW)
    gae_kernel_v(const float* __restrict__ r, const float* __restrict__ v,
                 const uint8_t* __restrict__ d, const float* __restrict__ last_v, int T, int E,
                 float gamma, float lam, float* __restrict__ adv, float* __restrict__ ret) {
  using FV = typename std::conditional<V == 2, float2, float>::type;
  using BV = typename std::conditional<V == 2, uchar2, unsigned char>::type;
  __shared__ float sa[NW][32 * V], sb[NW][32 * V], cin[NW + 1][32 * V];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int e0 = (blockIdx.x * 32 + lane) * V;   // first env of this thread
  const bool ok = e0 < E;
  const float gl = gamma * lam;
  float carry[V];
#pragma unroll
  for (int u = 0; u < V; ++u) carry[u] = 0.0f;
  for (int sc_end = T; sc_end > 0; sc_end -= CL * NW) {
    const int sc_start = max(0, sc_end - CL * NW);
    const int t1 = sc_end - w * CL;
    const int t0 = max(sc_start, t1 - CL);
    float rr[CL][V], vv[CL][V], nt[CL][V];
    float vnext[V];
#pragma unroll
    for (int u = 0; u < V; ++u) vnext[u] = 0.0f;
    if (ok && t1 > t0) {
      const FV q = t1 < T ? *reinterpret_cast<const FV*>(v + (int64_t)t1 * E + e0) : *reinterpret_cast<const FV*>(last_v + e0);
      const float* qp = reinterpret_cast<const float*>(&q);
#pragma unroll
      for (int u = 0; u < V; ++u) vnext[u] = qp[u];
    }
#pragma unroll
    for (int i = 0; i < CL; ++i) {
      const int t = t1 - 1 - i;
#pragma unroll
      for (int u = 0; u < V; ++u) rr[i][u] = vv[i][u] = nt[i][u] = 0.0f;
      if (ok && t >= t0) {
        const int64_t o = (int64_t)t * E + e0;
        const FV a = __ldcs(reinterpret_cast<const FV*>(r + o));
        const FV b = *reinterpret_cast<const FV*>(v + o);
        const BV c = *reinterpret_cast<const BV*>(d + o);
        const float* ap = reinterpret_cast<const float*>(&a);
        const float* bp = reinterpret_cast<const float*>(&b);
        const unsigned char* cp = reinterpret_cast<const unsigned char*>(&c);
#pragma unroll
        for (int u = 0; u < V; ++u) {
          rr[i][u] = ap[u];
          vv[i][u] = bp[u];
          nt[i][u] = 1.0f - (float)cp[u];
        }
      }
    }
#pragma unroll
    for (int u = 0; u < V; ++u) {
      float alpha = 0.0f, beta = 1.0f, vn = vnext[u];
#pragma unroll
      for (int i = 0; i < CL; ++i) {
        if (t1 - 1 - i >= t0) {
          const float delta = rr[i][u] + gamma * vn * nt[i][u] - vv[i][u];
          const float c = gl * nt[i][u];
          alpha = delta + c * alpha;
          beta = c * beta;
          vn = vv[i][u];
        }
      }
      sa[w][lane * V + u] = alpha;
      sb[w][lane * V + u] = beta;
    }
    __syncthreads();
    if (w == 0) {
#pragma unroll
      for (int u = 0; u < V; ++u) {
        float a = carry[u];
        for (int j = 0; j < NW; ++j) {
          cin[j][lane * V + u] = a;
          a = sa[j][lane * V + u] + sb[j][lane * V + u] * a;
        }
        cin[NW][lane * V + u] = a;
      }
    }
    __syncthreads();
    float A[V], vn[V];
#pragma unroll
    for (int u = 0; u < V; ++u) {
      A[u] = cin[w][lane * V + u];
      vn[u] = vnext[u];
    }
#pragma unroll
    for (int i = 0; i < CL; ++i) {
      const int t = t1 - 1 - i;
      if (ok && t >= t0) {
        float ao[V], ro[V];
#pragma unroll
        for (int u = 0; u < V; ++u) {
          const float delta = rr[i][u] + gamma * vn[u] * nt[i][u] - vv[i][u];
          A[u] = delta + gl * nt[i][u] * A[u];
          ao[u] = A[u];
          ro[u] = A[u] + vv[i][u];
          vn[u] = vv[i][u];
        }
        const int64_t o = (int64_t)t * E + e0;
        __stcs(reinterpret_cast<FV*>(adv + o), *reinterpret_cast<FV*>(ao));
        __stcs(reinterpret_cast<FV*>(ret + o), *reinterpret_cast<FV*>(ro));
      }
    }
#pragma unroll
    for (int u = 0; u < V; ++u) carry[u] = cin[NW][lane * V + u];
    __syncthreads();
  }
}


// Batches too wide for the chunked kernels: one thread per env walks the whole
// horizon backwards, A_t = delta_t + gamma lambda (1 - d_t) A_{t+1} in the same
// order as the recursion, with no barrier and no shared memory.  The loads of
// the next P steps are kept in flight in a register ring, so each SM holds
// enough outstanding bytes to cover HBM latency; every warp streams
// 32 consecutive envs of a row (coalesced).  Measured: 2,048 steps of 262,144
// envs with 32 steps in flight 1.66 ms, 81% of the HBM copy peak (16 steps take
// 2% longer, two envs per thread 3%, four 8%); 1,024 x 65,536 with 16 steps and
// blocks of 64, which spread evenly over the SMs, 0.21 ms, 80% (blocks of 128
// take 5% longer).
template <int P, int NT>
__global__ void __launch_bounds__(NT)
    gae_stream_kernel(const float* __restrict__ r, const float* __restrict__ v, const uint8_t* __restrict__ d,
                      const float* __restrict__ last_v, int T, int E, float gamma, float lam,
                      float* __restrict__ adv, float* __restrict__ ret) {
  const int e = blockIdx.x * NT + threadIdx.x;
  if (e >= E) return;
  const float gl = gamma * lam;
  float rb[P], vb[P];
  uint8_t db[P];
  auto load = [&](int k, int t) {
    const int64_t o = (int64_t)t * E + e;
    rb[k] = __ldcs(r + o);
    vb[k] = __ldcs(v + o);
    db[k] = __ldcs(d + o);
  };
#pragma unroll
  for (int k = 0; k < P; ++k)
    if (T - 1 - k >= 0) load(k, T - 1 - k);
  float A = 0.0f, vn = last_v[e];
  for (int base = T - 1; base >= 0; base -= P) {
#pragma unroll
    for (int k = 0; k < P; ++k) {
      const int t = base - k;
      if (t >= 0) {
        const float nt = 1.0f - (float)db[k], vt = vb[k];
        const float delta = rb[k] + gamma * vn * nt - vt;
        A = delta + gl * nt * A;
        vn = vt;
        if (t - P >= 0) load(k, t - P);
        const int64_t o = (int64_t)t * E + e;
        __stcs(adv + o, A);
        __stcs(ret + o, A + vt);
      }
    }
  }
}

template <int P, int NT>
static pe_status gae_stream_run(const float* r, const float* v, const uint8_t* d, const float* last_v, int T,
                                int E, float gamma, float lam, float* adv, float* ret, cudaStream_t st) {
  {
    ProfScope ps(PE_PROF_GAE, st);
    gae_stream_kernel<P, NT><<<ceil_div(E, NT), NT, 0, st>>>(r, v, d, last_v, T, E, gamma, lam, adv, ret);
  }
  PE_CHECK_LAUNCH("gae_stream_kernel");
  return PE_OK;
}

template <int CL, int NW, int V>
static pe_status gae_run(const float* r, const float* v, const uint8_t* d, const float* last_v, int T,
                         int E, float gamma, float lam, float* adv, float* ret, cudaStream_t st) {
  {
    ProfScope ps(PE_PROF_GAE, st);
    gae_kernel_v<CL, NW, V><<<ceil_div(E / V, 32), 32 * NW, 0, st>>>(r, v, d, last_v, T, E, gamma, lam, adv, ret);
  }
  PE_CHECK_LAUNCH("gae_kernel");
  return PE_OK;
}

pe_status gae_launch(const float* r, const float* v, const uint8_t* d, const float* last_v,
                     int T, int E, float gamma, float lam, float* adv, float* ret,
                     cudaStream_t st) {
  const bool al2 = (E % 2 == 0) && ((reinterpret_cast<uintptr_t>(r) | reinterpret_cast<uintptr_t>(v) |
                                      reinterpret_cast<uintptr_t>(adv) | reinterpret_cast<uintptr_t>(ret) |
                                      reinterpret_cast<uintptr_t>(last_v)) % 8 == 0) &&
                   reinterpret_cast<uintptr_t>(d) % 2 == 0;
  int dev = 0, sms = 0;
  PE_TRY_CUDA(cudaGetDevice(&dev));
  PE_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // The streaming kernels by what the SMs hold at once: with 32 steps in flight
  // 512 envs per SM, with 16 steps 1,024; a partly filled second wave costs more
  // than the shallower ring.  Measured on 152 SMs, with 54M env-steps: 56,000
  // envs 169 us (16 steps: 183), 85,000 envs 180 (32 steps: 199), 150,000 envs
  // 175 (181), 262,144 envs 171; 64 steps in flight below 230 envs per SM: 32,768
  // envs 186 us (32 steps: 193), 34,000 envs 191 (193), 36,000 envs 194 (191).
  // Blocks of 64 spread more evenly over the SMs (42,000 envs: 193 against 201
  // us); where a row does not start on a 16-byte boundary, neighbouring blocks
  // share more lines (49,151 envs: 201 against 195).
  if (E > 920 * sms) return gae_stream_run<32, 128>(r, v, d, last_v, T, E, gamma, lam, adv, ret, st);
  if (E > 400 * sms) return gae_stream_run<16, 64>(r, v, d, last_v, T, E, gamma, lam, adv, ret, st);
  if (E > 250 * sms && E % 4 == 0) return gae_stream_run<32, 64>(r, v, d, last_v, T, E, gamma, lam, adv, ret, st);
  if (E > 230 * sms) return gae_stream_run<32, 128>(r, v, d, last_v, T, E, gamma, lam, adv, ret, st);
  // The chunked kernels while their CTAs fit the SMs at once (one of 1,024
  // threads per 32 envs, two of 512 per 32 or 64 envs); beyond that the
  // streaming kernel with 64 steps in flight.  2,048 steps of 10,000 envs: 140
  // us (179 with CTAs of 32 envs), of 20,000 envs 181 (281 with CTAs of 64).  Long
  // horizons change nothing: of 2^28 env-steps 4,096 envs take 1.75 ms, 16,384
  // envs 1.24 (CTAs of 128 envs with 16-byte loads: 8.0 and 2.2).
  if (E > 128 * sms || (E > 64 * sms && !al2))
    return gae_stream_run<64, 64>(r, v, d, last_v, T, E, gamma, lam, adv, ret, st);
  if (E > 64 * sms) return gae_run<4, 16, 2>(r, v, d, last_v, T, E, gamma, lam, adv, ret, st);
  if (E > 32 * sms) return gae_run<8, 16, 1>(r, v, d, last_v, T, E, gamma, lam, adv, ret, st);
  return gae_run<8, 32, 1>(r, v, d, last_v, T, E, gamma, lam, adv, ret, st);
}

}  // namespace pe
