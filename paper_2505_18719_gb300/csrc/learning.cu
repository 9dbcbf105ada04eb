// The value model's output and the learning-phase quantities of the method, on the device:
//  * value head: V(o_t, v_t^in) of Algorithm 1 for a homogeneous value model (the same decoder
//    as the policy): the final RMSNorm of each env's last prefix row, then one linear output;
//  * GAE (Algorithm 1, "compute advantages"; §3.3): the reverse recursion over M steps,
//    one lane per env;
//  * the clipped PPO objective of Eq. 2 with action log-probs as the sum of the 7 token
//    log-probs (Eq. 1): one CTA, a fixed-order reduction, so the result is deterministic.
#include "misc.h"

namespace vla {

namespace {

// One CTA (256 threads) per env: V_b = sum_c h_c r g_c w_c + bias, r = rsqrt(mean h^2 + eps).
__global__ void __launch_bounds__(256) value_head_kernel(const float* h, int ldh, int d,
                                                         const bf16* __restrict__ gain,
                                                         const bf16* __restrict__ w, float eps,
                                                         float bias, float* __restrict__ out) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ float red[2][8];
  const float* row = h + static_cast<size_t>(blockIdx.x) * ldh;
  float ss = 0.f, dot = 0.f;
  for (int c = threadIdx.x; c < d; c += blockDim.x) {
    const float x = row[c];
    ss += x * x;
    dot += x * bf2f(gain[c]) * bf2f(w[c]);
  }
  ss = warp_sum(ss);
  dot = warp_sum(dot);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    red[0][warp] = ss;
    red[1][warp] = dot;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.f, t = 0.f;
    for (int i = 0; i < 8; ++i) {
      s += red[0][i];
      t += red[1][i];
    }
    out[blockIdx.x] = t * rsqrtf(s / static_cast<float>(d) + eps) + bias;
  }
}

// GAE: A_t = delta_t + c_t A_{t+1} with c_t = gamma lam (1 - done_t), t = M-1 .. 0, for 32 envs per
// CTA (lane = env).  The recurrence is a chain of M dependent FMAs per env, so everything else is
// taken off it: all 8 warps load a chunk of 64 steps ahead (coalesced over the envs) and put (delta_t,
// c_t) into shared memory, warp 0 walks the chunk (one FMA a step, same order and rounding as a plain
// loop), and all warps write A and A + V out while the next chunk's loads are in flight.  The
// one-thread-per-env loop over global memory paid a load's latency every step: 128 steps x 256 envs
// took 75.5 us with cold caches (23.8 us a call back to back), now 5.2 (about 9, the caller's share
// included); 1024 x 4096 took 552 us, now 23.1.
constexpr int kGaeT = 64;                 // steps per chunk
constexpr int kGaeWarps = 8;
constexpr int kGaeRows = kGaeT / kGaeWarps;  // steps of a chunk per warp

__global__ void __launch_bounds__(32 * kGaeWarps) gae_kernel(const float* r, const float* v, const float* done,
                                                             int M, int B, float gamma, float lam,
                                                             float* __restrict__ adv, float* __restrict__ ret) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ float2 dc[kGaeT][32];  // (delta, c)
  __shared__ float as[kGaeT][32];   // A
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = blockIdx.x * 32 + lane;
  const bool ok = b < B;
  const int n_chunks = (M + kGaeT - 1) / kGaeT;
  float xr[kGaeRows], xv[kGaeRows], xn[kGaeRows], xd[kGaeRows];
  // steps of chunk k: t0 + 0 .. kGaeT-1; this warp's are t0 + warp * kGaeRows + i
  auto load = [&](int k) {
    const int t0 = k * kGaeT + warp * kGaeRows;
#pragma unroll
    for (int i = 0; i < kGaeRows; ++i) {
      const bool in = ok && t0 + i < M;
      const size_t at = static_cast<size_t>(t0 + i) * B + b;
      xr[i] = in ? r[at] : 0.f;
      xv[i] = in ? v[at] : 0.f;
      xn[i] = in ? v[at + B] : 0.f;
      xd[i] = in ? done[at] : 0.f;
    }
  };
  float next = 0.f;
  load(n_chunks - 1);
  for (int k = n_chunks - 1; k >= 0; --k) {
    float vt[kGaeRows];
#pragma unroll
    for (int i = 0; i < kGaeRows; ++i) {
      const float live = 1.f - xd[i];
      dc[warp * kGaeRows + i][lane] = make_float2(xr[i] + gamma * live * xn[i] - xv[i], gamma * lam * live);
      vt[i] = xv[i];
    }
    __syncthreads();
    if (k > 0) load(k - 1);
    const int rows = min(kGaeT, M - k * kGaeT);
    if (warp == 0) {
      // 16 steps' operands in registers ahead of the chain; steps past M have delta = 0 and leave
      // the chain's initial 0 alone
#pragma unroll 1
      for (int t1 = kGaeT - 1; t1 >= 0; t1 -= 16) {
        float2 x[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = dc[t1 - i][lane];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          next = fmaf(x[i].y, next, x[i].x);
          as[t1 - i][lane] = next;
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kGaeRows; ++i) {
      const int t = warp * kGaeRows + i;
      if (!ok || t >= rows) continue;
      const size_t at = static_cast<size_t>(k * kGaeT + t) * B + b;
      const float a = as[t][lane];
      adv[at] = a;
      if (ret) ret[at] = a + vt[i];
    }
    // dc and as are written again only after the next barrier, or by the warps that have read them
  }
}

// One CTA of 1024 threads: thread j sums samples j, j + 1024, ... in order; then a fixed tree.
__global__ void __launch_bounds__(1024) ppo_clip_kernel(const float* lp_new,
                                                        const float* lp_old,
                                                        const float* adv, int N, int A,
                                                        float eps, float* __restrict__ objective,
                                                        float* __restrict__ ratio,
                                                        float* __restrict__ clip_frac) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ float red[2][32];
  float acc = 0.f, clipped = 0.f;
  for (int n = threadIdx.x; n < N; n += blockDim.x) {
    float dl = 0.f;
    for (int i = 0; i < A; ++i)
      dl += lp_new[static_cast<size_t>(n) * A + i] - lp_old[static_cast<size_t>(n) * A + i];
    const float rho = expf(dl);
    const float a = adv[n];
    const float rc = fminf(fmaxf(rho, 1.f - eps), 1.f + eps);
    acc += fminf(rho * a, rc * a);
    clipped += fabsf(rho - 1.f) > eps ? 1.f : 0.f;
    if (ratio) ratio[n] = rho;
  }
  acc = warp_sum(acc);
  clipped = warp_sum(clipped);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    red[0][warp] = acc;
    red[1][warp] = clipped;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.f, c = 0.f;
    for (int i = 0; i < static_cast<int>(blockDim.x >> 5); ++i) {
      s += red[0][i];
      c += red[1][i];
    }
    objective[0] = s / static_cast<float>(N);
    if (clip_frac) clip_frac[0] = c / static_cast<float>(N);
  }
}

}  // namespace

int value_head_launch(const float* h, int ldh, int B, int d, const bf16* gain, const bf16* w, float eps,
                      float bias, float* out, cudaStream_t s) {
  if (B <= 0) return VLA_OK;
  VLA_CUDA_TRY(launch_pdl(value_head_kernel, dim3(B), dim3(256), 0, s, h, ldh, d, gain, w, eps, bias, out));
  note_launch();
  VLA_CUDA_TRY(cudaGetLastError());
  return VLA_OK;
}

int gae_launch(const float* r, const float* v, const float* done, int M, int B, float gamma, float lam,
               float* adv, float* ret, cudaStream_t s) {
  if (M <= 0 || B <= 0) return VLA_OK;
  VLA_CUDA_TRY(launch_pdl(gae_kernel, dim3((B + 31) / 32), dim3(32 * kGaeWarps), 0, s, r, v, done, M, B, gamma, lam,
                          adv, ret));
  note_launch();
  VLA_CUDA_TRY(cudaGetLastError());
  return VLA_OK;
}

int ppo_clip_launch(const float* lp_new, const float* lp_old, const float* adv, int N, int A, float eps,
                    float* objective, float* ratio, float* clip_frac, cudaStream_t s) {
  if (N <= 0) return VLA_ERR_ARG;
  VLA_CUDA_TRY(launch_pdl(ppo_clip_kernel, dim3(1), dim3(1024), 0, s, lp_new, lp_old, adv, N, A, eps, objective,
                          ratio, clip_frac));
  note_launch();
  VLA_CUDA_TRY(cudaGetLastError());
  return VLA_OK;
}

}  // namespace vla
