// The value model's output and the learning-phase quantities of the method, on the device:
//  * value head: V(o_t, v_t^in) of Algorithm 1 for a homogeneous value model (the same decoder
//    as the policy): the final RMSNorm of each env's last prefix row, then one linear output;
//  * GAE (Algorithm 1, "compute advantages"; §3.3): the reverse recursion over M steps,
//    one lane per env;
//  * the clipped PPO objective of Eq. 2 with action log-probs as the sum of the 7 token
//    log-probs (Eq. 1): one cluster, a fixed-order reduction, so the result is deterministic.
#include <algorithm>

#include "misc.h"
#include "ptx.cuh"

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

// Blocks of `size` that hold n >= 1 items (no sum that overflows at the largest n).
__host__ __device__ constexpr int blocks_of(int n, int size) { return (n - 1) / size + 1; }
static_assert(blocks_of(1, 64) == 1 && blocks_of(64, 64) == 1 && blocks_of(65, 64) == 2 && blocks_of(0x7fffffff, 64) == 1 << 25,
              "blocks");

// GAE: A_t = delta_t + c_t A_{t+1} with c_t = gamma lam (1 - done_t), t = M-1 .. 0, for 32 envs per
// CTA (lane = env).  The recurrence is a chain of M dependent FMAs per env, so everything else is
// taken off it: all 8 warps load a chunk of 64 steps ahead (coalesced over the envs) and put (delta_t,
// c_t) into shared memory, warp 0 walks the chunk (one FMA a step, same order and rounding as a plain
// loop), and all warps write A and A + V out while the next chunk's loads are in flight.  The
// one-thread-per-env loop over global memory paid a load's latency every step: 128 steps x 256 envs
// took 75.5 us with cold caches (23.7 us a call back to back, 34 alone), now 5.2 (3.5 back to back, 13
// alone; 8 to 11 through the caller's tensors); 1024 x 4096 took 552 us, now 23.1.
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
  const int n_chunks = blocks_of(M, kGaeT);
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

// The clipped objective on one thread-block cluster: the samples go round-robin over its CTAs in
// tiles of 512, each tile's log-probs staged through shared memory (cp.async, all but one stage in
// flight; A floats per sample are then read at stride A), one sample per thread; the CTAs' sums meet in CTA
// 0 over distributed shared memory in a fixed order, so no scratch memory is shared between
// calls and repeated calls give identical results.  One CTA of 1024 threads walked all samples
// before: 32768 x 7 took 41.3 us with cold caches (21.8 us a call back to back, 32 alone; one SM's share of
// bandwidth and latency), now 7.6 (5.8 back to back, 16 alone; 11 to 14 through the caller's tensors) on 16
// CTAs; 1M samples x 7 took 1215 us, now 111, the bandwidth of those 16 SMs.
constexpr int kPpoTile = 512;   // samples per tile = threads
constexpr int kPpoMaxA = 16;    // more tokens per sample are read in place (no staging)

__device__ __forceinline__ void ppo_cp16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

constexpr int kPpoStageBytes = 2 * kPpoTile * 4;  // per token of a sample

template <int kPpoStages>
__global__ void __launch_bounds__(kPpoTile) ppo_clip_kernel(const float* lp_new, const float* lp_old,
                                                            const float* adv, int N, int A, int staged,
                                                            float eps, float* __restrict__ objective,
                                                            float* __restrict__ ratio,
                                                            float* __restrict__ clip_frac) {
  extern __shared__ __align__(16) float ppo_sm[];  // [stage][new, old][kPpoTile * A]
  __shared__ float red[2][kPpoTile / 32];
  __shared__ float2 cta_sum;
  pdl_launch_dependents();
  pdl_wait();
  const int n_cta = static_cast<int>(gridDim.x), rank = static_cast<int>(blockIdx.x);
  const int tid = threadIdx.x;
  const int tiles = blocks_of(N, kPpoTile);
  const int plane = kPpoTile * A;
  auto stage_load = [&](int tile, int st) {
    if (tile < tiles) {
      const size_t first = static_cast<size_t>(tile) * plane;  // a multiple of 512 floats
      const int n = min(kPpoTile, N - tile * kPpoTile) * A;
      float* dn = ppo_sm + static_cast<size_t>(st) * 2 * plane;
      const uint32_t sn = static_cast<uint32_t>(__cvta_generic_to_shared(dn)), so = sn + plane * 4;
      const int n4 = n >> 2;
      for (int i = tid; i < n4; i += kPpoTile) {
        ppo_cp16(sn + i * 16, lp_new + first + i * 4);
        ppo_cp16(so + i * 16, lp_old + first + i * 4);
      }
      for (int i = (n4 << 2) + tid; i < n; i += kPpoTile) {  // the last 0-3 floats
        dn[i] = lp_new[first + i];
        dn[plane + i] = lp_old[first + i];
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc = 0.f, clipped = 0.f;
  auto adv_of = [&](int tile) {
    return tile < tiles && tile * kPpoTile + tid < N ? adv[tile * kPpoTile + tid] : 0.f;
  };
  float a = adv_of(rank);
  if (staged)
    for (int s = 0; s < kPpoStages - 1; ++s) stage_load(rank + s * n_cta, s);
  int st = 0;
  for (int tile = rank; tile < tiles; tile += n_cta) {
    const int n = tile * kPpoTile + tid;
    const float a_next = adv_of(tile + n_cta);  // in flight during this tile
    const float *pn, *po;
    if (staged) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kPpoStages - 2) : "memory");
      __syncthreads();
      stage_load(tile + (kPpoStages - 1) * n_cta, (st + kPpoStages - 1) % kPpoStages);
      pn = ppo_sm + static_cast<size_t>(st) * 2 * plane + tid * A;
      po = pn + plane;
      st = (st + 1) % kPpoStages;
    } else {
      pn = lp_new + static_cast<size_t>(n) * A;
      po = lp_old + static_cast<size_t>(n) * A;
    }
    if (n < N) {
      float dl = 0.f;
      if (staged && (A & 3) == 0) {  // 16-byte reads: at a stride of 4, 8 or 16 floats scalar ones conflict
        for (int i = 0; i < A; i += 4) {
          const float4 x = *reinterpret_cast<const float4*>(pn + i), y = *reinterpret_cast<const float4*>(po + i);
          dl += x.x - y.x;
          dl += x.y - y.y;
          dl += x.z - y.z;
          dl += x.w - y.w;
        }
      } else {
  #pragma unroll 4
        for (int i = 0; i < A; ++i) dl += pn[i] - po[i];
      }
      const float rho = expf(dl);
      const float rc = fminf(fmaxf(rho, 1.f - eps), 1.f + eps);
      acc += fminf(rho * a, rc * a);
      clipped += fabsf(rho - 1.f) > eps ? 1.f : 0.f;
      if (ratio) ratio[n] = rho;
    }
    a = a_next;
  }
  acc = warp_sum(acc);
  clipped = warp_sum(clipped);
  const int warp = tid >> 5, lane = tid & 31;
  if (lane == 0) {
    red[0][warp] = acc;
    red[1][warp] = clipped;
  }
  __syncthreads();
  if (tid == 0) {
    float s = 0.f, c = 0.f;
    for (int i = 0; i < kPpoTile / 32; ++i) {
      s += red[0][i];
      c += red[1][i];
    }
    cta_sum = make_float2(s, c);
  }
  if (n_cta > 1) cluster_sync();
  if (rank == 0 && tid < 32) {
    float2 x = make_float2(0.f, 0.f);
    if (lane < n_cta) {
      if (lane == 0) {
        x = cta_sum;
      } else {
        const uint32_t at = mapa_shared(smem_u32(&cta_sum), lane);
        asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(x.x), "=f"(x.y) : "r"(at) : "memory");
      }
    }
    const float s = warp_sum(x.x), c = warp_sum(x.y);
    if (lane == 0) {
      objective[0] = s / static_cast<float>(N);
      if (clip_frac) clip_frac[0] = c / static_cast<float>(N);
    }
  }
  if (n_cta > 1) cluster_sync();  // the other CTAs' sums stay readable until CTA 0 has them
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
  // one tile per CTA up to 16 CTAs (the non-portable cluster maximum) or what the device can place: the
  // CTAs take the tiles in turn at any number; the staging needs 16-byte aligned log-probs.  Two tiles of
  // few tokens are read in place by one CTA: 1024 x 7 takes 2.7 us back to back and 12.4 alone, on two CTAs
  // 3.1 to 3.4 and 13.2 (1024 x 8: 4.0 and 14.0, on two CTAs 3.3 and 13.5).
  const int tiles = blocks_of(N, kPpoTile);
  const bool small = tiles <= 2 && A < 8;
  const int want = tiles <= 1 || small ? 1 : tiles <= 2 ? 2 : tiles <= 4 ? 4 : tiles <= 8 ? 8 : 16;
  const bool staged = !small && A <= kPpoMaxA && !(reinterpret_cast<uintptr_t>(lp_new) & 15) &&
                      !(reinterpret_cast<uintptr_t>(lp_old) & 15);
  static std::atomic<uint64_t> smem_done[2] = {}, cluster_done[2] = {};
  static std::atomic<int> cluster_size[2][64] = {};
  auto go = [&](auto kern, int stages, int max_a, int which) -> cudaError_t {
    const int smem = staged ? stages * kPpoStageBytes * A : 0;
    if (const cudaError_t e = set_smem_limit(kern, stages * kPpoStageBytes * max_a, smem_done[which])) return e;
    if (const cudaError_t e = allow_wide_clusters(kern, cluster_done[which])) return e;
    int n_cta = 1;  // asked with the most shared memory that a call takes
    if (const cudaError_t e = max_cluster_size(kern, dim3(kPpoTile), stages * kPpoStageBytes * max_a, 16, cluster_size[which], &n_cta))
      return e;
    n_cta = std::min(n_cta, want);
    return launch_pdl_cluster(kern, dim3(n_cta), dim3(kPpoTile), smem, s, n_cta, lp_new, lp_old, adv, N, A,
                              staged ? 1 : 0, eps, objective, ratio, clip_frac);
  };
  // as many stages as 192 KB hold
  VLA_CUDA_TRY(A <= 8 ? go(ppo_clip_kernel<6>, 6, 8, 0) : go(ppo_clip_kernel<3>, 3, kPpoMaxA, 1));
  note_launch();
  VLA_CUDA_TRY(cudaGetLastError());
  return VLA_OK;
}

}  // namespace vla
