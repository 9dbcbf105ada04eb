// Action head: final RMSNorm -> the 256 action-bin logits -> logsumexp -> Gumbel-max
// sample -> log-prob and bin-centre action (paper §3.1: each action token is one discrete
// bin of one action dimension, a_t = f(v_out); Eq. 1: per-token log-probs; Table 2: the
// sampling temperature).  Only the last 256 rows of lm_head are ever read.
//
// One kernel: a cluster of 8 CTAs takes 8 or 16 rows.  CTA c multiplies slice c of d (h * gain as three
// bf16 parts, which hold an fp32 value in full, times the bf16 bin rows: exact products on mma.sync,
// fp32 sums), the slices' [rows, 256] partial products meet over distributed shared memory, and CTA c
// then owns rows c (and c + 8): scale by 1 / RMS, logsumexp, argmax (ties to the lowest bin), outputs.
// Between decode steps the CTA that sampled a row's token also assembles the next step's row from it (its
// embedding and first RMSNorm), a launch less per step.
// Bound by the latency of its chain (rows, weights from L2, exchange, block reductions); two kernels,
// with fp32 FMAs on one CTA per 32 bins x 8 rows before, took 22.2 + 4.3 us at 64 rows x 4096 in a
// decode's launch list (cold caches), this one 15.0 with the next step's rows; alone 12.4.
#include "misc.h"
#include "ptx.cuh"

namespace vla {

namespace {

struct ArgMax {
  float v;
  int i;
};
// Larger value wins; equal values -> lower index.  Callers map NaN scores to -inf first (a NaN
// held in `a` would otherwise never be replaced, since no comparison with NaN is true).
__device__ __forceinline__ ArgMax better(ArgMax a, ArgMax b) {
  if (b.v > a.v || (b.v == a.v && b.i < a.i)) return b;
  return a;
}

// y -> bf16 parts hi + mid + lo (8 significant bits each: an fp32 value in full), two values packed.
// A part that would come from inf - inf or NaN is left zero: hi alone carries a non-finite value.
__device__ __forceinline__ void split3_pack2(float a, float b, uint32_t (&p)[3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    p[i] = pack_bf16x2(a, b);
    const float2 f = unpack_bf16x2(p[i]);
    a = isfinite(f.x) ? a - f.x : 0.f;
    b = isfinite(f.y) ? b - f.y : 0.f;
  }
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ float ld_cluster(uint32_t addr) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}

constexpr int kHeadCluster = 8;  // CTAs of a cluster: slices of d, then rows
constexpr int kHeadThreads = 256;
constexpr int kPartStride = 256 + 8;

// Slice of d per CTA (a multiple of the 32-wide step) and the row stride of the split rows in
// shared memory (bf16 elements): 16 words modulo 32, so a quarter warp's 16-byte reads of two rows
// hit all banks once.
__host__ __device__ constexpr int head_slice(int d) { return ((d + kHeadCluster - 1) / kHeadCluster + 31) / 32 * 32; }
__host__ __device__ constexpr int head_stride(int slice) { return (slice / 2) % 32 == 0 ? slice + 32 : slice; }
constexpr int kHeadMaxD = 6400;
// Up to 128 rows a cluster takes 8 of them (half of each MMA's 16 rows is padding): the calls are
// bound by latency, and one row per CTA halves the sampling's share of it.  Above, 16 rows per
// cluster halve the MMAs and the weight reads from L2.
constexpr int kHeadSmallRows = 128;
constexpr size_t head_smem(int d, int rows) {
  return static_cast<size_t>(rows) * head_stride(head_slice(d)) * 3 * 2 + static_cast<size_t>(rows) * kPartStride * 4;
}

// RPC: rows per CTA after the exchange, 8 * RPC rows per cluster.  FIRST: the rows come from two places
// (h_first).  Two CTAs per SM only where the grid needs them (RPC 2: 448 rows are 224 CTAs): the 128 registers
// that leaves cost a few spills.
template <int RPC, bool FIRST>
__global__ void __launch_bounds__(kHeadThreads, RPC) head_kernel(const HeadArgs a) {
  constexpr int ROWS = kHeadCluster * RPC;
  constexpr int DEPTH = RPC == 1 ? 4 : 3;  // 32-wide steps of weights in flight per warp
  extern __shared__ __align__(16) uint8_t head_sm[];
  __shared__ float ss_s[ROWS];
  __shared__ float z_s[256];
  __shared__ float red_f[8];
  __shared__ ArgMax red_a[8];
  __shared__ float red_m[8];
  __shared__ int fed_s;
  pdl_launch_dependents();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, tq = lane & 3;
  const int d = a.d, R = a.B * a.n_pos;
  const int rank = static_cast<int>(cluster_ctarank());
  const int r0 = static_cast<int>(blockIdx.x / kHeadCluster) * ROWS;
  const int slice = head_slice(d), stride = head_stride(slice);
  const int k0 = rank * slice;
  bf16* ys = reinterpret_cast<bf16*>(head_sm);  // [3][ROWS][stride]
  float* part = reinterpret_cast<float*>(head_sm + static_cast<size_t>(3) * ROWS * stride * 2);  // [ROWS][kPartStride]

  // this warp's bins 32 warp + 8 nt + g; lane tq of a row reads 8 consecutive k of each 32-wide step.
  // Which k an MMA element stands for does not matter as long as A and B agree: of the 8, elements 0-3
  // serve the step's first MMA and 4-7 its second.
  const bf16* wrow = a.head_rows + static_cast<size_t>(warp * 32 + g) * d;
  const int steps = slice / 32;
  uint4 wq[DEPTH][4];
  auto load_w = [&](int step, uint4 (&w)[4]) {
    const int k = k0 + step * 32 + tq * 8;
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
      w[nt] = (step < steps && k < d) ? *reinterpret_cast<const uint4*>(wrow + static_cast<size_t>(nt * 8) * d + k)
                                      : make_uint4(0u, 0u, 0u, 0u);
  };
  // the bin rows are the caller's weights: requested before the previous kernel is waited for (as a call's
  // first kernel the head is launched in stream order)
#pragma unroll
  for (int i = 0; i < DEPTH; ++i) load_w(i, wq[i]);

  pdl_wait();
  // rows r0 + i: h * gain of this CTA's slice as three bf16 parts, and its share of the sum of squares
#pragma unroll
  for (int j = 0; j < RPC; ++j) {
    const int i = warp * RPC + j, r = r0 + i;
    const float* hrow = a.h + static_cast<size_t>(r) * a.ldh;
    if (FIRST && r < R) {
      const int b = r / a.n_pos, pos = r - b * a.n_pos;
      hrow = pos == 0 ? a.h_first + static_cast<size_t>(b) * a.ldh
                      : a.h + static_cast<size_t>(b * (a.n_pos - 1) + pos - 1) * a.ldh;
    }
    float ss = 0.f;
#pragma unroll 4
    for (int c = lane * 4; c < slice; c += 128) {
      const int k = k0 + c;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      float2 w0 = make_float2(0.f, 0.f), w1 = w0;
      if (r < R && k < d) {
        v = __ldcg(reinterpret_cast<const float4*>(hrow + k));
        const uint2 ww = *reinterpret_cast<const uint2*>(a.final_norm + k);
        w0 = unpack_bf16x2(ww.x);
        w1 = unpack_bf16x2(ww.y);
      }
      ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
      uint32_t p0[3], p1[3];
      split3_pack2(v.x * w0.x, v.y * w0.y, p0);
      split3_pack2(v.z * w1.x, v.w * w1.y, p1);
#pragma unroll
      for (int q = 0; q < 3; ++q)
        *reinterpret_cast<uint2*>(ys + (static_cast<size_t>(q) * ROWS + i) * stride + c) = make_uint2(p0[q], p1[q]);
    }
    ss = warp_sum(ss);
    if (lane == 0) ss_s[i] = ss;
  }
  __syncthreads();

  float acc[4][4];
#pragma unroll
  for (int nt = 0; nt < 4; ++nt) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.f;
  for (int s0 = 0; s0 < steps; s0 += DEPTH) {
#pragma unroll
    for (int u = 0; u < DEPTH; ++u) {
      const int step = s0 + u;
      if (step >= steps) break;
      // a fresh accumulator per step, the small parts first: the tensor cores truncate their sums, so
      // a long chain of them drifts (1.8e-6 of the logits' norm at d = 4096); added up here in
      // rounded fp32 the error is 1.3e-7, that of a plain
      // chain of fp32 FMAs 2.2e-7
      float t[4][4];
#pragma unroll
      for (int nt = 0; nt < 4; ++nt) t[nt][0] = t[nt][1] = t[nt][2] = t[nt][3] = 0.f;
#pragma unroll
      for (int q = 2; q >= 0; --q) {
        const bf16* yp = ys + (static_cast<size_t>(q) * ROWS + g) * stride + step * 32 + tq * 8;
        const uint4 x = *reinterpret_cast<const uint4*>(yp);
        const uint4 y = RPC == 2 ? *reinterpret_cast<const uint4*>(yp + 8 * stride) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
          mma_bf16(t[nt], x.x, y.x, x.y, y.y, wq[u][nt].x, wq[u][nt].y);
          mma_bf16(t[nt], x.z, y.z, x.w, y.w, wq[u][nt].z, wq[u][nt].w);
        }
      }
#pragma unroll
      for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int c = 0; c < (RPC == 2 ? 4 : 2); ++c) acc[nt][c] += t[nt][c];
      load_w(step + DEPTH, wq[u]);
    }
  }
#pragma unroll
  for (int nt = 0; nt < 4; ++nt) {
    const int col = warp * 32 + nt * 8 + 2 * tq;
    *reinterpret_cast<float2*>(part + g * kPartStride + col) = make_float2(acc[nt][0], acc[nt][1]);
    if (RPC == 2) *reinterpret_cast<float2*>(part + (g + 8) * kPartStride + col) = make_float2(acc[nt][2], acc[nt][3]);
  }
  cluster_sync();

  // rows rank (and rank + 8): the eight slices' dot products, summed in slice order; the norm is a
  // per-row scale, applied to the sum
  const int k = tid;  // thread k owns bin k from here on
  float z_of[RPC];
#pragma unroll
  for (int j = 0; j < RPC; ++j) {
    const int i = rank + j * kHeadCluster;
    float z = 0.f, ss = 0.f;
#pragma unroll
    for (int c = 0; c < kHeadCluster; ++c) {
      z += ld_cluster(mapa_shared(smem_u32(part + i * kPartStride + k), c));
      ss += ld_cluster(mapa_shared(smem_u32(ss_s + i), c));
    }
    z_of[j] = z * rsqrtf(ss / static_cast<float>(d) + a.eps);
  }
  cluster_arrive();  // this CTA is done with the others' shared memory
#pragma unroll 1
  for (int j = 0; j < RPC; ++j) {
    const int r = r0 + rank + j * kHeadCluster;
    if (r >= R) break;
    const int b = r / a.n_pos;
    const int out_i = b * a.A + a.step + (r - b * a.n_pos);  // [B, A] output slot
    const float z = z_of[j];
    z_s[k] = z;
    const float T = a.temperature;
    const float zt = (T > 0.f) ? z / T : z;
    float s = zt;
    if (T > 0.f && a.uniforms) {
      float u = a.uniforms[static_cast<size_t>(out_i) * 256 + k];
      u = fminf(fmaxf(u, 5.9604644775390625e-8f), 0.99999994039535522f);  // [2^-24, 1-2^-24]
      s = zt - logf(-logf(u));
    }
    // A NaN score (from a NaN logit, which raises VLA_STATUS_NONFINITE below) loses to every bin.
    ArgMax am{isnan(s) ? -INFINITY : s, k};
    float mx = zt;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      ArgMax other{__shfl_xor_sync(0xffffffffu, am.v, o), __shfl_xor_sync(0xffffffffu, am.i, o)};
      am = better(am, other);
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if (lane == 0) {
      red_a[warp] = am;
      red_m[warp] = mx;
    }
    __syncthreads();
    ArgMax best = red_a[0];
    float zmax = red_m[0];
#pragma unroll
    for (int w = 1; w < 8; ++w) {
      best = better(best, red_a[w]);
      zmax = fmaxf(zmax, red_m[w]);
    }
    const float e = expf(zt - zmax);
    float se = warp_sum(e);
    float sez = warp_sum(e * (zt - zmax));  // for the entropy: sum_k p_k (zt_k - zmax) * sum_e
    __syncthreads();  // red_f reuse
    if (lane == 0) {
      red_f[warp] = se;
      red_m[warp] = sez;
    }
    __syncthreads();
    float sum_e = 0.f, sum_ez = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      sum_e += red_f[w];
      sum_ez += red_m[w];
    }
    const float lse = zmax + logf(sum_e);
    // rollout entropy of this token's bin distribution: H = lse - sum_k p_k zt_k
    if (tid == 0 && a.entropy_out) a.entropy_out[out_i] = logf(sum_e) - sum_ez / sum_e;

    if (a.logits_out) a.logits_out[static_cast<size_t>(out_i) * 256 + k] = z;
    if (!isfinite(z)) atomicOr(a.status, VLA_STATUS_NONFINITE);

    if (tid == 0) {
      const int ks = best.i;
      int kl = ks;  // bin whose log-prob is reported
      int fed = a.token_base + ks;
      if (a.forced) {
        int f = a.forced[out_i] - a.forced_base;
        if (f < 0 || f >= 256) {
          atomicOr(a.status, VLA_STATUS_BAD_FORCED);
          f = f < 0 ? 0 : 255;
        }
        kl = f;
        fed = a.token_base + f;
      }
      a.lp_out[out_i] = z_s[kl] / (T > 0.f ? T : 1.f) - lse;
      if (a.tokens_out) a.tokens_out[out_i] = a.token_base + ks;
      if (a.bins_out) a.bins_out[out_i] = ks;
      if (a.act_out) a.act_out[out_i] = static_cast<float>(2 * ks + 1 - 256) * (1.0f / 256.0f);
      // the env's last token stays pending (a scored one as given, its range is checked when it is fed)
      if (a.pending_out && out_i == b * a.A + a.A - 1) a.pending_out[b] = FIRST ? a.forced[out_i] : fed;
      fed_s = fed;
    }
    __syncthreads();  // the shared arrays are the next row's
    // the next step's input row: every CTA of the cluster has read row r of a.h
    if (a.next_embed)
      token_row_256(a.next_embed + static_cast<size_t>(fed_s) * d, d, a.next_h + static_cast<size_t>(r) * d, a.next_norm,
                    static_cast<size_t>(r) * d, red_f, a.status);
  }
  cluster_wait();  // the others are done with this CTA's shared memory
}

}  // namespace

int action_head_launch(const HeadArgs& a, cudaStream_t s) {
  if (a.B <= 0) return VLA_OK;
  if (a.d % 8 || a.ldh % 4 || (reinterpret_cast<uintptr_t>(a.h) & 15) ||
      (reinterpret_cast<uintptr_t>(a.h_first) & 15) || (reinterpret_cast<uintptr_t>(a.head_rows) & 15) ||
      (reinterpret_cast<uintptr_t>(a.final_norm) & 7))
    return VLA_ERR_UNSUPPORTED;
  if (a.d > kHeadMaxD) return VLA_ERR_UNSUPPORTED;
  const int R = a.B * a.n_pos;
  auto go = [&](auto kern, int rows, std::atomic<uint64_t>& attr_done) -> cudaError_t {
    if (const cudaError_t e = set_smem_limit(kern, static_cast<int>(head_smem(kHeadMaxD, rows)), attr_done)) return e;
    return launch_cluster_at(a.start, kern, dim3((R + rows - 1) / rows * kHeadCluster), dim3(kHeadThreads),
                             head_smem(a.d, rows), s, kHeadCluster, a);
  };
  static std::atomic<uint64_t> done[4];
  if (R <= kHeadSmallRows) {
    VLA_CUDA_TRY(a.h_first ? go(head_kernel<1, true>, kHeadCluster, done[0]) : go(head_kernel<1, false>, kHeadCluster, done[1]));
  } else {
    VLA_CUDA_TRY(a.h_first ? go(head_kernel<2, true>, 2 * kHeadCluster, done[2])
                           : go(head_kernel<2, false>, 2 * kHeadCluster, done[3]));
  }
  note_launch();
  VLA_CUDA_TRY(cudaGetLastError());
  return VLA_OK;
}

}  // namespace vla
