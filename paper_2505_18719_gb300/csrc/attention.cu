// Causal attention over the per-environment KV cache (paper §3.1: the policy's Llama-2
// self-attention; §3.3: the whole trajectory is one context, so every chunk attends to all
// earlier turns).
//
//  * attn_rows8 / attn_rows: chunks whose tiles all have at most 8 / 16 rows at consecutive positions of
//    one env (the score pass's teacher-forced action rows) over the fp16 + residual cache, one CTA per
//    (tile, head), mma.sync.  (Longer tiles, a prefill's, run on attn_tc.cu.)
//  * attn_decode: one query per env (the decode step, and each env's last row in a prefill's last
//    layer): full waves of whole (env, head) pairs on one CTA each, the pairs left over with their key
//    range split across CTAs (flash-decoding), whose partials (reference exponent, sum, unnormalised
//    output) the last one to finish merges in a fixed order.  attn_decode_short: many pairs over short
//    contexts.
//  * attn_chunk: tiles of 64 rows over a cache of fp16 alone, for the op entry point.
//
// The fp32 queries and the softmax weights are taken as two or three 16-bit parts; the output is the
// operand hi/lo pair that the O-projection GEMM reads (fp16 for the engine, bf16 for the op entry points).
//
// Keys visible to a query at position p are positions 0..p (all of them are in the cache:
// chunk rows write their K/V in the QKV epilogue before attention runs).
#include <algorithm>

#include "attention.h"
#include "ptx.cuh"

namespace vla {

namespace {


// ------------------------------------------------------------------------ chunk (tensor core)
// Flash-attention over one 64-row query tile of one env and one head: S = Q K^T and O += P V
// on mma.sync m16n8k16 (fp16 inputs, fp32 accumulation), online softmax in the exp2 domain.
// 4 warps x 16 query rows; K/V blocks of 64 keys double-buffered in shared memory with
// cp.async (rows past the last visible key are zero-filled, never read from the cache).
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2,
                                        uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2,
                                          uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
  const int n = valid ? 16 : 0;  // 0 source bytes -> 16 zero bytes
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// (a, b) -> fp16 pairs hi = fp16(x), lo = fp16(x - hi): P V is taken as P_hi V + P_lo V so the
// softmax weights keep ~22 bits.
__device__ __forceinline__ void split_h2(float a, float b, uint32_t& hi, uint32_t& lo) {
  const __half ha = __float2half_rn(a), hb = __float2half_rn(b);
  __half2 h2 = __halves2half2(ha, hb);
  __half2 l2 = __floats2half2_rn(a - __half2float(ha), b - __half2float(hb));
  hi = *reinterpret_cast<uint32_t*>(&h2);
  lo = *reinterpret_cast<uint32_t*>(&l2);
}

template <int HD>
__global__ void __launch_bounds__(128) attn_chunk_mma_kernel(const float* q,
                                                             bf16* __restrict__ out_hi,
                                                             bf16* __restrict__ out_lo,
                                                             const AttnTile* __restrict__ tiles,
                                                             KVLayout kv, int layer, int H,
                                                             float scale_log2, bool fp16) {
  constexpr int KB = 64;       // keys per block
  constexpr int LD = HD + 8;   // padded row (halves): 16-byte rows land in distinct banks
  constexpr int CPR = HD / 8;  // 16-byte chunks per row
  constexpr int NT_D = HD / 8; // n-tiles over the head dim
  extern __shared__ __align__(16) f16 sm_h[];
  f16* Ks = sm_h;              // [2][KB][LD]
  f16* Vs = Ks + 2 * KB * LD;  // [2][KB][LD]

  pdl_launch_dependents();
  pdl_wait();
  const AttnTile t = tiles[blockIdx.x];
  const int head = blockIdx.y;
  const int d = H * HD;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, tq = lane & 3;
  const f16* kbase = kv.base + static_cast<int64_t>(layer) * kv.layer_stride +
                     static_cast<int64_t>(t.env) * kv.env_stride +
                     static_cast<int64_t>(head) * kv.head_stride;
  const f16* vbase = kbase + kv.kv_stride;
  const int n_keys = t.pos0 + t.nrows;
  const int n_blocks = (n_keys + KB - 1) / KB;

  auto load_block = [&](int blk, int buf) {
    const int j0 = blk * KB;
    const uint32_t ks = static_cast<uint32_t>(__cvta_generic_to_shared(Ks + buf * KB * LD));
    const uint32_t vs = static_cast<uint32_t>(__cvta_generic_to_shared(Vs + buf * KB * LD));
    for (int i = tid; i < KB * CPR; i += 128) {
      const int r = i / CPR, c = (i - r * CPR) * 8;
      const bool ok = j0 + r < n_keys;
      const int64_t src = static_cast<int64_t>(ok ? j0 + r : 0) * HD + c;
      cp_async16(ks + (r * LD + c) * 2, kbase + src, ok);
      cp_async16(vs + (r * LD + c) * 2, vbase + src, ok);
    }
  };

  load_block(0, 0);
  cp_async_commit();

  // this thread's two rows and their positions (rows past nrows reuse the last position;
  // their results are never written)
  const int r0 = warp * 16 + g, r1 = r0 + 8;
  const int qpos0 = t.pos0 + min(r0, t.nrows - 1);
  const int qpos1 = t.pos0 + min(r1, t.nrows - 1);
  const int warp_last = t.pos0 + min(warp * 16 + 15, t.nrows - 1);
  const bool warp_active = warp * 16 < t.nrows;

  float o[NT_D][4];
#pragma unroll
  for (int i = 0; i < NT_D; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
  float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
  // Q A-fragments straight from the fp32 rows, as fp16 hi/lo pairs (S = Q_hi K + Q_lo K).
  uint32_t qh[HD / 16][4], ql[HD / 16][4];
  {
    const int ra = min(r0, t.nrows - 1), rb = min(r1, t.nrows - 1);
    const float* qa = q + static_cast<size_t>(t.row0 + ra) * d + head * HD + 2 * tq;
    const float* qb = q + static_cast<size_t>(t.row0 + rb) * d + head * HD + 2 * tq;
#pragma unroll
    for (int kk = 0; kk < HD / 16; ++kk) {
      const float2 x0 = *reinterpret_cast<const float2*>(qa + kk * 16);
      const float2 x1 = *reinterpret_cast<const float2*>(qb + kk * 16);
      const float2 x2 = *reinterpret_cast<const float2*>(qa + kk * 16 + 8);
      const float2 x3 = *reinterpret_cast<const float2*>(qb + kk * 16 + 8);
      split_h2(x0.x, x0.y, qh[kk][0], ql[kk][0]);
      split_h2(x1.x, x1.y, qh[kk][1], ql[kk][1]);
      split_h2(x2.x, x2.y, qh[kk][2], ql[kk][2]);
      split_h2(x3.x, x3.y, qh[kk][3], ql[kk][3]);
    }
  }

  for (int blk = 0; blk < n_blocks; ++blk) {
    if (blk + 1 < n_blocks) {
      load_block(blk + 1, (blk + 1) & 1);
      cp_async_commit();
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const int j0 = blk * KB;
    if (warp_active && j0 <= warp_last) {
      const int buf = blk & 1;
      const uint32_t ks = static_cast<uint32_t>(__cvta_generic_to_shared(Ks + buf * KB * LD));
      const uint32_t vs = static_cast<uint32_t>(__cvta_generic_to_shared(Vs + buf * KB * LD));
      float s[8][4];
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
        const int i = lane >> 3;
#pragma unroll
        for (int kk = 0; kk < HD / 16; kk += 2) {
          uint32_t b0, b1, b2, b3;
          const int key = nt * 8 + (lane & 7);
          const int dim = (kk + (i >> 1)) * 16 + (i & 1) * 8;
          ldsm_x4(ks + (key * LD + dim) * 2, b0, b1, b2, b3);
          mma16816(s[nt], qh[kk], b0, b1);
          mma16816(s[nt], ql[kk], b0, b1);
          mma16816(s[nt], qh[kk + 1], b2, b3);
          mma16816(s[nt], ql[kk + 1], b2, b3);
        }
      }
      // scale, causal mask, online softmax (rows r0: c 0,1; r1: c 2,3)
      float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int key = j0 + nt * 8 + 2 * tq + (c & 1);
          const int qp = (c < 2) ? qpos0 : qpos1;
          const float v = (key <= qp) ? s[nt][c] * scale_log2 : -INFINITY;
          s[nt][c] = v;
        }
        mx0 = fmaxf(mx0, fmaxf(s[nt][0], s[nt][1]));
        mx1 = fmaxf(mx1, fmaxf(s[nt][2], s[nt][3]));
      }
      mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1));
      mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
      mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
      mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
      const float mn0 = fmaxf(m0, mx0), mn1 = fmaxf(m1, mx1);  // finite: key j0 <= qpos
      const float a0 = exp2f(m0 - mn0), a1 = exp2f(m1 - mn1);
      m0 = mn0;
      m1 = mn1;
      float ps0 = 0.f, ps1 = 0.f;
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        s[nt][0] = exp2f(s[nt][0] - mn0);
        s[nt][1] = exp2f(s[nt][1] - mn0);
        s[nt][2] = exp2f(s[nt][2] - mn1);
        s[nt][3] = exp2f(s[nt][3] - mn1);
        ps0 += s[nt][0] + s[nt][1];
        ps1 += s[nt][2] + s[nt][3];
      }
      l0 = l0 * a0 + ps0;  // per-thread partial row sums; reduced across the quad at the end
      l1 = l1 * a1 + ps1;
#pragma unroll
      for (int nt = 0; nt < NT_D; ++nt) {
        o[nt][0] *= a0;
        o[nt][1] *= a0;
        o[nt][2] *= a1;
        o[nt][3] *= a1;
      }
      // O += P V: P re-used from the S accumulators as the A operand, as an fp16 hi/lo pair
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        uint32_t ph[4], pl[4];
        split_h2(s[2 * kk][0], s[2 * kk][1], ph[0], pl[0]);
        split_h2(s[2 * kk][2], s[2 * kk][3], ph[1], pl[1]);
        split_h2(s[2 * kk + 1][0], s[2 * kk + 1][1], ph[2], pl[2]);
        split_h2(s[2 * kk + 1][2], s[2 * kk + 1][3], ph[3], pl[3]);
        const int i = lane >> 3;
#pragma unroll
        for (int nt = 0; nt < NT_D; nt += 2) {
          uint32_t b0, b1, b2, b3;
          const int key = kk * 16 + (i & 1) * 8 + (lane & 7);
          const int dim = (nt + (i >> 1)) * 8;
          ldsm_x4_t(vs + (key * LD + dim) * 2, b0, b1, b2, b3);
          mma16816(o[nt], ph, b0, b1);
          mma16816(o[nt], pl, b0, b1);
          mma16816(o[nt + 1], ph, b2, b3);
          mma16816(o[nt + 1], pl, b2, b3);
        }
      }
    }
    __syncthreads();  // this buffer is refilled two blocks later
  }
  if (!warp_active) return;
  l0 += __shfl_xor_sync(0xffffffffu, l0, 1);
  l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
  l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
  l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
  const float inv0 = 1.f / l0, inv1 = 1.f / l1;
  // outputs are convex combinations of fp16 values, so the fp16 split never saturates here
  uint32_t sat = 0;
#pragma unroll
  for (int nt = 0; nt < NT_D; ++nt) {
    const int col = head * HD + nt * 8 + 2 * tq;
    if (r0 < t.nrows) {
      const size_t off = static_cast<size_t>(t.row0 + r0) * d + col;
      uint32_t hi, lo;
      split_pack2(o[nt][0] * inv0, o[nt][1] * inv0, hi, lo, fp16, sat);
      *reinterpret_cast<uint32_t*>(out_hi + off) = hi;
      *reinterpret_cast<uint32_t*>(out_lo + off) = lo;
    }
    if (r1 < t.nrows) {
      const size_t off = static_cast<size_t>(t.row0 + r1) * d + col;
      uint32_t hi, lo;
      split_pack2(o[nt][2] * inv1, o[nt][3] * inv1, hi, lo, fp16, sat);
      *reinterpret_cast<uint32_t*>(out_hi + off) = hi;
      *reinterpret_cast<uint32_t*>(out_lo + off) = lo;
    }
  }
}

// ------------------------------------------------------------------ few-row chunk (residual cache)
// Query tiles of at most 16 rows (the teacher-forced action rows of the score pass, Eq. 2, or any
// chunk that short) against keys 0..pos of their env, the cache read as fp16 + 4-bit residual
// (hi + lo, KVLayout).  One CTA per (tile, head), 4 warps, 128 registers and one 45 KB stage so
// that four CTAs share an SM (the other CTAs' blocks are in flight while one computes): key
// blocks of 64 staged in shared memory by cp.async (fp16 parts and residual codes; keys past the
// tile's last position are zero-filled, never read), the tile's query rows as an fp16 pair in
// shared memory (ldmatrix A fragments); warp w takes keys 16w .. 16w+15 of every block with one
// m16n8k16 row tile (rows past the tile's last repeat its last row and are not written), the low
// parts decoded from the codes beside each B fragment:
//   S = Q_hi K_hi + Q_lo K_hi + Q_hi K_lo,   O += P_hi V_hi + P_lo V_hi + P_hi V_lo,
// online softmax per warp in the exp2 domain (Q pre-scaled by log2(e) / sqrt(hd)); the four warps'
// (max, sum, O) merge through shared memory at the end.  Each cached byte is read once per (tile,
// head), against a 128-row tensor-core tile that would spend 7/8 of its MMAs on padding rows.
template <int HD>
struct RowsSmem {
  static constexpr int KB = 64;                 // keys per staged block
  static constexpr int LD = HD + 8;             // padded fp16 row (halves): ldmatrix rows in distinct banks
  static constexpr int RB = HD / 2;             // residual bytes of one row
  static constexpr int RBP = RB + 16;           // padded code row: the fragment reads hit distinct banks
  static constexpr int PLANE = KB * LD * 2;     // bytes of one staged fp16 block
  static constexpr int CODES = KB * RBP;        // bytes of one staged code block
  static constexpr int STAGE = 2 * PLANE + 2 * CODES;  // K | V | K codes | V codes
  static constexpr int QPLANE = 16 * LD * 2;            // the tile's 16 query rows, fp16 (hi or lo)
  static constexpr int SMEM = STAGE + 2 * QPLANE;       // one stage: four CTAs share an SM
  static_assert(STAGE % 16 == 0 && 4 * 16 * HD * 4 + 4 * 16 * 2 * 4 <= STAGE, "staging / merge layout");
};

template <int HD>
__global__ void __launch_bounds__(128, 4) attn_rows_kernel(const float* q, bf16* out_hi, bf16* out_lo,
                                                           const AttnTile* tiles, KVLayout kv, int layer, int H,
                                                           float scale_log2, bool fp16, bool write_lo) {
  using Sm = RowsSmem<HD>;
  constexpr int KB = Sm::KB, LD = Sm::LD, RB = Sm::RB, RBP = Sm::RBP, PLANE = Sm::PLANE;
  constexpr int CPR = HD / 8;   // 16-byte chunks of an fp16 row
  constexpr int NT_D = HD / 8;  // n-tiles over the head dim
  constexpr int RWP = RBP / 4;  // 32-bit words of a padded code row
  extern __shared__ __align__(16) uint8_t sm_rows[];
  uint8_t* qs = sm_rows + Sm::STAGE;  // Q_hi [16][LD], then Q_lo [16][LD]

  pdl_launch_dependents();
  pdl_wait();
  const AttnTile t = tiles[blockIdx.x];
  const int head = blockIdx.y;
  const int d = H * HD;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, tq = lane & 3;
  const int64_t e0 = static_cast<int64_t>(layer) * kv.layer_stride + static_cast<int64_t>(t.env) * kv.env_stride +
                     static_cast<int64_t>(head) * kv.head_stride;
  const f16* kbase = kv.base + e0;
  const f16* vbase = kbase + kv.kv_stride;
  const uint8_t* kres = kv.res + e0 / 2;
  const uint8_t* vres = kres + kv.kv_stride / 2;
  const int n_keys = t.pos0 + t.nrows;
  const int n_blocks = (n_keys + KB - 1) / KB;
  const int last_pos = n_keys - 1;

  auto load_block = [&](int blk) {
    const int j0 = blk * KB;
    const uint32_t s0 = smem_u32(sm_rows);
    for (int i = tid; i < KB * CPR; i += 128) {
      const int r = i / CPR, c = i - r * CPR;
      const bool ok = j0 + r < n_keys;
      const int64_t src = static_cast<int64_t>(ok ? j0 + r : 0) * HD + c * 8;
      cp_async16(s0 + (r * LD + c * 8) * 2, kbase + src, ok);
      cp_async16(s0 + PLANE + (r * LD + c * 8) * 2, vbase + src, ok);
    }
    for (int i = tid; i < KB * (RB / 16); i += 128) {
      const int r = i / (RB / 16), c = i - r * (RB / 16);
      const bool ok = j0 + r < n_keys;
      const int64_t src = static_cast<int64_t>(ok ? j0 + r : 0) * RB + c * 16;
      cp_async16(s0 + 2 * PLANE + r * RBP + c * 16, kres + src, ok);
      cp_async16(s0 + 2 * PLANE + Sm::CODES + r * RBP + c * 16, vres + src, ok);
    }
  };
  load_block(0);
  cp_async_commit();

  // the tile's 16 query rows (rows past the last repeat it) times log2(e) / sqrt(hd), as fp16
  // hi / lo planes: 8 threads per row, HD / 8 values each
  {
    constexpr int QPT = HD / 8;
    const int row = tid >> 3, c0 = (tid & 7) * QPT;
    const float* qr = q + static_cast<size_t>(t.row0 + min(row, t.nrows - 1)) * d + head * HD + c0;
    float4 x[QPT / 4];
#pragma unroll
    for (int i = 0; i < QPT / 4; ++i) x[i] = __ldcg(reinterpret_cast<const float4*>(qr) + i);
    uint32_t hi[QPT / 2], lo[QPT / 2];
#pragma unroll
    for (int i = 0; i < QPT / 4; ++i) {
      split_h2(x[i].x * scale_log2, x[i].y * scale_log2, hi[2 * i], lo[2 * i]);
      split_h2(x[i].z * scale_log2, x[i].w * scale_log2, hi[2 * i + 1], lo[2 * i + 1]);
    }
#pragma unroll
    for (int i = 0; i < QPT / 8; ++i) {
      reinterpret_cast<uint4*>(qs + (row * LD + c0) * 2)[i] = make_uint4(hi[4 * i], hi[4 * i + 1], hi[4 * i + 2], hi[4 * i + 3]);
      reinterpret_cast<uint4*>(qs + Sm::QPLANE + (row * LD + c0) * 2)[i] =
          make_uint4(lo[4 * i], lo[4 * i + 1], lo[4 * i + 2], lo[4 * i + 3]);
    }
  }
  // this thread's two rows (g and g + 8 of the tile) and their positions
  const int qpos0 = t.pos0 + min(g, t.nrows - 1), qpos1 = t.pos0 + min(g + 8, t.nrows - 1);
  const uint32_t qh_s = smem_u32(qs), ql_s = qh_s + Sm::QPLANE;
  // A-fragment address of this lane: row lane % 16, columns + 8 for lanes 16..31
  const uint32_t qa_off = ((lane & 15) * LD + (lane >> 4) * 8) * 2;

  float o[NT_D][4];
#pragma unroll
  for (int i = 0; i < NT_D; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
  float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
  const int im = lane >> 3;  // the ldmatrix sub-matrix this lane addresses

  for (int blk = 0; blk < n_blocks; ++blk) {
    cp_async_wait<0>();
    __syncthreads();
    const int k0 = blk * KB + warp * 16;  // this warp's first key
    if (k0 <= last_pos) {
      const uint32_t ks = smem_u32(sm_rows), vs = ks + PLANE;
      const uint32_t* kc = reinterpret_cast<const uint32_t*>(sm_rows + 2 * PLANE);
      const uint32_t* vc = reinterpret_cast<const uint32_t*>(sm_rows + 2 * PLANE + Sm::CODES);
      float s[2][4];
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
#pragma unroll
      for (int kk = 0; kk < HD / 16; kk += 2) {
        uint32_t qh0[4], ql0[4], qh1[4], ql1[4];
        ldsm_x4(qh_s + qa_off + kk * 32, qh0[0], qh0[1], qh0[2], qh0[3]);
        ldsm_x4(ql_s + qa_off + kk * 32, ql0[0], ql0[1], ql0[2], ql0[3]);
        ldsm_x4(qh_s + qa_off + kk * 32 + 32, qh1[0], qh1[1], qh1[2], qh1[3]);
        ldsm_x4(ql_s + qa_off + kk * 32 + 32, ql1[0], ql1[1], ql1[2], ql1[3]);
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
          // this thread's B elements are in key row warp*16 + nt*8 + g; the codes of dims
          // 16kk + 2tq (+1) sit in byte tq of the row's word 2kk (+1 for dims + 8)
          uint32_t b0, b1, b2, b3;
          const int key = warp * 16 + nt * 8 + (lane & 7);
          const int dim = (kk + (im >> 1)) * 16 + (im & 1) * 8;
          ldsm_x4(ks + (key * LD + dim) * 2, b0, b1, b2, b3);
          const uint4 cw = *reinterpret_cast<const uint4*>(kc + (warp * 16 + nt * 8 + g) * RWP + 2 * kk);
          const int sh = 8 * tq;
          const uint32_t l0b = kv_res_lo2(b0, (cw.x >> sh) & 15u, (cw.x >> (sh + 4)) & 15u);
          const uint32_t l1b = kv_res_lo2(b1, (cw.y >> sh) & 15u, (cw.y >> (sh + 4)) & 15u);
          const uint32_t l2b = kv_res_lo2(b2, (cw.z >> sh) & 15u, (cw.z >> (sh + 4)) & 15u);
          const uint32_t l3b = kv_res_lo2(b3, (cw.w >> sh) & 15u, (cw.w >> (sh + 4)) & 15u);
          mma16816(s[nt], qh0, b0, b1);
          mma16816(s[nt], ql0, b0, b1);
          mma16816(s[nt], qh0, l0b, l1b);
          mma16816(s[nt], qh1, b2, b3);
          mma16816(s[nt], ql1, b2, b3);
          mma16816(s[nt], qh1, l2b, l3b);
        }
      }
      // causal mask, online softmax (row g: c 0, 1; row g + 8: c 2, 3)
      float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int kpos = k0 + nt * 8 + 2 * tq + (c & 1);
          if (kpos > ((c < 2) ? qpos0 : qpos1)) s[nt][c] = -INFINITY;
        }
        mx0 = fmaxf(mx0, fmaxf(s[nt][0], s[nt][1]));
        mx1 = fmaxf(mx1, fmaxf(s[nt][2], s[nt][3]));
      }
      mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1));
      mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
      mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
      mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
      const float mn0 = fmaxf(m0, mx0), mn1 = fmaxf(m1, mx1);
      // a row with no visible key yet (in this warp's share) keeps max -inf: reference 0, weights 0
      const float u0 = mn0 == -INFINITY ? 0.f : mn0, u1 = mn1 == -INFINITY ? 0.f : mn1;
      const float a0 = exp2f(m0 - u0), a1 = exp2f(m1 - u1);
      m0 = mn0;
      m1 = mn1;
      float ps0 = 0.f, ps1 = 0.f;
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        s[nt][0] = exp2f(s[nt][0] - u0);
        s[nt][1] = exp2f(s[nt][1] - u0);
        s[nt][2] = exp2f(s[nt][2] - u1);
        s[nt][3] = exp2f(s[nt][3] - u1);
        ps0 += s[nt][0] + s[nt][1];
        ps1 += s[nt][2] + s[nt][3];
      }
      l0 = l0 * a0 + ps0;  // per-thread partial row sums, reduced across the quad at the end
      l1 = l1 * a1 + ps1;
#pragma unroll
      for (int nt = 0; nt < NT_D; ++nt) {
        o[nt][0] *= a0;
        o[nt][1] *= a0;
        o[nt][2] *= a1;
        o[nt][3] *= a1;
      }
      // O += P V: P from the S accumulators as the A operand (keys 0..7 of the warp's 16 in s[0],
      // 8..15 in s[1]), an fp16 hi / lo pair
      uint32_t ph[4], pl[4];
      split_h2(s[0][0], s[0][1], ph[0], pl[0]);
      split_h2(s[0][2], s[0][3], ph[1], pl[1]);
      split_h2(s[1][0], s[1][1], ph[2], pl[2]);
      split_h2(s[1][2], s[1][3], ph[3], pl[3]);
      // V^T fragments: this thread holds keys 2tq, 2tq + 1 (b0, b2) and 8 + 2tq, 9 + 2tq (b1, b3) of
      // the warp's 16 at dim 8n + g; that element's code is nibble g of the key row's word n
      const uint32_t* vrow = vc + (warp * 16 + 2 * tq) * RWP;
      const int key = warp * 16 + (im & 1) * 8 + (lane & 7);
      const int sh = 4 * g;
#pragma unroll
      for (int nt = 0; nt < NT_D; nt += 2) {
        uint32_t b0, b1, b2, b3;
        ldsm_x4_t(vs + (key * LD + (nt + (im >> 1)) * 8) * 2, b0, b1, b2, b3);
        const uint2 c00 = *reinterpret_cast<const uint2*>(vrow + nt);            // key 2tq
        const uint2 c01 = *reinterpret_cast<const uint2*>(vrow + RWP + nt);      // key 2tq + 1
        const uint2 c10 = *reinterpret_cast<const uint2*>(vrow + 8 * RWP + nt);  // key 8 + 2tq
        const uint2 c11 = *reinterpret_cast<const uint2*>(vrow + 9 * RWP + nt);  // key 9 + 2tq
        const uint32_t l0b = kv_res_lo2(b0, (c00.x >> sh) & 15u, (c01.x >> sh) & 15u);
        const uint32_t l1b = kv_res_lo2(b1, (c10.x >> sh) & 15u, (c11.x >> sh) & 15u);
        const uint32_t l2b = kv_res_lo2(b2, (c00.y >> sh) & 15u, (c01.y >> sh) & 15u);
        const uint32_t l3b = kv_res_lo2(b3, (c10.y >> sh) & 15u, (c11.y >> sh) & 15u);
        mma16816(o[nt], ph, b0, b1);
        mma16816(o[nt], pl, b0, b1);
        mma16816(o[nt], ph, l0b, l1b);
        mma16816(o[nt + 1], ph, b2, b3);
        mma16816(o[nt + 1], pl, b2, b3);
        mma16816(o[nt + 1], ph, l2b, l3b);
      }
    }
    __syncthreads();  // every warp is done with the stage: the next block's copies may land
    if (blk + 1 < n_blocks) {
      load_block(blk + 1);
      cp_async_commit();
    }
  }

  // merge the four warps' partials: O [warp][16][HD] and (max, sum) [warp][16] over the stages
  l0 += __shfl_xor_sync(0xffffffffu, l0, 1);
  l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
  l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
  l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
  float* mo = reinterpret_cast<float*>(sm_rows);
  float* mml = mo + 4 * 16 * HD;
  {
    float* oa = mo + (warp * 16 + g) * HD + 2 * tq;
    float* ob = oa + 8 * HD;
#pragma unroll
    for (int nt = 0; nt < NT_D; ++nt) {
      *reinterpret_cast<float2*>(oa + nt * 8) = make_float2(o[nt][0], o[nt][1]);
      *reinterpret_cast<float2*>(ob + nt * 8) = make_float2(o[nt][2], o[nt][3]);
    }
    if (tq == 0) {
      *reinterpret_cast<float2*>(mml + (warp * 16 + g) * 2) = make_float2(m0, l0);
      *reinterpret_cast<float2*>(mml + (warp * 16 + g + 8) * 2) = make_float2(m1, l1);
    }
  }
  __syncthreads();
  constexpr int CPT = HD / 8;  // output columns per thread: 8 threads per row
  const int row = tid >> 3, c0 = (tid & 7) * CPT;
  if (row >= t.nrows) return;
  float mw[4], lw[4], mx = -INFINITY;
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    const float2 ml = *reinterpret_cast<const float2*>(mml + (w * 16 + row) * 2);
    mw[w] = ml.x;
    lw[w] = ml.y;
    mx = fmaxf(mx, ml.x);  // finite: warp 0 holds key 0, visible to every row
  }
  float wt[4], lsum = 0.f;
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    wt[w] = exp2f(mw[w] - mx);  // 0 for a warp that saw no visible key of this row
    lsum += wt[w] * lw[w];
  }
  const float inv = 1.f / lsum;
  uint32_t sat = 0;  // convex combinations of cached values: the fp16 split never saturates
  uint32_t hi[CPT / 2], lo[CPT / 2];
#pragma unroll
  for (int c = 0; c < CPT; c += 2) {
    float v0 = 0.f, v1 = 0.f;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const float2 x = *reinterpret_cast<const float2*>(mo + (w * 16 + row) * HD + c0 + c);
      v0 += wt[w] * x.x;
      v1 += wt[w] * x.y;
    }
    split_pack2(v0 * inv, v1 * inv, hi[c / 2], lo[c / 2], fp16, sat);
  }
  const size_t off = static_cast<size_t>(t.row0 + row) * d + head * HD + c0;
#pragma unroll
  for (int i = 0; i < CPT / 8; ++i) {
    reinterpret_cast<uint4*>(out_hi + off)[i] = make_uint4(hi[4 * i], hi[4 * i + 1], hi[4 * i + 2], hi[4 * i + 3]);
    if (write_lo)
      reinterpret_cast<uint4*>(out_lo + off)[i] = make_uint4(lo[4 * i], lo[4 * i + 1], lo[4 * i + 2], lo[4 * i + 3]);
  }
}

// ---------------------------------------------------------------------------------- decode
// One query per (env, head, key range).  A warp takes 16 keys at a time on mma.sync, with the products
// arranged so that cached rows go from global memory into MMA operands without a shuffle or a
// conversion (which of a row's elements an MMA's k index stands for is free as long as both operands
// agree):
//   S   keys x 8 columns = K Q^T: lane (g, t) of the A operand reads 16-byte chunks 4 i + t of rows g
//       and g + 8;
//   O   dims x 8 columns = V^T P^T: lane (g, t) reads chunks 8 u + g of keys 2t, 2t + 1, 2t + 8, 2t + 9
//       and pairs two keys' elements with one byte permute.
// Columns 0 - 2 of the other operand carry three parts, as fp16, of the query or of the weights
// (together the fp32 value in full, both scaled by a power of two into the middle of fp16's range),
// columns 3 - 7 zeros; the cached value's low part (RES) multiplies the same columns.  Every MMA chain
// is at most four long and added up in fp32, since the tensor cores truncate their sums.  Each warp has
// its own ring of cp.async slots: bytes in flight cost shared memory, not registers.
// The warps of the CTA merge through shared memory into one partial (reference exponent, sum,
// unnormalised output) per range.  The last CTA of an (env, head) to finish (a ticket on
// counters[b * H + head], no waiting) merges the S partials in range order and writes the normalised
// output as the operand pair; with S == 1 the CTA writes it directly.
// Bound by the K/V bytes for many pairs and by the chain of one CTA's steps for few.  fp32 FMAs, one key
// per half warp and 16 keys' loads in registers, took about 1200 instructions per 16 keys and warp; this
// takes about 700.  Decode of 256 envs at 1100 positions (two 7B layers) 13500 -> 12320 us, 6.1 TB/s of
// weights and K/V; one layer's attention of 64 envs 83 -> 73 us, of 16 envs 34 -> 25.  (Rows loaded
// straight into registers, 12 warps per SM: 64 envs 2283 -> 2452 us a decode; two whole 10 KB stages per
// warp instead of three 5 KB slots: 2320 against 2294.)  Error of the output against 64 bits over 20 to
// 1100 keys: 1.8e-7 to 2.4e-7 (4.6e-7 for queries eight times as large), before 1.9e-7 to 2.8e-7 (5.8e-7).
constexpr int kDecodeWarps = 2;
constexpr int kSmemPerSm = 228 * 1024;
constexpr int kDecodeStatic = 2304;  // of a CTA's shared memory: the runtime's 1 KB and the static arrays

// Part `n` (0 .. 2) of x, 8 significant bits each: an fp32 value in full, NaN if x is not finite; 0 for
// n > 2.  Short parts leave the products with 11-bit values room in the tensor cores' sums, which cut
// terms off at the largest one's last bits.
__device__ __forceinline__ float part8(float x, int n) {
  const float p0 = bf2f(f2bf(x));
  const float r0 = x - p0;
  const float p1 = bf2f(f2bf(r0));
  return n == 0 ? p0 : n == 1 ? p1 : n == 2 ? r0 - p1 : 0.f;
}

// A warp's ring of three slots, each the keys or the values of 16 positions with their codes, in the order
// K 0, V 0, K 1, V 1 ..: a slot is refilled as soon as its product is done, so two others are in flight or
// landed.  16-byte chunks are stored xor-swizzled by row so that the operand reads hit distinct banks
// (value codes: two-way).
template <int HD, bool RES>
struct DecodeSlot {
  static constexpr int ROW = HD * 2, CODE = RES ? HD / 2 : 0;  // bytes of a row, of its codes
  static constexpr int BYTES = 16 * (ROW + CODE);
  static constexpr int RING = 3 * BYTES;
  __device__ static int k(int r, int c) { return r * ROW + ((c ^ ((r & 1) << 2)) << 4); }
  __device__ static int v(int r, int c) { return r * ROW + ((c ^ (((r >> 1) & 3) << 1)) << 4); }
  __device__ static int code(int r, int c) {
    return 16 * ROW + r * CODE + ((HD == 128 ? c ^ ((r >> 1) & 3) : c ^ ((r >> 2) & 1)) << 4);
  }
};

// One warp copies the keys (or values) of 16 positions from key0 on, with their codes, into the slot at
// shared address dst; positions from k_end on read the last one again (their weight is zero).  One commit
// group, empty when key0 is past the end.
template <int HD, bool RES, bool VALUE>
__device__ __forceinline__ void load_slot(uint32_t dst, const f16* base, const uint8_t* res, int key0, int k_end,
                                          int lane) {
  using St = DecodeSlot<HD, RES>;
  if (key0 < k_end) {
    constexpr int RC = HD / 8;  // chunks of a row
#pragma unroll
    for (int n = 0; n < 16 * RC / 32; ++n) {
      const int i = lane + 32 * n, r = i / RC, c = i % RC;
      cp_async16(dst + (VALUE ? St::v(r, c) : St::k(r, c)), base + static_cast<int64_t>(min(key0 + r, k_end - 1)) * HD + 8 * c,
                 true);
    }
    if (RES) {
      constexpr int CC = HD / 32;  // chunks of a row's codes
#pragma unroll
      for (int n = 0; n < 16 * CC / 32; ++n) {
        const int i = lane + 32 * n, r = i / CC, c = i % CC;
        cp_async16(dst + St::code(r, c), res + static_cast<int64_t>(min(key0 + r, k_end - 1)) * (HD / 2) + 16 * c, true);
      }
    }
  }
  cp_async_commit();
}

template <int HD, bool RES, int NW = kDecodeWarps>
__global__ void __launch_bounds__(NW * 32, decode_ctas_per_sm(HD)) attn_decode_kernel(const float* q, const RowInfo* rows,
                                                          KVLayout kv, int layer, int H,
                                                          int n_whole, int chunk, int S_rest, float scale_log2,
                                                          float* __restrict__ part_o,
                                                          float2* __restrict__ part_ml,
                                                          int* __restrict__ counters,
                                                          bf16* __restrict__ out_hi,
                                                          bf16* __restrict__ out_lo, bool fp16) {
  constexpr int KT = HD / 32;  // 16-byte chunks of a key row per lane
  constexpr int VT = HD / 64;  // 16-byte chunks of a value row per lane
  constexpr int NT = NW * 32;  // threads
  using St = DecodeSlot<HD, RES>;
  extern __shared__ __align__(128) uint8_t sm_dec[];
  __shared__ float s_m[NW], s_l[NW];
  __shared__ float s_o[NW][HD];

  pdl_launch_dependents();
  pdl_wait();
  // the first n_whole (env, head) pairs take one CTA each, the others S_rest ranges of `chunk` keys
  const bool whole = static_cast<int>(blockIdx.x) < n_whole;
  const int rest = static_cast<int>(blockIdx.x) - n_whole;
  const int S = whole ? 1 : S_rest;
  const int split = whole ? 0 : rest % S_rest;
  const int bh = whole ? blockIdx.x : n_whole + rest / S_rest;
  const int b = bh / H, head = bh - b * H;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  uint8_t* ring = sm_dec + warp * St::RING;
  // the queries and row table come from the kernels just before (programmatic dependent
  // launch): read them at L2, never through the non-coherent read-only path
  const int env = __ldcg(&rows[b].env), pos = __ldcg(&rows[b].pos);
  const int d = H * HD;
  const int k_begin = split * chunk;
  const int k_end = S == 1 ? pos + 1 : min(k_begin + chunk, pos + 1);

  const f16* kbase = kv.base + static_cast<int64_t>(layer) * kv.layer_stride +
                     static_cast<int64_t>(env) * kv.env_stride +
                     static_cast<int64_t>(head) * kv.head_stride;
  const f16* vbase = kbase + kv.kv_stride;
  // RES: the residual codes of the same elements (half a byte each), read with the fp16 parts
  const uint8_t* kres = RES ? kv.res + (kbase - kv.base) / 2 : nullptr;
  const uint8_t* vres = RES ? kres + kv.kv_stride / 2 : nullptr;

  auto load_k = [&](int key0, int slot) {
    load_slot<HD, RES, false>(smem_u32(ring + slot * St::BYTES), kbase, kres, key0, k_end, lane);
  };
  auto load_v = [&](int key0, int slot) {
    load_slot<HD, RES, true>(smem_u32(ring + slot * St::BYTES), vbase, vres, key0, k_end, lane);
  };
  const int key_first = k_begin + warp * 16;
  load_k(key_first, 0);
  load_v(key_first, 1);
  load_k(key_first + NW * 16, 2);

  // the query times log2(e) / sqrt(hd), its largest element scaled to [2^9, 2^10): part g of this
  // lane's dims as the B operand
  uint32_t qb[KT][4];
  float q_inv;  // undoes the scaling
  {
    float x[KT][8];
    float amax = 0.f;
#pragma unroll
    for (int i = 0; i < KT; ++i) {
      const float4* qp = reinterpret_cast<const float4*>(q + static_cast<size_t>(b) * d + head * HD + 32 * i + 8 * t);
      const float4 a = __ldcg(qp), c = __ldcg(qp + 1);
      const float v[8] = {a.x, a.y, a.z, a.w, c.x, c.y, c.z, c.w};
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        x[i][e] = v[e] * scale_log2;
        amax = fmaxf(amax, fabsf(x[i][e]));
      }
    }
    amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 1));
    amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 2));
    const int ex = static_cast<int>(__float_as_uint(amax) >> 23);  // biased exponent (255: not finite)
    const int se = min(max(263 - ex, 1), 253);
    const float q_scale = __uint_as_float(static_cast<uint32_t>(se) << 23);
    q_inv = __uint_as_float(static_cast<uint32_t>(254 - se) << 23);
#pragma unroll
    for (int i = 0; i < KT; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        qb[i][e] = pack_f16x2(part8(x[i][2 * e] * q_scale, g), part8(x[i][2 * e + 1] * q_scale, g));
  }
  // m: the running maximum less 10, so that the weights lie in (0, 2^10]; l: this lane's share of
  // their sum; o[u][w][h]: dim 64 u + 8 g + 2 w + h, this lane's columns added up
  float m = -INFINITY, l = 0.f, o[VT][4][2];
#pragma unroll
  for (int u = 0; u < VT; ++u)
#pragma unroll
    for (int w = 0; w < 4; ++w) o[u][w][0] = o[u][w][1] = 0.f;

  int slot = 0;  // of this step's keys; its values are in the next one
  for (int key0 = key_first; key0 < k_end; key0 += NW * 16) {
    cp_async_wait<2>();
    __syncwarp();
    const uint8_t* sb = ring + slot * St::BYTES;
    float s0 = 0.f, s1 = 0.f;  // this lane's columns of keys g and g + 8
#pragma unroll
    for (int i = 0; i < KT; ++i) {
      const uint4 ka = *reinterpret_cast<const uint4*>(sb + St::k(g, 4 * i + t));
      const uint4 kb = *reinterpret_cast<const uint4*>(sb + St::k(g + 8, 4 * i + t));
      float c[4] = {0.f, 0.f, 0.f, 0.f};
      if (RES) {
        const uint4 la = kv_res_lo8(ka, *reinterpret_cast<const uint32_t*>(sb + St::code(g, i) + 4 * t));
        const uint4 lb = kv_res_lo8(kb, *reinterpret_cast<const uint32_t*>(sb + St::code(g + 8, i) + 4 * t));
        mma16816(c, {la.x, lb.x, la.y, lb.y}, qb[i][0], qb[i][1]);
        mma16816(c, {la.z, lb.z, la.w, lb.w}, qb[i][2], qb[i][3]);
      }
      mma16816(c, {ka.x, kb.x, ka.y, kb.y}, qb[i][0], qb[i][1]);
      mma16816(c, {ka.z, kb.z, ka.w, kb.w}, qb[i][2], qb[i][3]);
      s0 += c[0] + c[1];
      s1 += c[2] + c[3];
    }
    __syncwarp();  // every lane has read the slot
    load_v(key0 + NW * 16, slot);
    slot = slot == 2 ? 0 : slot + 1;
    // columns 0, 1 are with t = 0 and column 2 with t = 1; then each lane takes keys 2t, 2t + 1,
    // 2t + 8, 2t + 9
    s0 += __shfl_xor_sync(0xffffffffu, s0, 1);
    s1 += __shfl_xor_sync(0xffffffffu, s1, 1);
    float p[4];
    p[0] = __shfl_sync(0xffffffffu, s0, 8 * t);
    p[1] = __shfl_sync(0xffffffffu, s0, 8 * t + 4);
    p[2] = __shfl_sync(0xffffffffu, s1, 8 * t);
    p[3] = __shfl_sync(0xffffffffu, s1, 8 * t + 4);
    float mx = -INFINITY;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      p[j] = key0 + 2 * t + (j & 1) + 8 * (j >> 1) < k_end ? p[j] * q_inv : -INFINITY;
      mx = fmaxf(mx, p[j]);
    }
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    const float m_new = fmaxf(m, mx - 10.f);
    const float alpha = exp2f(m - m_new);
    m = m_new;
#pragma unroll
    for (int j = 0; j < 4; ++j) p[j] = exp2f(p[j] - m_new);
    l = l * alpha + ((p[0] + p[1]) + (p[2] + p[3]));
    cp_async_wait<2>();
    __syncwarp();
    sb = ring + slot * St::BYTES;
    const uint32_t b0 = pack_f16x2(part8(p[0], g), part8(p[1], g));
    const uint32_t b1 = pack_f16x2(part8(p[2], g), part8(p[3], g));
#pragma unroll
    for (int u = 0; u < VT; ++u) {
      uint32_t hw[4][4], lw[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int r = 2 * t + (j & 1) + 8 * (j >> 1);
        const uint4 hv = *reinterpret_cast<const uint4*>(sb + St::v(r, 8 * u + g));
        hw[j][0] = hv.x;
        hw[j][1] = hv.y;
        hw[j][2] = hv.z;
        hw[j][3] = hv.w;
        if (RES) {
          const uint4 lv = kv_res_lo8(hv, *reinterpret_cast<const uint32_t*>(sb + St::code(r, 2 * u + (g >> 2)) + 4 * (g & 3)));
          lw[j][0] = lv.x;
          lw[j][1] = lv.y;
          lw[j][2] = lv.z;
          lw[j][3] = lv.w;
        }
      }
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        // rows g and g + 8 of the product: dims 2w and 2w + 1 of the chunk
        float c[4] = {0.f, 0.f, 0.f, 0.f};
        if (RES)
          mma16816(c, {__byte_perm(lw[0][w], lw[1][w], 0x5410), __byte_perm(lw[0][w], lw[1][w], 0x7632),
                       __byte_perm(lw[2][w], lw[3][w], 0x5410), __byte_perm(lw[2][w], lw[3][w], 0x7632)}, b0, b1);
        mma16816(c, {__byte_perm(hw[0][w], hw[1][w], 0x5410), __byte_perm(hw[0][w], hw[1][w], 0x7632),
                     __byte_perm(hw[2][w], hw[3][w], 0x5410), __byte_perm(hw[2][w], hw[3][w], 0x7632)}, b0, b1);
        o[u][w][0] = fmaf(o[u][w][0], alpha, c[0] + c[1]);
        o[u][w][1] = fmaf(o[u][w][1], alpha, c[2] + c[3]);
      }
    }
    __syncwarp();
    load_k(key0 + 2 * NW * 16, slot);
    slot = slot == 2 ? 0 : slot + 1;
  }
  // the warps' states -> shared memory: sums over the lanes of a row
  l += __shfl_xor_sync(0xffffffffu, l, 1);
  l += __shfl_xor_sync(0xffffffffu, l, 2);
  if (lane == 0) {
    s_m[warp] = m;
    s_l[warp] = l;
  }
#pragma unroll
  for (int u = 0; u < VT; ++u)
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const float a = o[u][w][0] + __shfl_xor_sync(0xffffffffu, o[u][w][0], 1);
      const float c = o[u][w][1] + __shfl_xor_sync(0xffffffffu, o[u][w][1], 1);
      if (t == 0) *reinterpret_cast<float2*>(&s_o[warp][64 * u + 8 * g + 2 * w]) = make_float2(a, c);
    }
  __syncthreads();
  // merge the warps' states in order
  float M = -INFINITY;
#pragma unroll
  for (int w = 0; w < NW; ++w) M = fmaxf(M, s_m[w]);
  float L = 0.f, wt[NW];
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    wt[w] = s_m[w] != -INFINITY ? exp2f(s_m[w] - M) : 0.f;  // -inf: a warp without keys
    L += s_l[w] * wt[w];
  }
  const size_t out_off = static_cast<size_t>(b) * d + head * HD;
  const size_t part0 = static_cast<size_t>(bh - n_whole) * S;  // S > 1: this pair's partials
  uint32_t sat = 0;  // convex combinations of fp16 values: the fp16 split never saturates
  for (int c = threadIdx.x; c < HD; c += NT) {
    float acc = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) acc += s_o[w][c] * wt[w];
    if (S == 1)
      store_split1(out_hi, out_lo, out_off + c, acc / L, fp16, sat);
    else
      part_o[(part0 + split) * HD + c] = acc;
  }
  if (S == 1) return;
  if (threadIdx.x == 0) part_ml[part0 + split] = make_float2(M, L);

  // ticket: the partial is published (fence) before the counter moves
  __shared__ int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = (atomicAdd(counters + bh, 1) == S - 1);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  float Mx = -INFINITY;
#pragma unroll 8
  for (int s = 0; s < S; ++s) Mx = fmaxf(Mx, __ldcg(&part_ml[part0 + s].x));
  float Lt = 0.f;
  float acc[(HD + NT - 1) / NT];
#pragma unroll
  for (int i = 0; i < (HD + NT - 1) / NT; ++i) acc[i] = 0.f;
#pragma unroll 8
  for (int s = 0; s < S; ++s) {
    const float2 ml = __ldcg(&part_ml[part0 + s]);
    const float w = ml.x != -INFINITY ? exp2f(ml.x - Mx) : 0.f;  // -inf: a range without keys, its partials 0
    Lt += ml.y * w;
#pragma unroll
    for (int i = 0; i < (HD + NT - 1) / NT; ++i) {
      const int c = threadIdx.x + i * NT;
      if (c < HD) acc[i] += __ldcg(&part_o[(part0 + s) * HD + c]) * w;
    }
  }
#pragma unroll
  for (int i = 0; i < (HD + NT - 1) / NT; ++i) {
    const int c = threadIdx.x + i * NT;
    if (c < HD) {
      store_split1(out_hi, out_lo, out_off + c, acc[i] / Lt, fp16, sat);
    }
  }
  if (threadIdx.x == 0) counters[bh] = 0;  // ready for the next launch
}

// One query per (env, head) over a short context, when there are many pairs: a CTA lives for one or two steps
// of 16 keys per warp, so its time is latency and what counts is how many are resident.  fp32 FMAs on 72
// registers let 14 CTAs share an SM (the kernel above: 6 or 8; decode_short has both sides).  LPK lanes read one key row, 16 bytes
// (and 4 bytes of codes) each; a lane group has 4 keys and values in flight; its dot products meet by
// shuffles; the groups' online softmax states merge through shared memory in a fixed order.
template <int HD, bool RES, int NW = kDecodeWarps>
__global__ void __launch_bounds__(NW * 32, RES ? 14 : 1) attn_decode_short_kernel(
    const float* q, const RowInfo* rows, KVLayout kv, int layer, int H, float scale_log2, bf16* __restrict__ out_hi,
    bf16* __restrict__ out_lo, bool fp16) {
  constexpr int LPK = HD / 8;    // lanes per key row
  constexpr int KPI = 32 / LPK;  // key rows per warp instruction
  constexpr int U = 4;           // key rows per lane group loaded ahead
  __shared__ float s_m[NW][KPI], s_l[NW][KPI];
  __shared__ float s_o[NW][KPI][HD];

  pdl_launch_dependents();
  pdl_wait();
  const int b = blockIdx.x / H, head = blockIdx.x - b * H;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sub = lane / LPK, part = lane - sub * LPK;
  const int env = __ldcg(&rows[b].env), k_end = __ldcg(&rows[b].pos) + 1;
  const size_t off = static_cast<size_t>(b) * H * HD + head * HD;

  float qv[8];
  {
    const float4* qp = reinterpret_cast<const float4*>(q + off + part * 8);
    const float4 a = __ldcg(qp), c = __ldcg(qp + 1);
    const float v[8] = {a.x, a.y, a.z, a.w, c.x, c.y, c.z, c.w};
#pragma unroll
    for (int e = 0; e < 8; ++e) qv[e] = v[e] * scale_log2;
  }
  const f16* kbase = kv.base + static_cast<int64_t>(layer) * kv.layer_stride + static_cast<int64_t>(env) * kv.env_stride +
                     static_cast<int64_t>(head) * kv.head_stride;
  const f16* vbase = kbase + kv.kv_stride;
  const uint8_t* kres = RES ? kv.res + (kbase - kv.base) / 2 : nullptr;
  const uint8_t* vres = RES ? kres + kv.kv_stride / 2 : nullptr;

  float m = -INFINITY, l = 0.f, o[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) o[e] = 0.f;
  for (int key0 = warp * KPI * U; key0 < k_end; key0 += NW * KPI * U) {
    uint4 kk[U], vv[U];
    uint32_t kc[U], vc[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int key = key0 + u * KPI + sub;
      kk[u] = vv[u] = make_uint4(0u, 0u, 0u, 0u);
      kc[u] = vc[u] = 0u;
      if (key < k_end) {
        kk[u] = *reinterpret_cast<const uint4*>(kbase + static_cast<int64_t>(key) * HD + part * 8);
        vv[u] = *reinterpret_cast<const uint4*>(vbase + static_cast<int64_t>(key) * HD + part * 8);
        if (RES) {
          kc[u] = *reinterpret_cast<const uint32_t*>(kres + static_cast<int64_t>(key) * (HD / 2) + part * 4);
          vc[u] = *reinterpret_cast<const uint32_t*>(vres + static_cast<int64_t>(key) * (HD / 2) + part * 4);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t w[4] = {kk[u].x, kk[u].y, kk[u].z, kk[u].w};
      float acc = 0.f;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 f = unpack_f16x2(w[e]);
        acc = fmaf(qv[2 * e], f.x, acc);
        acc = fmaf(qv[2 * e + 1], f.y, acc);
      }
      if (RES) {
        const uint4 kl = kv_res_lo8(kk[u], kc[u]);
        const uint32_t wl[4] = {kl.x, kl.y, kl.z, kl.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 f = unpack_f16x2(wl[e]);
          acc = fmaf(qv[2 * e], f.x, acc);
          acc = fmaf(qv[2 * e + 1], f.y, acc);
        }
      }
#pragma unroll
      for (int x = LPK / 2; x > 0; x >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, x);
      if (key0 + u * KPI + sub < k_end) {  // the same for all lanes of a key row
        const float m_new = fmaxf(m, acc);
        const float alpha = exp2f(m - m_new), p = exp2f(acc - m_new);
        m = m_new;
        l = l * alpha + p;
        const uint32_t v4[4] = {vv[u].x, vv[u].y, vv[u].z, vv[u].w};
        uint32_t vl4[4] = {0u, 0u, 0u, 0u};
        if (RES) {
          const uint4 vl = kv_res_lo8(vv[u], vc[u]);
          vl4[0] = vl.x;
          vl4[1] = vl.y;
          vl4[2] = vl.z;
          vl4[3] = vl.w;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 f = unpack_f16x2(v4[e]), fl = unpack_f16x2(vl4[e]);
          o[2 * e] = fmaf(p, f.x + fl.x, o[2 * e] * alpha);
          o[2 * e + 1] = fmaf(p, f.y + fl.y, o[2 * e + 1] * alpha);
        }
      }
    }
  }
  if (part == 0) {
    s_m[warp][sub] = m;
    s_l[warp][sub] = l;
  }
#pragma unroll
  for (int e = 0; e < 8; ++e) s_o[warp][sub][part * 8 + e] = o[e];
  __syncthreads();
  // merge the groups' states in order (-inf: a group without keys)
  float M = -INFINITY;
  for (int w = 0; w < NW; ++w)
    for (int k = 0; k < KPI; ++k) M = fmaxf(M, s_m[w][k]);
  float L = 0.f;
  for (int w = 0; w < NW; ++w)
    for (int k = 0; k < KPI; ++k)
      if (s_m[w][k] != -INFINITY) L += s_l[w][k] * exp2f(s_m[w][k] - M);
  uint32_t sat = 0;  // convex combinations of cached values: the fp16 split never saturates
  for (int c = threadIdx.x; c < HD; c += NW * 32) {
    float acc = 0.f;
    for (int w = 0; w < NW; ++w)
      for (int k = 0; k < KPI; ++k)
        if (s_m[w][k] != -INFINITY) acc += s_o[w][k][c] * exp2f(s_m[w][k] - M);
    store_split1(out_hi, out_lo, off + c, acc / L, fp16, sat);
  }
}

// ------------------------------------------------------------------ up to 8 rows (residual cache)
// Query tiles of at most 8 rows (the teacher-forced action rows of the score pass) with the decode kernel's
// layout and ring: the 8 columns of the small operand are the rows, and an fp32 value is an fp16 pair,
//   S = K_hi Q_hi + K_hi Q_lo + K_lo Q_hi,   O = V_hi P_hi + V_hi P_lo + V_lo P_hi.
// A lane's S values are keys g, g + 8 of rows 2t, 2t + 1; one 8 x 8 transpose (movmatrix) turns the weights
// into the operand of the second product.  One CTA of two warps per (tile, head).
// 64 envs x 32 heads, 6 rows, 296 positions: 71 us against 101 for attn_rows_kernel (one 45 KB stage
// per CTA: its copies wait for its products).
__device__ __forceinline__ uint32_t transpose8(uint32_t x) {
  uint32_t y;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}

constexpr int kRows8 = 8;
template <int HD, int NW = kDecodeWarps>
__global__ void __launch_bounds__(NW * 32, decode_ctas_per_sm(HD) - 1) attn_rows8_kernel(const float* q, bf16* out_hi, bf16* out_lo,
                                                             const AttnTile* tiles, KVLayout kv, int layer, int H,
                                                             float scale_log2, bool fp16, bool write_lo) {
  constexpr int KT = HD / 32, VT = HD / 64;
  using St = DecodeSlot<HD, true>;
  extern __shared__ __align__(128) uint8_t sm_dec[];
  __shared__ uint4 s_q[2][KT][32];  // the queries as B operands, fp16 hi and lo, per lane
  __shared__ float s_m[NW][8], s_l[NW][8];
  static_assert(NW * 8 * HD * 4 <= NW * St::RING, "the warps' outputs reuse the ring");

  pdl_launch_dependents();
  const int head = blockIdx.y;
  const int d = H * HD;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, t = lane & 3;
  uint8_t* ring = sm_dec + warp * St::RING;
  const AttnTile tile = tiles[blockIdx.x];  // copied in before the first kernel of this call started
  pdl_wait();
  const int k_end = tile.pos0 + tile.nrows;
  const int64_t e0 = static_cast<int64_t>(layer) * kv.layer_stride + static_cast<int64_t>(tile.env) * kv.env_stride +
                     static_cast<int64_t>(head) * kv.head_stride;
  const f16* kbase = kv.base + e0;
  const f16* vbase = kbase + kv.kv_stride;
  const uint8_t* kres = kv.res + e0 / 2;
  const uint8_t* vres = kres + kv.kv_stride / 2;
  auto load_k = [&](int key0, int slot) {
    load_slot<HD, true, false>(smem_u32(ring + slot * St::BYTES), kbase, kres, key0, k_end, lane);
  };
  auto load_v = [&](int key0, int slot) {
    load_slot<HD, true, true>(smem_u32(ring + slot * St::BYTES), vbase, vres, key0, k_end, lane);
  };
  const int key_first = warp * 16;
  load_k(key_first, 0);
  load_v(key_first, 1);
  load_k(key_first + NW * 16, 2);

  // row g of the tile (past the last: the last again, not written) times log2(e) / sqrt(hd)
  for (int i = warp; i < KT; i += NW) {
    const float4* qp = reinterpret_cast<const float4*>(q + static_cast<size_t>(tile.row0 + min(g, tile.nrows - 1)) * d +
                                                       head * HD + 32 * i + 8 * t);
    const float4 a = __ldcg(qp), c = __ldcg(qp + 1);
    uint4 hi, lo;
    split_h2(a.x * scale_log2, a.y * scale_log2, hi.x, lo.x);
    split_h2(a.z * scale_log2, a.w * scale_log2, hi.y, lo.y);
    split_h2(c.x * scale_log2, c.y * scale_log2, hi.z, lo.z);
    split_h2(c.z * scale_log2, c.w * scale_log2, hi.w, lo.w);
    s_q[0][i][lane] = hi;
    s_q[1][i][lane] = lo;
  }
  __syncthreads();

  // of rows 2t and 2t + 1: last visible position, running maximum less 10, this lane's share of the sum;
  // o[u][w]: dims 64 u + 8 g + 2 w (first two) and + 1, rows 2t, 2t + 1
  int last[2];
  float m[2], l[2], o[VT][4][4];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    last[j] = tile.pos0 + min(2 * t + j, tile.nrows - 1);
    m[j] = -INFINITY;
    l[j] = 0.f;
  }
#pragma unroll
  for (int u = 0; u < VT; ++u)
#pragma unroll
    for (int w = 0; w < 4; ++w) o[u][w][0] = o[u][w][1] = o[u][w][2] = o[u][w][3] = 0.f;

  int slot = 0;  // of this step's keys; its values are in the next one
  for (int key0 = key_first; key0 < k_end; key0 += NW * 16) {
    cp_async_wait<2>();
    __syncwarp();
    const uint8_t* sb = ring + slot * St::BYTES;
    float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < KT; ++i) {
      const uint4 ka = *reinterpret_cast<const uint4*>(sb + St::k(g, 4 * i + t));
      const uint4 kb = *reinterpret_cast<const uint4*>(sb + St::k(g + 8, 4 * i + t));
      const uint4 la = kv_res_lo8(ka, *reinterpret_cast<const uint32_t*>(sb + St::code(g, i) + 4 * t));
      const uint4 lb = kv_res_lo8(kb, *reinterpret_cast<const uint32_t*>(sb + St::code(g + 8, i) + 4 * t));
      const uint4 qh = s_q[0][i][lane], ql = s_q[1][i][lane];
      float c[4] = {0.f, 0.f, 0.f, 0.f};
      mma16816(c, {la.x, lb.x, la.y, lb.y}, qh.x, qh.y);
      mma16816(c, {la.z, lb.z, la.w, lb.w}, qh.z, qh.w);
      mma16816(c, {ka.x, kb.x, ka.y, kb.y}, ql.x, ql.y);
      mma16816(c, {ka.z, kb.z, ka.w, kb.w}, ql.z, ql.w);
      mma16816(c, {ka.x, kb.x, ka.y, kb.y}, qh.x, qh.y);
      mma16816(c, {ka.z, kb.z, ka.w, kb.w}, qh.z, qh.w);
#pragma unroll
      for (int e = 0; e < 4; ++e) s[e] += c[e];
    }
    __syncwarp();  // every lane has read the slot
    load_v(key0 + NW * 16, slot);
    slot = slot == 2 ? 0 : slot + 1;
    float alpha[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      if (key0 + g > last[j]) s[j] = -INFINITY;
      if (key0 + g + 8 > last[j]) s[2 + j] = -INFINITY;
      float mx = fmaxf(s[j], s[2 + j]);
#pragma unroll
      for (int x = 4; x <= 16; x <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, x));
      const float m_new = fmaxf(m[j], mx - 10.f);
      const float ref = m_new != -INFINITY ? m_new : 0.f;  // no key of this row yet
      alpha[j] = exp2f(m[j] - ref);
      m[j] = m_new;
      s[j] = exp2f(s[j] - ref);
      s[2 + j] = exp2f(s[2 + j] - ref);
      l[j] = l[j] * alpha[j] + (s[j] + s[2 + j]);
    }
    uint32_t ph[2], pl[2];
    split_h2(s[0], s[1], ph[0], pl[0]);
    split_h2(s[2], s[3], ph[1], pl[1]);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      ph[j] = transpose8(ph[j]);
      pl[j] = transpose8(pl[j]);
    }
    cp_async_wait<2>();
    __syncwarp();
    sb = ring + slot * St::BYTES;
#pragma unroll
    for (int u = 0; u < VT; ++u) {
      uint32_t hw[4][4], lw[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int r = 2 * t + (j & 1) + 8 * (j >> 1);
        const uint4 hv = *reinterpret_cast<const uint4*>(sb + St::v(r, 8 * u + g));
        const uint4 lv = kv_res_lo8(hv, *reinterpret_cast<const uint32_t*>(sb + St::code(r, 2 * u + (g >> 2)) + 4 * (g & 3)));
        hw[j][0] = hv.x;
        hw[j][1] = hv.y;
        hw[j][2] = hv.z;
        hw[j][3] = hv.w;
        lw[j][0] = lv.x;
        lw[j][1] = lv.y;
        lw[j][2] = lv.z;
        lw[j][3] = lv.w;
      }
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        float c[4] = {0.f, 0.f, 0.f, 0.f};
        const uint32_t vh[4] = {__byte_perm(hw[0][w], hw[1][w], 0x5410), __byte_perm(hw[0][w], hw[1][w], 0x7632),
                                __byte_perm(hw[2][w], hw[3][w], 0x5410), __byte_perm(hw[2][w], hw[3][w], 0x7632)};
        mma16816(c, {__byte_perm(lw[0][w], lw[1][w], 0x5410), __byte_perm(lw[0][w], lw[1][w], 0x7632),
                     __byte_perm(lw[2][w], lw[3][w], 0x5410), __byte_perm(lw[2][w], lw[3][w], 0x7632)}, ph[0], ph[1]);
        mma16816(c, vh, pl[0], pl[1]);
        mma16816(c, vh, ph[0], ph[1]);
#pragma unroll
        for (int e = 0; e < 4; ++e) o[u][w][e] = fmaf(o[u][w][e], alpha[e & 1], c[e]);
      }
    }
    __syncwarp();
    load_k(key0 + 2 * NW * 16, slot);
    slot = slot == 2 ? 0 : slot + 1;
  }
  // the warps' states -> shared memory, the outputs over the rings
  cp_async_wait<0>();
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int x = 4; x <= 16; x <<= 1) l[j] += __shfl_xor_sync(0xffffffffu, l[j], x);
  if (g == 0) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      s_m[warp][2 * t + j] = m[j];
      s_l[warp][2 * t + j] = l[j];
    }
  }
  __syncthreads();
  float* mo = reinterpret_cast<float*>(sm_dec);  // [warp][row][HD]
#pragma unroll
  for (int u = 0; u < VT; ++u)
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      float* dst = mo + (warp * 8 + 2 * t) * HD + 64 * u + 8 * g + 2 * w;
      *reinterpret_cast<float2*>(dst) = make_float2(o[u][w][0], o[u][w][2]);
      *reinterpret_cast<float2*>(dst + HD) = make_float2(o[u][w][1], o[u][w][3]);
    }
  __syncthreads();
  constexpr int CPT = 8;  // output columns of a thread at a time
  uint32_t sat = 0;       // convex combinations of cached values: the fp16 split never saturates
  for (int k = tid; k < tile.nrows * (HD / CPT); k += NW * 32) {
    const int row = k / (HD / CPT), c0 = k % (HD / CPT) * CPT;
    float mx = -INFINITY, wt[NW], lsum = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) mx = fmaxf(mx, s_m[w][row]);  // finite: warp 0 holds key 0
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      wt[w] = exp2f(s_m[w][row] - mx);  // 0 for a warp that saw no visible key of this row
      lsum += wt[w] * s_l[w][row];
    }
    const float inv = 1.f / lsum;
    uint32_t hi[CPT / 2], lo[CPT / 2];
#pragma unroll
    for (int c = 0; c < CPT; c += 2) {
      float v0 = 0.f, v1 = 0.f;
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        const float2 x = *reinterpret_cast<const float2*>(mo + (w * 8 + row) * HD + c0 + c);
        v0 += wt[w] * x.x;
        v1 += wt[w] * x.y;
      }
      split_pack2(v0 * inv, v1 * inv, hi[c / 2], lo[c / 2], fp16, sat);
    }
    const size_t off = static_cast<size_t>(tile.row0 + row) * d + head * HD + c0;
    *reinterpret_cast<uint4*>(out_hi + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    if (write_lo) *reinterpret_cast<uint4*>(out_lo + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  }
}

}  // namespace

int attn_chunk_launch(const float* q, bf16* out_hi, bf16* out_lo, const AttnTile* tiles,
                      int n_tiles, KVLayout kv, int layer, int H, int hd, cudaStream_t stream, bool fp16) {
  if (n_tiles <= 0) return VLA_OK;
  const float scale_log2 = 1.4426950408889634f / sqrtf(static_cast<float>(hd));
  dim3 grid(n_tiles, H);
  if (hd == 128) {
    const int smem = (4 * 64) * (128 + 8) * 2;
    static std::atomic<uint64_t> attr_done{0};
    VLA_CUDA_TRY(set_smem_limit(attn_chunk_mma_kernel<128>, smem, attr_done));
    VLA_CUDA_TRY(launch_pdl(attn_chunk_mma_kernel<128>, grid, dim3(128), smem, stream, q, out_hi, out_lo,
                            tiles, kv, layer, H, scale_log2, fp16));
  } else if (hd == 64) {
    const int smem = (4 * 64) * (64 + 8) * 2;
    static std::atomic<uint64_t> attr_done{0};
    VLA_CUDA_TRY(set_smem_limit(attn_chunk_mma_kernel<64>, smem, attr_done));
    VLA_CUDA_TRY(launch_pdl(attn_chunk_mma_kernel<64>, grid, dim3(128), smem, stream, q, out_hi, out_lo,
                            tiles, kv, layer, H, scale_log2, fp16));
  } else {
    return VLA_ERR_UNSUPPORTED;
  }
  note_launch();
  VLA_CUDA_TRY(cudaGetLastError());
  return VLA_OK;
}

int attn_rows_launch(const float* q, bf16* out_hi, bf16* out_lo, const AttnTile* tiles, int n_tiles, int max_rows,
                     KVLayout kv, int layer, int H, int hd, cudaStream_t stream, bool fp16, bool write_lo) {
  if (n_tiles <= 0) return VLA_OK;
  if (max_rows > kAttnRowsMax || !kv.res || (hd != 64 && hd != 128)) return VLA_ERR_UNSUPPORTED;
  if ((reinterpret_cast<uintptr_t>(kv.base) & 15) || (reinterpret_cast<uintptr_t>(kv.res) & 15)) return VLA_ERR_ARG;
  const float scale_log2 = 1.4426950408889634f / sqrtf(static_cast<float>(hd));
  const dim3 grid(n_tiles, H);
  if (max_rows <= kRows8) {
    auto go = [&](auto kern, int smem, std::atomic<uint64_t>& attr_done) {
      if (const cudaError_t e = set_smem_limit(kern, smem, attr_done)) return e;
      return launch_pdl(kern, grid, dim3(kDecodeWarps * 32), smem, stream, q, out_hi, out_lo, tiles, kv, layer, H,
                        scale_log2, fp16, write_lo);
    };
    static std::atomic<uint64_t> done128{0}, done64{0};
    if (hd == 128)
      VLA_CUDA_TRY(go(attn_rows8_kernel<128>, kDecodeWarps * DecodeSlot<128, true>::RING, done128));
    else
      VLA_CUDA_TRY(go(attn_rows8_kernel<64>, kDecodeWarps * DecodeSlot<64, true>::RING, done64));
    note_launch();
    VLA_CUDA_TRY(cudaGetLastError());
    return VLA_OK;
  }
  if (hd == 128) {
    static std::atomic<uint64_t> attr_done{0};
    VLA_CUDA_TRY(set_smem_limit(attn_rows_kernel<128>, RowsSmem<128>::SMEM, attr_done));
    VLA_CUDA_TRY(launch_pdl(attn_rows_kernel<128>, grid, dim3(128), RowsSmem<128>::SMEM, stream, q, out_hi, out_lo,
                            tiles, kv, layer, H, scale_log2, fp16, write_lo));
  } else {
    static std::atomic<uint64_t> attr_done{0};
    VLA_CUDA_TRY(set_smem_limit(attn_rows_kernel<64>, RowsSmem<64>::SMEM, attr_done));
    VLA_CUDA_TRY(launch_pdl(attn_rows_kernel<64>, grid, dim3(128), RowsSmem<64>::SMEM, stream, q, out_hi, out_lo,
                            tiles, kv, layer, H, scale_log2, fp16, write_lo));
  }
  note_launch();
  VLA_CUDA_TRY(cudaGetLastError());
  return VLA_OK;
}

int attn_decode_short_launch(const float* q, bf16* out_hi, bf16* out_lo, const RowInfo* rows, int B, KVLayout kv,
                             int layer, int H, int hd, cudaStream_t stream, bool fp16) {
  if (B <= 0) return VLA_OK;
  const float scale_log2 = 1.4426950408889634f / sqrtf(static_cast<float>(hd));
  auto go = [&](auto kern) {
    return launch_pdl(kern, dim3(static_cast<unsigned>(B) * H), dim3(kDecodeWarps * 32), 0, stream, q, rows, kv, layer, H,
                      scale_log2, out_hi, out_lo, fp16);
  };
  const bool res = kv.res != nullptr;
  if (hd == 128) {
    VLA_CUDA_TRY(res ? go(attn_decode_short_kernel<128, true>) : go(attn_decode_short_kernel<128, false>));
  } else if (hd == 64) {
    VLA_CUDA_TRY(res ? go(attn_decode_short_kernel<64, true>) : go(attn_decode_short_kernel<64, false>));
  } else {
    return VLA_ERR_UNSUPPORTED;
  }
  note_launch();
  VLA_CUDA_TRY(cudaGetLastError());
  return VLA_OK;
}

int attn_decode_launch(const float* q, bf16* out_hi, bf16* out_lo, const RowInfo* rows, int B,
                       int max_ctx, KVLayout kv, int layer, int H, int hd, int n_whole, int S,
                       float* part_o, float2* part_ml, int* counters, cudaStream_t stream, bool fp16, int num_sms) {
  if (B <= 0) return VLA_OK;
  if (n_whole < 0 || n_whole > B * H || S < 1) return VLA_ERR_ARG;
  const int c = ((max_ctx + S - 1) / S + 15) / 16 * 16;  // equal key ranges, multiples of 16
  const float scale_log2 = 1.4426950408889634f / sqrtf(static_cast<float>(hd));
  const int64_t grid = n_whole + static_cast<int64_t>(B * H - n_whole) * S;
  auto go = [&](auto kern, int ring, std::atomic<uint64_t>& attr_done) {
    int smem = kDecodeWarps * ring;
    // A grid within one wave is spread evenly: CTAs start as the previous kernel's leave, and the first
    // SMs to empty would take all they can hold (16 envs x 32 heads: 6 CTAs on some SMs, none on others,
    // 31 us against 25), so each asks for its share of the shared memory.  The price is that nothing else
    // fits beside them, the next projection's early CTAs among it: decode of 64 envs of 8 small layers takes
    // 3294 us so and 3364 without.
    const int64_t per_sm = (grid + num_sms - 1) / num_sms;
    if (per_sm < decode_ctas_per_sm(hd)) smem = std::max(smem, static_cast<int>(kSmemPerSm / per_sm - kDecodeStatic) / 128 * 128);
    if (const cudaError_t e = set_smem_limit(kern, kSmemPerSm - kDecodeStatic, attr_done)) return e;
    return launch_pdl(kern, dim3(static_cast<unsigned>(grid)), dim3(kDecodeWarps * 32), smem, stream,
                      q, rows, kv, layer, H, n_whole, c, S, scale_log2, part_o, part_ml, counters, out_hi, out_lo, fp16);
  };
  const bool res = kv.res != nullptr;
  static std::atomic<uint64_t> done[4];
  if (hd == 128) {
    VLA_CUDA_TRY(res ? go(attn_decode_kernel<128, true>, DecodeSlot<128, true>::RING, done[0])
                     : go(attn_decode_kernel<128, false>, DecodeSlot<128, false>::RING, done[1]));
  } else if (hd == 64) {
    VLA_CUDA_TRY(res ? go(attn_decode_kernel<64, true>, DecodeSlot<64, true>::RING, done[2])
                     : go(attn_decode_kernel<64, false>, DecodeSlot<64, false>::RING, done[3]));
  } else {
    return VLA_ERR_UNSUPPORTED;
  }
  note_launch();
  VLA_CUDA_TRY(cudaGetLastError());
  return VLA_OK;
}

}  // namespace vla
