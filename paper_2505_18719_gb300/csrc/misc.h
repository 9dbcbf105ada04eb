// Internal interface of the row kernels (kernels_misc.cu) and the action head (action_head.cu).
#pragma once
#include "common.cuh"

namespace vla {

// First RMSNorm of assembled rows: weight w, the operand pair y_hi / y_lo [rows, d].
struct FirstNorm {
  const bf16* w;
  float eps;
  bf16* y_hi;
  bf16* y_lo;
  bool fp16;
};
// One 256-thread CTA: the bf16 row src as fp32 to h, and its RMSNorm to the pair at element `off`, summed in
// rmsnorm_kernel's order (the second read of src comes from L1).  red: 8 floats of shared memory, free on
// entry; free again once every thread has returned and met at a barrier.
__device__ __forceinline__ void token_row_256(const bf16* src, int d, float* h, const FirstNorm& nm, size_t off, float* red,
                                              uint32_t* status) {
  float ss = 0.f;
  for (int c = threadIdx.x * 4; c < d; c += 1024) {
    const uint2 x = *reinterpret_cast<const uint2*>(src + c);
    const float2 a = unpack_bf16x2(x.x), b = unpack_bf16x2(x.y);
    const float4 v = make_float4(a.x, a.y, b.x, b.y);
    *reinterpret_cast<float4*>(h + c) = v;
    ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
  }
  ss = warp_sum(ss);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  float tot = 0.f;
  for (int i = 0; i < 8; ++i) tot += red[i];
  const float r = rsqrtf(tot / static_cast<float>(d) + nm.eps);
  uint32_t sat = 0;
  for (int c = threadIdx.x * 4; c < d; c += 1024) {
    const uint2 x = *reinterpret_cast<const uint2*>(src + c), ww = *reinterpret_cast<const uint2*>(nm.w + c);
    const float2 a = unpack_bf16x2(x.x), b = unpack_bf16x2(x.y), w0 = unpack_bf16x2(ww.x), w1 = unpack_bf16x2(ww.y);
    uint2 hi, lo;
    split_pack2(a.x * r * w0.x, a.y * r * w0.y, hi.x, lo.x, nm.fp16, sat);
    split_pack2(b.x * r * w1.x, b.y * r * w1.y, hi.y, lo.y, nm.fp16, sat);
    *reinterpret_cast<uint2*>(nm.y_hi + off + c) = hi;
    *reinterpret_cast<uint2*>(nm.y_lo + off + c) = lo;
  }
  report_saturation(status, sat);
}

// h[r] (f32 [rows, d]) = source row of RowInfo r: visual (bf16 row idx), text (embed[ids[idx]])
// or token (embed[tokens[idx]]).  Ids outside [0, vocab) -> VLA_STATUS_BAD_TOKEN, row 0.
// The rows' RMSNorm with weight norm.w goes to norm.y_hi / y_lo [rows, d] as the operand pair.  The first kernel
// of a call: launched in stream order.
int assemble_launch(const RowInfo* rows, int n_rows, const bf16* visual, const int* ids,
                    const int* tokens, const bf16* embed, int d, int vocab, float* h, const FirstNorm& norm,
                    uint32_t* status, cudaStream_t s);

// The RMSNorm of rows whose sums of squares are known: sum_i ss[i * M + m], i < n_ss.
int norm_scale_launch(const float* h, int ldh, const bf16* w, const float* ss, int n_ss, int M, int d, float eps,
                      bf16* y_hi, bf16* y_lo, cudaStream_t s, bool fp16, uint32_t* status);

// y[m] = h[m] / sqrt(mean(h[m]^2) + eps) * w, h f32 [M, d] (row stride ldh), written as the
// operand pair (y_hi, y_lo) [M, d] with y_hi + y_lo ~ y, fp16 if `fp16` else bf16; a finite
// value beyond the fp16 range is stored as +-65504 and sets VLA_STATUS_SATURATED in *status.
int rmsnorm_launch(const float* h, int ldh, const bf16* w, int M, int d, float eps, bf16* y_hi,
                   bf16* y_lo, cudaStream_t s, bool fp16, uint32_t* status);

// dst[i] = fp16(src[i]) for n bf16 values (n % 8 == 0, both 16-byte aligned).  A value outside
// the finite fp16 range (|x| > 65504, or not finite) is clamped to +-65504 and sets
// *out_of_range to 1.  A bf16 value (8 significant bits) with 2^-14 <= |x| <= 65504 is exact
// in fp16 (11); a smaller one rounds to a multiple of 2^-24, an absolute error <= 2^-25.
int bf16_to_f16_launch(const bf16* src, f16* dst, size_t n, int* out_of_range, int num_sms,
                       cudaStream_t s);

// dst0[i] = src0[idx[i]] and dst1[i] = src1[idx[i]], rows of width d (f32).
int gather_rows2_launch(const float* src0, const float* src1, const int* idx, int n, int d, float* dst0, float* dst1,
                        cudaStream_t s);

struct HeadArgs {
  Start start = Start::kEarly;  // kInOrder for the first kernel of a call
  const float* h = nullptr;   // input rows, row (b * n_pos + j) has stride ldh
  // set (score): row j = 0 of env b is h_first's row b, row j > 0 is h's row b * (n_pos - 1) + j - 1
  const float* h_first = nullptr;
  int ldh = 0;
  int B = 0, n_pos = 1;       // grid: B x n_pos
  int step = 0;               // action index of j = 0 (decode: current step; score: 0)
  int A = 7;                  // actions per env (row stride of the [B, A] outputs)
  const bf16* final_norm = nullptr;
  const bf16* head_rows = nullptr;  // [256, d]
  int d = 0;
  float eps = 1e-6f;
  float temperature = 1.f;
  const float* uniforms = nullptr;  // [B, A, 256] (sample mode) or null (score mode)
  const int* forced = nullptr;      // [B, A] ids whose log-prob is reported (null: the sample)
  int forced_base = 0;              // subtracted from forced ids to get bins (vocab-256 or 0)
  int token_base = 0;               // vocab - 256
  int* tokens_out = nullptr;        // [B, A] sampled ids
  int* bins_out = nullptr;          // [B, A] sampled bins
  float* lp_out = nullptr;          // [B, A]
  float* act_out = nullptr;         // [B, A]
  float* logits_out = nullptr;      // [B, A, 256]
  float* entropy_out = nullptr;     // [B, A] entropy of each token's bin distribution
  int* pending_out = nullptr;       // [B] each env's token of action A - 1
  uint32_t* status = nullptr;
  // decode steps with a next one (n_pos == 1): the row of the token fed next, per env, as assemble_launch
  // would write it (next_embed null: none)
  const bf16* next_embed = nullptr;
  float* next_h = nullptr;
  FirstNorm next_norm{};
};
int action_head_launch(const HeadArgs& a, cudaStream_t s);

// learning.cu
int value_head_launch(const float* h, int ldh, int B, int d, const bf16* gain, const bf16* w, float eps,
                      float bias, float* out, cudaStream_t s);
int gae_launch(const float* r, const float* v, const float* done, int M, int B, float gamma, float lam,
               float* adv, float* ret, cudaStream_t s);
int ppo_clip_launch(const float* lp_new, const float* lp_old, const float* adv, int N, int A, float eps,
                    float* objective, float* ratio, float* clip_frac, cudaStream_t s);

}  // namespace vla
