// Internal interface of the attention kernels (attention.cu).
#pragma once
#include "common.cuh"

namespace vla {

// A tile of up to 64 consecutive query rows of one env: packed rows row0 .. row0+nrows-1
// at positions pos0 .. pos0+nrows-1.
struct AttnTile {
  int env, row0, nrows, pos0;
};

// q: f32 [rows, H*hd]; out: hi/lo operand pair [rows, H*hd], fp16 if `fp16` else bf16; keys
// from the fp16 cache of `layer`.
int attn_chunk_launch(const float* q, bf16* out_hi, bf16* out_lo, const AttnTile* tiles,
                      int n_tiles, KVLayout kv, int layer, int H, int hd, cudaStream_t stream,
                      bool fp16);

// The same on the tcgen05 tensor cores with the cache read as fp16 + 4-bit residual (kv.res
// required): tiles of up to 128 rows; status gets VLA_STATUS_TIMEOUT if a pipeline wait runs out.
// write_lo = false leaves out_lo untouched (for a consumer that reads the hi plane alone).
int attn_chunk_tc_launch(const float* q, bf16* out_hi, bf16* out_lo, const AttnTile* tiles, int n_tiles,
                         KVLayout kv, int layer, int H, int hd, uint32_t* status, cudaStream_t stream, bool fp16,
                         int num_sms, bool write_lo);

// The same for tiles of at most 16 rows, max_rows the most that one has (kv.res required; not checked on
// the device: the caller guarantees nrows <= max_rows), on mma.sync with one CTA per (tile, head): each
// cached byte is read once per tile and head.  write_lo as attn_chunk_tc_launch.
constexpr int kAttnRowsMax = 16;
int attn_rows_launch(const float* q, bf16* out_hi, bf16* out_lo, const AttnTile* tiles, int n_tiles, int max_rows,
                     KVLayout kv, int layer, int H, int hd, cudaStream_t stream, bool fp16, bool write_lo);

// One query per env row b (rows[b] gives env and position).  The first n_whole of the B * H (env, head)
// pairs run on one CTA each, the others on S CTAs with equal key ranges: their partials in part_o
// [(B * H - n_whole) * S * hd] f32 and part_ml, counters [B * H] int zero at launch and zero again when
// the kernel completes (none of the three is touched with S == 1).  The output pair is fp16 if `fp16`,
// else bf16.
int attn_decode_launch(const float* q, bf16* out_hi, bf16* out_lo, const RowInfo* rows, int B,
                       int max_ctx, KVLayout kv, int layer, int H, int hd, int n_whole, int S,
                       float* part_o, float2* part_ml, int* counters, cudaStream_t stream,
                       bool fp16, int num_sms);
// CTAs of the kernel that an SM holds.
constexpr int decode_ctas_per_sm(int hd) { return hd == 64 ? 8 : 6; }

// The same on the kernel for many (env, head) pairs over short contexts, one CTA per pair.
int attn_decode_short_launch(const float* q, bf16* out_hi, bf16* out_lo, const RowInfo* rows, int B, KVLayout kv,
                             int layer, int H, int hd, cudaStream_t stream, bool fp16);
// Where it is the faster one when the cache comes from HBM.  A decode's time on attn_decode_launch's kernel
// over that on this one, in 8 layers of 8 64-wide heads (envs x 8 pairs) and two 7B layers (envs x 32 pairs), at
// 24 / 100 / 130 / 200 positions, 152 SMs:
//   64-wide   512 pairs .97 / .93 / .91 / .87   640 1.04 / 1.02 / 1.00 / .97   768 1.05 / 1.06 / 1.04 / 1.01
//             1024 1.06 / 1.05 / 1.03 / 1.00    1536 1.08 / 1.04 / 1.02 / .99  2048 1.12 / 1.09 / 1.08
//   128-wide  992 at 60 to 100 .99               1056 1.03 / 1.02 / .99 / .98   1824 1.04 / 1.02 / 1.00 / .98
//             3072 1.08 / 1.02 / 1.00 / .98     4096 1.10 / 1.06 / 1.05 / 1.02 8192 1.14 / 1.08 / 1.05
// (256 envs x 8 positions: 3738 against 3271 us, and 3348 against 2807 in the 7B layers.)
constexpr bool decode_short(int pairs, int max_ctx, int hd, int num_sms) {
  const int few = (hd == 64 ? 4 : 7) * num_sms, many = (hd == 64 ? 5 : 24) * num_sms;
  return pairs > few && max_ctx <= (hd == 64 ? (pairs > many ? 160 : 112) : (pairs > many ? 192 : 128));
}

}  // namespace vla
