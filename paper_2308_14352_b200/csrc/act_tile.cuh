// Activation tiles of the weight-streaming kernel (ffn_tma.cu): the tokens of one pass over an
// expert (at most 16), stored so that ONE bulk copy brings the part a stage
// needs and every shared-memory read of it is free of bank conflicts.
//
//   tile     [K / 128 segments], at act_tile_offset(first slot of the pass)
//   segment  [tokens][256 bytes: 128 inputs as fp16]; in passes of at most 8 tokens then 64 bytes: (4 and 2 bits) every
//            token's share of the code offset, -2^(b-1) * 2^-24 * (sum of its 128 inputs), as fp32,
//            [8][2]: two halves to be added up, which one 16-byte read brings for a lane's two tokens (hidden vectors of
//            a gated layer, whose producers hold 64 channels each, fill one half at a time; others the first, the
//            second being zero)
//   row      sixteen 16-byte chunks; chunk (q ^ (token & 1)) * 4 + t holds what lane t of an MMA quad
//            needs for the two MMAs 2q and 2q+1 of the segment (its inputs 32t .. 32t+31), so the
//            eight lanes of one shared-memory phase (two tokens x four t) cover all 32 banks.
//
// Inside a chunk the eight inputs follow the order in which the kernel takes the code fields out of
// a packed word w: first the fields that sit at the same bit position of both 16-bit halves of w,
// then those of w >> 8 at that position (an MMA takes both), then the next position:
//   8 bits (2 words of 4 per chunk)  0 2 | 1 3 | 4 6 | 5 7
//   4 bits (1 word of 8 per chunk)   0 4 | 2 6 | 1 5 | 3 7
//   2 bits (half a word of 16)       0 8 | 4 12 | 1 9 | 5 13   and   2 10 | 6 14 | 3 11 | 7 15
#pragma once
#include "common.cuh"
#include "ffn_tile.cuh"

namespace emoe {

constexpr int ACT_PASS_MAX = 16;  // tokens per pass
__host__ __device__ __forceinline__ constexpr int act_seg_bytes(int ntok) { return ntok * 256 + (ntok <= 8 ? 64 : 0); }
// bytes per slot of an activation buffer with rows of K inputs: a tile of n tokens takes n rows plus the offset shares
__host__ __device__ __forceinline__ constexpr size_t act_slot_bytes(int K) { return static_cast<size_t>(K) * 2 + static_cast<size_t>(K / 128) * 64; }
__host__ __device__ __forceinline__ size_t act_tile_offset(int slot0, int K) { return static_cast<size_t>(slot0) * act_slot_bytes(K); }

// the share of the code offset of token `tok` from the sum of its inputs (half 0 or 1: of those 64; -1: of all); `at`:
// behind the segment's rows
__device__ __forceinline__ void act_tile_offset_share(unsigned char* at, int tok, int half, float sum, int bits) {
  const float share = -static_cast<float>(1 << (bits - 1)) * 5.9604644775390625e-8f * sum;
  if (half < 0) reinterpret_cast<float2*>(at)[tok] = make_float2(share, 0.0f);
  else reinterpret_cast<float*>(at)[2 * tok + half] = share;
}

// byte offset of input n (inside its segment) in the row of token `tok`
template <int BITS>
__device__ __forceinline__ int act_tile_pos(int n, int tok) {
  const int t = (n >> 5) & 3, i = n & 31;
  int q, elem;
  if (BITS == 2) {
    const int c = i & 3;
    q = 2 * (i >> 4) + (c >> 1);
    elem = ((c & 1) << 2) | (((i >> 2) & 1) << 1) | ((i >> 3) & 1);
  } else {
    const int o = i & 7;
    q = i >> 3;
    elem = BITS == 8 ? ((o & 4) | ((o & 1) << 1) | ((o >> 1) & 1)) : (((o & 1) << 2) | (o & 2) | (o >> 2));
  }
  return (((q ^ (tok & 1)) * 4 + t) << 4) + elem * 2;
}

// One activation row (bf16, natural order) into the tile of its pass, by the threads of a CTA:
// `rank` of the token among the `cnt` tokens of its expert, whose first slot is `begin`.
__device__ __forceinline__ void act_tile_row(const __nv_bfloat16* __restrict__ src_row, unsigned char* __restrict__ tiles, int begin,
                                             int cnt, int rank, int d, int bits, int* __restrict__ check_word) {
  const int p0 = rank / ACT_PASS_MAX * ACT_PASS_MAX, tok = rank - p0, ntok = min(ACT_PASS_MAX, cnt - p0);
  unsigned char* tile = tiles + act_tile_offset(begin + p0, d);
  const int seg_bytes = act_seg_bytes(ntok);
  bool beyond = false;
  // one thread moves 16 consecutive inputs: half b of lane t's 32 inputs of a segment; the eight
  // threads of a segment are neighbours and add up its sum
  for (int u = threadIdx.x; u < d / 16; u += blockDim.x) {
    const int seg = u >> 3, t = (u >> 1) & 3, b = u & 1;
    const uint4* src = reinterpret_cast<const uint4*>(src_row + u * 16);
    uint4 a = src[0], c = src[1];
    beyond |= bf16x2_beyond_f16(a.x) | bf16x2_beyond_f16(a.y) | bf16x2_beyond_f16(a.z) | bf16x2_beyond_f16(a.w) |
              bf16x2_beyond_f16(c.x) | bf16x2_beyond_f16(c.y) | bf16x2_beyond_f16(c.z) | bf16x2_beyond_f16(c.w);
    a = make_uint4(bf16x2_to_f16x2_sat(a.x), bf16x2_to_f16x2_sat(a.y), bf16x2_to_f16x2_sat(a.z), bf16x2_to_f16x2_sat(a.w));
    c = make_uint4(bf16x2_to_f16x2_sat(c.x), bf16x2_to_f16x2_sat(c.y), bf16x2_to_f16x2_sat(c.z), bf16x2_to_f16x2_sat(c.w));
    uint4 lo, hi;  // chunks q = 2b and 2b + 1
    if (bits == 8) {
      lo = make_uint4(prmt(a.x, a.y, 0x5410u), prmt(a.x, a.y, 0x7632u), prmt(a.z, a.w, 0x5410u), prmt(a.z, a.w, 0x7632u));
      hi = make_uint4(prmt(c.x, c.y, 0x5410u), prmt(c.x, c.y, 0x7632u), prmt(c.z, c.w, 0x5410u), prmt(c.z, c.w, 0x7632u));
    } else if (bits == 4) {
      lo = make_uint4(prmt(a.x, a.z, 0x5410u), prmt(a.y, a.w, 0x5410u), prmt(a.x, a.z, 0x7632u), prmt(a.y, a.w, 0x7632u));
      hi = make_uint4(prmt(c.x, c.z, 0x5410u), prmt(c.y, c.w, 0x5410u), prmt(c.x, c.z, 0x7632u), prmt(c.y, c.w, 0x7632u));
    } else {
      lo = make_uint4(prmt(a.x, c.x, 0x5410u), prmt(a.z, c.z, 0x5410u), prmt(a.x, c.x, 0x7632u), prmt(a.z, c.z, 0x7632u));
      hi = make_uint4(prmt(a.y, c.y, 0x5410u), prmt(a.w, c.w, 0x5410u), prmt(a.y, c.y, 0x7632u), prmt(a.w, c.w, 0x7632u));
    }
    unsigned char* row = tile + static_cast<size_t>(seg) * seg_bytes + tok * 256;
    const int x = tok & 1;
    *reinterpret_cast<uint4*>(row + ((((2 * b) ^ x) * 4 + t) << 4)) = lo;
    *reinterpret_cast<uint4*>(row + ((((2 * b + 1) ^ x) * 4 + t) << 4)) = hi;
    if (ntok <= 8 && bits != 8) {
      float sum = 0.0f;
      const uint32_t v[8] = {a.x, a.y, a.z, a.w, c.x, c.y, c.z, c.w};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&v[i]));
        sum += f.x + f.y;
      }
      const unsigned group = 0xffu << (threadIdx.x & 24);
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) sum += __shfl_xor_sync(group, sum, o);
      if ((u & 7) == 0) act_tile_offset_share(tile + static_cast<size_t>(seg) * seg_bytes + ntok * 256, tok, -1, sum, bits);
    }
  }
  // a value the fp16 operand cannot hold was saturated: the result is no longer the definition's
  if (beyond) atomicOr(check_word, CHECK_F16_RANGE);
}

}  // namespace emoe
