// Grouped expert FFN on packed weights: TMA-staged weight stream + tensor-core multiply-adds, for
// bf16 activations with up to some tens of tokens per expert (decode, small prefill).  Paper
// Sections 1/2.1 (each activated expert is an independent FFN) on the Section 3.2 storage (b-bit
// codes + scale channel, w~ = q * s formed in registers).
//
// The codes are the A operand of mma.m16n8k16 (rows = output channels), tokens the N dimension,
// products accumulate in fp32 per 128-input segment, then total += scale * segment.  The work is
// bound by streaming packed weights from HBM and, at 4 and 2 bits, by the logic pipe (one
// instruction per pair of codes, at half the issue rate), so both are kept lean:
//   * the kernel is persistent and runs BOTH projections of a layer.  The items are the first projection's (activated
//     expert, block of output rows), then the second's (.., split-K slice), most expensive bitwidth first.  A CTA takes every
//     n-th of the first and, where the second has more than three items per CTA, whichever is next of those (fixed shares let the
//     slowest CTA end a tenth of the launch behind the others; Mixtral-like layer, 4 tokens 133 -> 125 us).  The stream runs ahead across items, so
//     it never drains between tiles; an item of the second projection waits until the expert's
//     hidden vectors are complete (release / acquire on a counter in the expert's plan record);
//   * a stage holds two 64-row x 128-byte boxes of packed codes (two TMA tensor copies, 128-byte
//     swizzle: the consumers' reads are conflict free), the rows' scales (cp.async) and the matching
//     slice of the pass's activation tile (ONE bulk copy: the tile is stored segment-major, see
//     act_tile.cuh).  Stages are cut from a ring in shared memory, each as large as it needs to
//     be, because the activation part varies from 0.3 to 17 KB.  Two CTAs with some four stages
//     each in flight reach the copy rate of the HBM (6.5 to 6.9 TB/s measured with idle consumers;
//     one feeding thread per SM tops out at 5.2);
//   * two feeding warps: one for the codes, one for activations and scales, so that a wait for hidden
//     vectors does not keep the weight stream from running ahead.  They come first in the CTA: the
//     schedulers favour old warps.  Items are decoded 32 at a time by the lanes of the first; a
//     feeding thread between eight computing warps needs about twenty cycles per instruction,
//     and whatever it does per stage shows;
//   * eight consumer warps take one 16-row tile of the stage each, or four warps two (see the launch): eight rows of either box (gated projection: of
//     w1 and the same eight of w3, so that the activation is formed in one lane).  The two rows of a lane then always lie
//     one box apart, and with the lane's places worked out once per pass and the scales of a stage read as whole words a
//     segment costs few instructions beside its unpacking (4 bits, 4 tokens of the Mixtral-like layer: 156 -> 149 per
//     16 rows x 128 inputs, expert launch 129 -> 121 us; 768 x 3072, 32 experts, 64 tokens 37 -> 35 us);
//   * up to 8 tokens per pass, 4 and 2 bits: a code field is read in place as the mantissa of a SUBNORMAL fp16
//     number ((q + 2^(b-1)) * 2^(p-24) for a field at bit p): one logic instruction per pair of
//     codes, one shift per word.  Fields at different positions go to accumulators of their own,
//     which are brought together once per segment; the offset's share 2^(b-1) * sum(x) comes with
//     the activation tile.  This costs the sums some bits: 0.3 % (4 bits) and 1.7 % (2 bits) of the hidden
//     values round to the other side of a bf16 tie, with exact codes 0.007 %.  At 8 bits it would be 1 % where
//     the codes bring 0.007 %, so these are taken exactly, as all are with 9 to 16 tokens per
//     pass (one fp16x2 subtraction more per pair, there shared by two token tiles).
// 128 bytes of a row are 128 / 256 / 512 inputs at 8 / 4 / 2 bits, so a stage covers 1 / 2 / 4
// scale segments.  Every wait is bounded: a wait that runs out sets a bit in the context's
// check word and the CTA winds down without touching the stage.
//
// Measured (expert launch alone; one feeding and four computing warps per CTA, three CTAs -> eight computing warps, fixed items
// -> now): Mixtral-like layer (d 4096, f 14336), 23 tokens 245 -> 223 -> 200 us (4.1 TB/s of packed bytes), 4 tokens 143 -> 121
// (4.3); of 8-bit experts 4.7 -> 4.7 -> 5.35 TB/s, 4 bits 2.8 -> 3.5 -> 4.1, 2 bits 1.8 -> 2.1 -> 2.5; 768 x 3072, 32 experts, 64 tokens
// 37 -> 35.5 us.  With the consumers idle the same launch takes 103 us at 4 tokens, with nothing loaded 113.
#include <cuda.h>

#include <climits>

#include "act_tile.cuh"
#include "common.cuh"
#include "ffn_tile.cuh"
#include "pipe.cuh"

namespace emoe {
namespace {

// A CTA has W consumer warps, eight or four, which take one or two 16-row tiles of every stage, and the weight and the
// activation warp.
__host__ __device__ constexpr int st_threads(int w) { return (w + 2) * 32; }
constexpr int ST_PLAN_CACHE = 64;                // plan records a CTA keeps in shared memory
constexpr int ST_CTAS = 2;                       // per SM
constexpr int ST_BOX_ROWS = 64;
__host__ __device__ constexpr int st_tiles(int w) { return ST_BOX_ROWS / (8 * w); }  // 16-row tiles of a warp: eight rows of each box per tile
constexpr int ST_BOX_BYTES = ST_BOX_ROWS * 128;  // 8 KB
constexpr int ST_X_OFFSET = 2 * ST_BOX_BYTES + 2 * ST_BOX_ROWS * 16;  // a stage: two boxes, 16 bytes of scales per row, the activation slice
constexpr int ST_RING = 96 * 1024;
constexpr int ST_SLOTS = 8;                      // stages in flight at most (barriers, records)
constexpr int ST_HID_BYTES = ACT_PASS_MAX * 256;  // one segment of hidden values on their way out
constexpr int ST_SMEM = ST_RING + 2 * ST_HID_BYTES + 1024;  // + slack to align the base to 1024
static_assert(ST_X_OFFSET + 4 * (ACT_PASS_MAX * 256) + 1023 <= ST_RING / 2, "two of the largest stages fit the ring");

// MMA row g of a 16-row tile -> row of the shared-memory box, chosen per bitwidth so that the
// lanes of one shared-memory transaction fall into different 16-byte columns after the swizzle.
template <int BITS>
__device__ __forceinline__ int box_row_of(int g) {
  if (BITS == 8) return g;
  if (BITS == 4) return ((g & 1) << 2) | (g >> 1);
  return ((g & 3) << 1) | (g >> 2);
}

struct TmaArgs {
  int phase_begin, phase_end;  // projections this launch runs: [0,1), [1,2) or both, [0,2)
  LayerDims L;
  const CUtensorMap* tmaps;  // [E][3]
  const unsigned char* xs;   // input tiles of the first projection (act_tile.cuh)
  int* plan;                 // header {activated experts, item counters} + one PlanRec per activated expert
  unsigned char* hidden;     // output tiles of the first projection, input of the second
  float* o_part;
  int ksplit;         // split-K slices of the second projection
  int row_blocks[2];  // row blocks of an expert per projection
  int ngroups[2];     // scale groups per row, per projection
  unsigned gmul;      // scale group of segment s: (s * gmul) >> 20 (2^20 / segments per group, rounded up; 0: one group per row)
  int n_pairs;
  int claim_above;    // items of the second projection per CTA beyond which they are claimed
  int* check_word;
  // floor(2^32 / d) + 1 for the divisors of the item index, per projection: n / d = umulhi(n, magic) for the
  // small n and d met here (n * d < 2^32), instead of an integer division in front of every item's first copy
  uint32_t mg_units[2], mg_ksplit[2], mg_rb[2];
};

__host__ __device__ inline uint32_t div_magic(uint32_t d) { return d <= 1 ? 0u : static_cast<uint32_t>((1ull << 32) / d) + 1u; }
__device__ __forceinline__ int fast_div(int n, int d, uint32_t magic) { return d <= 1 ? n : static_cast<int>(__umulhi(static_cast<uint32_t>(n), magic)); }
// exact for rows of up to 2^17 inputs: s * (segments per group) stays below 2^20
__device__ __forceinline__ int group_of_seg(const TmaArgs& a, int seg) { return static_cast<int>((static_cast<unsigned>(seg) * a.gmul) >> 20); }

// One item of a CTA's list: a block of output rows of an expert (and a slice of the inputs in the second
// projection), all tokens of the expert in passes of at most ACT_PASS_MAX.
struct __align__(16) ItemRec {
  int flags;            // ITEM_*; bits 8.. the width of the codes
  int nst, seg0, last;  // stages per pass, first segment, segments of the last stage (0: an empty split-K slice)
  int begin, cnt;       // the expert's slots
  int rbz, ai;          // row block | slice << 16, plan record
  const char* scales[2];   // scale channels of the item's matrices (second: w3 of a gated projection)
  const CUtensorMap* map;  // packed codes; a gated projection's w3 follows
  int row0, pad;
};
constexpr int ITEM_STOP = 1;
constexpr int ITEM_SECOND = 2;  // of the second projection
constexpr int ST_QUEUE = 64;    // records kept: decoded 32 at a time, nobody is more than ST_SLOTS stages behind
static_assert(ST_QUEUE >= 64, "a half of the queue is rewritten while the other is in use");

// How long the second projection of an expert waits for its hidden vectors (polls of ~0.1 us).
constexpr unsigned DEP_WAIT_LIMIT = 1u << 20;

// ---- codes -> A operand registers --------------------------------------------------------------
// The MMA `m` (0..7) of a segment takes two pairs of codes per row (registers lo, hi), class
// code_class(m) of field positions; see act_tile.cuh for the order of the inputs.
template <int BITS>
__device__ __forceinline__ constexpr int code_class(int m) { return BITS == 2 ? (m & 3) : (m & 1); }
template <int BITS>
__device__ __forceinline__ constexpr int field_pos(int m) { return BITS == 8 ? 0 : (BITS == 4 ? 4 * (m & 1) : 2 * (m & 3)); }
template <int BITS>
__device__ __forceinline__ constexpr int word_of(int m) { return BITS == 8 ? m : (BITS == 4 ? m >> 1 : m >> 2); }
template <int BITS>
__device__ __forceinline__ constexpr uint32_t field_mask() { return BITS == 8 ? 0x00FF00FFu : (BITS == 4 ? 0x000F000Fu : 0x00030003u); }
template <int BITS>
__device__ __forceinline__ constexpr uint32_t sign_bits() { return BITS == 8 ? 0x00800080u : (BITS == 4 ? 0x00080008u : 0x00020002u); }

// offset codes as subnormal fp16 numbers: (q + 2^(b-1)) * 2^(pos - 24)
template <int BITS>
__device__ __forceinline__ uint32_t code_sub(uint32_t w, int pos) { return and_xor(w, field_mask<BITS>() << pos, sign_bits<BITS>() << pos); }
// exact codes: the field under the exponent that makes its lowest bit weigh 1, the constant subtracted
template <int BITS>
__device__ __forceinline__ uint32_t code_exact(uint32_t w, int pos) {
  const uint32_t one = (static_cast<uint32_t>(25 - pos) << 10) * 0x00010001u;  // 2^(10-pos): mantissa bit pos weighs 1
  const uint32_t c = one | (sign_bits<BITS>() << pos);                         // 2^(10-pos) + 2^(b-1)
  return f16x2_sub(and_xor(w, field_mask<BITS>() << pos, c), c);
}
// what passes of up to 8 tokens take
template <int BITS>
__device__ __forceinline__ uint32_t code_one(uint32_t w, int pos) { return BITS == 8 ? code_exact<BITS>(w, pos) : code_sub<BITS>(w, pos); }

// Where a lane finds its operands in a stage, from the stage's start.  Everything that does not change from stage to stage
// is worked out once per pass: a segment's reads then are a register and a constant each.
struct StageLane {
  int row;      // its first row of codes, at the 16-byte column of segment 0 under the swizzle (the second: ROW2 behind it)
  int d1, d2;   // to the columns of the next segment and of the one after that (the swizzle makes them differ from lane to lane)
  int xe, xo;   // the even and the odd chunks of the activation tile
  int init;     // the code offset's shares
  int sc;       // the scales of its first row (the second's: SCALE2 behind it)
};
constexpr int ROW2 = ST_BOX_BYTES, SCALE2 = ST_BOX_ROWS * 16;  // a warp takes eight rows of each of the stage's two boxes

// One segment (128 inputs) of the warp's tiles: codes at wp (8 bits: and wp + d1), activations at x0 / x1 (even and odd
// chunks), the offset's shares at init; sc: the rows' scales.
template <int BITS, int NT, int TILES>
__device__ __forceinline__ void consume_segment(const unsigned char* wp, int d1, const unsigned char* x0, const unsigned char* x1,
                                                const unsigned char* init, const float (&sc)[TILES][2], float (&tot)[TILES][NT][4]) {
  constexpr int NW = BITS;  // 32-bit words of the lane's 32 codes of a row
  uint32_t w[TILES][2][NW];
#pragma unroll
  for (int j = 0; j < TILES; ++j)
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const unsigned char* at = wp + i * ROW2 + j * 1024;
      if constexpr (BITS == 2) {
        const uint2 v = *reinterpret_cast<const uint2*>(at);
        w[j][i][0] = v.x, w[j][i][1] = v.y;
      } else {
        const uint4 v = *reinterpret_cast<const uint4*>(at);
        w[j][i][0] = v.x, w[j][i][1] = v.y, w[j][i][2] = v.z, w[j][i][3] = v.w;
        if constexpr (BITS == 8) {
          const uint4 u = *reinterpret_cast<const uint4*>(at + d1);
          w[j][i][4] = u.x, w[j][i][5] = u.y, w[j][i][6] = u.z, w[j][i][7] = u.w;
        }
      }
    }
  if constexpr (NT == 1) {
    constexpr int NC = BITS == 2 ? 4 : 2;
    float acc[TILES][NC][4];
    float2 off = make_float2(0.0f, 0.0f);
    if constexpr (BITS != 8) {
      const float4 o = *reinterpret_cast<const float4*>(init);
      off = make_float2(o.x + o.y, o.z + o.w);
    }
#pragma unroll
    for (int j = 0; j < TILES; ++j) {
      acc[j][0][0] = acc[j][0][2] = off.x;
      acc[j][0][1] = acc[j][0][3] = off.y;
#pragma unroll
      for (int c = 1; c < NC; ++c)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[j][c][i] = 0.0f;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint4 b = *reinterpret_cast<const uint4*>((q & 1 ? x1 : x0) + 128 * (q >> 1));
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int m = 2 * q + h, pos = field_pos<BITS>(m);
#pragma unroll
        for (int j = 0; j < TILES; ++j) {
          const uint32_t u0 = w[j][0][word_of<BITS>(m)], u1 = w[j][1][word_of<BITS>(m)];
          mma_f16(acc[j][code_class<BITS>(m)], code_one<BITS>(u0, pos), code_one<BITS>(u1, pos), code_one<BITS>(u0 >> 8, pos),
                  code_one<BITS>(u1 >> 8, pos), h ? b.z : b.x, h ? b.w : b.y);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < TILES; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float v;
        if constexpr (BITS == 8) v = acc[j][0][i] + acc[j][1][i];
        else if constexpr (BITS == 4) v = fmaf(acc[j][1][i], 0.0625f, acc[j][0][i]);
        else v = fmaf(fmaf(acc[j][3][i], 0.25f, acc[j][2][i]), 0.0625f, fmaf(acc[j][1][i], 0.25f, acc[j][0][i]));
        tot[j][0][i] = fmaf(sc[j][i >> 1], v, tot[j][0][i]);
      }
  } else {
    float acc[TILES][NT][4];
#pragma unroll
    for (int j = 0; j < TILES; ++j)
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[j][nt][i] = 0.0f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint32_t c[TILES][2][4];
#pragma unroll
      for (int j = 0; j < TILES; ++j)
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int m = 2 * q + h, pos = field_pos<BITS>(m);
            const uint32_t u = w[j][i][word_of<BITS>(m)];
            c[j][i][2 * h] = code_exact<BITS>(u, pos);
            c[j][i][2 * h + 1] = code_exact<BITS>(u >> 8, pos);
          }
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        const uint4 b = *reinterpret_cast<const uint4*>((q & 1 ? x1 : x0) + 128 * (q >> 1) + nt * 2048);
#pragma unroll
        for (int j = 0; j < TILES; ++j) mma_f16(acc[j][nt], c[j][0][0], c[j][1][0], c[j][0][1], c[j][1][1], b.x, b.y);
#pragma unroll
        for (int j = 0; j < TILES; ++j) mma_f16(acc[j][nt], c[j][0][2], c[j][1][2], c[j][0][3], c[j][1][3], b.z, b.w);
      }
    }
#pragma unroll
    for (int j = 0; j < TILES; ++j)
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) tot[j][nt][i] = fmaf(sc[j][i >> 1], acc[j][nt][i], tot[j][nt][i]);
  }
}

// This warp's share of an expert's hidden vectors is written: make it visible to the bulk copies
// of other SMs (release), then count it.
__device__ __forceinline__ void count_item_done(PlanRec* recs, int ai, int lane) {
  // the hidden values live in global memory: the fence restricted to that space costs some 40 cycles where the
  // unrestricted one (which also settles the shared-memory side) was measured at 800 to 1300
  asm volatile("fence.proxy.async.global;" ::: "memory");
  __syncwarp();
  if (lane == 0)  // release: the hidden values this warp stored are visible before the count is
    asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(&recs[ai].done), "r"(1) : "memory");
}

// the hidden vector is rounded to bf16 (the layer's activation type), then carried as fp16; a
// saturated value is recognised by its bit pattern (+-65504 is not a bf16 number, so a hidden value
// can only be there by saturation)
__device__ __forceinline__ __half hidden_half(float h) { return f32_to_f16_sat(__bfloat162float(__float2bfloat16_rn(h))); }
__device__ __forceinline__ bool half_saturated(__half v) { return (__half_as_ushort(v) & 0x7fffu) == 0x7bffu; }

// Hidden values of a first-projection item: the lane's results (row gp of either box x tokens 2t, 2t+1 of
// every 8-token tile) into the warp-shared tile segment in shared memory, in the order the second
// projection reads them.
template <int BITS, int NT>
__device__ __forceinline__ void hidden_to_smem(bool gated, int rb, int ntok, int row, int lane, const float (&tot)[NT][4],
                                               unsigned char* hid, int* check_word) {
  const int t = lane & 3;
  bool beyond = false;
  if (gated) {
    const int n = (rb & 1) * 64 + row;  // channel inside its 128-input segment
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      if (nt * 8 >= ntok) break;
      __half hv[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float av = tot[nt][i], bv = tot[nt][i + 2];
        hv[i] = hidden_half(av / (1.0f + expf(-av)) * bv);
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int tok = nt * 8 + 2 * t + i;
        if (tok < ntok) {
          *reinterpret_cast<__half*>(hid + tok * 256 + act_tile_pos<BITS>(n, tok)) = hv[i];
          beyond |= half_saturated(hv[i]);
        }
      }
    }
  } else {
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      if (nt * 8 >= ntok) break;
      __half hv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) hv[i] = hidden_half(fmaxf(tot[nt][i], 0.0f));
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int tok = nt * 8 + 2 * t + (i & 1);
        if (tok < ntok) {
          *reinterpret_cast<__half*>(hid + tok * 256 + act_tile_pos<BITS>(row + 64 * (i >> 1), tok)) = hv[i];
          beyond |= half_saturated(hv[i]);
        }
      }
    }
  }
  if (beyond) atomicOr(check_word, CHECK_F16_RANGE);  // saturated above: reported, not silent
}

// The staged segment to global memory, a warp per token: 8 bytes per lane, and the sum of the
// token's values for the offset codes of the second projection.
__device__ __forceinline__ void hidden_to_global(const TmaArgs& a, bool gated, int rb, int slot0, int ntok, int bits, int warp,
                                                 int warps, int lane, const unsigned char* hid) {
  const int seg = gated ? rb >> 1 : rb, half = gated ? rb & 1 : 0;
  unsigned char* tile = a.hidden + act_tile_offset(slot0, a.L.d_ff) + static_cast<size_t>(seg) * act_seg_bytes(ntok);
  const bool mine = !gated || ((lane >> 2) & 1) == half;  // a gated item fills half of the segment: inputs of lanes t = 2*half, 2*half+1
  for (int tok = warp; tok < ntok; tok += warps) {
    float sum = 0.0f;
    if (mine) {
      const uint2 v = *reinterpret_cast<const uint2*>(hid + tok * 256 + lane * 8);
      *reinterpret_cast<uint2*>(tile + tok * 256 + lane * 8) = v;
      const float2 p = __half22float2(*reinterpret_cast<const __half2*>(&v.x)), q = __half22float2(*reinterpret_cast<const __half2*>(&v.y));
      sum = (p.x + p.y) + (q.x + q.y);
    }
    if (ntok <= 8 && bits != 8) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      if (lane == 0) {
        act_tile_offset_share(tile + ntok * 256, tok, gated ? half : -1, sum, bits);
      }
    }
  }
}

template <int BITS, int NT>
__device__ __forceinline__ void store_output(const TmaArgs& a, int rb, int z, int slot0, int ntok, int row, int lane,
                                             const float (&tot)[NT][4]) {
  const int t = lane & 3;
  const int N = a.L.d_model;
  float* dst = a.o_part + (static_cast<size_t>(z) * a.n_pairs + slot0) * N + rb * 128 + row;
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    if (nt * 8 >= ntok) break;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int tok = nt * 8 + 2 * t + (i & 1);
      if (tok < ntok) dst[static_cast<size_t>(tok) * N + ST_BOX_ROWS * (i >> 1)] = tot[nt][i];
    }
  }
}

// Item li of a projection, decoded by one thread.  The items are listed by expert, most expensive bitwidth first.
__device__ __forceinline__ void decode_item(const TmaArgs& a, const PlanRec* s_plan, const PlanRec* recs, int phase, int li, ItemRec* out) {
  const bool gated = phase == 0 && a.L.act == EMOE_ACT_SWIGLU;
  const int row_blocks = a.row_blocks[phase], ksplit = phase == 0 ? 1 : a.ksplit;
  const int mat_first = phase == 0 ? 0 : (a.L.act == EMOE_ACT_SWIGLU ? 2 : 1);
  const int ai = fast_div(li, ksplit * row_blocks, a.mg_units[phase]);
  const PlanRec& rec = ai < ST_PLAN_CACHE ? s_plan[ai] : recs[ai];
  const int lz = fast_div(li, ksplit, a.mg_ksplit[phase]);  // (expert, row block) index
  const int z = li - lz * ksplit;
  const int rb = lz - fast_div(lz, row_blocks, a.mg_rb[phase]) * row_blocks;
  const int bits = rec.bits;
  const int sh = bits == 8 ? 0 : (bits == 4 ? 1 : 2);  // log2 of the 128-input segments per stage
  const int seg_total = (phase == 0 ? a.L.d_model : a.L.d_ff) >> 7;
  const int steps_total = (seg_total + (1 << sh) - 1) >> sh;
  const int spz = fast_div(steps_total + ksplit - 1, ksplit, a.mg_ksplit[phase]);
  const int step_begin = z * spz;
  const int nsteps = max(0, min(steps_total, step_begin + spz) - step_begin);
  const int nst = max(nsteps, 1);  // an empty split-K slice still has to store its zeros
  out->flags = (phase == 1 ? ITEM_SECOND : 0) | (bits << 8);
  out->nst = nst;
  out->seg0 = step_begin << sh;
  out->last = nsteps > 0 ? min(1 << sh, seg_total - ((step_begin + nst - 1) << sh)) : 0;
  out->begin = rec.begin;
  out->cnt = rec.cnt;
  out->rbz = rb | (z << 16);
  out->ai = ai;
  out->scales[0] = static_cast<const char*>(mat_first == 0 ? rec.scales[0] : (mat_first == 1 ? rec.scales[1] : rec.scales[2]));
  out->scales[1] = gated ? static_cast<const char*>(rec.scales[1]) : out->scales[0];
  out->map = a.tmaps + static_cast<size_t>(rec.e) * 3 + mat_first;
  out->row0 = rb * (gated ? ST_BOX_ROWS : 2 * ST_BOX_ROWS);
}

__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

// How a row's scales lie: one fp16 number per segment and an even number of them, so that a stage's are whole aligned
// 4-byte words; fp16 or fp32 in any other number.
constexpr int SC_PAIRS = 0, SC_F16 = 1, SC_F32 = 2;
template <int SC>
__device__ __forceinline__ float scale_at(const unsigned char* p) {
  if constexpr (SC != SC_F32) return __half2float(*reinterpret_cast<const __half*>(p));
  else return *reinterpret_cast<const float*>(p);
}
__device__ __forceinline__ float2 scale_pair(uint32_t w) { return __half22float2(*reinterpret_cast<const __half2*>(&w)); }

// what the consumer warps share
struct Pipe {
  const unsigned char* ring;
  unsigned char* hid_stage;
  const ItemRec* queue;
  uint32_t bar_full, bar_empty, bar_hid;
  PlanRec* recs;
  bool fused;
  volatile int* abort_flag;
};
// where a consumer warp stands
struct Cursor {
  int it;          // next stage
  int phys;        // ... and the first place in the ring for it
  int n_hidden;    // first-projection items stored so far
  int pending_ai;  // expert whose finished item is still to be counted (-1: none)
};

// bytes of a stage in the ring
__device__ __forceinline__ int stage_bytes(int nseg, int xseg) { return nseg > 0 ? ST_X_OFFSET + ((nseg * xseg + 1023) & ~1023) : 0; }

// One pass of an item by a consumer warp, its first stage having arrived: all its stages, then the results.
template <int BITS, int SC, int NT, int W>
__device__ __forceinline__ bool consume_pass(const TmaArgs& a, const Pipe& pp, int k, int p0, int warp, int lane, Cursor& cur) {
  constexpr int SEGS = 8 / BITS, TILES = st_tiles(W);
  const ItemRec& rec = pp.queue[k % ST_QUEUE];
  const int nst = rec.nst, seg0 = rec.seg0, last = rec.last, cnt = rec.cnt, tok0 = rec.begin + p0;
  const int ntok = min(ACT_PASS_MAX, cnt - p0);
  const int phase = rec.flags & ITEM_SECOND ? 1 : 0;
  const bool gated = phase == 0 && a.L.act == EMOE_ACT_SWIGLU;
  constexpr int ssz = SC == SC_F32 ? 4 : 2;
  const int g = lane >> 2, t = lane & 3;
  const int gp = box_row_of<BITS>(g), row = 8 * TILES * warp + gp;  // in its box; of the warp's next tile: eight further down
  StageLane p;
  // a tile has eight rows of either box: of w1 and the same of w3, or of one matrix and those 64 further down.  8 bits:
  // columns 2t and 2t+1; 4 bits: column t of the segment's four; 2 bits: half of column t/2 of its two
  p.row = row * 128 + (((BITS == 8 ? 2 * t : (BITS == 4 ? t : t >> 1)) ^ gp) << 4) + (BITS == 2 ? (t & 1) << 3 : 0);
  p.d1 = (p.row ^ (BITS == 8 ? 16 : (BITS == 4 ? 64 : 32))) - p.row;
  p.d2 = (p.row ^ 64) - p.row;  // (2 bits)
  p.xe = ST_X_OFFSET + g * 256 + t * 16 + ((g & 1) << 6);
  p.xo = p.xe ^ 64;
  p.init = ST_X_OFFSET + ntok * 256 + t * 16;
  const int xstride = act_seg_bytes(ntok);
  const int need_full = stage_bytes(SEGS, xstride), need_last = stage_bytes(last, xstride);
  float tot[TILES][NT][4];
#pragma unroll
  for (int j = 0; j < TILES; ++j)
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int i = 0; i < 4; ++i) tot[j][nt][i] = 0.0f;
  // scales: 16 bytes per row of the stage, from the 4-byte boundary at or below the first one
  p.sc = 2 * ST_BOX_BYTES + row * 16;
  const int row_off = (rec.row0 + row) * a.ngroups[phase] * ssz;
#pragma unroll 1
  for (int s = 0; s < nst; ++s) {
    const int slot = cur.it % ST_SLOTS, need = s == nst - 1 ? need_last : need_full;
    if (cur.phys + need > ST_RING) cur.phys = 0;  // as the weight warp places it
    const unsigned char* stage = pp.ring + cur.phys;
    cur.phys += need;
    if (s > 0 && !__all_sync(0xffffffffu, mbar_wait(pp.bar_full + 8 * slot, (cur.it / ST_SLOTS) & 1, a.check_word, pp.abort_flag)))
      return false;
    const int seg = seg0 + s * SEGS, nseg = s == nst - 1 ? last : SEGS;
    const unsigned char *wp = stage + p.row, *x0 = stage + p.xe, *x1 = stage + p.xo, *init = stage + p.init, *sc = stage + p.sc;
    uint32_t sw[TILES][2][2];
    int g0 = 0;
    if constexpr (SC == SC_PAIRS) {
#pragma unroll
      for (int j = 0; j < TILES; ++j)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const unsigned char* at = sc + i * SCALE2 + j * 128;
          if constexpr (BITS == 8) {
            sw[j][i][0] = *reinterpret_cast<const unsigned short*>(at + 2 * (seg & 1));
          } else if constexpr (BITS == 4) {
            sw[j][i][0] = *reinterpret_cast<const uint32_t*>(at);
          } else {
            const uint2 v = *reinterpret_cast<const uint2*>(at);
            sw[j][i][0] = v.x, sw[j][i][1] = v.y;
          }
        }
    } else {
      g0 = group_of_seg(a, seg);
      sc += (row_off + g0 * ssz) & 3;
    }
#pragma unroll
    for (int sg = 0; sg < SEGS; ++sg) {
      if (sg >= nseg) break;
      float f[TILES][2];
      const int d = SC == SC_PAIRS || sg == 0 ? 0 : (group_of_seg(a, seg + sg) - g0) * ssz;
#pragma unroll
      for (int j = 0; j < TILES; ++j)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          if constexpr (SC == SC_PAIRS) {
            const float2 u = scale_pair(sw[j][i][sg >> 1]);
            f[j][i] = sg & 1 ? u.y : u.x;
          } else {
            f[j][i] = scale_at<SC>(sc + d + i * SCALE2 + j * 128);
          }
        }
      const unsigned char* w = BITS == 2 ? wp + (sg & 1 ? p.d1 : 0) + (sg & 2 ? p.d2 : 0) : wp + (BITS == 4 && sg ? p.d1 : 0);
      consume_segment<BITS, NT, TILES>(w, p.d1, x0 + sg * xstride, x1 + sg * xstride, init + sg * xstride, f, tot);
    }
    // shared memory of the stage is no longer needed
    __syncwarp();
    if (lane == 0) mbar_arrive(pp.bar_empty + 8 * slot);
    ++cur.it;
    if (s == 0 && cur.pending_ai >= 0) {
      count_item_done(pp.recs, cur.pending_ai, lane);
      cur.pending_ai = -1;
    }
  }
  const bool last_pass = p0 + ACT_PASS_MAX >= cnt;
  const int rb = rec.rbz & 0xffff, z = rec.rbz >> 16, ai = rec.ai;
  if (NT == 1 && BITS != 8) {  // the subnormal codes weigh 2^-24
#pragma unroll
    for (int j = 0; j < TILES; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) tot[j][0][i] *= 16777216.0f;
  }
  if (phase == 0) {
    // two staging buffers in turn: a warp can be one item ahead of the slowest, not two
    unsigned char* hid = pp.hid_stage + (cur.n_hidden & 1) * ST_HID_BYTES;
#pragma unroll
    for (int j = 0; j < TILES; ++j) hidden_to_smem<BITS, NT>(gated, rb, ntok, row + 8 * j, lane, tot[j], hid, a.check_word);
    __syncwarp();
    if (lane == 0) mbar_arrive(pp.bar_hid);
    if (!__all_sync(0xffffffffu, mbar_wait(pp.bar_hid, cur.n_hidden & 1, a.check_word, pp.abort_flag))) return false;
    ++cur.n_hidden;
    hidden_to_global(a, gated, rb, tok0, ntok, BITS, warp, W, lane, hid);
    if (pp.fused && last_pass) cur.pending_ai = ai;
  } else {
#pragma unroll
    for (int j = 0; j < TILES; ++j) store_output<BITS, NT>(a, rb, z, tok0, ntok, row + 8 * j, lane, tot[j]);
  }
  return true;
}

template <int SC, int W>
__global__ void __launch_bounds__(st_threads(W), ST_CTAS) ffn_tma_kernel(const __grid_constant__ TmaArgs a) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bars[3 * ST_SLOTS + 1];  // full, empty, issued (weight warp -> activation warp), hidden segment staged
  __shared__ ItemRec queue[ST_QUEUE];
  __shared__ __align__(16) PlanRec s_plan[ST_PLAN_CACHE];
  __shared__ int s_active, s_vstart[ST_SLOTS], s_offset[ST_SLOTS];
  __shared__ int wait_words[PIPE_WORDS];
  volatile int* abort_flag = wait_words + PIPE_ABORT;
  // an offset from the array, not a rounded address: the compiler then knows that every access is to shared memory
  unsigned char* ring = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* hid_stage = ring + ST_RING;
  // The feeding warps come first: the schedulers favour the oldest warp, and a feeding warp that has to wait for
  // eight computing ones to stall leaves them without work soon after.
  const int lane = threadIdx.x & 31, warp_id = threadIdx.x >> 5, warp = warp_id < 2 ? W + warp_id : warp_id - 2;
  const uint32_t bar_full = smem_u32(bars), bar_empty = smem_u32(bars + ST_SLOTS), bar_issued = smem_u32(bars + 2 * ST_SLOTS), bar_hid = smem_u32(bars + 3 * ST_SLOTS);

  if (threadIdx.x == 0) {
    wait_words[PIPE_ABORT] = wait_words[PIPE_FRONT] = 0;
    for (int s = 0; s < ST_SLOTS; ++s) {
      mbar_init(bar_full + 8 * s, 34);          // weight warp and activation warp (+ the bytes of their copies), every lane's scale copies
      mbar_init(bar_issued + 8 * s, 1);
      mbar_init(bar_empty + 8 * s, W);   // one arrival per consumer warp
    }
    mbar_init(bar_hid, W);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // Everything above overlaps the tail of the kernel in front.
  if (warp == W) {
    // The tensor maps are older than every kernel of the chain: pull them towards L2 now, so that
    // the first copy of an expert's matrix does not wait for its descriptor to come from HBM.
    const int n_maps = 3 * a.L.E;
    const int i = (static_cast<int>(blockIdx.x) * 32 + lane) % ((n_maps + 31) / 32 * 32);
    if (i < n_maps) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.tmaps + i));
  }
  pdl_wait();
  pdl_trigger();
  {  // the plan into shared memory: header and records in one round trip
    const int4* src = reinterpret_cast<const int4*>(reinterpret_cast<const char*>(a.plan) + PLAN_HEADER_BYTES);
    const int n = min(a.L.E, ST_PLAN_CACHE) * static_cast<int>(sizeof(PlanRec) / 16);
    for (int i = threadIdx.x; i < n; i += st_threads(W)) reinterpret_cast<int4*>(s_plan)[i] = __ldcg(src + i);
    if (threadIdx.x == 0) s_active = __ldcg(a.plan);
    __syncthreads();
  }

  const LayerDims& L = a.L;
  PlanRec* recs = reinterpret_cast<PlanRec*>(reinterpret_cast<char*>(a.plan) + PLAN_HEADER_BYTES);
  // both projections in this launch: an item of the second projection waits until the expert's
  // hidden vectors are complete (PlanRec::done, raised by the consumers of the first projection)
  const bool fused = a.phase_begin == 0 && a.phase_end == 2;

  if (warp == W) {
    // ---------------- weight warp: items, ring, packed codes ----------------
    // The ring: stages lie one behind the other, a stage that would run over the end starts at the
    // beginning again.  head and vstart are positions on an endless tape; a stage may be written
    // once nothing live lies within a ring's length behind its end.  This thread feeds eight
    // computing warps: whatever it does per stage is kept to a few instructions.
    // Every CTA takes every n-th item of the first projection and, going on so, one of the second; these are known without
    // asking and decoded 32 at a time.  From then on whoever is free claims the next one (one claim ahead, so that nobody
    // waits for the answer).  Up to three items of the second projection per CTA (one beside the tcgen05 kernel, where few experts are left
    // to stream and have 1 to 32 tokens each) the fixed shares go on to the end: a claimed
    // item is decoded alone, in front of its first copy, and the shares are as even as claims could make them (us per layer, fixed /
    // claimed, at 1.7 to 2 items per CTA: 1024 x 4096, 8 experts, 64 tokens 36.4/39.4; 768 x 3072, 16 experts, 96 tokens 37.1/39.7;
    // 512 x 2048, 32 experts, 192 tokens 35.0/36.9; at 3.5 to 4: 2048 x 8192, 4 experts, 16 tokens 48.1/46.9, 768 x 3072, 32 experts, 192
    // tokens 53.0/49.9, Mixtral-like layer, 8 tokens 188/179; beside the tcgen05 kernel, Zipf exponent 1.1: 1024 x 4096, 64 experts, 300 tokens
    // 101/98, 500 tokens 109/110, 128 experts, 1000 tokens 144/140, 1280 x 4480, 128 experts, 1000 tokens 210/200; even loads there leave
    // more than three).
    const int n = static_cast<int>(gridDim.x), me = static_cast<int>(blockIdx.x);
    const int n_items0 = a.phase_begin == 0 ? s_active * a.row_blocks[0] : 0, n_items1 = a.phase_end == 2 ? s_active * a.row_blocks[1] * a.ksplit : 0;
    const bool claims = n_items1 > a.claim_above * n;
    const int n_fixed = n_items0 + (claims ? n : n_items1);
    int it = 0, oldest = 0, head = 0, phys = 0;
    int more = 1, claim = n_items1;
    for (int k0 = 0; more; k0 += 32) {
      const int item = me + (k0 + lane) * n;
      ItemRec* out = &queue[(k0 + lane) % ST_QUEUE];
      if (item < n_fixed) decode_item(a, s_plan, recs, item < n_items0 ? 0 : 1, item < n_items0 ? item : item - n_items0, out);
      else out->flags = ITEM_STOP;
      __syncwarp();
      if (lane == 0) {
        for (int k = k0; k < k0 + 32 && more; ++k) {
          if (claims && me + (k + 1) * n >= n_fixed) {  // this item is the last known one, or a claimed one
            const int now = claim;
            claim = n + atomicAdd(a.plan + 1, 1);
            if (me + k * n >= n_fixed && now < n_items1) decode_item(a, s_plan, recs, 1, now, &queue[k % ST_QUEUE]);
          }
          const ItemRec& rec = queue[k % ST_QUEUE];
          const int flags = rec.flags;
          if (flags & ITEM_STOP) {  // tell the others that nothing else comes
            const int slot = it % ST_SLOTS;
            if (it < ST_SLOTS || mbar_wait(bar_empty + 8 * slot, ((it / ST_SLOTS) & 1) ^ 1, a.check_word, abort_flag)) {
              mbar_arrive(bar_full + 8 * slot);
              mbar_arrive(bar_issued + 8 * slot);
            }
            more = 0;
            break;
          }
          const int bits = flags >> 8, nst = rec.nst, last = rec.last, cnt = rec.cnt, row0 = rec.row0;
          const bool gated = !(flags & ITEM_SECOND) && L.act == EMOE_ACT_SWIGLU;
          const CUtensorMap* map0 = rec.map;
          const CUtensorMap* map1 = gated ? map0 + 1 : map0;
          const int row1 = gated ? row0 : row0 + ST_BOX_ROWS;
          const int c_first = rec.seg0 * 16 * bits;  // byte column: 128 inputs = 16 * bits bytes
          for (int p0 = 0; p0 < cnt && more; p0 += ACT_PASS_MAX) {
            const int xseg = act_seg_bytes(min(ACT_PASS_MAX, cnt - p0));
            const int need_full = stage_bytes(8 / bits, xseg), need_last = stage_bytes(last, xseg);
            for (int s = 0, c0 = c_first; s < nst; ++s, ++it, c0 += 128) {
              const int need = s == nst - 1 ? need_last : need_full;
              if (phys + need > ST_RING) {  // does not fit in front of the end of the ring
                head += ST_RING - phys;
                phys = 0;
              }
              while (oldest < it && (it - oldest >= ST_SLOTS || head + need > s_vstart[oldest % ST_SLOTS] + ST_RING)) {
                if (!mbar_wait(bar_empty + 8 * (oldest % ST_SLOTS), (oldest / ST_SLOTS) & 1, a.check_word, abort_flag)) {
                  more = 0;
                  break;
                }
                ++oldest;
              }
              if (!more) break;
              const int slot = it % ST_SLOTS;
              const uint32_t full = bar_full + 8 * slot;
              if (need > 0) {
                const uint32_t st = smem_u32(ring + phys);
                mbar_expect_tx(full, 2 * ST_BOX_BYTES);
                tma_load_2d(st, map0, c0, row0, full);
                tma_load_2d(st + ST_BOX_BYTES, map1, c0, row1, full);
              } else {
                mbar_arrive(full);
              }
              s_vstart[slot] = head;
              s_offset[slot] = phys;
              mbar_arrive(bar_issued + 8 * slot);  // over to the activation warp
              head += need;
              phys += need;
            }
          }
        }
      }
      more = __shfl_sync(0xffffffffu, more, 0);
    }
  } else if (warp == W + 1) {
    // ---------------- activation warp: the activation slice and the scales of every stage ----------------
    // On its own so that a wait for hidden vectors does not keep the weight stream from running ahead.
    int ready_ai = -1;  // the expert whose hidden vectors are known to be complete
    bool ok = true;
    int it = 0;
    for (int k = 0; ok; ++k) {
      if (!__all_sync(0xffffffffu, mbar_wait(bar_issued + 8 * (it % ST_SLOTS), (it / ST_SLOTS) & 1, a.check_word, abort_flag))) break;
      const ItemRec& rec = queue[k % ST_QUEUE];
      const int flags = rec.flags;
      if (flags & ITEM_STOP) {
        mbar_arrive(bar_full + 8 * (it % ST_SLOTS));
        if (lane == 0) mbar_arrive(bar_full + 8 * (it % ST_SLOTS));
        break;
      }
      const int phase = flags & ITEM_SECOND ? 1 : 0, bits = flags >> 8, nst = rec.nst, last = rec.last, cnt = rec.cnt, seg0 = rec.seg0;
      const bool gated = phase == 0 && L.act == EMOE_ACT_SWIGLU;
      constexpr int ssz = SC == SC_F32 ? 4 : 2;
      // the lane's rows of the stage: lane, lane + 32, ...
      const int row_bytes = a.ngroups[phase] * ssz;
      const char* sc_a = rec.scales[0];
      const char* sc_b = rec.scales[1];
      const char* sc_row[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        sc_row[i] = (gated && i >= 2 ? sc_b : sc_a) + static_cast<size_t>(rec.row0 + (gated ? (lane + 32 * i) & 63 : lane + 32 * i)) * row_bytes;
      {  // pull the item's scales towards L2, where the copies below find them
        for (int b = lane * 128; b < (gated ? ST_BOX_ROWS : 2 * ST_BOX_ROWS) * row_bytes && (phase == 0 || a.ksplit == 1); b += 32 * 128) {
          asm volatile("prefetch.global.L2 [%0];" ::"l"(sc_a + static_cast<size_t>(rec.row0) * row_bytes + b));
          if (gated) asm volatile("prefetch.global.L2 [%0];" ::"l"(sc_b + static_cast<size_t>(rec.row0) * row_bytes + b));
        }
      }
      if (fused && phase == 1 && rec.ai != ready_ai && last > 0) {
        // The codes of the stage are on their way; the hidden vectors may still be in the making on other
        // SMs.  (Every lane acquires the counter itself.)
        const int expect = a.row_blocks[0] * W;  // every consumer warp counts once per item
        const int* done = &recs[rec.ai].done;
        bool ready = false;
        for (unsigned i = 0; i < DEP_WAIT_LIMIT; ++i) {
          int v;
          asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(done) : "memory");
          ready = __all_sync(0xffffffffu, v >= expect);
          if (ready || __any_sync(0xffffffffu, *abort_flag)) break;
          __nanosleep(100);
        }
        if (!ready) {
          if (lane == 0) {
            *abort_flag = 1;
            atomicOr(a.check_word, CHECK_WAIT_TIMEOUT);
          }
          break;
        }
        asm volatile("fence.proxy.async.global;" ::: "memory");  // generic-proxy stores (global memory) -> bulk-copy reads
        ready_ai = rec.ai;
      }
      const int K = phase == 0 ? L.d_model : L.d_ff;
      const unsigned char* base = phase == 0 ? a.xs : a.hidden;
      for (int p0 = 0; p0 < cnt && ok; p0 += ACT_PASS_MAX) {
        const uint32_t xseg = act_seg_bytes(min(ACT_PASS_MAX, cnt - p0));
        const unsigned char* src = base + act_tile_offset(rec.begin + p0, K) + static_cast<size_t>(seg0) * xseg;
        for (int s = 0; s < nst; ++s, ++it) {
          const int slot = it % ST_SLOTS;
          if ((s > 0 || p0 > 0) &&
              !__all_sync(0xffffffffu, mbar_wait(bar_issued + 8 * slot, (it / ST_SLOTS) & 1, a.check_word, abort_flag))) {
            ok = false;
            break;
          }
          const uint32_t full = bar_full + 8 * slot;
          const int nseg = s == nst - 1 ? last : 8 / bits;
          if (nseg > 0) {
            const uint32_t st = smem_u32(ring + s_offset[slot]);
            if (lane == 0) {
              mbar_expect_tx(full, nseg * xseg);
              bulk_load(st + ST_X_OFFSET, src, nseg * xseg, full);
            }
            src += nseg * xseg;
            const int seg = seg0 + s * (8 / bits);
            const uint32_t dst = st + 2 * ST_BOX_BYTES + lane * 16;
            if constexpr (SC == SC_PAIRS) {  // one word, or two at 2 bits
              const int b0 = (seg * 2) & ~3;
#pragma unroll
              for (int i = 0; i < 4; ++i) cp_async4(dst + 512 * i, sc_row[i] + b0);
              if (nseg > 2) {
#pragma unroll
                for (int i = 0; i < 4; ++i) cp_async4(dst + 512 * i + 4, sc_row[i] + b0 + 4);
              }
            } else {  // the words that hold the stage's scales, from the 4-byte boundary at or below the first
              const int g0 = group_of_seg(a, seg) * ssz, g1 = (group_of_seg(a, seg + nseg - 1) + 1) * ssz;
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const char* from = reinterpret_cast<const char*>(reinterpret_cast<uintptr_t>(sc_row[i] + g0) & ~static_cast<uintptr_t>(3));
#pragma unroll 1
                for (int w = 0; from + w < sc_row[i] + g1; w += 4) cp_async4(dst + 512 * i + w, from + w);
              }
            }
            asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(full) : "memory");
          } else {
            mbar_arrive(full);
            if (lane == 0) mbar_arrive(full);
          }
        }
      }
    }
  } else {
    // ---------------- consumer warps ----------------
    const Pipe pp = {ring, hid_stage, queue, bar_full, bar_empty, bar_hid, recs, fused, abort_flag};
    // A finished first-projection item is counted one stage late: by then its stores have long
    // been acknowledged and the fence in front of the count costs nothing.  It is never held back
    // across a wait, because the stage waited for may be the one that waits for this count.
    Cursor cur = {0, 0, 0, -1};
    bool ok = true;
    for (int k = 0, p0 = 0; ok;) {
      const int slot = cur.it % ST_SLOTS;
      const uint32_t par = (cur.it / ST_SLOTS) & 1;
      if (cur.pending_ai >= 0 && !__all_sync(0xffffffffu, mbar_try_wait(bar_full + 8 * slot, par))) {
        count_item_done(recs, cur.pending_ai, lane);
        cur.pending_ai = -1;
      }
      if (!__all_sync(0xffffffffu, mbar_wait(bar_full + 8 * slot, par, a.check_word, abort_flag))) break;
      const ItemRec& rec = queue[k % ST_QUEUE];
      const int flags = rec.flags, cnt = rec.cnt;
      if (flags & ITEM_STOP) break;
      if (cnt - p0 <= 8) {
        switch (flags >> 8) {
          case 2: ok = consume_pass<2, SC, 1, W>(a, pp, k, p0, warp, lane, cur); break;
          case 4: ok = consume_pass<4, SC, 1, W>(a, pp, k, p0, warp, lane, cur); break;
          default: ok = consume_pass<8, SC, 1, W>(a, pp, k, p0, warp, lane, cur); break;
        }
      } else {
        switch (flags >> 8) {
          case 2: ok = consume_pass<2, SC, 2, W>(a, pp, k, p0, warp, lane, cur); break;
          case 4: ok = consume_pass<4, SC, 2, W>(a, pp, k, p0, warp, lane, cur); break;
          default: ok = consume_pass<8, SC, 2, W>(a, pp, k, p0, warp, lane, cur); break;
        }
      }
      p0 += ACT_PASS_MAX;
      if (p0 >= cnt) {
        p0 = 0;
        ++k;
      }
    }
    if (cur.pending_ai >= 0) count_item_done(recs, cur.pending_ai, lane);
  }
  if (*abort_flag) {
    // a wait ran out: give copies that may still be in flight time to land before the CTA's
    // shared memory is released
#pragma unroll 1
    for (int i = 0; i < 2000; ++i) __nanosleep(100);
  }
}

template <int SC, int W>
cudaError_t launch_sc(const TmaArgs& a, long long items, cudaStream_t st) {
  static int ctas_per_device[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!ctas_per_device[dev]) {
    e = cudaFuncSetAttribute(ffn_tma_kernel<SC, W>, cudaFuncAttributeMaxDynamicSharedMemorySize, ST_SMEM);
    if (e != cudaSuccess) return e;
    int per_sm = 0, sms = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ffn_tma_kernel<SC, W>, st_threads(W), ST_SMEM);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    ctas_per_device[dev] = (per_sm > 0 ? per_sm : 1) * sms;
  }
  const int grid = items < ctas_per_device[dev] ? static_cast<int>(items) : ctas_per_device[dev];
  return launch_chain(ffn_tma_kernel<SC, W>, dim3(grid), dim3(st_threads(W)), ST_SMEM, st, a);
}

}  // namespace

bool ffn_tma_supported(const LayerDims& L) {
  // tensor maps use 128-byte x 64-row boxes: every packed row must hold at least 128 bytes at
  // the narrowest width (2 bits)
  return ffn_mma_supported(L) && L.d_model >= 512 && L.d_ff >= 512 && L.d_model <= (1 << 17) && L.d_ff <= (1 << 17);
}

int ffn_tma_ksplit(const LayerDims& L, int T) {
  const int row_blocks = (L.d_model + 2 * ST_BOX_ROWS - 1) / (2 * ST_BOX_ROWS);
  const long long pairs = static_cast<long long>(T) * L.top_k;
  const long long active = pairs < L.E ? pairs : L.E;
  const long long ctas = row_blocks * active;
  const int steps_min = (L.d_ff + 511) / 512;  // stages at the widest span (2 bits)
  // enough slices that the second projection's items outnumber the resident CTAs (2 per SM)
  // several times: short items at the end of the launch keep its tail short
  long long z = (12 * GPU_SMS + ctas - 1) / ctas;
  // A handful of tokens leaves most SMs without an item: the slices are then cut as fine as the
  // 8-bit stages allow (narrower experts get empty slices, which only store zeros), so that the
  // second projection of the one or two activated experts is a short step on many SMs instead
  // of a chain of stages on a few.
  const int steps_max = (L.d_ff + 127) / 128;
  const int cap = ctas * 4 <= GPU_SMS ? steps_max : steps_min;
  if (z > cap) z = cap;
  if (z > 16) z = 16;
  // ... but not so fine that the items of both projections outnumber the resident CTAs where coarser slices would not: a
  // second item is a second chain of steps (12 tokens, 8 experts, 512 x 1152: 25 us per layer with nine slices, 21 with
  // seven; 24 tokens on 512 x 2048 28 and 22)
  const int rows0 = L.act == EMOE_ACT_SWIGLU ? ST_BOX_ROWS : 2 * ST_BOX_ROWS;
  const long long room = (ST_CTAS * GPU_SMS - active * ((L.d_ff + rows0 - 1) / rows0)) / ctas;
  if (z > room && room >= 2) z = room;
  if (z < 1) z = 1;
  return static_cast<int>(z);
}

cudaError_t launch_ffn_tma(int phase_begin, int phase_end, const LayerDims& L, const void* tmaps, const void* xs, int* plan,
                           void* hidden, float* o_part, int ksplit, int n_pairs, bool uneven, int* check_word, cudaStream_t st) {
  if (phase_begin < 0 || phase_end > 2 || phase_begin >= phase_end) return cudaErrorInvalidValue;
  const int rows_first = L.act == EMOE_ACT_SWIGLU ? ST_BOX_ROWS : 2 * ST_BOX_ROWS;
  TmaArgs a;
  a.phase_begin = phase_begin;
  a.phase_end = phase_end;
  a.L = L;
  a.tmaps = static_cast<const CUtensorMap*>(tmaps);
  a.xs = static_cast<const unsigned char*>(xs);
  a.plan = plan;
  a.hidden = static_cast<unsigned char*>(hidden);
  a.o_part = o_part;
  a.ksplit = ksplit;
  a.row_blocks[0] = L.d_ff / rows_first;
  a.row_blocks[1] = L.d_model / (2 * ST_BOX_ROWS);
  a.ngroups[0] = L.group > 0 ? L.d_model / L.group : 1;
  a.ngroups[1] = L.group > 0 ? L.d_ff / L.group : 1;
  a.gmul = L.group > 0 ? ((1u << 20) + static_cast<unsigned>(L.group / 128) - 1) / static_cast<unsigned>(L.group / 128) : 0u;
  a.n_pairs = n_pairs;
  a.claim_above = uneven ? 1 : 3;
  a.check_word = check_word;
  for (int p = 0; p < 2; ++p) {
    const int ks = p == 0 ? 1 : ksplit;
    a.mg_units[p] = div_magic(static_cast<uint32_t>(ks * a.row_blocks[p]));
    a.mg_ksplit[p] = div_magic(static_cast<uint32_t>(ks));
    a.mg_rb[p] = div_magic(static_cast<uint32_t>(a.row_blocks[p]));
  }
  const long long active_max = n_pairs < L.E ? n_pairs : L.E;
  long long per_expert = 0;
  if (phase_begin == 0) per_expert += a.row_blocks[0];
  if (phase_end == 2) per_expert += static_cast<long long>(a.row_blocks[1]) * ksplit;
  const long long items = active_max * per_expert;
  // Few tokens per activated expert: four warps with two tiles each, which read the activations once for both and meet a stage
  // half as often.  Passes of more than 8 tokens need the eight warps to hide their latencies, the sooner the shorter the rows, and an uneven
  // load has such passes at any mean.  So on rows below 1024 four warps only up to 16 pairs; beyond, for one token per 256
  // inputs less one on average, six at most.  us per layer, eight / four warps, even and skewed (Zipf exponent 1.1) loads: 512 x 2048, 16 experts,
  // 32 tokens 29.5/28.9 and 24.3/26.6; 768 x 3072, 32 experts, 12 tokens 36.0/34.8 and 30.5/29.8, 64 tokens 42.6/41.8 and 41.9/43.8;
  // 1024 x 4096, 64 experts, 128 tokens 90.1/86.0 and 72.5/74.5, 256 tokens 114/116 and 96.5/100; 1536 x 5632, 32 experts, 64 tokens
  // 89.1/86.1 and 68.1/69.9, 192 tokens 110/110 and 121/122; 2048 x 6144, 16 experts, 32 tokens 71.6/68.6 and 56.5/55.6, 80 tokens 79.5/78.6
  // and 76.2/76.2; 3072 x 8192 gated, 8 experts, two picks, 20 tokens 109/106 and 104/102.
  const int few_mean = L.d_model / 256 - 1 < 6 ? L.d_model / 256 - 1 : 6;
  const bool few = n_pairs <= (L.d_model < 1024 ? 16 : few_mean * active_max);
  if (!L.scale_f16) return few ? launch_sc<SC_F32, 4>(a, items, st) : launch_sc<SC_F32, 8>(a, items, st);
  const bool pairs = L.group == 128 && a.ngroups[0] % 2 == 0 && a.ngroups[1] % 2 == 0;
  if (pairs) return few ? launch_sc<SC_PAIRS, 4>(a, items, st) : launch_sc<SC_PAIRS, 8>(a, items, st);
  return few ? launch_sc<SC_F16, 4>(a, items, st) : launch_sc<SC_F16, 8>(a, items, st);
}

// Host-side tensor-map encoder (driver entry point looked up once; no link against libcuda).
// dtype: 0 = bytes, 1 = fp16.  2-D row-major image [outer][inner], box [box_outer][box_inner],
// 128-byte swizzle (box_inner * element size must be 128 bytes or less).
int encode_tmap_2d(void* out_map, int dtype, const void* base, uint64_t inner, uint64_t outer, uint64_t row_stride_bytes,
                   uint32_t box_inner, uint32_t box_outer, bool swizzle128) {
  typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                               const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                               CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static EncodeFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess || !p) return -1;
    fn = reinterpret_cast<EncodeFn>(p);
  }
  if (row_stride_bytes % 16 != 0 || (reinterpret_cast<uintptr_t>(base) & 15) != 0) return -2;
  const cuuint64_t dims[2] = {inner, outer};
  const cuuint64_t strides[1] = {row_stride_bytes};
  const cuuint32_t box[2] = {box_inner, box_outer};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = fn(static_cast<CUtensorMap*>(out_map), dtype == 1 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8,
                        2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        swizzle128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : -3;
}

// One tensor map per scale channel whose rows are a multiple of 16 bytes: a [N][row_bytes] byte image,
// boxes of 128 rows x 32 bytes, no swizzle (the int8 streaming kernel's scale windows).
int encode_scale_tmap(void* out_map, const void* scales, int N, int row_bytes) {
  if (row_bytes < 32 || row_bytes % 16 != 0 || N < 128) return -2;
  return encode_tmap_2d(out_map, 0, scales, static_cast<uint64_t>(row_bytes), static_cast<uint64_t>(N),
                        static_cast<uint64_t>(row_bytes), 32, 128, false);
}

// One tensor map per packed matrix: a [N][row_bytes] byte image, 64-row x 128-byte boxes, 128-byte swizzle.
int encode_weight_tmap(void* out_map, const void* packed, int N, int K, int bits) {
  const uint64_t row_bytes = static_cast<uint64_t>(K) * bits / 8;
  if (row_bytes < 128 || N < ST_BOX_ROWS) return -2;
  return encode_tmap_2d(out_map, 0, packed, row_bytes, static_cast<uint64_t>(N), row_bytes, 128, ST_BOX_ROWS);
}

}  // namespace emoe
