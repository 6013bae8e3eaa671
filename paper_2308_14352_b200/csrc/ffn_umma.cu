// Grouped expert GEMM on packed weights with tcgen05 tensor-core MMAs, for experts that hold
// many tokens (prefill, large decode batches).  Paper Sections 1/2.1 (each activated expert is
// an independent FFN) on the Section 3.2 storage (b-bit codes + scale channel, w~ = q * s).
//
// Shape of one work unit: 128 weight rows (UMMA M, "swap-AB": the weight rows are the M side; in a gated first
// projection 64 rows of w1 and the same 64 of w3, so that one pass over the inputs suffices) x a group of
// up to 320 tokens of one expert (N, accumulators in as many tensor-memory columns) x all inputs.  The
// dequantised A operand, the expensive part, is shared by the whole group, and it never touches
// shared memory: the dequantisation warps write it into TENSOR MEMORY (tcgen05.st, 32 columns per
// 64-input stage, a ring of four stages behind the accumulators) and the MMA takes it from there
// (the [a_tmem] operand form).  With A in shared memory too, the operand reads of the MMAs, the
// stores of the dequantisation and the TMA writes together asked for more than the 128 bytes per
// cycle an SM has.
//   warp 0    producer of the activations: boxes of 64 tokens x 64 inputs (fp16, K-major, 128-byte swizzle)
//             into a 4-deep ring;
//   warp 10   producer of the packed codes: boxes of 64 rows x 128 bytes (the decode kernel's tensor maps)
//             into a 3-deep ring.  A warp of its own: one thread feeding both rings asked for a box only
//             when the activations in front of it had found a free stage, and the dequantisation
//             waited for every box (a quarter of its time);
//   warps 2-9 two sets of four, a thread per weight row, taking turns at the steps: read the row's
//             packed bytes, dequantise to fp16 (code -> exact fp16 integer by mantissa insertion, then one
//             multiply by the group scale: |error| <= 2^-12 relative, the only approximation of
//             this path), and store the 64 values as 32 columns of the row's tensor-memory
//             lane; later the epilogue: tensor memory -> registers -> activation -> shared memory -> global
//             memory, where a thread writes 16 bytes of one token (gated: a w1 row and its w3 row lie 16 lanes apart in
//             one warp and swap halves by shuffles);
//   warps 11-18 (EXACT, see the kernel) scales and epilogue, two sets of four, while the others go on with the next unit;
//   warp 1    one thread issues tcgen05.mma (M128, N = the group's tokens rounded up to 16, in two halves
//             beyond 256, K16, fp16 x fp16 -> fp32) per 16 inputs and commits each stage back (EXACT: warp 19 every other one).
// A step costs two cycles per token in the tensor pipe and some 330 to 450 in the dequantisation, so groups of
// about 256 tokens and more are tensor-bound; an expert's tokens are split evenly (choose_cut, TileWalk).
// Measured (4096 x 14336 gated, 8 experts, 2048 tokens, 4 bits, both launches): 2040 us with one issuing lane in a branch
// and groups of whole 128-token tiles, 1053 us now: 1.37 PFLOP/s, 0.85 of the measured dense rate.  Few tokens are bound by
// what the roles of a CTA say to one another: an MMA of 16 to 32 tokens takes 19 to 23 cycles, its step some 450.
// Activations travel as fp16 (exact for bf16 values inside the fp16 range, saturated outside);
// the hidden vector is rounded to bf16 first, as the definition asks, then stored as fp16.
// The reduction index is enumerated in the order the unpack emits code pairs; the activation
// buffers are written in that same order (scatter.cuh, first-projection epilogue).
// Every wait is bounded (see pipe.cuh); tensor memory is always released before exit.
#include <cuda.h>

#include "common.cuh"
#include "ffn_tile.cuh"
#include "pipe.cuh"
#include "umma.cuh"

namespace emoe {
namespace {

constexpr int UM_ROWS = 128;               // weight rows per unit (UMMA M)
constexpr int UM_ROW = 64;                 // inputs of a 128-byte row of fp16
constexpr int UM_TILE_BYTES = 128 * 128;   // a [128 rows][128 B] packed tile
constexpr int UM_GROUP_TOK = 320;          // tokens that share one dequantised A stage, at most (accumulator columns)
constexpr int UM_OUT_BYTES = 32 * 128 * 2;  // hidden values of a set on their way out: 32 tokens x 128 channels (gated: two turns of 64)
constexpr int UM_EXACT_TOK = 64;           // EXACT: tokens of a group, at most
constexpr int UM_SETS = 4;                 // EXACT: sets of accumulators (two instead: 3 % more time)
constexpr int UM_CAPS = 4;                 // limits of a group that are considered: 128, 192, 256, 320 tokens
template <bool EXACT>
__host__ __device__ __forceinline__ constexpr int um_cap(int c) { return EXACT ? UM_EXACT_TOK : 128 + 64 * c; }
constexpr int UM_SCALE_SETS = 2;            // EXACT: sets of four warps for scales and epilogue: every other unit, or (SCALE_TOK
constexpr int UM_SCALE_TOK = 32;            // tokens, whose sums a thread holds, and more) half of the tokens each
constexpr int UM_SCALE_WARPS = 4 * UM_SCALE_SETS;
constexpr int UM_SCALE_AHEAD = 2;           // EXACT: scales of a row on their way
constexpr int UM_TMEM_COLS = 512;
// What the two forms of the kernel (see there) are made of
template <bool EXACT>
struct Um {
  static constexpr int SETS = 2;         // of four dequantising warps
  static constexpr int UNPACK_WARPS = 4 * SETS;
  static constexpr int RAW_WARP = 2 + UNPACK_WARPS;
  static constexpr int ISSUERS = EXACT ? 2 : 1;      // warp 1 and one behind the scaling warps
  static constexpr int ISSUER2 = RAW_WARP + 1 + (EXACT ? UM_SCALE_WARPS : 0);
  static constexpr int THREADS = (ISSUER2 + ISSUERS - 1) * 32;
  static constexpr int BK = EXACT ? 128 : 64;        // inputs per operand stage
  static constexpr int HALVES = BK / UM_ROW;
  static constexpr int STAGES = 4;                   // operand stages: A in tensor memory, B in shared memory
  static constexpr int A_COLS = BK / 2;              // an A stage, behind the accumulators
  static constexpr int RAW_STAGES = EXACT ? 8 : 3;
  static constexpr int BOX_TOK = EXACT ? 16 : 64;    // tokens per box of the activations' tensor map
  static constexpr int BOX_BYTES = BOX_TOK * 128;
  static constexpr int ACC_COLS = EXACT ? UM_SETS * UM_EXACT_TOK : UM_GROUP_TOK;
  static constexpr int B_HALF_BYTES = (EXACT ? UM_EXACT_TOK : UM_GROUP_TOK) * 128;
  static constexpr int B_STAGE_BYTES = HALVES * B_HALF_BYTES;
  static constexpr int OUT_SETS = EXACT ? UM_SCALE_SETS : SETS;  // sets of storing warps
  static constexpr int SMEM_BYTES = RAW_STAGES * UM_TILE_BYTES + STAGES * B_STAGE_BYTES + OUT_SETS * UM_OUT_BYTES + 1024;  // + alignment slack
};
static_assert(Um<false>::ACC_COLS + Um<false>::STAGES * Um<false>::A_COLS <= UM_TMEM_COLS && Um<true>::ACC_COLS + Um<true>::STAGES * Um<true>::A_COLS <= UM_TMEM_COLS, "tensor memory");
static_assert(Um<false>::SMEM_BYTES <= 227 * 1024 - 1024 && Um<true>::SMEM_BYTES <= 227 * 1024 - 1024, "shared memory");

// a / (1 + exp(-a)) without a branch, so that the 16 columns of a thread overlap (the operator's slow path
// kept them apart: 18000 cycles for 256 tokens x 64 channels, 10600 without): the approximate reciprocal, one product and
// Markstein's correction of the quotient by its remainder (IBM J. Res. Dev. 34, 1990).  The denominator is held
// below 2^126, where the reciprocal is still a normal number; an infinite a keeps the plain product.
__device__ __forceinline__ float silu_branchless(float a) {
  const float d = 1.0f + fminf(expf(-a), 8.507059173023462e37f);
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  const float q = a * r;
  const float c = fmaf(fmaf(-q, d, a), r, q);
  return c == c ? c : q;
}

// position of input k in the activation buffers of this path: the unpack emits the code pairs
// (c, c+4) of an 8-code word at 4 bits and (c, c+8) of a 16-code word at 2 bits
template <int BITS>
__device__ __forceinline__ int pair_pos(int k) {
  if (BITS == 8) return k;
  constexpr int B = BITS == 4 ? 8 : 16;
  const int o = k & (B - 1);
  return (k & ~(B - 1)) + (o < B / 2 ? 2 * o : 2 * (o - B / 2) + 1);
}
__device__ __forceinline__ int pair_pos_rt(int bits, int k) {
  return bits == 8 ? k : (bits == 4 ? pair_pos<4>(k) : pair_pos<2>(k));
}

__device__ __forceinline__ uint32_t h2_fma(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t r;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
}
__device__ __forceinline__ uint32_t h2_add(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ uint32_t h2_mul(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

// ---- dequantise one 16-byte chunk of a packed row to fp16 (q * s; EXACT: q), 8 values per output chunk ----
template <bool EXACT>
__device__ __forceinline__ uint32_t h2_scale(uint32_t q, uint32_t s2) { return EXACT ? q : h2_mul(q, s2); }
// 8 bits: 16 codes -> 2 chunks.  byte ^ 0x80 = q + 128 goes into the mantissa of 1024.
template <bool EXACT>
__device__ __forceinline__ void dequant_chunk8(const uint4& raw, uint32_t s2, uint4 (&out)[2]) {
  const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
  uint32_t o[8];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t u = w[i] ^ 0x80808080u;
    o[2 * i] = h2_scale<EXACT>(h2_add(prmt(u, 0x64646464u, 0x5140u), 0xE480E480u), s2);      // -(1024 + 128)
    o[2 * i + 1] = h2_scale<EXACT>(h2_add(prmt(u, 0x64646464u, 0x5342u), 0xE480E480u), s2);
  }
  out[0] = make_uint4(o[0], o[1], o[2], o[3]);
  out[1] = make_uint4(o[4], o[5], o[6], o[7]);
}
// 4 bits: one 8-code word -> one chunk, pair order (c, c+4).
template <bool EXACT>
__device__ __forceinline__ uint4 dequant_word4(uint32_t w, uint32_t s2) {
  const uint32_t hi = w >> 8;
  const uint32_t t0 = h2_add(and_xor(w, 0x000F000Fu, 0x64086408u), 0xE408E408u);               // v - 1032
  const uint32_t t1 = h2_fma(and_xor(w, 0x00F000F0u, 0x64806480u), 0x2C002C00u, 0xD480D480u);  // v/16 - 72
  const uint32_t t2 = h2_add(and_xor(hi, 0x000F000Fu, 0x64086408u), 0xE408E408u);
  const uint32_t t3 = h2_fma(and_xor(hi, 0x00F000F0u, 0x64806480u), 0x2C002C00u, 0xD480D480u);
  return make_uint4(h2_scale<EXACT>(t0, s2), h2_scale<EXACT>(t1, s2), h2_scale<EXACT>(t2, s2), h2_scale<EXACT>(t3, s2));
}
// 2 bits: one 16-code word -> two chunks, pair order (c, c+8).
template <bool EXACT>
__device__ __forceinline__ void dequant_word2(uint32_t w, uint32_t s2, uint4 (&out)[2]) {
  // field at mantissa bit p of 1024: v = 1024 + (q + 2) * 2^p;  q = v * 2^-p - (1024 * 2^-p + 2)
  const uint32_t msk[5] = {0x00030003u, 0x000C000Cu, 0x00300030u, 0x00C000C0u, 0x03000300u};
  const uint32_t mag[5] = {0x64026402u, 0x64086408u, 0x64206420u, 0x64806480u, 0x66006600u};
  const uint32_t mul[5] = {0x3C003C00u, 0x34003400u, 0x2C002C00u, 0x24002400u, 0x1C001C00u};
  const uint32_t add[5] = {0xE402E402u, 0xDC08DC08u, 0xD420D420u, 0xCC80CC80u, 0xC600C600u};
  uint32_t o[8];
  const uint32_t hi = w >> 10;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int p = c < 5 ? c : c - 5;
    o[c] = h2_scale<EXACT>(h2_fma(and_xor(c < 5 ? w : hi, msk[p], mag[p]), mul[p], add[p]), s2);
  }
  out[0] = make_uint4(o[0], o[1], o[2], o[3]);
  out[1] = make_uint4(o[4], o[5], o[6], o[7]);
}
// The 64 inputs of operand stage j of a packed row, two per register
template <int BITS, bool EXACT>
__device__ __forceinline__ void dequant_stage(const unsigned char* rrow, int rin, int j, uint32_t s2, uint32_t (&v)[32]) {
  if constexpr (BITS == 8) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      uint4 o[2];
      dequant_chunk8<EXACT>(*reinterpret_cast<const uint4*>(rrow + (((4 * j + c) ^ (rin & 7)) << 4)), s2, o);
      v[8 * c + 0] = o[0].x, v[8 * c + 1] = o[0].y, v[8 * c + 2] = o[0].z, v[8 * c + 3] = o[0].w;
      v[8 * c + 4] = o[1].x, v[8 * c + 5] = o[1].y, v[8 * c + 6] = o[1].z, v[8 * c + 7] = o[1].w;
    }
  } else if constexpr (BITS == 4) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const uint4 raw = *reinterpret_cast<const uint4*>(rrow + (((2 * j + c) ^ (rin & 7)) << 4));
      const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint4 o = dequant_word4<EXACT>(w[i], s2);
        v[16 * c + 4 * i + 0] = o.x, v[16 * c + 4 * i + 1] = o.y, v[16 * c + 4 * i + 2] = o.z, v[16 * c + 4 * i + 3] = o.w;
      }
    }
  } else {
    const uint4 raw = *reinterpret_cast<const uint4*>(rrow + ((j ^ (rin & 7)) << 4));
    const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      uint4 o[2];
      dequant_word2<EXACT>(w[i], s2, o);
      v[8 * i + 0] = o[0].x, v[8 * i + 1] = o[0].y, v[8 * i + 2] = o[0].z, v[8 * i + 3] = o[0].w;
      v[8 * i + 4] = o[1].x, v[8 * i + 5] = o[1].y, v[8 * i + 6] = o[1].z, v[8 * i + 7] = o[1].w;
    }
  }
}

struct UmmaArgs {
  int phase;
  LayerDims L;
  const CUtensorMap* wmaps;  // [E][3] packed-weight tensor maps (boxes of 64 rows x 128 bytes)
  int* plan;                 // header + PlanRec per activated expert
  __half* hidden16;          // first projection's output (fp16, pair order), rows hid_stride values apart
  int hid_stride;
  float* o;                  // second projection's output [n_pairs][d_model]
  int zmax;                  // second projection: most slices of the inputs per unit (slice z into plane z of o)
  int n_pairs;
  bool maybe_empty;          // the plan may well hold nobody
  size_t plane_stride;       // floats between the planes of o
  int* check_word;
};

// the work units of this CTA: linear index = blockIdx.x, += gridDim.x over
// (activated expert, group of tokens, row block[, slice of the inputs]) with the row block running fastest.  An
// expert's tokens are split evenly over as few groups as the accumulators allow: a last group with
// what full ones leave over would pay for the dequantisation of a whole one.
// Run by whole warps: the lanes hold the records of 32 experts and the sums of their units, so that the next unit costs a few
// shuffles.  (One expert after the other, each record asked for when the one in front had arrived, a step of 148 units over
// experts of 24 blocks was six trips to L2: 4000 cycles in front of every unit, for which nothing ran.)
// KEEP: the scale channels too; otherwise they are read when they are asked for (registers are short, and nobody waits).
template <bool KEEP>
struct TileWalk {
  const PlanRec* recs;
  int mat0, mat1;        // matrices of the projection (mat1: w3 of a gated one)
  const void *my_sp0, *my_sp1;
  int n_active, row_blocks, cap, z_log, lane;  // 2^z_log slices
  int lin;               // the next unit, from the chunk's first on
  int chunk;             // first of the 32 experts at hand
  int my_end, my_units;  // lane's expert: units up to and including it, its own
  int my_tok;            // tokens of its groups but the last: at most cap, which is a multiple of 16
  int my_e, my_begin, my_cnt, my_bits, owner;
  int e, begin, cnt, bits;  // of the unit at hand
  __device__ __forceinline__ void load_chunk(int limit) {
    const int i = chunk + lane;
    int4 r = make_int4(0, 0, 0, 0);
    if (i < limit) r = *reinterpret_cast<const int4*>(recs + i);
    my_e = r.x, my_begin = r.y, my_cnt = r.z, my_bits = r.w;
    if (KEEP && i < limit) {
      my_sp0 = recs[i].scales[mat0];
      my_sp1 = recs[i].scales[mat1];
    }
  }
  // asks for the first records beside their number
  __device__ __forceinline__ void open(const int* plan, int E, int m0, int m1) {
    mat0 = m0, mat1 = m1;
    my_sp0 = my_sp1 = nullptr;
    recs = reinterpret_cast<const PlanRec*>(reinterpret_cast<const char*>(plan) + PLAN_HEADER_BYTES);
    lane = threadIdx.x & 31;
    chunk = 0;
    n_active = *reinterpret_cast<const volatile int*>(plan);
    load_chunk(E);
    if (lane >= n_active) my_cnt = 0;  // what an earlier call left behind
  }
  __device__ __forceinline__ void sum_units() {
    const int groups = (my_cnt + cap - 1) / cap;
    my_tok = groups > 0 ? ((my_cnt + groups - 1) / groups + 15) & ~15 : 0;
    my_units = groups * row_blocks << z_log;
    my_end = my_units;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, my_end, o);
      if (lane >= o) my_end += v;
    }
  }
  __device__ __forceinline__ void start(int rb, int2 choice) {
    cap = choice.x;
    z_log = 31 - __clz(choice.y);
    row_blocks = rb;
    lin = blockIdx.x;
    sum_units();
  }
  // advances to the CTA's next unit (tok0 = its first token inside the expert, ntok = how many); false when there is none
  __device__ __forceinline__ bool next(int& tok0, int& ntok, int& rb, int& z) {
    __syncwarp();
    for (;;) {
      const int total = __shfl_sync(0xffffffffu, my_end, 31);
      if (lin < total) break;
      if (chunk + 32 >= n_active) return false;
      lin -= total;
      chunk += 32;
      load_chunk(n_active);
      sum_units();
    }
    owner = __ffs(__ballot_sync(0xffffffffu, my_end > lin)) - 1;
    int local = lin - __shfl_sync(0xffffffffu, my_end - my_units, owner);
    e = __shfl_sync(0xffffffffu, my_e, owner);
    begin = __shfl_sync(0xffffffffu, my_begin, owner);
    cnt = __shfl_sync(0xffffffffu, my_cnt, owner);
    bits = __shfl_sync(0xffffffffu, my_bits, owner);
    const int tok_group = __shfl_sync(0xffffffffu, my_tok, owner);
    int tt = 0;  // an expert has few groups: no division
    for (; local >= row_blocks << z_log; local -= row_blocks << z_log) ++tt;
    rb = local >> z_log;  // the slices of a row block lie next to each other
    z = local & ((1 << z_log) - 1);
    tok0 = tt * tok_group;
    ntok = max(0, min(tok_group, cnt - tok0));  // (rounding to 16 may leave the last of many groups without tokens)
    lin += gridDim.x;
    return true;
  }
  // scale channel of the expert's first or second matrix (whole warps; `other` may differ from lane to lane)
  __device__ __forceinline__ const char* scales(bool other) const {
    if (!KEEP) return static_cast<const char*>(recs[chunk + owner].scales[other ? mat1 : mat0]);
    const unsigned long long p0 = __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(my_sp0), owner);
    const unsigned long long p1 = __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(my_sp1), owner);
    return reinterpret_cast<const char*>(other ? p1 : p0);
  }
};

// How a launch is cut (every warp works it out for itself): most tokens of a group, slices of the second projection's inputs.  Larger groups share
// the dequantisation, smaller ones and slices fill the last round of CTAs.  The estimate, in cycles: a
// step of 64 inputs takes two per token or the 330 of the dequantisation (EXACT: 500 for one of 128), a unit 1500 + 12
// per token to start and store; a further plane of sums costs the combine step its bandwidth (3400 B per cycle).
template <bool EXACT>
__device__ __forceinline__ int2 choose_cut(const UmmaArgs& a, const TileWalk<!EXACT>& walk, int row_blocks, int kb_total) {
  int groups[UM_CAPS] = {}, tokens = 0;
  for (int i = walk.lane; i < max(walk.n_active, 32); i += 32) {
    const int cnt = i < 32 ? walk.my_cnt : walk.recs[i].cnt;
    tokens += cnt;
#pragma unroll
    for (int c = 0; c < UM_CAPS; ++c) groups[c] += (cnt + um_cap<EXACT>(c) - 1) / um_cap<EXACT>(c);
  }
  tokens = __reduce_add_sync(0xffffffffu, tokens);
  int2 best = make_int2(um_cap<EXACT>(0), 1);
  float best_cost = 3.0e38f;
#pragma unroll
  for (int c = 0; c < (EXACT ? 1 : UM_CAPS); ++c) {
    const int g = __reduce_add_sync(0xffffffffu, groups[c]);
    const float tok = static_cast<float>(tokens) / static_cast<float>(max(g, 1));
    for (int z = 1; z <= a.zmax; z *= 2) {
      if (z > 1 && (kb_total % z != 0 || kb_total / z % (512 / Um<EXACT>::BK) != 0)) break;  // a slice starts on a packed box at every width
      const int rounds = (g * row_blocks * z + static_cast<int>(gridDim.x) - 1) / static_cast<int>(gridDim.x);
      const float steps = static_cast<float>(kb_total / z) * fmaxf(EXACT ? 500.0f : 330.0f, 2.0f * tok);
      const float unit = EXACT ? steps + 1000.0f : steps + 1500.0f + 12.0f * tok;
      const float cost = static_cast<float>(rounds) * unit + static_cast<float>(z - 1) * static_cast<float>(tokens) * static_cast<float>(a.L.d_model) * (8.0f / 3400.0f);
      if (cost < best_cost) {
        best_cost = cost;
        best = make_int2(um_cap<EXACT>(c), z);
      }
    }
  }
  return best;
}

// where a dequantisation warp stands in the rings
struct RingPos {
  int raw_it, ab_it;
  int next;  // steps from ab_it to the set's next one
};
// The accumulators of a CTA's n-th run of MMAs: a unit, or (EXACT) one scale group of a unit, UM_SETS of which have columns of
// their own in turn.
template <bool EXACT>
struct AccSlot {
  int index, parity, col;
  __device__ __forceinline__ explicit AccSlot(int n) {
    index = EXACT ? n % UM_SETS : 0;
    parity = EXACT ? (n / UM_SETS) & 1 : n & 1;
    col = index * UM_EXACT_TOK;
  }
};
struct UmBars {
  uint32_t raw_full, raw_empty, ab_full, ab_empty, acc_full, acc_empty;
};

// One unit's steps by a dequantisation warp (the sets take turns at the steps of a CTA).  srow: the row's scales from the
// unit's first step on, spg steps per scale.
template <int BITS, bool EXACT>
__device__ __forceinline__ bool dequant_unit(const UmmaArgs& a, const UmBars& b, const unsigned char* raw_ring, uint32_t a_col, const void* sp,
                                             size_t srow, int ngroups, int spg, int kb0, int kb_len, int box, int rin, uint32_t on, RingPos& pos,
                                             volatile int* abort_flag) {
  using U = Um<EXACT>;
  constexpr int KBS = (1024 / BITS) / U::BK;  // steps per box
  const bool sf16 = a.L.scale_f16 != 0;
  // scales of this set's step, its next one and the one after: a load has two steps to come back from L2; the group
  // index of the step two ahead is kept by counting
  const int first = kb0 + pos.next;
  float sv = 1.0f, sv_n1 = 1.0f, sv_n2 = 1.0f;  // EXACT: the codes alone, whole numbers
  if (!EXACT) {
    sv = load_scale_ro(sp, sf16, srow + min(first / spg, ngroups - 1));
    sv_n1 = load_scale_ro(sp, sf16, srow + min((first + U::SETS) / spg, ngroups - 1));
  }
  int g2 = (first + 2 * U::SETS) / spg, c2 = (first + 2 * U::SETS) % spg;
  bool tiny_scale = false;  // q * s below the smallest normal fp16 number would lose bits in the fp16 operand
  for (int kb = 0; kb < kb_len; kb += KBS) {
    const int rs = pos.raw_it % U::RAW_STAGES;
    if (!mbar_wait_warp(b.raw_full + 8 * rs, (pos.raw_it / U::RAW_STAGES) & 1, a.check_word, abort_flag)) return false;
    const unsigned char* rrow = raw_ring + rs * UM_TILE_BYTES + box * (UM_TILE_BYTES / 2) + rin * 128;
    const int steps = min(KBS, kb_len - kb);
    int j = pos.next;
#pragma unroll 1
    for (; j < steps; j += U::SETS) {
      const int it = pos.ab_it + j, s = it % U::STAGES;
      if (!EXACT) {
        sv_n2 = load_scale_ro(sp, sf16, srow + min(g2, ngroups - 1));
        c2 += U::SETS;
        if (c2 >= spg) {
          c2 -= spg;
          ++g2;
        }
      }
      tiny_scale |= sv != 0.0f && fabsf(sv) < 6.104e-5f;
      const uint32_t s2 = static_cast<uint32_t>(__half_as_ushort(__float2half_rn(sv))) * 0x00010001u;
      uint32_t v[32];
      dequant_stage<BITS, EXACT>(rrow, rin, j * U::HALVES, s2, v);  // while the stage may still be in use
      if (!mbar_wait_warp(b.ab_empty + 8 * s, ((it / U::STAGES) & 1) ^ 1, a.check_word, abort_flag)) return false;
      tc_fence_after();  // the MMAs that read this stage's columns are complete
      tmem_st32(a_col + s * U::A_COLS, v);
      if constexpr (U::HALVES == 2) {
        dequant_stage<BITS, EXACT>(rrow, rin, j * 2 + 1, s2, v);
        tmem_st32(a_col + s * U::A_COLS + UM_ROW / 2, v);
      }
      tmem_st_wait();
      sv = sv_n1;
      sv_n1 = sv_n2;
      tc_fence_before();
      mbar_arrive_if(on, b.ab_full + 8 * s);  // (the wait in front keeps the warp together)
    }
    pos.next = j - steps;
    pos.ab_it += steps;
    __syncwarp();
    mbar_arrive_if(on, b.raw_empty + 8 * rs);
    ++pos.raw_it;
  }
  if (tiny_scale) atomicOr(a.check_word, CHECK_F16_RANGE);
  return true;
}

// The four storing warps of a set meet at barriers of their own (the hidden values change hands between them), so they
// have to leave together: each warp's waits may end differently once another role has given up, and a warp that had
// left would keep its neighbours at the next barrier for ever.  So they vote once per unit, behind its last wait.
// (4096 x 14336 gated, 2048 tokens: 1400 us per call with the vote and without; 1450 where the result is not known to be
// the same in every lane.)
__device__ __forceinline__ bool set_agrees(int part, bool ok) {
  uint32_t all;
  __syncwarp();
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, %2, 128, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
               : "=r"(all)
               : "r"(static_cast<uint32_t>(ok)), "r"(1 + part)
               : "memory");
  return __all_sync(0xffffffffu, all != 0);
}
__device__ __forceinline__ void set_sync(int part) { asm volatile("bar.sync %0, 128;" ::"r"(1 + part) : "memory"); }

// EXACT: A holds the codes themselves, whole numbers that fp16 holds exactly; eight more warps take the sums of each scale
// group out of tensor memory and add them, times the row's scale, in fp32 registers, as the streaming kernel does.
// Groups of up to 64 tokens, four sets of accumulators in turn, steps of 128 inputs (the usual scale group).  What bounds it is the
// hand-over between the roles, hence: two issuing warps; every other unit to the other set of scaling warps, whose
// epilogue then hides behind the next unit; two runs read at a time; scales asked for two groups ahead; activations in boxes of 16
// tokens (boxes of 64 were four times the L2 traffic at few tokens).  Its 20 warps leave 96 registers a thread, of which 40 bytes
// spill (none in the rounded form's 142).  One set of scaling warps of 64 tokens each: 10 us more at 4096 x
// 14336 and at 768 x 3072 alike; three sets of dequantising warps: nothing.
// us per layer, before -> after: 768 x 3072, 32 experts, 512 tokens 84.7 -> 65.9, 777 tokens 90.7 -> 74.5, 2048 tokens 121 -> 99
// (and 64.9 and 90 with the early start of the second projection); Mixtral-like layer, 23 tokens 440 -> 242 (231).
template <bool EXACT>
__global__ void __launch_bounds__(Um<EXACT>::THREADS, 1)
    ffn_umma_kernel(const UmmaArgs a, const __grid_constant__ CUtensorMap tmap_b) {
  using U = Um<EXACT>;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bars[2 * U::RAW_STAGES + 2 * U::STAGES + (1 + UM_SCALE_SETS) * UM_SETS];
  __shared__ uint32_t tmem_base_slot;
  __shared__ int wait_words[PIPE_WORDS];
  volatile int* abort_flag = wait_words + PIPE_ABORT;
  // an offset from the array, not a rounded address: the compiler then knows that every access is to shared memory
  unsigned char* raw_ring = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char* b_ring = raw_ring + U::RAW_STAGES * UM_TILE_BYTES;
  const int lane = threadIdx.x & 31, warp = uniform_warp();

  if (a.maybe_empty) {  // nobody is full enough, the common case of an even load: gone before anything is set up
    pdl_trigger();  // (the kernel behind waits for this one's end, and with it for the one in front)
    pdl_wait();
    if (*reinterpret_cast<const volatile int*>(a.plan) == 0) return;
  }
  UmBars b;
  b.raw_full = smem_u32(bars);
  b.raw_empty = b.raw_full + 8 * U::RAW_STAGES;
  b.ab_full = b.raw_empty + 8 * U::RAW_STAGES;
  b.ab_empty = b.ab_full + 8 * U::STAGES;
  b.acc_full = b.ab_empty + 8 * U::STAGES;
  b.acc_empty = b.acc_full + 8 * UM_SCALE_SETS * UM_SETS;

  if (threadIdx.x == 0) {
    wait_words[PIPE_ABORT] = 0;
    wait_words[PIPE_FRONT] = a.phase != 0;
    for (int s = 0; s < U::RAW_STAGES; ++s) {
      mbar_init(b.raw_full + 8 * s, 1);
      mbar_init(b.raw_empty + 8 * s, U::UNPACK_WARPS);
    }
    for (int s = 0; s < U::STAGES; ++s) {
      mbar_init(b.ab_full + 8 * s, 1 + 4);  // the activations' producer (+ bytes) and the set that fills A
      mbar_init(b.ab_empty + 8 * s, 1);
    }
    for (int i = 0; i < UM_SETS; ++i) {
      for (int h = 0; h < UM_SCALE_SETS; ++h) mbar_init(b.acc_full + 8 * (UM_SETS * h + i), 1);
      mbar_init(b.acc_empty + 8 * i, EXACT ? UM_SCALE_WARPS : U::UNPACK_WARPS);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(smem_u32(&tmem_base_slot), UM_TMEM_COLS);  // accumulators + four A stages
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_slot;
  // Barrier set-up and the tensor-memory allocation overlap the kernel in front.  The second projection needs nothing of the first
  // but its hidden values: the plan was complete before the first started (it waits itself before it lets this one in), so only
  // the producer of the activations waits, and codes, scales and dequantisation are under way where the first has left an SM
  // (768 x 3072, 32 experts, 777 tokens: 72.8 -> 64.9 us per layer; Mixtral-like layer, 64 tokens 257 -> 241).
  // (where the plan may be empty, everybody has waited above, in both launches)
  if (a.phase == 0) pdl_wait();
  else __threadfence();  // nothing that an earlier kernel left in this SM's L1 is taken for the plan
  pdl_trigger();

  const LayerDims& L = a.L;
  const int N = a.phase == 0 ? L.d_ff : L.d_model;
  const int K = a.phase == 0 ? L.d_model : L.d_ff;
  const bool gated = a.phase == 0 && L.act == EMOE_ACT_SWIGLU;
  const int mat_first = a.phase == 0 ? 0 : (L.act == EMOE_ACT_SWIGLU ? 2 : 1);
  const int row_blocks = gated ? N / (UM_ROWS / 2) : (N + UM_ROWS - 1) / UM_ROWS;
  const int kb_total = K / U::BK;

  TileWalk<!EXACT> walk;
  walk.open(a.plan, L.E, mat_first, gated ? 1 : mat_first);
  const int2 cut = choose_cut<EXACT>(a, walk, row_blocks, kb_total);
  if (a.phase == 1 && blockIdx.x == 0 && threadIdx.x == 0) a.plan[3] = cut.y;  // for the combine step
  const int spg = (L.group > 0 ? L.group : K) / U::BK;  // steps per scale: a group is a multiple of 128 inputs, or the whole row
  const int kb_len = kb_total / cut.y;  // steps of a unit
  walk.start(row_blocks, cut);
  int tok_first, ntok, rb, z;

  if (warp == 0) {
    // ---------------- producer of the activations ----------------
    if (a.phase != 0) {
      pdl_wait();
      if (lane == 0) abort_flag[PIPE_FRONT] = 0;
    }
    const uint32_t on = elect_one();
    int it = 0;
    bool ok = true;
    while (ok && walk.next(tok_first, ntok, rb, z)) {
      const int tok0 = walk.begin + tok_first;
      const int boxes = (ntok + U::BOX_TOK - 1) / U::BOX_TOK;
      for (int kb = z * kb_len; kb < (z + 1) * kb_len; ++kb, ++it) {
        const int s = it % U::STAGES;
        if (!mbar_wait_warp(b.ab_empty + 8 * s, ((it / U::STAGES) & 1) ^ 1, a.check_word, abort_flag)) {
          ok = false;
          break;
        }
        const uint32_t full = b.ab_full + 8 * s;
        mbar_expect_tx_if(on, full, U::HALVES * boxes * U::BOX_BYTES);
        for (int t = 0; t < boxes; ++t)
#pragma unroll
          for (int h = 0; h < U::HALVES; ++h)
            tma_load_2d_if(on, smem_u32(b_ring + s * U::B_STAGE_BYTES + h * U::B_HALF_BYTES + t * U::BOX_BYTES), &tmap_b, kb * U::BK + h * UM_ROW,
                           tok0 + t * U::BOX_TOK, full);
      }
    }
  } else if (warp == U::RAW_WARP) {
    // ---------------- producer of the packed codes ----------------
    const uint32_t on = elect_one();
    int it = 0;
    bool ok = true;
    while (ok && walk.next(tok_first, ntok, rb, z)) {
      const CUtensorMap* map0 = a.wmaps + static_cast<size_t>(walk.e) * 3 + mat_first;
      const CUtensorMap* map1 = gated ? map0 + 1 : map0;  // second box: w3, or the next 64 rows
      const int row0 = rb * (gated ? 64 : 128), row1 = gated ? row0 : row0 + 64;
      const int kbs = (1024 / walk.bits) / U::BK;  // steps per box (128 bytes of a row)
      const int kb_end = (z + 1) * kb_len;
      int c0 = z * kb_len / kbs * 128;
      for (int kb = z * kb_len; kb < kb_end; kb += kbs, ++it, c0 += 128) {
        const int s = it % U::RAW_STAGES;
        if (!mbar_wait_warp(b.raw_empty + 8 * s, ((it / U::RAW_STAGES) & 1) ^ 1, a.check_word, abort_flag)) {
          ok = false;
          break;
        }
        const uint32_t full = b.raw_full + 8 * s;
        mbar_expect_tx_if(on, full, UM_TILE_BYTES);
        const uint32_t dst = smem_u32(raw_ring + s * UM_TILE_BYTES);
        tma_load_2d_if(on, dst, map0, c0, row0, full);
        tma_load_2d_if(on, dst + UM_TILE_BYTES / 2, map1, c0, row1, full);
      }
      if (z == 0) {  // this warp is some boxes ahead: pull the unit's scales towards L2
        const int row_bytes = K / (L.group > 0 ? L.group : K) * (L.scale_f16 ? 2 : 4);
        const int bytes = min(gated ? 64 : 128, N - row0) * row_bytes;
        const char* sc0 = walk.scales(false) + static_cast<size_t>(row0) * row_bytes;
        const char* sc1 = walk.scales(true) + static_cast<size_t>(row0) * row_bytes;
        for (int i = lane * 128; i < bytes; i += 32 * 128) {
          asm volatile("prefetch.global.L2 [%0];" ::"l"(sc0 + i));
          if (gated) asm volatile("prefetch.global.L2 [%0];" ::"l"(sc1 + i));
        }
        __syncwarp();
      }
    }
  } else if (warp == 1 || (EXACT && warp == U::ISSUER2)) {
    // ---------------- MMA issuers ----------------
    // kind::f16, fp16 x fp16 -> fp32, A from tensor memory, B K-major from shared memory, M = 128; N = the unit's tokens
    // rounded up to 16, in two halves where they are more than one MMA takes.
    // The predicate of every MMA is elect's own: combined with any other condition it may mean several lanes, which
    // the compiler then serves one after the other (62 to 90 cycles per MMA; 27 as it stands).
    const uint32_t on = elect_one();
    const uint32_t idesc = (1u << 4) | ((UM_ROWS >> 4) << 24);
    const uint32_t tmem = static_cast<uint32_t>(warp_uniform(static_cast<int>(tmem_base)));
    const int len = warp_uniform(kb_len), group_len = EXACT ? warp_uniform(spg) : len;
    // EXACT, one step per scale: two issuers take every other step, because what a step costs beside its MMAs (waits, commits) is
    // twice the MMAs.  Both are then within STAGES steps of each other; with more steps per scale they would not
    // be, a barrier's parity could mean another phase, and one does them all.
    const uint32_t turns = EXACT && group_len == 1 ? U::ISSUERS : 1, turn = warp == 1 ? 0 : 1;
    uint32_t s = turn, s_par = 0, acc = EXACT ? turn : 0, acc_par = 1, unit = 0;
    int kb = turn;
    bool ok = turn < turns;
    while (ok && warp_uniform(walk.next(tok_first, ntok, rb, z))) {
      const int cols = warp_uniform((ntok + 15) & ~15);
      const int n1 = cols <= 256 ? cols : ((cols / 2 + 15) & ~15), n2 = cols - n1;
      const uint32_t id1 = idesc | ((n1 >> 3) << 17), id2 = idesc | ((n2 >> 3) << 17);
      const bool both = EXACT && cols > UM_SCALE_TOK;
      const uint32_t full = b.acc_full + (EXACT && !both ? 8 * UM_SETS * (unit & 1) : 0);
      ++unit;
      int left = EXACT ? warp_uniform(group_len - z * kb_len % spg) : len;  // steps to the end of the scale group
      bool fresh = true;                                                    // the accumulators start anew
      for (; kb < len; kb += turns) {
        const uint32_t d_t = tmem + acc * UM_EXACT_TOK;
        if (fresh) {
          ok = mbar_wait_warp(b.acc_empty + 8 * acc, acc_par, a.check_word, abort_flag);
          if (!ok) break;
        }
        ok = mbar_wait_warp(b.ab_full + 8 * s, s_par, a.check_word, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint32_t a_t = tmem + U::ACC_COLS + s * U::A_COLS;
        const uint32_t bs = smem_u32(b_ring) + s * U::B_STAGE_BYTES;
        if (n1 > 0) {
#pragma unroll
          for (int k4 = 0; k4 < U::BK / 16; ++k4)  // 16 inputs: 8 columns of A, 32 bytes (2 descriptor units) of B
            umma_f16_ts_if(on, d_t, a_t + 8 * k4, umma_desc(bs + k4 / 4 * U::B_HALF_BYTES) + 2 * (k4 % 4), id1, k4 > 0 || !fresh ? 1u : 0u);
        }
        if (!EXACT && n2 > 0) {
#pragma unroll
          for (int k4 = 0; k4 < U::BK / 16; ++k4)
            umma_f16_ts_if(on, d_t + n1, a_t + 8 * k4, umma_desc(bs + n1 * 128) + 2 * k4, id2, k4 > 0 || !fresh ? 1u : 0u);
        }
        umma_commit_if(on, b.ab_empty + 8 * s);  // the stage may be refilled once these MMAs have read it
        s = (s + turns) % U::STAGES;
        s_par ^= s < turns;
        fresh = --left == 0 || kb + 1 == len;
        if (fresh) {
          umma_commit_if(on, full + 8 * acc);
          if (both) umma_commit_if(on, full + 8 * (UM_SETS + acc));
          left = group_len;
          acc = EXACT ? (acc + turns) % UM_SETS : 0;
          acc_par ^= acc < turns;
        }
      }
      kb -= len;
    }
  } else {
    // ---------------- dequantise (a thread per weight row) and epilogue ----------------
    const int quarter = warp & 3;          // TMEM lanes this warp may access: 32 * quarter ...
    const int r = 32 * quarter + lane;     // row of the tile = row of the operand = TMEM lane
    const int G = L.group > 0 ? L.group : K;
    const int ngroups = K / G;
    const uint32_t lane_base = tmem_base + (static_cast<uint32_t>(32 * quarter) << 16);
    // gated: the upper 16 lanes of a warp hold the w3 rows that belong to the w1 rows of the lower 16
    const bool second = gated && lane >= 16;
    const int rin = gated ? 16 * quarter + (lane & 15) : r & 63, box = gated ? lane >> 4 : r >> 6;  // row in which packed box
    const uint32_t on = elect_one();
    // dequantises the unit at hand; nrow: the thread's output channel
    RingPos pos = {0, 0, (warp - 2) >> 2};
    auto dequant = [&](const void* sp, size_t srow) {
      const uint32_t a_col = lane_base + U::ACC_COLS;
      switch (walk.bits) {
        case 2: return dequant_unit<2, EXACT>(a, b, raw_ring, a_col, sp, srow, ngroups, spg, z * kb_len, kb_len, box, rin, on, pos, abort_flag);
        case 4: return dequant_unit<4, EXACT>(a, b, raw_ring, a_col, sp, srow, ngroups, spg, z * kb_len, kb_len, box, rin, on, pos, abort_flag);
        default: return dequant_unit<8, EXACT>(a, b, raw_ring, a_col, sp, srow, ngroups, spg, z * kb_len, kb_len, box, rin, on, pos, abort_flag);
      }
    };
    if (EXACT && warp < U::RAW_WARP) {
      while (walk.next(tok_first, ntok, rb, z) && dequant(nullptr, 0)) {}
    } else {
    const int part = EXACT ? (warp - U::RAW_WARP - 1) >> 2 : (warp - 2) >> 2;  // the set of storing warps
    unsigned char* out_stage = b_ring + U::STAGES * U::B_STAGE_BYTES + part * UM_OUT_BYTES;
    const int set_tid = 32 * quarter + lane;
    int turn = 0;  // gated: the half of the buffer
    int run_it = 0, unit = 0;
    uint32_t full_bits = 0;  // EXACT: the parity at which the set expects each accumulator
    for (; walk.next(tok_first, ntok, rb, z); ++unit) {
      const bool both = EXACT && ntok > UM_SCALE_TOK;
      if (EXACT && !both && (unit & 1) != part) {  // the other set's
        run_it += (z * kb_len % spg + kb_len + spg - 1) / spg;
        continue;
      }
      const int bits = walk.bits;
      const int nrow = gated ? rb * 64 + rin : rb * UM_ROWS + r;  // output channel
      const size_t srow = static_cast<size_t>(min(nrow, N - 1)) * ngroups;
      const void* sp = walk.scales(second);
      const int kb0 = z * kb_len;
      bool ok = true;
      if constexpr (!EXACT) ok = dequant(sp, srow);
      // ---- epilogue: this warp's 32 rows x its set's share of the chunks of 32 token columns (EXACT: all of them) ----
      uint32_t tot[32];  // EXACT: the scaled sums of the set's tokens
      int acc_index = 0;
      const int set_col = both ? UM_SCALE_TOK * part : 0;
      if constexpr (EXACT) {
        float* f = reinterpret_cast<float*>(tot);
#pragma unroll
        for (int c = 0; c < UM_SCALE_TOK; ++c) f[c] = 0.0f;
        // scales on their way: the loads of a warp's rows touch 32 lines and take as long as a run or more, and the slowest of
        // eight warps counts
        const bool sf16 = L.scale_f16 != 0;
        uint32_t q[UM_SCALE_AHEAD];
        int gi = kb0 / spg;
        auto ask = [&]() {
          const size_t at = srow + min(gi++, ngroups - 1);
          return sf16 ? static_cast<uint32_t>(__ldg(static_cast<const unsigned short*>(sp) + at)) : __ldg(static_cast<const uint32_t*>(sp) + at);
        };
#pragma unroll
        for (int i = 0; i < UM_SCALE_AHEAD; ++i) q[i] = ask();
        int left = spg - kb0 % spg;  // steps to the end of the scale group
        int kb = kb0;
        const int kb_end = kb0 + kb_len;
        auto full = [&](int n) {
          const AccSlot<EXACT> acc(n);
          const bool there = mbar_wait_warp(b.acc_full + 8 * (acc.index + UM_SETS * part), (full_bits >> acc.index) & 1, a.check_word, abort_flag);
          full_bits ^= 1u << acc.index;
          return there;
        };
        auto scale_of = [&](uint32_t raw) { return sf16 ? __half2float(__ushort_as_half(static_cast<unsigned short>(raw))) : __uint_as_float(raw); };
        // two runs at a time: waiting, reading and giving back take a warp some 500 cycles whether it is for one or two
        while (kb < kb_end) {
#pragma unroll
          for (int i = 0; i < UM_SCALE_AHEAD; i += 2) {
            if (kb >= kb_end) break;
            const bool two = kb + left < kb_end;
            ok = full(run_it) && (!two || full(run_it + 1));
            if (!ok) break;
            tc_fence_after();
            const AccSlot<EXACT> acc0(run_it), acc1(run_it + (two ? 1 : 0));
            const float sv0 = scale_of(q[i]), sv1 = two ? scale_of(q[i + 1]) : 0.0f;
            q[i] = ask();
            q[i + 1] = ask();
#pragma unroll
            for (int h = 0; h < UM_SCALE_TOK / 16; ++h) {
              if (set_col + 16 * h < ntok) {
                uint32_t va[16], vb[16];
                tmem_ld16(lane_base + acc0.col + set_col + 16 * h, va);
                tmem_ld16(lane_base + acc1.col + set_col + 16 * h, vb);
                tmem_ld_wait();
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                  f[16 * h + c] = fmaf(sv0, __uint_as_float(va[c]), f[16 * h + c]);
                  if (two) f[16 * h + c] = fmaf(sv1, __uint_as_float(vb[c]), f[16 * h + c]);
                }
              }
            }
            tc_fence_before();
            const int arrivals = both ? 1 : UM_SCALE_SETS;
            mbar_arrive_if(on, b.acc_empty + 8 * acc0.index, arrivals);
            if (two) mbar_arrive_if(on, b.acc_empty + 8 * acc1.index, arrivals);
            kb += left + (two ? spg : 0);
            left = spg;
            run_it += two ? 2 : 1;
          }
          if (!ok) break;
        }
      } else {
        const AccSlot<EXACT> acc(run_it);
        acc_index = acc.index;
        ok = mbar_wait_warp(b.acc_full + 8 * acc.index, acc.parity, a.check_word, abort_flag) && ok;
        tc_fence_after();
      }
      if (!set_agrees(part, ok)) break;  // no bounded wait from here to the end of the unit
      const size_t slot0 = static_cast<size_t>(walk.begin) + static_cast<size_t>(tok_first);
      const int u_row0 = rb * (gated ? 64 : UM_ROWS);  // first channel of the unit
      const int hpos = a.phase == 0 ? pair_pos_rt(bits, nrow) : 0;  // (moves a channel inside its 16)
      auto store_chunk = [&](int cc, uint32_t(&va)[32]) {
        const int live = min(32, ntok - cc);  // token columns of this chunk that exist
        // one compact unrolled loop per case (the conditions are uniform)
        if (gated) {
          // the lanes of a w1 row and of its w3 row swap halves: the first computes columns 0..15, the second 16..31
          const int c0 = second ? 16 : 0;
          unsigned char* stage = out_stage + turn * (UM_OUT_BYTES / 2);  // [32 tokens][64 channels], 64-byte halves swapped from token 16 on
          unsigned char* mine = stage + c0 * 128 + (((hpos - u_row0) * 2) ^ (second ? 64 : 0));
          bool beyond = false;
#pragma unroll
          for (int b4 = 0; b4 < 16; b4 += 4) {
            if (b4 < live) {
#pragma unroll
              for (int c = b4; c < b4 + 4; ++c) {
                const uint32_t other = __shfl_xor_sync(0xffffffffu, second ? va[c] : va[16 + c], 16);
                const float av = __uint_as_float(second ? other : va[c]), bv = __uint_as_float(second ? va[16 + c] : other);
                // the hidden vector is a bf16 tensor
                const float h = __bfloat162float(__float2bfloat16_rn(silu_branchless(av) * bv));
                beyond |= c0 + c < live && beyond_f16(h);  // columns past the last token read whatever lies behind it
                *reinterpret_cast<__half*>(mine + c * 128) = __float2half_rn(fminf(fmaxf(h, -65504.0f), 65504.0f));
              }
            }
          }
          if (beyond) atomicOr(a.check_word, CHECK_F16_RANGE);  // saturated above: reported, not silent
          set_sync(part);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int tok = (set_tid >> 3) + 16 * i, piece = set_tid & 7;
            if (tok < live)
              *reinterpret_cast<uint4*>(a.hidden16 + (slot0 + cc + tok) * a.hid_stride + u_row0 + 8 * piece) =
                  *reinterpret_cast<const uint4*>(stage + tok * 128 + ((piece * 16) ^ (i ? 64 : 0)));
          }
          turn ^= 1;  // whoever writes this half again has passed the next barrier, and with it everybody's reads
        } else if (a.phase != 0) {
          float* dst = a.o + z * a.plane_stride + (slot0 + cc) * N + nrow;
          if (nrow < N) {
#pragma unroll
            for (int b8 = 0; b8 < 32; b8 += 8) {
              if (b8 < live) {
#pragma unroll
                for (int c = b8; c < b8 + 8; ++c) {
                  if (c < live) *dst = __uint_as_float(va[c]);
                  dst += N;
                }
              }
            }
          }
        } else {
          unsigned char* mine = out_stage + (hpos - u_row0) * 2;  // [32 tokens][128 channels]
          float most = 0.0f;
#pragma unroll
          for (int b8 = 0; b8 < 32; b8 += 8) {
            if (b8 < live) {
#pragma unroll
              for (int c = b8; c < b8 + 8; c += 2) {
                const __nv_bfloat162 h2 = __floats2bfloat162_rn(fmaxf(__uint_as_float(va[c]), 0.0f), fmaxf(__uint_as_float(va[c + 1]), 0.0f));
                const float h0 = __low2float(h2), h1 = __high2float(h2);
                if (c < live) most = fmaxf(most, h0);
                if (c + 1 < live) most = fmaxf(most, h1);
                const __half2 f2 = __floats2half2_rn(fminf(h0, 65504.0f), fminf(h1, 65504.0f));
                *reinterpret_cast<__half*>(mine + c * 256) = __low2half(f2);
                *reinterpret_cast<__half*>(mine + (c + 1) * 256) = __high2half(f2);
              }
            }
          }
          if (nrow < N && beyond_f16(most)) atomicOr(a.check_word, CHECK_F16_RANGE);
          set_sync(part);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int tok = (set_tid >> 4) + 8 * i, ch = 8 * (set_tid & 15);
            if (tok < live && u_row0 + ch < N)
              *reinterpret_cast<uint4*>(a.hidden16 + (slot0 + cc + tok) * a.hid_stride + u_row0 + ch) =
                  *reinterpret_cast<const uint4*>(out_stage + tok * 256 + ch * 2);
          }
          set_sync(part);  // the buffer has been read
        }
      };
      if constexpr (EXACT) {
        store_chunk(set_col, tot);
      } else {
#pragma unroll 1
        for (int cc = 32 * part; cc < ntok; cc += 32 * U::SETS) {
          uint32_t va[32];
          __syncwarp();
          tmem_ld32(lane_base + cc, va);
          tmem_ld_wait();
          store_chunk(cc, va);
        }
      }
      if (!EXACT) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(b.acc_empty + 8 * acc_index);
        ++run_it;
      }
    }
    }
  }

  // wind-down: everybody meets, then the allocating warp releases tensor memory
  if (*abort_flag)
    for (int i = 0; i < 2000; ++i) __nanosleep(100);  // let copies in flight land
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, UM_TMEM_COLS);
  }
}

}  // namespace

bool ffn_umma_supported(const LayerDims& L) {
  // the same tensor maps as the TMA path (a last packed box that is not full is completed with zeros nobody reads)
  return ffn_tma_supported(L);
}

cudaError_t launch_ffn_umma(int phase, const LayerDims& L, const void* wmaps, int* plan, const void* in16, int in_stride,
                            void* hidden16, int hid_stride, float* o, int n_pairs, int zmax, bool exact, bool maybe_empty, int* check_word,
                            cudaStream_t st) {
  const int N = phase == 0 ? L.d_ff : L.d_model;
  const int K = phase == 0 ? L.d_model : L.d_ff;
  CUtensorMap tmap_b;
  if (encode_tmap_2d(&tmap_b, /*fp16*/ 1, in16, static_cast<uint64_t>(K), static_cast<uint64_t>(n_pairs),
                     static_cast<uint64_t>(in_stride) * 2, UM_ROW, exact ? Um<true>::BOX_TOK : Um<false>::BOX_TOK) != 0)
    return cudaErrorInvalidValue;
  static int sms_of_device[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!sms_of_device[dev]) {
    e = cudaFuncSetAttribute(ffn_umma_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, Um<false>::SMEM_BYTES);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(ffn_umma_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, Um<true>::SMEM_BYTES);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms_of_device[dev], cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
  }
  const bool gated = phase == 0 && L.act == EMOE_ACT_SWIGLU;
  const long long row_blocks = gated ? N / (UM_ROWS / 2) : (N + UM_ROWS - 1) / UM_ROWS;
  // upper bound of the tile count: every pair alone in a token tile
  long long tiles = row_blocks * (static_cast<long long>(n_pairs < L.E ? n_pairs : L.E) + n_pairs / (exact ? UM_EXACT_TOK : 128)) * (phase == 1 && zmax > 1 ? zmax : 1);
  const int grid = static_cast<int>(tiles < sms_of_device[dev] ? tiles : sms_of_device[dev]);
  UmmaArgs a;
  a.phase = phase;
  a.L = L;
  a.wmaps = static_cast<const CUtensorMap*>(wmaps);
  a.plan = plan;
  a.hidden16 = reinterpret_cast<__half*>(hidden16);
  a.hid_stride = hid_stride;
  a.o = o;
  a.zmax = phase == 0 || zmax < 1 ? 1 : zmax;
  a.n_pairs = n_pairs;
  a.maybe_empty = maybe_empty;
  a.plane_stride = static_cast<size_t>(n_pairs) * L.d_model;
  a.check_word = check_word;
  if (exact) return launch_chain(ffn_umma_kernel<true>, dim3(grid), dim3(Um<true>::THREADS), Um<true>::SMEM_BYTES, st, a, tmap_b);
  return launch_chain(ffn_umma_kernel<false>, dim3(grid), dim3(Um<false>::THREADS), Um<false>::SMEM_BYTES, st, a, tmap_b);
}

}  // namespace emoe
