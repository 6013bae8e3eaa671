// Grouped GEMV on packed expert weights, CUDA-core path (paper Sections 1/2.1: each
// activated expert is an independent FFN; Section 3.2: weights are stored as b-bit codes
// with a scale channel and decompressed as q * s — here in registers).
//
// The path for fp32 activations (fp32 products and sums throughout) and the fallback for shapes the
// tensor-core paths do not take.  At these sizes a layer is a few microseconds of arithmetic, so
// the time is latency: the second projection's weights are fetched while the first still runs, and all of the work is
// on the SMs at once.
//   * a CTA takes some blocks of 32 rows of one expert and a slice of at most 1024 inputs (second projection: one
//     slice per CTA, summed by the combine step; first projection: all slices in turn).  Their codes come into shared
//     memory by asynchronous 16-byte copies of all threads, all of them asked for at once (a bulk copy takes longer to its first
//     byte); the number of blocks is such that every CTA is resident at once;
//   * up to four tokens at a time have their activations in shared memory as fp32 (from global memory each
//     step of the loop below waited for the L1 or L2); the loads of a pass are in flight together;
//   * a warp is cut into groups of lanes; a group owns four rows of a block and its lanes take 128-bit words of them (16 / 32 / 64
//     weights each), so that an activation read serves four rows (two: the reads of shared memory bound passes of four tokens);
//   * the fields of a 32-bit word are masked into bytes together, a byte becomes a float by one byte
//     permute into the mantissa of 2^23 and one (exact) subtraction for two of them, shared by the tokens; products and sums go
//     by twos as well.
// Measured (us per layer of a forward call; two rows per group, codes through registers, a variant of the loop per width and number
// of tokens -> bulk copies, tokens staged one after the other, one token as two -> now): 768 x 3072, 8 experts, fp32, 16 tokens 41.8 ->
// 34.5 -> 30.5; 1024 x 4096, 4 experts, two picks, 64 tokens 211 -> 148 -> 136; 4096 x 14336 gated, 8 experts, two picks, one token
// 204 -> 228 -> 194, 4 tokens 405 -> 436 -> 368, 64 tokens 3690 -> 3240 -> 2630; 64 x 128, 4 experts, two picks, 64 tokens (bf16) 23.8 -> 26.9 -> 22.2.
#include "common.cuh"
#include "ffn_tile.cuh"

namespace emoe {
namespace {

constexpr int GEMV_WARPS = 4;
constexpr int GEMV_THREADS = GEMV_WARPS * 32;
constexpr int GEMV_TOK = 4;       // tokens of a pass
constexpr int GEMV_SLICE = 1024;  // inputs staged at a time
constexpr int GEMV_R = 4;         // rows of a group of lanes
constexpr int GEMV_LANES = 16;    // lanes of a group: a slice is one to four words per lane at 2 bits to 8, and a lane's share about 64 weights per row
constexpr int GEMV_ROWS = GEMV_WARPS * (32 / GEMV_LANES) * GEMV_R;  // rows of a block, which a CTA takes at a time
constexpr int GEMV_CTAS = 4;      // per SM (registers)
constexpr int GEMV_BLOCKS = 4;    // of a CTA, at most
constexpr int GEMV_SMEM = 226 * 1024;  // of an SM, with what the system keeps per CTA taken off below
constexpr int GEMV_GROUP = 16;    // inputs per scale, at least: a 128-bit word of 8-bit codes
// codes, scales and activations of one block of a gated first projection: the most a CTA takes (several blocks: a third of an SM)
constexpr int GEMV_CTA_SMEM = 2 * GEMV_ROWS * (GEMV_SLICE + 4 * (GEMV_SLICE / GEMV_GROUP + 1)) + 4 * GEMV_TOK * GEMV_SLICE;
static_assert(GEMV_SMEM / 3 <= GEMV_CTA_SMEM && GEMV_CTA_SMEM <= GEMV_SMEM, "shared memory");

// two fp32 numbers in a register pair: sums and products of both by one instruction
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pair_of(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float pair_sum(f32x2 v) {
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
  return lo + hi;
}

// How codes of b bits are taken: field f of a 32-bit word's four bytes at a time (one, two or four fields to a byte), as bytes
// q + 2^(b-1).  The width is data here, not a variant of the code: with a variant per width and number of tokens the CTAs of an
// SM ran nine loops, and a third of all cycles went into waiting for instructions.
struct Width {
  int bits;
  uint32_t mask, flip;  // of a field, and its sign bit, in every byte
  f32x2 minus;          // -(2^23 + 2^(b-1)), twice
};
__device__ __forceinline__ Width width_of(int bits) {
  Width w;
  w.bits = bits;
  w.mask = ((1u << bits) - 1) * 0x01010101u;
  w.flip = (1u << (bits - 1)) * 0x01010101u;
  const float m = -(8388608.0f + static_cast<float>(1 << (bits - 1)));
  w.minus = pair_of(m, m);
  return w;
}
// bytes 2h and 2h + 1 as fp32: each in the mantissa of 2^23 by a byte permute, the constant subtracted from both (exact)
template <int H>
__device__ __forceinline__ f32x2 code_pair(uint32_t bytes, f32x2 minus) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pair_of(__uint_as_float(prmt(bytes, 0x4B000000u, 0x7540u + 2 * H)), __uint_as_float(prmt(bytes, 0x4B000000u, 0x7541u + 2 * H)))), "l"(minus));
  return r;
}

struct GemvArgs {
  int phase;
  LayerDims L;
  const ExpertDev* experts;
  const void* x;
  const int32_t* perm;
  const int32_t* off;
  void* hidden;  // [slot][d_ff], activation type
  float* o;      // [ksplit][n_pairs][d_model]
  int slice;     // inputs of a slice
  int nslices, ksplit, n_pairs;
  int blocks;    // blocks of rows per CTA (one where there are several slices in turn)
  int G, ngroups;  // inputs per scale, scales of a row
  int groups;    // scales of a row that a slice touches, at most
};

// shared memory: [matrices][rows][slice] codes, [matrices][rows][groups] scales, [GEMV_TOK][slice] activations
struct Staged {
  unsigned char* codes;
  float* scales;
  float* xs;
};

// a slice of the inputs of an expert's rows
struct Slice {
  int k0, len, bytes;  // its first input, inputs, bytes of a row
  int g0, ng;          // first scale, scales
  int wpg, gshift;     // 128-bit words per scale, its logarithm (negative: not a power of two)
};
__device__ __forceinline__ Slice slice_of(const GemvArgs& a, int sl, int bits) {
  const int K = a.phase == 0 ? a.L.d_model : a.L.d_ff;
  Slice s;
  s.k0 = sl * a.slice;
  s.len = min(a.slice, K - s.k0);
  s.bytes = s.len * bits / 8;
  s.g0 = a.nslices == 1 ? 0 : s.k0 / a.G;
  s.ng = a.nslices == 1 ? a.ngroups : (s.k0 + s.len - 1) / a.G - s.g0 + 1;
  s.wpg = a.G * bits / 128;
  s.gshift = (s.wpg & (s.wpg - 1)) == 0 ? 31 - __clz(s.wpg) : -1;
  return s;
}

// where one matrix's rows of a lane group lie
struct Rows {
  const unsigned char* w;  // first row
  const float* s;          // its scales
  int row_bytes, srow;     // distance to the second row
};

// acc[r][m] += sum_k q[r][k] * s[r][k/G] * x_m[k] over the words l, l + L, ... of a slice of the group's rows.
// xs: [MT][32-bit word of a 128-bit one][field][128-bit word][byte], tokens xstride floats apart.
template <int MT>
__device__ __forceinline__ void rows_dot(const Rows& m, const Width& wd, const Slice& sc, const float* xs, int xstride, int l, float (&acc)[GEMV_R][MT]) {
  const int nv = sc.bytes >> 4, j0 = sc.k0 * wd.bits / 128;
#pragma unroll 1
  for (int j = l; j < nv; j += GEMV_LANES) {
    uint32_t w[GEMV_R][4];
    float s[GEMV_R];
    f32x2 part[GEMV_R][MT];  // the sums over even and over odd bytes
    const int g = sc.ng == 1 ? 0 : (sc.gshift >= 0 ? (j0 + j) >> sc.gshift : (j0 + j) / sc.wpg) - sc.g0;
#pragma unroll
    for (int r = 0; r < GEMV_R; ++r) {
      const uint4 v = *reinterpret_cast<const uint4*>(m.w + r * m.row_bytes + 16 * j);
      w[r][0] = v.x, w[r][1] = v.y, w[r][2] = v.z, w[r][3] = v.w;
      s[r] = m.s[r * m.srow + g];
#pragma unroll
      for (int t = 0; t < MT; ++t) part[r][t] = 0ull;
    }
    const float* xp = xs + j * 4;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll 1
      for (int f = 0; f < 8; f += wd.bits) {
        ulonglong2 xv[MT];
#pragma unroll
        for (int t = 0; t < MT; ++t) xv[t] = *reinterpret_cast<const ulonglong2*>(xp + t * xstride);
        xp += nv * 4;
#pragma unroll
        for (int r = 0; r < GEMV_R; ++r) {
          const uint32_t by = and_xor(w[r][i] >> f, wd.mask, wd.flip);
          const f32x2 q0 = code_pair<0>(by, wd.minus), q1 = code_pair<1>(by, wd.minus);
#pragma unroll
          for (int t = 0; t < MT; ++t) {
            asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(part[r][t]) : "l"(q0), "l"(xv[t].x));
            asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(part[r][t]) : "l"(q1), "l"(xv[t].y));
          }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < GEMV_R; ++r)
#pragma unroll
      for (int t = 0; t < MT; ++t) acc[r][t] = fmaf(s[r], pair_sum(part[r][t]), acc[r][t]);
  }
}

// The activations of MT tokens (the last of ntok repeated) in the slice of `len` inputs from k0 on, in the order rows_dot takes
// them.  The loads of all tokens are in flight together.
template <int MT>
__device__ __forceinline__ void stage_inputs(const GemvArgs& a, const Width& wd, int slot0, int ntok, int k0, int len, float* xs) {
  const LayerDims& L = a.L;
  const int K = a.phase == 0 ? L.d_model : L.d_ff, nv = len * wd.bits / 128;
  const int sh = wd.bits == 8 ? 0 : (wd.bits == 4 ? 1 : 2);  // log2 of the fields
  const void* src = a.phase == 0 ? a.x : a.hidden;
  size_t at[MT];
#pragma unroll
  for (int t = 0; t < MT; ++t) {
    const int slot = slot0 + min(t, ntok - 1);
    at[t] = static_cast<size_t>(a.phase == 0 ? a.perm[slot] : slot);
  }
#pragma unroll
  for (int t = 0; t < MT; ++t) at[t] = (a.phase == 0 && L.top_k != 1 ? static_cast<int>(at[t]) / L.top_k : at[t]) * K + k0;
  for (int k = 4 * threadIdx.x; k < len; k += 4 * GEMV_THREADS) {
    float4 v[MT];
    if (L.act_bf16) {
      uint2 b[MT];
#pragma unroll
      for (int t = 0; t < MT; ++t) b[t] = *reinterpret_cast<const uint2*>(static_cast<const __nv_bfloat16*>(src) + at[t] + k);
#pragma unroll
      for (int t = 0; t < MT; ++t)
        v[t] = make_float4(__uint_as_float(b[t].x << 16), __uint_as_float(b[t].x & 0xffff0000u), __uint_as_float(b[t].y << 16), __uint_as_float(b[t].y & 0xffff0000u));
    } else {
#pragma unroll
      for (int t = 0; t < MT; ++t) v[t] = *reinterpret_cast<const float4*>(static_cast<const float*>(src) + at[t] + k);
    }
    // input k of the slice: 128-bit word k / (16 << sh), and in it 32-bit word, byte and field
    const int word = k >> (4 + sh), i = (k >> (2 + sh)) & 3, o = k & ((4 << sh) - 1);
#pragma unroll
    for (int t = 0; t < MT; ++t) {
      float* to = xs + t * a.slice;
      if (sh == 0) {
        *reinterpret_cast<float4*>(to + (i * nv + word) * 4) = v[t];
      } else if (sh == 1) {  // two fields, two bytes
        float* p = to + (i * 2 * nv + word) * 4 + (o >> 1);
        *reinterpret_cast<float2*>(p) = make_float2(v[t].x, v[t].z);
        *reinterpret_cast<float2*>(p + nv * 4) = make_float2(v[t].y, v[t].w);
      } else {  // four fields, one byte
        float* p = to + (i * 4 * nv + word) * 4 + (o >> 2);
        p[0] = v[t].x;
        p[nv * 4] = v[t].y;
        p[nv * 8] = v[t].z;
        p[nv * 12] = v[t].w;
      }
    }
  }
}

__device__ __forceinline__ void cp_async16(void* to, const void* from) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(to))), "l"(from) : "memory");
}

// asks for the codes of a slice of the CTA's rows
template <bool GATED>
__device__ __forceinline__ void fetch_codes(const GemvArgs& a, const ExpertDev& ex, const Slice& sc, int n0, int rows, const Staged& sm) {
  const int K = a.phase == 0 ? a.L.d_model : a.L.d_ff, mat = a.phase == 0 ? 0 : (a.L.act == EMOE_ACT_RELU ? 1 : 2);
  const size_t row_bytes = static_cast<size_t>(K) * ex.bits / 8;
#pragma unroll
  for (int i = 0; i < (GATED ? 2 : 1); ++i) {
    const int m = GATED ? i : mat;
    const uint8_t* from = (m == 0 ? ex.packed[0] : (m == 1 ? ex.packed[1] : ex.packed[2])) + n0 * row_bytes + static_cast<size_t>(sc.k0) * ex.bits / 8;
    unsigned char* to = sm.codes + i * a.blocks * GEMV_ROWS * a.slice;
    if (sc.len == K) {  // whole rows follow each other
      for (int u = 16 * threadIdx.x; u < rows * sc.bytes; u += 16 * GEMV_THREADS) cp_async16(to + u, from + u);
    } else {
      const int words = sc.bytes >> 4;
      for (int u = threadIdx.x; u < rows * words; u += GEMV_THREADS) {
        const int r = u / words, c = 16 * (u - r * words);
        cp_async16(to + r * sc.bytes + c, from + r * row_bytes + c);
      }
    }
  }
}
// ... and their scales; `staging` runs between the first loads and the first store
template <bool GATED, typename F>
__device__ __forceinline__ void fetch_scales(const GemvArgs& a, const ExpertDev& ex, const Slice& sc, int n0, int rows, const Staged& sm, F staging) {
  const int mat = a.phase == 0 ? 0 : (a.L.act == EMOE_ACT_RELU ? 1 : 2);
  const auto scale = [&](int m, int u) {
    const int r = sc.ng == 1 ? u : u / sc.ng;
    const void* scales = m == 0 ? ex.scales[0] : (m == 1 ? ex.scales[1] : ex.scales[2]);
    return load_scale_ro(scales, a.L.scale_f16, static_cast<size_t>(n0 + r) * a.ngroups + sc.g0 + u - r * sc.ng);
  };
  const int n = rows * sc.ng, tid = threadIdx.x;
  float first[GATED ? 2 : 1];
#pragma unroll
  for (int i = 0; i < (GATED ? 2 : 1); ++i) first[i] = tid < n ? scale(GATED ? i : mat, tid) : 0.0f;
  staging();
#pragma unroll
  for (int i = 0; i < (GATED ? 2 : 1); ++i) {
    float* to = sm.scales + i * a.blocks * GEMV_ROWS * a.groups;
    if (tid < n) to[tid] = first[i];
    for (int u = tid + GEMV_THREADS; u < n; u += GEMV_THREADS) to[u] = scale(GATED ? i : mat, u);
  }
}

// the sums of a block's rows in the staged slice, for MT tokens
template <bool GATED, int MT>
__device__ __forceinline__ void block_dot(const GemvArgs& a, const Width& wd, int b, const Slice& sc, const Staged& sm, float (&v)[GEMV_R][MT], float (&u)[GEMV_R][MT]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, l = lane & (GEMV_LANES - 1);
  const int r = b * GEMV_ROWS + (warp * (32 / GEMV_LANES) + lane / GEMV_LANES) * GEMV_R;
  const Rows m0 = {sm.codes + r * sc.bytes, sm.scales + r * sc.ng, sc.bytes, sc.ng};
  rows_dot<MT>(m0, wd, sc, sm.xs, a.slice, l, v);
  if (GATED) {
    const Rows m1 = {m0.w + a.blocks * GEMV_ROWS * a.slice, m0.s + a.blocks * GEMV_ROWS * a.groups, sc.bytes, sc.ng};
    rows_dot<MT>(m1, wd, sc, sm.xs, a.slice, l, u);
  }
}

// Adds up the V values of every lane over its group of lanes; lane i keeps value i % V.  Half of the values go to
// the partner in each of the first steps.
template <int V>
__device__ __forceinline__ float sum_lanes(const float (&v)[V], int l) {
  static_assert(V == 1 || V == 2 || V == 4 || V == 8 || V == 16, "");
  float x[V];
#pragma unroll
  for (int i = 0; i < V; ++i) x[i] = v[i];
  int o = 1;
#pragma unroll
  for (int n = V; n > 1; n >>= 1, o <<= 1) {  // value 2i stays in the lanes without bit o, 2i + 1 in those with it
    const bool odd = l & o;
#pragma unroll
    for (int i = 0; i < n / 2; ++i) {
      const float keep = odd ? x[2 * i + 1] : x[2 * i], give = odd ? x[2 * i] : x[2 * i + 1];
      x[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  for (; o < GEMV_LANES; o <<= 1) x[0] += __shfl_xor_sync(0xffffffffu, x[0], o);
  return x[0];
}

// adds the lanes up and stores a block's results
template <bool GATED, int MT>
__device__ __forceinline__ void store_block(const GemvArgs& a, int z, int n0, int slot0, int ntok, float (&v)[GEMV_R][MT], float (&u)[GEMV_R][MT]) {
  const LayerDims& L = a.L;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, l = lane & (GEMV_LANES - 1);
  const int N = a.phase == 0 ? L.d_ff : L.d_model;
  float f[GEMV_R * MT], h[GEMV_R * MT];
#pragma unroll
  for (int i = 0; i < GEMV_R * MT; ++i) f[i] = v[i / MT][i % MT], h[i] = u[i / MT][i % MT];
  const float x = sum_lanes(f, l), y = GATED ? sum_lanes(h, l) : 0.0f;
  const int i = l % (GEMV_R * MT), t = i % MT;
  const int n = n0 + (warp * (32 / GEMV_LANES) + lane / GEMV_LANES) * GEMV_R + i / MT;
  if (l >= GEMV_R * MT || t >= ntok) return;
  const size_t slot = static_cast<size_t>(slot0 + t);
  if (a.phase == 0) {
    const float r = GATED ? x / (1.0f + expf(-x)) * y : fmaxf(x, 0.0f);
    if (L.act_bf16) static_cast<__nv_bfloat16*>(a.hidden)[slot * N + n] = __float2bfloat16_rn(r);
    else static_cast<float*>(a.hidden)[slot * N + n] = r;
  } else {
    a.o[(static_cast<size_t>(z) * a.n_pairs + slot) * N + n] = x;
  }
}

// What a CTA does; the codes of its first slice are on their way.
struct Work {
  int begin, cnt;      // the expert's slots
  int n0, rows;        // its rows
  int sl0, sl1, z;     // slices and plane
};

template <bool GATED, int MT>
__device__ __forceinline__ void token_pass(const GemvArgs& a, const ExpertDev& ex, const Width& wd, const Work& w, int c0, int ntok, const Staged& sm, Slice& sc,
                                           bool& first) {
  const int slot0 = w.begin + c0;
  const bool one = w.sl1 - w.sl0 == 1;
  float v[GEMV_R][MT], u[GEMV_R][MT];
  for (int b = 0; b < w.rows / GEMV_ROWS; ++b) {
#pragma unroll
    for (int r = 0; r < GEMV_R; ++r)
#pragma unroll
      for (int t = 0; t < MT; ++t) v[r][t] = u[r][t] = 0.0f;
    for (int sl = w.sl0; sl < w.sl1; ++sl) {
      if (b == 0) {  // (with several slices there is one block)
        __syncthreads();  // what is staged has been used
        if (!one && !first) {
          sc = slice_of(a, sl, wd.bits);
          fetch_codes<GATED>(a, ex, sc, w.n0, w.rows, sm);
        }
        const auto staging = [&] { stage_inputs<MT>(a, wd, slot0, ntok, sc.k0, sc.len, sm.xs); };
        if (first || !one) fetch_scales<GATED>(a, ex, sc, w.n0, w.rows, sm, staging);
        else staging();
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        first = false;
      }
      block_dot<GATED, MT>(a, wd, b, sc, sm, v, u);
    }
    store_block<GATED, MT>(a, w.z, w.n0 + b * GEMV_ROWS, slot0, ntok, v, u);
  }
}

template <bool GATED>
__device__ __forceinline__ void expert_rows(const GemvArgs& a, const ExpertDev& ex, const Work& w, Slice sc, const Staged& sm) {
  const Width wd = width_of(ex.bits);
  bool first = true;
  for (int c0 = blockIdx.z * GEMV_TOK; c0 < w.cnt; c0 += gridDim.z * GEMV_TOK) {
    const int ntok = min(GEMV_TOK, w.cnt - c0);
    if (ntok > 2) token_pass<GATED, 4>(a, ex, wd, w, c0, ntok, sm, sc, first);
    else if (ntok == 2) token_pass<GATED, 2>(a, ex, wd, w, c0, ntok, sm, sc, first);
    else token_pass<GATED, 1>(a, ex, wd, w, c0, ntok, sm, sc, first);
  }
}

template <bool GATED>  // first projection of a gated layer: two matrices
__global__ void __launch_bounds__(GEMV_THREADS, GEMV_CTAS) ffn_gemv_kernel(const __grid_constant__ GemvArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int rows_max = (GATED ? 2 : 1) * a.blocks * GEMV_ROWS;
  Staged sm;
  sm.codes = smem;
  sm.xs = reinterpret_cast<float*>(smem + rows_max * a.slice);
  sm.scales = sm.xs + GEMV_TOK * a.slice;
  const int N = a.phase == 0 ? a.L.d_ff : a.L.d_model;
  const int e = a.phase == 0 ? blockIdx.y : blockIdx.y / a.ksplit;
  Work w;
  w.n0 = static_cast<int>(blockIdx.x) * a.blocks * GEMV_ROWS;
  w.rows = min(a.blocks * GEMV_ROWS, N - w.n0);
  // second projection: slices z, z + 1, ... of this plane
  w.z = a.phase == 0 ? 0 : blockIdx.y % a.ksplit;
  const int per = a.phase == 0 ? a.nslices : (a.nslices + a.ksplit - 1) / a.ksplit;
  w.sl0 = w.z * per;
  w.sl1 = min(a.nslices, w.sl0 + per);
  // The table of experts is older than the kernel in front, and for the second projection so are the offsets: the first
  // projection had waited for them when it let this kernel start.  What does not depend on the kernel in front is fetched
  // beside it; only activated experts are touched.
  const ExpertDev ex = a.experts[e];
  if (a.phase == 0) {
    pdl_wait();
    pdl_trigger();  // behind the wait: the second projection relies on what it lets through being complete (common.cuh)
  }
  w.begin = __ldcg(a.off + e);
  w.cnt = __ldcg(a.off + e + 1) - w.begin;
  const bool idle = w.cnt <= static_cast<int>(blockIdx.z) * GEMV_TOK;
  const Slice sc = slice_of(a, w.sl0, ex.bits);
  if (!idle && w.sl0 < w.sl1) fetch_codes<GATED>(a, ex, sc, w.n0, w.rows, sm);  // (the last planes may be without a slice)
  if (a.phase == 1) {
    pdl_wait();
    pdl_trigger();
  }
  if (idle) return;
  expert_rows<GATED>(a, ex, w, sc, sm);
}

// slices of a projection over K inputs: as long as shared memory holds, of equal length, whole 128-bit words at every width
int gemv_slices(int K) { return (K + GEMV_SLICE - 1) / GEMV_SLICE; }

}  // namespace

// planes of the second projection's partial sums
int ffn_gemv_ksplit(const LayerDims& L) {
  const int n = gemv_slices(L.d_ff);
  return n < 16 ? n : 16;
}

cudaError_t launch_ffn_gemv(int phase, const LayerDims& L, const ExpertDev* experts, const void* x, const int32_t* perm, const int32_t* off,
                            void* hidden, float* o, int ksplit, int n_pairs, cudaStream_t st) {
  const int N = phase == 0 ? L.d_ff : L.d_model, K = phase == 0 ? L.d_model : L.d_ff;
  const bool gated = phase == 0 && L.act == EMOE_ACT_SWIGLU;
  const int G = L.group > 0 ? L.group : K;
  GemvArgs a{phase, L, experts, x, perm, off, hidden, o, 0, 0, ksplit, n_pairs, 1, G, K / G, 0};
  const int want = gemv_slices(K);
  a.slice = ((K + want - 1) / want + 63) / 64 * 64;
  a.nslices = (K + a.slice - 1) / a.slice;
  a.groups = a.nslices == 1 ? K / G : (a.slice + G - 1) / G + 1;
  const int turns = phase == 0 ? a.nslices : (a.nslices + ksplit - 1) / ksplit;  // slices a CTA takes one after another
  const int gy = phase == 0 ? L.E : L.E * ksplit, row_blocks = N / GEMV_ROWS;
  const size_t per_block = static_cast<size_t>(gated ? 2 : 1) * GEMV_ROWS * (a.slice + 4 * a.groups), fixed = sizeof(float) * GEMV_TOK * a.slice;
  // Blocks of rows per CTA: a CTA's start (offsets, activations, first codes) costs about a block's time, and so does every
  // wave of CTAs.  At least three CTAs of an SM have to be resident.
  const auto resident = [&](int blocks) {
    const long long by_smem = GEMV_SMEM / static_cast<long long>(fixed + blocks * per_block + 1280);
    return by_smem < GEMV_CTAS ? by_smem : GEMV_CTAS;
  };
  const long long active = static_cast<long long>(n_pairs < L.E ? n_pairs : L.E) * (gy / L.E);
  const auto waves = [&](int blocks) {
    const long long at_once = resident(blocks) * GPU_SMS;
    return (active * ((row_blocks + blocks - 1) / blocks) + at_once - 1) / at_once;
  };
  for (int b = 2; b <= GEMV_BLOCKS && turns == 1 && resident(b) >= 3; ++b)
    if (waves(b) * (b + 1) <= waves(a.blocks) * (a.blocks + 1)) a.blocks = b;
  const int gx = (row_blocks + a.blocks - 1) / a.blocks;
  // passes of four tokens side by side while there is room for their CTAs
  const int passes = (n_pairs / L.E + GEMV_TOK - 1) / GEMV_TOK + (n_pairs < L.E ? 1 : 0);
  const long long room = resident(a.blocks) * GPU_SMS / (gx * active);
  const int gz = room < 1 ? 1 : static_cast<int>(room < passes ? room : passes);
  const size_t smem = fixed + a.blocks * per_block;
  if (smem > GEMV_CTA_SMEM) return cudaErrorInvalidValue;
  const dim3 grid(gx, gy, gz < 16 ? gz : 16), block(GEMV_THREADS);
  const cudaError_t e = gated ? allow_smem<ffn_gemv_kernel<true>>(GEMV_CTA_SMEM) : allow_smem<ffn_gemv_kernel<false>>(GEMV_CTA_SMEM);
  if (e != cudaSuccess) return e;
  return gated ? launch_chain(ffn_gemv_kernel<true>, grid, block, smem, st, a) : launch_chain(ffn_gemv_kernel<false>, grid, block, smem, st, a);
}

}  // namespace emoe
