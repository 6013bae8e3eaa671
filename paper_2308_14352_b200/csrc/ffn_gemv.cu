// Grouped GEMV on packed expert weights, CUDA-core path (paper Sections 1/2.1: each
// activated expert is an independent FFN; Section 3.2: weights are stored as b-bit codes
// with a scale channel and decompressed as q * s — here in registers).
//
// The path for fp32 activations (fp32 products and sums throughout) and the fallback for shapes the
// tensor-core paths do not take.  At these sizes a layer is a few microseconds of arithmetic, so
// the time is latency: the work is cut fine enough that all of it is on the SMs at once.
//   * a CTA takes a few rows of one expert, a slice of at most 1024 inputs (second projection: one
//     slice per CTA, summed by the combine step; first projection: all slices in turn) and up to
//     four tokens, whose activations it stages in shared memory as fp32 (read from there by every
//     warp; from global memory each step of the loop below waited for the L1 or L2);
//   * a warp is cut into groups of lanes; a group owns two rows and its lanes stream them with
//     128-bit loads (16 / 32 / 64 weights each), the next loads on their way while one set is used;
//   * the fields of a 32-bit word are masked into bytes together, a byte becomes a float by one byte
//     permute into the mantissa of 2^23 and one (exact) subtraction, shared by the tokens.
// Measured: Switch-base-like layers with 8 experts and 16 fp32 tokens, forward call of eight layers 878 -> 340 us
// (one row per warp, all inputs in turn, activations from global memory before); what is left is the
// latency of five launches and of the first loads of each.
#include "common.cuh"
#include "ffn_tile.cuh"

namespace emoe {
namespace {

constexpr int GEMV_WARPS = 4;
constexpr int GEMV_THREADS = GEMV_WARPS * 32;
constexpr int GEMV_TOK = 4;       // tokens of a pass
constexpr int GEMV_SLICE = 1024;  // inputs staged at a time
constexpr int GEMV_R = 2;         // rows of a group of lanes
constexpr int GEMV_LANES = 16;    // lanes of a group: a slice is one to four words per lane at 2 bits to 8, and a lane's share about 64 weights per row
constexpr int GEMV_ROWS = GEMV_WARPS * (32 / GEMV_LANES) * GEMV_R;  // rows of a CTA

// The codes of a 32-bit word (two's-complement fields, low bits first) as bytes q + 2^(b-1): code i is byte i / S of
// out[i % S], S = 8 / BITS fields to a byte.
template <int BITS>
__device__ __forceinline__ void code_bytes(uint32_t word, uint32_t (&out)[8 / BITS]) {
  constexpr uint32_t mask = ((1u << BITS) - 1) * 0x01010101u, flip = (1u << (BITS - 1)) * 0x01010101u;
#pragma unroll
  for (int i = 0; i < 8 / BITS; ++i) out[i] = and_xor(word >> (BITS * i), mask, flip);
}
// code i of the word as fp32: its byte in the mantissa of 2^23 by one byte permute, the constant subtracted (exact)
template <int BITS>
__device__ __forceinline__ float code_f32(const uint32_t (&bytes)[8 / BITS], int i) {
  constexpr int S = 8 / BITS;
  return __uint_as_float(prmt(bytes[i % S], 0x4B000000u, 0x7540u + i / S)) - (8388608.0f + static_cast<float>(1 << (BITS - 1)));
}

__device__ __forceinline__ float load_scale(const void* scales, bool f16, size_t idx) {
  return f16 ? __half2float(__ldg(reinterpret_cast<const __half*>(scales) + idx)) : __ldg(reinterpret_cast<const float*>(scales) + idx);
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
};

// where one matrix's rows of a lane group lie
struct Rows {
  const uint4* w;      // first row, first word of the row
  const void* scales;
  size_t srow;         // index of the first row's first scale
};

// acc[r][m] += sum_k q[r][k] * s[r][k/G] * x_m[k] over the words l, l + L, ... of the slice [j0, j0 + nv) of two rows.
// xs: [MT][chunk of 4 inputs][word] in shared memory, tokens GEMV_SLICE floats apart.
template <int BITS, int MT>
__device__ __forceinline__ void rows_dot(const Rows& m, int nvec, bool scale_f16, int ngroups, int gshift, int wpg, int j0, int nv, const float* xs,
                                         int l, float (&acc)[GEMV_R][MT]) {
  constexpr int PER = 32 / BITS;
  uint4 nw[GEMV_R];
  if (l < nv)
#pragma unroll
    for (int r = 0; r < GEMV_R; ++r) nw[r] = __ldg(m.w + static_cast<size_t>(r) * nvec + j0 + l);
#pragma unroll 1
  for (int j = l; j < nv; j += GEMV_LANES) {
    uint32_t w[GEMV_R][4];
    float s[GEMV_R], part[GEMV_R][MT];
    const int g = gshift >= 0 ? (j0 + j) >> gshift : (j0 + j) / wpg;  // words per scale group
#pragma unroll
    for (int r = 0; r < GEMV_R; ++r) {
      w[r][0] = nw[r].x, w[r][1] = nw[r].y, w[r][2] = nw[r].z, w[r][3] = nw[r].w;
      s[r] = load_scale(m.scales, scale_f16, m.srow + static_cast<size_t>(r) * ngroups + g);
#pragma unroll
      for (int t = 0; t < MT; ++t) part[r][t] = 0.0f;
    }
    if (j + GEMV_LANES < nv)
#pragma unroll
      for (int r = 0; r < GEMV_R; ++r) nw[r] = __ldg(m.w + static_cast<size_t>(r) * nvec + j0 + j + GEMV_LANES);
    const float* xp = xs + j * 4;
    constexpr int AT_ONCE = BITS / 2;  // 32-bit words: 16 weights (the kernel holds nine variants of this loop: unrolled further, it waits for its instructions)
#pragma unroll 1
    for (int i0 = 0; i0 < 4; i0 += AT_ONCE) {
#pragma unroll
      for (int i = 0; i < AT_ONCE; ++i) {
        uint32_t by[GEMV_R][8 / BITS];
#pragma unroll
        for (int r = 0; r < GEMV_R; ++r) code_bytes<BITS>(w[r][i], by[r]);
#pragma unroll
        for (int c = 0; c < PER / 4; ++c) {
          float4 xv[MT];
#pragma unroll
          for (int t = 0; t < MT; ++t) xv[t] = *reinterpret_cast<const float4*>(xp + t * GEMV_SLICE);
          xp += nv * 4;
#pragma unroll
          for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int r = 0; r < GEMV_R; ++r) {
              const float q = code_f32<BITS>(by[r], 4 * c + k);
#pragma unroll
              for (int t = 0; t < MT; ++t) part[r][t] = fmaf(q, k == 0 ? xv[t].x : (k == 1 ? xv[t].y : (k == 2 ? xv[t].z : xv[t].w)), part[r][t]);
            }
        }
      }
#pragma unroll
      for (int r = 0; r < GEMV_R; ++r)
#pragma unroll
        for (int i = 0; i + AT_ONCE < 4; ++i) w[r][i] = w[r][i + AT_ONCE];
    }
#pragma unroll
    for (int r = 0; r < GEMV_R; ++r)
#pragma unroll
      for (int t = 0; t < MT; ++t) acc[r][t] = fmaf(s[r], part[r][t], acc[r][t]);
  }
}

// the rows' sums over the slices [sl0, sl1) for MT tokens in slots slot0 ..
template <int BITS, bool GATED, int MT>
__device__ __forceinline__ void expert_pass(const GemvArgs& a, const ExpertDev& ex, int slot0, int ntok, int sl0, int sl1, int n0, float* xs) {
  const LayerDims& L = a.L;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int N = a.phase == 0 ? L.d_ff : L.d_model, K = a.phase == 0 ? L.d_model : L.d_ff;
  const int nvec = K * BITS / 128;
  const int n = n0 + (warp * (32 / GEMV_LANES) + lane / GEMV_LANES) * GEMV_R, l = lane & (GEMV_LANES - 1);
  const int G = L.group > 0 ? L.group : K, ngroups = K / G;
  const int wpg = G * BITS / 128;
  const int gshift = (wpg & (wpg - 1)) == 0 ? 31 - __clz(wpg) : -1;
  const int mat = a.phase == 0 ? 0 : (L.act == EMOE_ACT_RELU ? 1 : 2);
  const Rows m0 = {reinterpret_cast<const uint4*>(ex.packed[mat]) + static_cast<size_t>(n) * nvec, ex.scales[mat], static_cast<size_t>(n) * ngroups};
  const Rows m1 = {reinterpret_cast<const uint4*>(ex.packed[1]) + static_cast<size_t>(n) * nvec, ex.scales[1], static_cast<size_t>(n) * ngroups};
  float v[GEMV_R][MT], u[GEMV_R][MT];
#pragma unroll
  for (int r = 0; r < GEMV_R; ++r)
#pragma unroll
    for (int t = 0; t < MT; ++t) v[r][t] = u[r][t] = 0.0f;
  for (int sl = sl0; sl < sl1; ++sl) {
    const int k0 = sl * a.slice, len = min(a.slice, K - k0), nv = len * BITS / 128;
    __syncthreads();  // the slice in front is used up
    for (int i = threadIdx.x; i < MT * (len / 4); i += GEMV_THREADS) {
      const int t = i / (len / 4), c4 = i - t * (len / 4);  // token, chunk of four inputs
      const int slot = slot0 + min(t, ntok - 1);
      const size_t row = a.phase == 0 ? static_cast<size_t>(L.top_k == 1 ? a.perm[slot] : a.perm[slot] / L.top_k) : static_cast<size_t>(slot);
      const size_t at = row * K + k0 + 4 * c4;
      const void* src = a.phase == 0 ? a.x : a.hidden;
      float4 f;
      if (L.act_bf16) {
        const uint2 b = *reinterpret_cast<const uint2*>(static_cast<const __nv_bfloat16*>(src) + at);
        f = make_float4(__uint_as_float(b.x << 16), __uint_as_float(b.x & 0xffff0000u), __uint_as_float(b.y << 16), __uint_as_float(b.y & 0xffff0000u));
      } else {
        f = *reinterpret_cast<const float4*>(static_cast<const float*>(src) + at);
      }
      constexpr int CH = 32 / BITS;  // chunks of a 128-bit word; chunk-major, so that neighbouring words' readers read neighbouring 16 bytes
      *reinterpret_cast<float4*>(xs + t * GEMV_SLICE + ((c4 % CH) * nv + c4 / CH) * 4) = f;
    }
    __syncthreads();
    rows_dot<BITS, MT>(m0, nvec, L.scale_f16, ngroups, gshift, wpg, k0 * BITS / 128, nv, xs, l, v);
    if (GATED) rows_dot<BITS, MT>(m1, nvec, L.scale_f16, ngroups, gshift, wpg, k0 * BITS / 128, nv, xs, l, u);
  }
#pragma unroll
  for (int o = GEMV_LANES >> 1; o > 0; o >>= 1)
#pragma unroll
    for (int r = 0; r < GEMV_R; ++r)
#pragma unroll
      for (int t = 0; t < MT; ++t) {
        v[r][t] += __shfl_xor_sync(0xffffffffu, v[r][t], o);
        if (GATED) u[r][t] += __shfl_xor_sync(0xffffffffu, u[r][t], o);
      }
  // every lane of the group holds all sums: lane i stores the i-th
#pragma unroll
  for (int r = 0; r < GEMV_R; ++r)
#pragma unroll
    for (int t = 0; t < MT; ++t) {
      if (((r * MT + t) & (GEMV_LANES - 1)) != l || t >= ntok) continue;
      const size_t slot = static_cast<size_t>(slot0 + t);
      if (a.phase == 0) {
        const float h = GATED ? v[r][t] / (1.0f + expf(-v[r][t])) * u[r][t] : fmaxf(v[r][t], 0.0f);
        if (L.act_bf16) static_cast<__nv_bfloat16*>(a.hidden)[slot * N + n + r] = __float2bfloat16_rn(h);
        else static_cast<float*>(a.hidden)[slot * N + n + r] = h;
      } else {
        a.o[(static_cast<size_t>(blockIdx.y % a.ksplit) * a.n_pairs + slot) * N + n + r] = v[r][t];
      }
    }
}

template <int BITS, bool GATED>
__device__ __forceinline__ void expert_rows(const GemvArgs& a, const ExpertDev& ex, int begin, int cnt, float* xs) {
  const int n0 = static_cast<int>(blockIdx.x) * GEMV_ROWS;
  // second projection: slices z, z + 1, ... of this plane
  const int z = a.phase == 0 ? 0 : blockIdx.y % a.ksplit, per = a.phase == 0 ? a.nslices : (a.nslices + a.ksplit - 1) / a.ksplit;
  const int sl0 = z * per, sl1 = min(a.nslices, sl0 + per);
  for (int c0 = blockIdx.z * GEMV_TOK; c0 < cnt; c0 += gridDim.z * GEMV_TOK) {
    const int ntok = min(GEMV_TOK, cnt - c0);
    if (ntok > 2) expert_pass<BITS, GATED, 4>(a, ex, begin + c0, ntok, sl0, sl1, n0, xs);
    else if (ntok == 2) expert_pass<BITS, GATED, 2>(a, ex, begin + c0, ntok, sl0, sl1, n0, xs);
    else expert_pass<BITS, GATED, 1>(a, ex, begin + c0, ntok, sl0, sl1, n0, xs);
  }
}

template <bool GATED>  // first projection of a gated layer: two matrices
__global__ void __launch_bounds__(GEMV_THREADS, GATED ? 4 : 5) ffn_gemv_kernel(const __grid_constant__ GemvArgs a) {
  __shared__ __align__(16) float xs[GEMV_TOK * GEMV_SLICE];
  pdl_wait();
  pdl_trigger();
  const int e = a.phase == 0 ? blockIdx.y : blockIdx.y / a.ksplit;
  const int begin = a.off[e];
  const int cnt = a.off[e + 1] - begin;
  if (cnt <= 0) return;  // only activated experts are touched
  const ExpertDev ex = a.experts[e];
  switch (ex.bits) {
    case 2: expert_rows<2, GATED>(a, ex, begin, cnt, xs); break;
    case 4: expert_rows<4, GATED>(a, ex, begin, cnt, xs); break;
    case 8: expert_rows<8, GATED>(a, ex, begin, cnt, xs); break;
    default: break;
  }
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
  GemvArgs a{phase, L, experts, x, perm, off, hidden, o, 0, 0, ksplit, n_pairs};
  const int want = gemv_slices(K);
  a.slice = ((K + want - 1) / want + 63) / 64 * 64;
  a.nslices = (K + a.slice - 1) / a.slice;
  // passes of four tokens side by side: what even routing would fill (empty CTAs cost more than a second turn of a full one)
  const int passes = (n_pairs / L.E + GEMV_TOK - 1) / GEMV_TOK + (n_pairs < L.E ? 1 : 0);
  const dim3 grid(N / GEMV_ROWS, phase == 0 ? L.E : L.E * ksplit, passes < 16 ? passes : 16);
  if (phase == 0 && L.act == EMOE_ACT_SWIGLU) return launch_chain(ffn_gemv_kernel<true>, grid, dim3(GEMV_THREADS), 0, st, a);
  return launch_chain(ffn_gemv_kernel<false>, grid, dim3(GEMV_THREADS), 0, st, a);
}

}  // namespace emoe
