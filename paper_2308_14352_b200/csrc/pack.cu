// Expert-wise quantisation kernels (paper Section 3.2, "Choosing the algorithm"):
// channel-wise linear quantisation to INT2/INT4/INT8 codes plus a scale channel, from an fp32
// matrix (emoe_pack_expert) or from a matrix already stored at another width
// (emoe_requantize_expert: the bitwidth selection of Section 3.2 lowers the width of chosen
// experts; the weight is decompressed in registers, w~ = q * s rounded once to fp32, and the fp32
// original is not needed).  Units are (output channel, group) pairs: find the unit's max-abs, derive the
// scale, quantise, pack.  Sixteen consecutive weights per lane (64 bytes read from fp32, 4 / 8 / 16 bytes
// written by one store) wherever the groups allow it:
//   groups of 32 to 512, powers of two: the matrix is dense, so its units follow each other in memory and a warp takes
//     512 weights at a time, group / 16 lanes per unit (groups of 64, 14336 x 12288: 843 us with a warp per unit, 152 so);
//   other groups of 16 n > 256 (per-channel scales): one to eight warps of a CTA per unit (8 to 4 bits 203 -> 135 us);
//   8 to 4 or 2 bits in groups of 64 or 128: integer arithmetic (requant8, 139 -> 85 us);
//   4 to 2 bits in groups of 128: a table of the 16 codes;
//   any other multiple of 4: a warp per unit, four weights per lane.
// HBM-bound by definition: 4 (or b_in / 8) bytes read and b_out / 8 bytes written per weight.  Packing
// from fp32 at 14336 x 12288 to 4 bits takes 137 us, 5.8 TB/s; the narrowing of codes stays bound by its
// instructions (3.1 TB/s at 8 to 4 bits).
//
// Two readings of "the range expressible by the bitwidth" (Section 3.2): symmetric codes
// -qmax .. qmax with qmax = 2^(b-1) - 1 and scale = max-abs / qmax (the default), or every code of
// the field, -2^(b-1) .. 2^(b-1) - 1, with scale = max-abs / 2^(b-1) ("full range": four levels at
// 2 bits instead of three).
//
// The quotient w / s is an IEEE division in the definition.  The kernels multiply by 1 / s
// instead and keep the result when it cannot differ from the definition's: the product lies
// within 1.8e-7 relative of the rounded quotient, so unless it comes within 1e-4 of a half-integer
// (or leaves the range where that bound holds) both round to the same integer; otherwise the
// division is carried out.  Bit-exact with the definition either way.
#include "common.cuh"

namespace emoe {
namespace {

constexpr float ROUND_MAGIC = 12582912.0f;  // 1.5 * 2^23, bit pattern 0x4B400000

template <int BITS>
struct PackWord;  // the codes of 4 consecutive weights
template <>
struct PackWord<8> { typedef uint32_t type; };
template <>
struct PackWord<4> { typedef uint16_t type; };
template <>
struct PackWord<2> { typedef uint8_t type; };

__device__ __forceinline__ uint32_t max_s16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("max.s16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ uint32_t min_s16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("min.s16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

// bytes of w by selector nibbles; one with its top bit set gives eight copies of the byte's sign (which the intrinsic
// of this instruction does not pass on)
__device__ __forceinline__ uint32_t sign_bytes(uint32_t w, uint32_t selector) {
  uint32_t r;
  asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(w), "r"(selector));
  return r;
}

// largest magnitude among the 16 signed bytes of four words
__device__ __forceinline__ int max_abs_code(const uint32_t (&w)[4]) {
  uint32_t mx = 0u, mn = 0u;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t even = sign_bytes(w[i], 0xA280u), odd = sign_bytes(w[i], 0xB391u);
    mx = max_s16x2(mx, max_s16x2(even, odd));
    mn = min_s16x2(mn, min_s16x2(even, odd));
  }
  const int top = max(static_cast<int>(mx << 16) >> 16, static_cast<int>(mx) >> 16);
  const int bottom = min(static_cast<int>(mn << 16) >> 16, static_cast<int>(mn) >> 16);
  return max(top, -bottom);
}

__device__ __forceinline__ float amax4(const float4& v) {
  return fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
}

// Where the weights come from.  load4(n, k): weights k .. k+3 of row n (k a multiple of 4);
// `unit` is the row's group index n * ngroups + g.
struct SourceF32 {
  static constexpr int IN_BITS = 32;
  const float* W;
  int K;
  __device__ __forceinline__ float4 load4(int n, int k, long long) const {
    return *reinterpret_cast<const float4*>(W + static_cast<size_t>(n) * K + k);
  }
  // 16 consecutive weights from linear index w0 (a multiple of 16) of the dense matrix: first the
  // loads (several steps are requested before the first is used), then the values
  static constexpr int STEPS = 1;  // steps of 512 weights a warp has in flight: more warps instead (14336 x 12288 to 4 bits: two steps 147 us, one 137)
  struct Raw {
    float4 f[4];
  };
  __device__ __forceinline__ void load_raw(long long w0, long long, Raw& r, float&) const {
    const float4* p = reinterpret_cast<const float4*>(W + w0);
#pragma unroll
    for (int i = 0; i < 4; ++i) r.f[i] = p[i];
  }
  __device__ __forceinline__ void zero_raw(Raw& r, float&) const {
#pragma unroll
    for (int i = 0; i < 4; ++i) r.f[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  // max-abs of the 16 weights, and of the unit from the largest of them
  __device__ __forceinline__ float magnitude(const Raw& r) const {
    return fmaxf(fmaxf(amax4(r.f[0]), amax4(r.f[1])), fmaxf(amax4(r.f[2]), amax4(r.f[3])));
  }
  __device__ __forceinline__ float amax_of(float mag, float) const { return mag; }
  __device__ __forceinline__ float scale_of(long long) const { return 1.0f; }
  __device__ __forceinline__ void load_codes(long long w0, Raw& r) const {
    float unused;
    load_raw(w0, 0, r, unused);
  }
  __device__ __forceinline__ void decode(const Raw& r, float, float (&v)[16]) const {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v[4 * i] = r.f[i].x;
      v[4 * i + 1] = r.f[i].y;
      v[4 * i + 2] = r.f[i].z;
      v[4 * i + 3] = r.f[i].w;
    }
  }
};
template <int BIN>
struct SourcePacked {
  static constexpr int IN_BITS = BIN;
  const uint8_t* packed;
  const void* scales;
  int K, scale_f16;
  __device__ __forceinline__ float scale_of(long long unit) const {
    return scale_f16 ? __half2float(reinterpret_cast<const __half*>(scales)[unit]) : reinterpret_cast<const float*>(scales)[unit];
  }
  __device__ __forceinline__ float4 load4(int n, int k, long long unit) const {
    const uint8_t* row = packed + static_cast<size_t>(n) * (static_cast<size_t>(K) * BIN / 8);
    uint32_t w;  // the codes of the 4 weights, low fields first
    if (BIN == 8) w = *reinterpret_cast<const uint32_t*>(row + k);
    else if (BIN == 4) w = *reinterpret_cast<const uint16_t*>(row + (k >> 1));
    else w = row[k >> 2];
    const float s = scale_f16 ? __half2float(reinterpret_cast<const __half*>(scales)[unit])
                              : reinterpret_cast<const float*>(scales)[unit];
    float v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int q = static_cast<int>(w << (32 - BIN * (c + 1))) >> (32 - BIN);  // sign-extended field
      v[c] = __fmul_rn(static_cast<float>(q), s);
    }
    return make_float4(v[0], v[1], v[2], v[3]);
  }
  static constexpr int STEPS = 2;  // as measured: more steps in flight buy nothing here (the kernel is bound by its instruction count)
  struct Raw {
    uint32_t w[BIN / 2];  // the 16 codes, low fields first
  };
  __device__ __forceinline__ void load_raw(long long w0, long long unit, Raw& r, float& s) const {
    load_codes(w0, r);
    s = scale_of(unit);
  }
  __device__ __forceinline__ void load_codes(long long w0, Raw& r) const {
    const uint8_t* p = packed + w0 * BIN / 8;
    if (BIN == 8) {
      const uint4 q = *reinterpret_cast<const uint4*>(p);
      r.w[0] = q.x, r.w[1] = q.y, r.w[2] = q.z, r.w[3] = q.w;
    } else if (BIN == 4) {
      const uint2 q = *reinterpret_cast<const uint2*>(p);
      r.w[0] = q.x, r.w[1] = q.y;
    } else {
      r.w[0] = *reinterpret_cast<const uint32_t*>(p);
    }
  }
  __device__ __forceinline__ void zero_raw(Raw& r, float& s) const {
#pragma unroll
    for (int i = 0; i < BIN / 2; ++i) r.w[i] = 0u;
    s = 0.0f;
  }
  // max-abs of the 16 codes; the unit's max-abs weight is the product with its scale (rounding is monotone)
  __device__ __forceinline__ float magnitude(const Raw& r) const {
    int m = 0;
    if constexpr (BIN == 8) {
      m = max_abs_code(r.w);
    } else {
      constexpr int PER_WORD = 32 / BIN;
#pragma unroll
      for (int c = 0; c < 16; ++c) m = max(m, abs(static_cast<int>(r.w[c / PER_WORD] << (32 - BIN * (c % PER_WORD + 1))) >> (32 - BIN)));
    }
    return static_cast<float>(m);
  }
  __device__ __forceinline__ float amax_of(float mag, float s) const { return __fmul_rn(mag, s); }
  __device__ __forceinline__ void decode(const Raw& r, float s, float (&v)[16]) const {
    constexpr int PER_WORD = 32 / BIN;
    if constexpr (BIN == 8) {
      // a byte with its sign bit flipped is q + 128; dropped into the low mantissa byte of
      // 1.5 * 2^23 it is the float 12582912 + 128 + q, exactly
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const uint32_t word = r.w[c >> 2] ^ 0x80808080u;
        const uint32_t f = __byte_perm(word, 0x4B400000u, 0x7640u | (c & 3));
        v[c] = __fmul_rn(__uint_as_float(f) - (ROUND_MAGIC + 128.0f), s);
      }
    } else {
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const uint32_t word = r.w[c / PER_WORD];
        const int q = static_cast<int>(word << (32 - BIN * (c % PER_WORD + 1))) >> (32 - BIN);
        v[c] = __fmul_rn(__int_as_float(0x4B400000 + q) - ROUND_MAGIC, s);  // the integer as a float, exactly
      }
    }
  }
};

// scale = max-abs / representable range, IEEE division; stored in the scale channel's type
__device__ __forceinline__ float store_scale(float amax, float range, int scale_f16, void* scales, long long unit, bool writer) {
  float s = __fdiv_rn(amax, range);
  if (scale_f16) {
    const __half h = __float2half_rn(s);
    s = __half2float(h);
    if (writer) reinterpret_cast<__half*>(scales)[unit] = h;
  } else if (writer) {
    reinterpret_cast<float*>(scales)[unit] = s;
  }
  return s;
}

// What the codes of one unit are made with: the stored scale, its reciprocal for the fast
// quotient (NaN where the error bound of the product does not hold: the division then decides
// every code), and the clamp.
struct QuantParams {
  float s, r, qlo, qhi;
};
__device__ __forceinline__ QuantParams quant_params(float s, float amax, float qlo, float qhi) {
  QuantParams p;
  p.s = s;
  // scale 0: reciprocal 0, every product is 0 and every code is 0, as the definition says
  p.r = s == 0.0f ? 0.0f : ((s > 1e-30f && s < 1e30f) ? __frcp_rn(s) : __int_as_float(0x7fc00000));
  // The rounding by addition needs |w * r| well below 2^22.  No weight of the unit exceeds its
  // max-abs and the product is monotone, so one test per unit covers them all (it fails only
  // where the stored scale lost its precision to fp16's subnormal range).
  if (!(__fmul_rn(amax, p.r) < 200.0f)) p.r = __int_as_float(0x7fc00000);
  p.qlo = qlo;
  p.qhi = qhi;
  return p;
}
// Adding and subtracting 1.5 * 2^23 rounds a float of magnitude below 2^22 to the nearest integer,
// ties to even (the addition's own rounding); after the addition the integer sits in the low
// mantissa bits in two's complement.
// one code (its low bits are the field): round-half-even of the fp32 quotient e / s, clamped
__device__ __forceinline__ uint32_t quantise1(float e, const QuantParams& p) {
  const float t = __fmul_rn(e, p.r);  // never contracted into the addition below
  float q = __fsub_rn(__fadd_rn(t, ROUND_MAGIC), ROUND_MAGIC);
  const float d = fabsf(fabsf(t - q) - 0.5f);
  if (!(d >= 1e-4f)) q = rintf(__fdiv_rn(e, p.s));  // also every weight of a unit whose reciprocal is NaN
  q = fminf(fmaxf(q, p.qlo), p.qhi);
  return __float_as_uint(__fadd_rn(q, ROUND_MAGIC));
}

// codes of 4 weights: round half to even on the quotient by the stored scale, clamp, pack
template <int BITS>
__device__ __forceinline__ uint32_t quantise4(const float4& v, const QuantParams& p) {
  constexpr int MASK = (1 << BITS) - 1;
  const float e[4] = {v.x, v.y, v.z, v.w};
  uint32_t word = 0;
#pragma unroll
  for (int c = 0; c < 4; ++c) word |= (quantise1(e[c], p) & MASK) << (BITS * c);
  return word;
}

// the codes of 16 consecutive weights, by one store
template <int BITS>
__device__ __forceinline__ void store_codes(const float (&v)[16], const QuantParams& p, uint8_t* out) {
  constexpr int MASK = (1 << BITS) - 1, PER_WORD = 32 / BITS;
  uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int c = 0; c < 16; ++c) w[c / PER_WORD] |= (quantise1(v[c], p) & MASK) << (BITS * (c % PER_WORD));
  if (BITS == 8) *reinterpret_cast<uint4*>(out) = make_uint4(w[0], w[1], w[2], w[3]);
  else if (BITS == 4) *reinterpret_cast<uint2*>(out) = make_uint2(w[0], w[1]);
  else *reinterpret_cast<uint32_t*>(out) = w[0];
}

// ---- 8-bit codes to narrower ones: bound by instructions per weight, so the weights stay integers ----
// A new code is the old one times the quotient of the scales, rounded; with that quotient as a fixed-point number of
// 24 fractional bits an integer multiply-add leaves it in the result's top byte.  The fixed-point product is
// within 2^-16 of the value the definition rounds (two products, one division and one reciprocal, each rounded once,
// and half a unit of the quotient), so both round alike unless that value lies as close to a half-integer: the
// products on both sides of every half-integer are looked at once per unit, and a warp that finds a close one (even
// maxima make near-ties) takes the general code.
struct FixedQuotient {
  int mul;
  bool close;  // a threshold this lane looked at may be decided differently by the definition
};
// m: the unit's largest code; the lane looks at the thresholds of the codes k0, k0 + stride, ... up to the largest
template <int BITS>
__device__ __forceinline__ FixedQuotient fixed_quotient(int m, float s_in, const QuantParams& p, int k0, int stride) {
  constexpr int K_MAX = 1 << (BITS - 1), HALF = 1 << 23, NEAR = 256;  // NEAR: 2^-16
  FixedQuotient f;
  const float rho = __fmul_rn(s_in, p.r);
  f.close = !(__fmul_rn(static_cast<float>(m), rho) < 100.0f);  // also where the reciprocal is NaN
  f.mul = f.close ? 0 : __float2int_rn(__fmul_rn(rho, 16777216.0f));
  f.close |= ((m * f.mul + HALF) >> 24) > -static_cast<int>(p.qlo);  // a negative code would have to be clamped
  const float inv = 1.0f / rho;
  for (int k = k0; k <= K_MAX; k += stride) {
    const int edge = (k << 24) - HALF;
    const int a = min(static_cast<int>(ceilf((static_cast<float>(k) - 0.5f) * inv)), m + 1);  // first code that becomes k
    f.close |= (a <= m && a * f.mul - edge <= NEAR) || edge - (a - 1) * f.mul <= NEAR;
  }
  return f;
}
// 16 codes by the fixed-point quotient; out: their packed bytes (16 * BITS / 8 of them)
template <int BITS>
__device__ __forceinline__ void store_fixed(const uint32_t (&w8)[4], int mul, int hi, uint8_t* out, bool live) {
  uint32_t c[16];  // the new code in the top byte
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int q = static_cast<int>(sign_bytes(w8[i >> 2], (i & 3) * 0x1111u + 0x8880u));
    c[i] = static_cast<uint32_t>(min(q * mul + (1 << 23), hi));
  }
  // top bytes of every second code (4 bits) or fourth code (2 bits), then shifted into each other
  auto top4 = [](uint32_t a, uint32_t b, uint32_t d, uint32_t e) {
    return __byte_perm(__byte_perm(a, b, 0x0073u), __byte_perm(d, e, 0x0073u), 0x5410u);
  };
  if constexpr (BITS == 4) {
    uint32_t w[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const uint32_t lo = top4(c[8 * i], c[8 * i + 2], c[8 * i + 4], c[8 * i + 6]), up = top4(c[8 * i + 1], c[8 * i + 3], c[8 * i + 5], c[8 * i + 7]);
      w[i] = (lo & 0x0F0F0F0Fu) | ((up << 4) & 0xF0F0F0F0u);
    }
    if (live) *reinterpret_cast<uint2*>(out) = make_uint2(w[0], w[1]);
  } else {
    uint32_t w = 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) w |= (top4(c[i], c[i + 4], c[i + 8], c[i + 12]) & 0x03030303u) << (2 * i);
    if (live) *reinterpret_cast<uint32_t*>(out) = w;
  }
}

// Groups of 16 * LANES weights (LANES = 4 or 8).  A warp handles four steps of 512 weights at a time; LANES lanes share
// a unit's codes, LANES / 4 of them prepare a unit each of the lane group's four steps, so that the
// scale arithmetic is spread instead of repeated.  14336 x 12288, groups of 128, 8 to 4 bits: 139 us with a float product,
// two roundings and their test per weight, 85 us like this.
template <int BITS, int LANES>
__device__ __forceinline__ void requant8(const SourcePacked<8>& src, long long n_units, long long warp, long long warps, int lane, float qlo,
                                         float qhi, float range, int scale_f16, uint8_t* packed, void* scales) {
  constexpr int STEPS = 4, PARTS = LANES / STEPS, UNITS = 32 / LANES;  // units per step
  const int hi = (static_cast<int>(qhi) << 24) | 0xffffff;
  const int in_unit = lane & (LANES - 1), group = lane / LANES, own = in_unit / PARTS;  // own: the step whose unit this lane prepares
  const long long n_steps = (n_units + UNITS - 1) / UNITS;
  for (long long st0 = warp * STEPS; st0 < n_steps; st0 += warps * STEPS) {
    SourcePacked<8>::Raw raws[STEPS];
    float unused;
#pragma unroll
    for (int u = 0; u < STEPS; ++u) {
      const long long unit = (st0 + u) * UNITS + group;
      if (unit < n_units) src.load_codes((unit * LANES + in_unit) * 16, raws[u]);
      else src.zero_raw(raws[u], unused);
    }
    const long long own_unit = (st0 + own) * UNITS + group;
    const float s_in = own_unit < n_units ? src.scale_of(own_unit) : 0.0f;
    uint32_t mag[STEPS / 2] = {};  // max-abs codes of two steps each
#pragma unroll
    for (int u = 0; u < STEPS; ++u) mag[u >> 1] |= static_cast<uint32_t>(max_abs_code(raws[u].w)) << (16 * (u & 1));
#pragma unroll
    for (int o = LANES / 2; o > 0; o >>= 1)
#pragma unroll
      for (int i = 0; i < STEPS / 2; ++i) mag[i] = max_s16x2(mag[i], __shfl_xor_sync(0xffffffffu, mag[i], o));
    const int m = static_cast<int>(((own & 2) ? mag[1] : mag[0]) >> (16 * (own & 1))) & 0xffff;
    const float amax = __fmul_rn(static_cast<float>(m), s_in);
    const float s_out = store_scale(amax, range, scale_f16, scales, own_unit, own_unit < n_units && in_unit % PARTS == 0);
    const FixedQuotient f = fixed_quotient<BITS>(m, s_in, quant_params(s_out, amax, qlo, qhi), 1 + in_unit % PARTS, PARTS);
    const bool general = __any_sync(0xffffffffu, f.close);
#pragma unroll
    for (int u = 0; u < STEPS; ++u) {
      const long long unit = (st0 + u) * UNITS + group;
      const int from = group * LANES + u * PARTS;
      const bool live = unit < n_units;
      uint8_t* out = packed + (unit * LANES + in_unit) * (2 * BITS);
      if (!general) {
        store_fixed<BITS>(raws[u].w, __shfl_sync(0xffffffffu, f.mul, from), hi, out, live);
      } else {
        const float si = __shfl_sync(0xffffffffu, s_in, from), so = __shfl_sync(0xffffffffu, s_out, from), am = __shfl_sync(0xffffffffu, amax, from);
        float v[16];
        src.decode(raws[u], si, v);
        if (live) store_codes<BITS>(v, quant_params(so, am, qlo, qhi), out);
      }
    }
  }
}

// how the units of a matrix are handled (16 weights per lane in the first two): a power of two of lanes each, the whole
// matrix being one run of units; some of a CTA's warps each; any group, four weights per lane
__host__ __device__ __forceinline__ bool dense_groups(int G) { return G >= 32 && G <= 512 && (G & (G - 1)) == 0; }
__host__ __device__ __forceinline__ bool wide_groups(int G) { return G % 16 == 0 && G > 256; }
__host__ __device__ __forceinline__ int warps_per_unit(int G) { return G > 2048 ? 8 : (G > 1024 ? 4 : (G > 512 ? 2 : 1)); }

// one kernel per way of handling the units, so that none pays for the registers of another
struct QuantArgs {
  int N, K, G, ngroups, scale_f16;
  float qlo, qhi, range;  // clamp of the codes; max-abs is divided by range
  uint8_t* packed;
  void* scales;
};

template <int BITS, int LANES>
__global__ void __launch_bounds__(256, 4) requant8_kernel(const SourcePacked<8> src, const QuantArgs a) {
  const int lane = threadIdx.x & 31;
  const long long n_units = static_cast<long long>(a.N) * a.ngroups;
  const long long warps = (static_cast<long long>(gridDim.x) * blockDim.x) >> 5;
  const long long warp = (static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  requant8<BITS, LANES>(src, n_units, warp, warps, lane, a.qlo, a.qhi, a.range, a.scale_f16, a.packed, a.scales);
}

// 4 to 2 bits, groups of 128
__global__ void __launch_bounds__(256, 4) requant4to2_kernel(const SourcePacked<4> src, const QuantArgs a) {
  const int lane = threadIdx.x & 31;
  const long long n_units = static_cast<long long>(a.N) * a.ngroups;
  const long long warps = (static_cast<long long>(gridDim.x) * blockDim.x) >> 5;
  const long long warp = (static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  // A 4-bit unit holds at most 16 different weights: the unit's 8 lanes quantise two of the 16
  // possible codes each (with the very function every other path uses), share the results as a
  // table of 16 x 2 bits, and every stored code is then a table lookup.  The unit's max-abs is
  // s * max |q| (rounding is monotone), found on the integer codes.
  constexpr int STEPS = SourcePacked<4>::STEPS;
  const long long n_steps = (n_units + 3) >> 2;
  for (long long st0 = warp * STEPS; st0 < n_steps; st0 += warps * STEPS) {
    SourcePacked<4>::Raw raws[STEPS];
    float s_ins[STEPS];
#pragma unroll
    for (int u = 0; u < STEPS; ++u) {
      const long long unit = (st0 + u) * 4 + (lane >> 3);
      if (unit < n_units) src.load_raw(unit * 128 + (lane & 7) * 16, unit, raws[u], s_ins[u]);
      else src.zero_raw(raws[u], s_ins[u]);
    }
#pragma unroll
    for (int u = 0; u < STEPS; ++u) {
      const long long unit = (st0 + u) * 4 + (lane >> 3);
      const bool live = unit < n_units;
      const uint32_t rx = raws[u].w[0], ry = raws[u].w[1];
      const float s_in = s_ins[u];
      int m = 0;
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const uint32_t word = c < 8 ? rx : ry;
        const int q = static_cast<int>(word << (28 - 4 * (c & 7))) >> 28;
        m = max(m, abs(q));
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
      const float amax = __fmul_rn(static_cast<float>(m), s_in);
      const QuantParams p = quant_params(store_scale(amax, a.range, a.scale_f16, a.scales, unit, live && (lane & 7) == 0), amax, a.qlo, a.qhi);
      uint32_t lut = 0;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int nib = 2 * (lane & 7) + i;
        const int q = (nib ^ 8) - 8;  // the field's value
        lut |= (quantise1(__fmul_rn(static_cast<float>(q), s_in), p) & 3u) << (2 * nib);
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) lut |= __shfl_xor_sync(0xffffffffu, lut, o);
      uint32_t out = 0;
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const uint32_t word = c < 8 ? rx : ry;
        const uint32_t nib2 = ((word >> (4 * (c & 7))) << 1) & 30u;
        out |= ((lut >> nib2) & 3u) << (2 * c);
      }
      if (live) *reinterpret_cast<uint32_t*>(a.packed + (unit * 128 + (lane & 7) * 16) / 4) = out;
    }
  }
}

// LANES: lanes per unit (8: groups of 128), or 0: as the group says
template <int BITS, typename Source, int LANES>
__global__ void __launch_bounds__(256, 5) quantise_dense_kernel(const Source src, const QuantArgs a) {
  const int lane = threadIdx.x & 31;
  const long long n_units = static_cast<long long>(a.N) * a.ngroups;
  const long long warps = (static_cast<long long>(gridDim.x) * blockDim.x) >> 5;
  const long long warp = (static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  // K is a whole number of units, so unit u holds the weights G u .. G u + G - 1 of the dense
  // matrix and the bytes G b u / 8 .. of the a.packed one, whatever its row
  constexpr int STEPS = Source::STEPS;
  const int G = LANES ? 16 * LANES : a.G, lanes = G >> 4, shift = __ffs(lanes) - 1, in_unit = lane & (lanes - 1), per_step = 32 >> shift;
  const long long n_steps = (n_units + per_step - 1) >> (5 - shift);
  for (long long st0 = warp * STEPS; st0 < n_steps; st0 += warps * STEPS) {
    typename Source::Raw raws[STEPS];
    float s_ins[STEPS];
#pragma unroll
    for (int u = 0; u < STEPS; ++u) {
      const long long unit = (st0 + u) * per_step + (lane >> shift);
      if (unit < n_units) src.load_raw(unit * G + in_unit * 16, unit, raws[u], s_ins[u]);
      else src.zero_raw(raws[u], s_ins[u]);
    }
#pragma unroll
    for (int u = 0; u < STEPS; ++u) {
      const long long unit = (st0 + u) * per_step + (lane >> shift);
      const bool live = unit < n_units;
      float v[16];
      src.decode(raws[u], s_ins[u], v);
      float amax = 0.0f;
#pragma unroll
      for (int c = 0; c < 16; ++c) amax = fmaxf(amax, fabsf(v[c]));
      for (int o = lanes >> 1; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
      const QuantParams p = quant_params(store_scale(amax, a.range, a.scale_f16, a.scales, unit, live && in_unit == 0), amax, a.qlo, a.qhi);
      if (live) store_codes<BITS>(v, p, a.packed + (unit * G + in_unit * 16) * BITS / 8);
    }
  }
}

template <int BITS, typename Source>
__global__ void __launch_bounds__(256) quantise_wide_kernel(const Source src, const QuantArgs a) {
  const int lane = threadIdx.x & 31, G = a.G;
  const long long n_units = static_cast<long long>(a.N) * a.ngroups;
  // long units of any multiple of 16 weights (per-channel a.scales): as many of the CTA's warps on a unit as
  // give every lane its 16 weights, which then are read once; a longer unit is read a second time for its codes
  __shared__ float s_mag[8];
  const int wpu = warps_per_unit(G), slot = (threadIdx.x >> 5) / wpu, sub = (threadIdx.x >> 5) % wpu;
  const int first = (sub * 32 + lane) * 16, stride = wpu * 512, upb = 8 / wpu;
  for (long long base = static_cast<long long>(blockIdx.x) * upb; base < n_units; base += static_cast<long long>(gridDim.x) * upb) {
    const long long unit = min(base + slot, n_units - 1);  // (a unit beyond the last: the last one once more)
    const long long w0 = unit * G;
    const float s_in = src.scale_of(unit);
    typename Source::Raw raw, next;
    float mag = 0.0f, unused;
    if (first < G) src.load_codes(w0 + first, raw);
    else src.zero_raw(raw, unused);
    mag = src.magnitude(raw);
    for (int i = first + stride; i < G; i += stride) {
      src.load_codes(w0 + i, next);
      mag = fmaxf(mag, src.magnitude(next));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mag = fmaxf(mag, __shfl_xor_sync(0xffffffffu, mag, o));
    if (wpu > 1) {
      if (lane == 0) s_mag[threadIdx.x >> 5] = mag;
      __syncthreads();
      for (int i = 0; i < wpu; ++i) mag = fmaxf(mag, s_mag[slot * wpu + i]);
      __syncthreads();
    }
    const float amax = src.amax_of(mag, s_in);
    const QuantParams p = quant_params(store_scale(amax, a.range, a.scale_f16, a.scales, unit, sub == 0 && lane == 0), amax, a.qlo, a.qhi);
    FixedQuotient f = {0, true};
    if constexpr (Source::IN_BITS == 8 && BITS < 8) {
      f = fixed_quotient<BITS>(static_cast<int>(mag), s_in, p, 1 + (lane & 7), 8);
      f.close = __any_sync(0xffffffffu, f.close);
    }
    for (int i = first; i < G; i += stride) {
      if (i != first) src.load_codes(w0 + i, raw);
      uint8_t* out = a.packed + (w0 + i) * BITS / 8;
      if constexpr (Source::IN_BITS == 8 && BITS < 8) {
        if (!f.close) {
          store_fixed<BITS>(raw.w, f.mul, (static_cast<int>(a.qhi) << 24) | 0xffffff, out, true);
          continue;
        }
      }
      float v[16];
      src.decode(raw, s_in, v);
      store_codes<BITS>(v, p, out);
    }
  }
}

template <int BITS, typename Source>
__global__ void __launch_bounds__(256) quantise_kernel(const Source src, const QuantArgs a) {
  typedef typename PackWord<BITS>::type word_t;
  const int lane = threadIdx.x & 31;
  const long long n_units = static_cast<long long>(a.N) * a.ngroups;
  const long long warps = (static_cast<long long>(gridDim.x) * blockDim.x) >> 5;
  const long long warp = (static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int G = a.G, ngroups = a.ngroups;
  const size_t row_bytes = static_cast<size_t>(a.K) * BITS / 8;
  for (long long unit = warp; unit < n_units; unit += warps) {
    const int n = static_cast<int>(unit / ngroups);
    const int g = static_cast<int>(unit % ngroups);
    const int k_first = g * G;
    // every lane owns 4 consecutive weights per 128-weight step; the first step stays in registers
    float4 first = make_float4(0.f, 0.f, 0.f, 0.f);
    float amax = 0.0f;
    for (int i = lane * 4; i < G; i += 128) {
      const float4 v = src.load4(n, k_first + i, unit);
      if (i < 128) first = v;
      amax = fmaxf(amax, amax4(v));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    const QuantParams p = quant_params(store_scale(amax, a.range, a.scale_f16, a.scales, unit, lane == 0), amax, a.qlo, a.qhi);
    word_t* out = reinterpret_cast<word_t*>(a.packed + static_cast<size_t>(n) * row_bytes + static_cast<size_t>(g) * G * BITS / 8);
    for (int i = lane * 4; i < G; i += 128) {
      const float4 v = i < 128 ? first : src.load4(n, k_first + i, unit);  // later steps come from L1/L2
      out[i >> 2] = static_cast<word_t>(quantise4<BITS>(v, p));
    }
  }
}

template <int BITS, typename Source>
cudaError_t launch_bits(const Source& src, int N, int K, int group, int scale_f16, int full_range, uint8_t* packed, void* scales,
                        cudaStream_t st) {
  QuantArgs a;
  a.N = N;
  a.K = K;
  a.G = group > 0 ? group : K;
  a.ngroups = K / a.G;
  a.scale_f16 = scale_f16;
  a.qhi = static_cast<float>((1 << (BITS - 1)) - 1);
  a.qlo = full_range ? -static_cast<float>(1 << (BITS - 1)) : -a.qhi;
  a.range = full_range ? static_cast<float>(1 << (BITS - 1)) : a.qhi;
  a.packed = packed;
  a.scales = scales;
  const bool dense = dense_groups(a.G), wide = !dense && wide_groups(a.G);
  const bool fixed8 = Source::IN_BITS == 8 && BITS < 8 && (a.G == 128 || a.G == 64);
  const long long units = static_cast<long long>(N) * a.ngroups;
  const long long step_units = dense ? 512 / a.G * (fixed8 ? 4 : Source::STEPS) : 1;  // units a warp takes at a time
  const long long warps_needed = (units + step_units - 1) / step_units * (wide ? warps_per_unit(a.G) : 1);
  const int threads = 256;
  long long blocks = (warps_needed * 32 + threads - 1) / threads;
  const long long cap = 148LL * 8 * 4;  // a few waves of resident blocks; each warp then loops over its units
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  const dim3 grid(static_cast<unsigned>(blocks));
  if constexpr (Source::IN_BITS == 8 && BITS < 8) {
    if (fixed8) {
      if (a.G == 128) requant8_kernel<BITS, 8><<<grid, threads, 0, st>>>(src, a);
      else requant8_kernel<BITS, 4><<<grid, threads, 0, st>>>(src, a);
      return cudaGetLastError();
    }
  }
  if constexpr (Source::IN_BITS == 4 && BITS == 2) {
    if (a.G == 128) {
      requant4to2_kernel<<<grid, threads, 0, st>>>(src, a);
      return cudaGetLastError();
    }
  }
  if (a.G == 128) quantise_dense_kernel<BITS, Source, 8><<<grid, threads, 0, st>>>(src, a);
  else if (dense) quantise_dense_kernel<BITS, Source, 0><<<grid, threads, 0, st>>>(src, a);
  else if (wide) quantise_wide_kernel<BITS, Source><<<grid, threads, 0, st>>>(src, a);
  else quantise_kernel<BITS, Source><<<grid, threads, 0, st>>>(src, a);
  return cudaGetLastError();
}

template <typename Source>
cudaError_t launch_quantise(const Source& src, int N, int K, int bits, int group, int scale_f16, int full_range,
                            uint8_t* packed, void* scales, cudaStream_t st) {
  switch (bits) {
    case 2: return launch_bits<2>(src, N, K, group, scale_f16, full_range, packed, scales, st);
    case 4: return launch_bits<4>(src, N, K, group, scale_f16, full_range, packed, scales, st);
    case 8: return launch_bits<8>(src, N, K, group, scale_f16, full_range, packed, scales, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_pack(const float* W, int N, int K, int bits, int group, int scale_f16, int full_range, uint8_t* packed,
                        void* scales, cudaStream_t st) {
  return launch_quantise(SourceF32{W, K}, N, K, bits, group, scale_f16, full_range, packed, scales, st);
}

cudaError_t launch_requant(const uint8_t* in_packed, const void* in_scales, int N, int K, int bits_in, int bits_out,
                           int group, int scale_f16, int full_range, uint8_t* packed, void* scales, cudaStream_t st) {
  switch (bits_in) {
    case 2: return launch_quantise(SourcePacked<2>{in_packed, in_scales, K, scale_f16}, N, K, bits_out, group, scale_f16, full_range, packed, scales, st);
    case 4: return launch_quantise(SourcePacked<4>{in_packed, in_scales, K, scale_f16}, N, K, bits_out, group, scale_f16, full_range, packed, scales, st);
    case 8: return launch_quantise(SourcePacked<8>{in_packed, in_scales, K, scale_f16}, N, K, bits_out, group, scale_f16, full_range, packed, scales, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace emoe
