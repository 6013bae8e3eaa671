// Router logits and Top-K gating as device functions (paper Section 2.1: a trained router sends
// every token to its Top-K experts), shared by the kernels that route: the router kernel, the
// one-launch routing kernel and the one-launch decode layer.
#pragma once
#include <math_constants.h>

#include <type_traits>

#include "common.cuh"

namespace emoe {

constexpr int ROUTER_THREADS = 256;
constexpr int ROUTER_DC = 1024;  // d_model chunk held in shared memory (1 and 8 tokens per CTA)
// tokens per CTA -> chunk: 32 tokens take chunks of 256 so that their rows still fit shared memory
__host__ __device__ constexpr int router_dc(int tt) { return tt > 8 ? 256 : ROUTER_DC; }

// The router comes first in a call, so the kernel in front of it may be the one that writes its inputs (the previous
// layer, whose last kernel lets this one start before it has stored y): nothing is read before pdl_wait().  Until
// then the lines are only pulled towards L2, which keeps no stale copy of them, by thread tid of nt.
__device__ __forceinline__ void prefetch_l2(const void* from, size_t bytes, int tid, int nt) {
  for (size_t b = 128 * static_cast<size_t>(tid); b < bytes; b += 128 * static_cast<size_t>(nt))
    asm volatile("prefetch.global.L2 [%0];" ::"l"(static_cast<const char*>(from) + b));
}
// rows t0 .. t0 + rows - 1 of x, and this CTA's share of the router weights
__device__ __forceinline__ void router_prefetch(const void* x, int x_bf16, int t0, int rows, int d, const float* Wr, int E, int tid, int nt) {
  const size_t row_bytes = static_cast<size_t>(d) * (x_bf16 ? 2 : 4), w_bytes = static_cast<size_t>(d) * E * 4;
  prefetch_l2(static_cast<const char*>(x) + t0 * row_bytes, rows * row_bytes, tid, nt);
  prefetch_l2(Wr, w_bytes, static_cast<int>(blockIdx.x) * nt + tid, static_cast<int>(gridDim.x) * nt);
}

// Logits of the CTA's TT tokens into zs[TT][EP] (shared memory).
template <int TT>
__device__ __forceinline__ void router_logits(float* smem, const void* __restrict__ x, int x_bf16, int T, int d,
                                              const float* __restrict__ Wr, const float* __restrict__ bias,
                                              int bias_stride, int E, int EP, int ep_shift, float* __restrict__ logits) {
  constexpr int DC = router_dc(TT);
  float* xs = smem;                          // [TT][DC]
  float* red = xs + TT * DC;                 // [S][TT][EP]
  float* zs = red + ROUTER_THREADS * TT;     // [TT][EP]
  const int tid = threadIdx.x;
  const int e = tid & (EP - 1);
  const int slice = tid >> ep_shift;
  const int S = ROUTER_THREADS >> ep_shift;
  const int t0 = blockIdx.x * TT;

  float acc[TT];
#pragma unroll
  for (int tt = 0; tt < TT; ++tt) acc[tt] = 0.0f;

  router_prefetch(x, x_bf16, t0, min(TT, T - t0), d, Wr, E, tid, ROUTER_THREADS);
  pdl_wait();
  for (int c0 = 0; c0 < d; c0 += DC) {
    const int dc = min(DC, d - c0);
    __syncthreads();
    for (int tt = 0; tt < TT; ++tt) {
      const int t = t0 + tt;
      for (int i = tid; i < dc; i += ROUTER_THREADS) {
        float v = 0.0f;
        if (t < T) {
          const size_t src = static_cast<size_t>(t) * d + c0 + i;
          v = x_bf16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(x)[src])
                     : reinterpret_cast<const float*>(x)[src];
        }
        xs[tt * DC + i] = v;
      }
    }
    __syncthreads();
    if (e < E) {
      // many independent router-weight loads in flight per thread (the loop is L2-latency bound;
      // with one token per CTA the registers allow 24)
      constexpr int U = TT == 1 ? 24 : 8;
      for (int i = slice; i < dc; i += U * S) {
        float w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int ii = i + u * S;
          w[u] = ii < dc ? __ldcg(Wr + static_cast<size_t>(c0 + ii) * E + e) : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int ii = min(i + u * S, dc - 1);
#pragma unroll
          for (int tt = 0; tt < TT; ++tt) acc[tt] = fmaf(xs[tt * DC + ii], w[u], acc[tt]);
        }
      }
    }
  }
#pragma unroll
  for (int tt = 0; tt < TT; ++tt) red[(slice * TT + tt) * EP + e] = acc[tt];
  __syncthreads();
  for (int idx = tid; idx < TT * EP; idx += ROUTER_THREADS) {
    const int tt = idx >> ep_shift, ee = idx & (EP - 1);
    const int t = t0 + tt;
    float z = 0.0f;
    for (int s = 0; s < S; ++s) z += red[(s * TT + tt) * EP + ee];
    if (ee < E && t < T) {
      if (bias) z += bias[static_cast<size_t>(t) * bias_stride + ee];
      if (logits) logits[static_cast<size_t>(t) * E + ee] = z;
    }
    zs[idx] = z;
  }
  __syncthreads();
}

// Logits of one token into zs[EP]: bound by the round trips to memory, so everything a thread reads is requested at
// once, with nothing staged in front: ROUTER_ONE_FLY pieces of four experts' weights per thread and the activation that
// belongs to each (up to 32 K products per round trip).  E a power of two, at least four: a thread keeps to four
// experts.  4 tokens x 4096 x 8 experts, back to back: 12.3 us with chunks staged in shared memory, 8.0 so.
constexpr int ROUTER_ONE_THREADS = 512, ROUTER_ONE_FLY = 16;
__host__ __device__ constexpr int router_one_rows(int E) { return ROUTER_ONE_THREADS * 4 / (E > 128 ? E : 128); }  // partial sums per expert
__host__ __device__ constexpr int router_one_smem(int E) { return (router_one_rows(E) + 1) * E * 4; }
// Can also run on fewer threads (NT), which then take the work of several in turn: the sums are the same to the bit.
__host__ __device__ __forceinline__ bool router_one_supported(int E, const void* Wr) {
  return E >= 4 && (E & (E - 1)) == 0 && reinterpret_cast<uintptr_t>(Wr) % 16 == 0;
}
template <int NT, int FLY>
__device__ __forceinline__ void router_logits_one(float* smem, const void* __restrict__ x, int x_bf16, int d, const float* __restrict__ Wr,
                                                  const float* __restrict__ bias, int bias_stride, int E, int ep_shift,
                                                  float* __restrict__ logits) {
  float* zs = smem;        // [E]
  float* red = smem + E;   // [rows][E]
  const int tid = threadIdx.x, t = blockIdx.x, sh = ep_shift - 2, quads = 1 << sh;
  const int n = d << sh;   // pieces
  router_prefetch(x, x_bf16, t, 1, d, Wr, E, tid, NT);
  pdl_wait();
  const auto product = [&](const auto* xrow, int vt) {
    float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int base = vt; base < n; base += FLY * ROUTER_ONE_THREADS) {
      float4 w[FLY];
      std::decay_t<decltype(*xrow)> v[FLY];
#pragma unroll
      for (int u = 0; u < FLY; ++u) {  // nothing is converted between the loads: they are to leave together
        const int i = base + u * ROUTER_ONE_THREADS;
        if (i < n) {
          w[u] = __ldcg(reinterpret_cast<const float4*>(Wr) + i);
          v[u] = __ldcg(xrow + (i >> sh));
        }
      }
#pragma unroll
      for (int u = 0; u < FLY; ++u) {
        if (base + u * ROUTER_ONE_THREADS >= n) break;
        const float xv = static_cast<float>(v[u]);
        acc.x = fmaf(xv, w[u].x, acc.x);
        acc.y = fmaf(xv, w[u].y, acc.y);
        acc.z = fmaf(xv, w[u].z, acc.z);
        acc.w = fmaf(xv, w[u].w, acc.w);
      }
    }
    return acc;
  };
  for (int vt = tid; vt < ROUTER_ONE_THREADS; vt += NT) {
    float4 acc = x_bf16 ? product(static_cast<const __nv_bfloat16*>(x) + static_cast<size_t>(t) * d, vt)
                        : product(static_cast<const float*>(x) + static_cast<size_t>(t) * d, vt);
    for (int o = 16; o >= quads; o >>= 1) {  // lanes with the same experts
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
      acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
      acc.z += __shfl_xor_sync(0xffffffffu, acc.z, o);
      acc.w += __shfl_xor_sync(0xffffffffu, acc.w, o);
    }
    if ((vt & 31) < quads)
      *reinterpret_cast<float4*>(red + static_cast<size_t>(vt / max(32, quads)) * E + 4 * (vt & (quads - 1))) = acc;
  }
  __syncthreads();
  for (int e = tid; e < E; e += NT) {
    float z = 0.0f;
    for (int row = 0; row < router_one_rows(E); ++row) z += red[row * E + e];
    if (bias) z += bias[static_cast<size_t>(t) * bias_stride + e];
    if (logits) logits[static_cast<size_t>(t) * E + e] = z;
    zs[e] = z;
  }
  __syncthreads();
}

// Logits of the CTA's TT tokens into zs[TT][EP] as a register-tiled product, for batches: a thread holds TT/2 tokens x
// four experts and an interleaved part of the inputs, so that an activation is read once per four
// experts and a router weight once per TT/2 tokens; with one expert per thread (router_logits) every
// product needed a shared-memory read of its own.  Chunks of BC inputs: the weights arrive by
// cp.async two chunks ahead, the activations one chunk ahead in registers (they become fp32,
// [input][token], on their way into shared memory).  E a multiple of four.
constexpr int ROUTER_BATCH_THREADS = 512;  // sixteen warps: the loop waits for shared memory with fewer
__host__ __device__ constexpr int router_batch_chunk(int EP) { return EP <= 16 ? 512 : (EP == 32 ? 256 : (EP <= 128 ? 128 : 64)); }
__host__ __device__ constexpr int router_batch_stages(int EP) { return EP > 64 ? 2 : 3; }
// weights' stages (the partial sums follow in the same memory), activations, logits
__host__ __device__ constexpr int router_batch_floats_w(int tt, int EP) {
  return router_batch_stages(EP) * router_batch_chunk(EP) * EP > 2 * ROUTER_BATCH_THREADS * tt ? router_batch_stages(EP) * router_batch_chunk(EP) * EP
                                                                                         : 2 * ROUTER_BATCH_THREADS * tt;
}
__host__ __device__ constexpr int router_batch_smem(int tt, int EP) {
  return (router_batch_floats_w(tt, EP) + tt * router_batch_chunk(EP) + tt * EP) * 4;
}
// the most that any number of experts with chunks of bc inputs takes
constexpr int router_batch_most(int tt, int bc) {
  int most = 0;
  for (int EP = 4; EP <= EMOE_MAX_EXPERTS; EP *= 2)
    if (router_batch_chunk(EP) == bc && router_batch_smem(tt, EP) > most) most = router_batch_smem(tt, EP);
  return most;
}

template <int TT, int BC>
__device__ __forceinline__ void router_logits_batch(float* smem, const void* __restrict__ x, int x_bf16, int T, int d,
                                                    const float* __restrict__ Wr, const float* __restrict__ bias, int bias_stride, int E,
                                                    int EP, int ep_shift, float* __restrict__ logits) {
  constexpr int TG = 2, TPT = TT / TG;  // token groups, tokens per thread
  const int stages = router_batch_stages(EP);
  float* ws = smem;                                   // [stages][BC][E]
  float* xs = smem + router_batch_floats_w(TT, EP);   // [BC][TT]
  float* zs = xs + TT * BC;                           // [TT][EP]
  float* red = smem;                                  // [S][TT][EP]
  const int tid = threadIdx.x, t0 = blockIdx.x * TT;
  const int eg_shift = ep_shift - 2;                  // groups of four experts
  const int eg = tid & ((1 << eg_shift) - 1), tg = (tid >> eg_shift) & (TG - 1), ks = tid >> (eg_shift + 1);
  const int S = ROUTER_BATCH_THREADS >> (eg_shift + 1);
  const int nchunks = (d + BC - 1) / BC;
  unsigned long long acc[TPT / 2][4];  // pairs of tokens: two fp32 products and sums per instruction
#pragma unroll
  for (int t = 0; t < TPT / 2; ++t)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[t][i] = 0ull;
  auto fetch_w = [&](int c) {  // rows c*BC .. of Wr are one contiguous block; one commit group per chunk, empty past the end
    if (c < nchunks) {
      const int n16 = min(BC, d - c * BC) * E / 4;
      const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(ws + (c % stages) * BC * EP));
      const float* src = Wr + static_cast<size_t>(c) * BC * E;
      for (int i = tid; i < n16; i += ROUTER_BATCH_THREADS)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16 * i), "l"(src + 4 * i) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // activations: a thread moves eight inputs of one token at a time; neighbouring threads take neighbouring tokens
  constexpr int NST = TT * BC / 8 / ROUTER_BATCH_THREADS > 0 ? TT * BC / 8 / ROUTER_BATCH_THREADS : 1;
  uint4 pre[NST][2];
  auto fetch_x = [&](int c) {
#pragma unroll
    for (int i = 0; i < NST; ++i) {
      const int u = tid + i * ROUTER_BATCH_THREADS, tok = t0 + u % TT, k = c * BC + u / TT * 8;
      const bool in = u < TT * BC / 8 && tok < T && k < d;
      pre[i][0] = pre[i][1] = make_uint4(0u, 0u, 0u, 0u);
      if (in) {
        const size_t at = static_cast<size_t>(tok) * d + k;
        if (x_bf16) {
          pre[i][0] = __ldcg(reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(x) + at));
        } else {
          pre[i][0] = __ldcg(reinterpret_cast<const uint4*>(reinterpret_cast<const float*>(x) + at));
          pre[i][1] = __ldcg(reinterpret_cast<const uint4*>(reinterpret_cast<const float*>(x) + at) + 1);
        }
      }
    }
  };
  router_prefetch(x, x_bf16, t0, min(TT, T - t0), d, Wr, E, tid, ROUTER_BATCH_THREADS);
  pdl_wait();
  for (int c = 0; c + 1 < stages; ++c) fetch_w(c);
  fetch_x(0);
  for (int c = 0; c < nchunks; ++c) {
    const int dc = min(BC, d - c * BC);
    if (stages == 3) asm volatile("cp.async.wait_group 1;" ::: "memory");
    else asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // the chunk's weights are here, and the chunk in front is used up
    fetch_w(c + stages - 1);
#pragma unroll
    for (int i = 0; i < NST; ++i) {
      const int u = tid + i * ROUTER_BATCH_THREADS, tok = u % TT, k = u / TT * 8;
      if (u >= TT * BC / 8) break;
      const uint32_t w[8] = {pre[i][0].x, pre[i][0].y, pre[i][0].z, pre[i][0].w, pre[i][1].x, pre[i][1].y, pre[i][1].z, pre[i][1].w};
#pragma unroll
      for (int j = 0; j < 8; ++j)
        xs[(k + j) * TT + tok] = __uint_as_float(!x_bf16 ? w[j] : ((j & 1) ? w[j >> 1] & 0xffff0000u : w[j >> 1] << 16));
    }
    __syncthreads();
    if (c + 1 < nchunks) fetch_x(c + 1);
    if (4 * eg < E) {
      const float* wp = ws + (c % stages) * BC * EP + 4 * eg;
      const float* xp = xs + tg * TPT;
#pragma unroll 4
      for (int i = ks; i < dc; i += S) {
        const float4 w = *reinterpret_cast<const float4*>(wp + i * E);
        unsigned long long xv[TPT / 2], wv[4];
#pragma unroll
        for (int t = 0; t < TPT / 2; t += 2) {
          const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(xp + i * TT + 2 * t);
          xv[t] = v.x;
          xv[t + 1] = v.y;
        }
        asm("mov.b64 %0, {%1, %1};" : "=l"(wv[0]) : "f"(w.x));
        asm("mov.b64 %0, {%1, %1};" : "=l"(wv[1]) : "f"(w.y));
        asm("mov.b64 %0, {%1, %1};" : "=l"(wv[2]) : "f"(w.z));
        asm("mov.b64 %0, {%1, %1};" : "=l"(wv[3]) : "f"(w.w));
#pragma unroll
        for (int t = 0; t < TPT / 2; ++t)
#pragma unroll
          for (int j = 0; j < 4; ++j) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[t][j]) : "l"(xv[t]), "l"(wv[j]));
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // partial sums [part][token][expert], added in order
#pragma unroll
  for (int t = 0; t < TPT / 2; ++t) {
    float lo[4], hi[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) asm("mov.b64 {%0, %1}, %2;" : "=f"(lo[j]), "=f"(hi[j]) : "l"(acc[t][j]));
    float* to = red + (ks * TT + tg * TPT + 2 * t) * EP + 4 * eg;
    *reinterpret_cast<float4*>(to) = make_float4(lo[0], lo[1], lo[2], lo[3]);
    *reinterpret_cast<float4*>(to + EP) = make_float4(hi[0], hi[1], hi[2], hi[3]);
  }
  __syncthreads();
  for (int idx = tid; idx < TT * EP; idx += ROUTER_BATCH_THREADS) {
    const int tt = idx >> ep_shift, ee = idx & (EP - 1);
    const int t = t0 + tt;
    float z = 0.0f;
    for (int s = 0; s < S; ++s) z += red[(s * TT + tt) * EP + ee];
    if (ee < E && t < T) {
      if (bias) z += bias[static_cast<size_t>(t) * bias_stride + ee];
      if (logits) logits[static_cast<size_t>(t) * E + ee] = z;
    }
    zs[idx] = z;
  }
  __syncthreads();
}

// Softmax and Top-K of one token by one warp from its row of logits zrow[EP] (shared memory):
// K rounds of arg-max, ties to the lower expert index.  Lane r < top_k returns the r-th pick.
// MAXJ: values per lane (one suffices up to 32 experts).
template <int MAXJ>
__device__ __forceinline__ void router_pick_of(const float* zrow, int E, int top_k, int renorm, int lane, int& out_id,
                                               float& out_gate) {
  float zv[MAXJ], pe[MAXJ];
  float m = -CUDART_INF_F;
#pragma unroll
  for (int j = 0; j < MAXJ; ++j) {
    const int ee = lane + 32 * j;
    zv[j] = ee < E ? zrow[ee] : -CUDART_INF_F;
    m = fmaxf(m, zv[j]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  float denom = 0.0f;
#pragma unroll
  for (int j = 0; j < MAXJ; ++j) {
    pe[j] = (lane + 32 * j) < E ? expf(zv[j] - m) : 0.0f;
    denom += pe[j];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) denom += __shfl_xor_sync(0xffffffffu, denom, o);

  unsigned taken = 0;
  float psel = 0.0f;
  int my_id = 0;     // lane r keeps the r-th pick
  float my_p = 0.0f;
  for (int r = 0; r < top_k; ++r) {
    float bv = -CUDART_INF_F;
    int bi = 0x7fffffff;
#pragma unroll
    for (int j = 0; j < MAXJ; ++j) {
      const int ee = lane + 32 * j;
      if (ee < E && !((taken >> j) & 1u) && (zv[j] > bv || bi == 0x7fffffff)) {
        bv = zv[j];
        bi = ee;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (oi != 0x7fffffff && (bi == 0x7fffffff || ov > bv || (ov == bv && oi < bi))) {
        bv = ov;
        bi = oi;
      }
    }
    float p = 0.0f;
#pragma unroll
    for (int j = 0; j < MAXJ; ++j)
      if (lane + 32 * j == bi) {
        taken |= 1u << j;
        p = pe[j];
      }
    p = __shfl_sync(0xffffffffu, p, bi & 31) / denom;
    psel += p;
    if (lane == r) {
      my_id = bi;
      my_p = p;
    }
  }
  out_id = my_id;
  out_gate = renorm ? my_p / psel : my_p;
}

__device__ __forceinline__ void router_pick(const float* zrow, int E, int top_k, int renorm, int lane, int& out_id, float& out_gate) {
  if (E <= 32) router_pick_of<1>(zrow, E, top_k, renorm, lane, out_id, out_gate);
  else router_pick_of<EMOE_MAX_EXPERTS / 32>(zrow, E, top_k, renorm, lane, out_id, out_gate);
}

}  // namespace emoe
