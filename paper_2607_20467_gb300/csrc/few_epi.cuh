// The epilogues of the GEMMs whose MMA has the weights on its M side (gemm_few.cu, gemm_mid.cu):
// a tile's sums lie in shared memory as [token][weight row] and leave token by token.
#pragma once

#include "common.cuh"
#include "tc_ptx.cuh"

namespace dcl {
namespace {

constexpr int FW_TILE = 128;           // weight rows of a CTA's tile
constexpr int FW_PITCH = FW_TILE + 4;  // fp32 per token of a staged sum

struct FewArgs {
  int nkb;  // K blocks
  int N, M;
  FewEpi ep;
};

// h += v without a return value (one add per element: no order to depend on)
__device__ __forceinline__ void red_add_v4(float* p, const float4& v) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
               : "memory");
}

// Four consecutive rows' sums (address `at` in every CTA of the cluster) of NP tokens, `step`
// bytes apart, added in K order.  All S * NP loads are issued before any is used, 16 bytes
// each: distributed shared memory is slow per access (adding rank after rank, 4 bytes a
// load, the pass took 5 us).
template <int S, int NP>
__device__ __forceinline__ void cluster_sums(uint32_t at, uint32_t step, int n, float4 (&x)[NP]) {
  float4 v[S][NP];
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const uint32_t from = S == 1 ? at : map_cluster(at, s);
#pragma unroll
    for (int i = 0; i < NP; ++i)
      if (i < n) v[s][i] = S == 1 ? ld_shared_v4(from + i * step) : ld_cluster_v4(from + i * step);
  }
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    x[i] = v[0][i];
#pragma unroll
    for (int s = 1; s < S; ++s) {
      x[i].x += v[s][i].x;
      x[i].y += v[s][i].y;
      x[i].z += v[s][i].z;
      x[i].w += v[s][i].w;
    }
  }
}

__device__ __forceinline__ void store_bf16x4(__nv_bfloat16* o, float a, float b, float c, float d) {
  *reinterpret_cast<uint2*>(o) = make_uint2(pack_bf16x2(a, b), pack_bf16x2(c, d));
}

// Tokens t0 .. t1 - 1 of the tile, by the 128 epilogue threads (et), four consecutive rows per
// thread.  sum: the staged sums [token][FW_PITCH], at the same shared address in each of the
// cluster's S CTAs.
template <int EPI, int S>
__device__ __forceinline__ void few_finish(const FewArgs& a, uint32_t sum, int u, int tok0, int t0, int t1, int et,
                                           const int* pos_s, const int* seq_s) {
  const FewEpi& ep = a.ep;
  const int n0 = u * FW_TILE;
  constexpr int NP = S >= 4 ? 2 : 4;  // tokens in flight per thread
  constexpr uint32_t TOK = FW_PITCH * 4;
  auto at = [&](int t, int r) { return sum + (uint32_t)t * TOK + (uint32_t)(4 * r); };
  if constexpr (EPI == EPI_BF16 || EPI == EPI_RESID_F32) {  // a warp per token
    const int r = 4 * (et & 31), n = n0 + r;
    if (n >= a.N) return;
#pragma unroll 1
    for (int t = t0 + (et >> 5); t < t1; t += 4 * NP) {
      float4 x[NP];
      const int m = (t1 - t + 3) >> 2;
      cluster_sums<S, NP>(at(t, r), 4 * TOK, m, x);
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        if (i >= m) continue;
        const size_t o = (size_t)(tok0 + t + 4 * i) * ep.ldo + n;
        if constexpr (EPI == EPI_BF16)
          store_bf16x4(static_cast<__nv_bfloat16*>(ep.out) + o, x[i].x, x[i].y, x[i].z, x[i].w);
        else
          red_add_v4(static_cast<float*>(ep.out) + o, x[i]);
      }
    }
  } else if constexpr (EPI == EPI_SWIGLU) {  // gate rows j .. j + 3 and up rows 64 + j ..; half a warp per token
    const int j = 4 * (et & 15);
#pragma unroll 1
    for (int t = t0 + (et >> 4); t < t1; t += 8 * NP) {
      float4 g[NP], v[NP];
      const int m = (t1 - t + 7) >> 3;
      cluster_sums<S, NP>(at(t, j), 8 * TOK, m, g);
      cluster_sums<S, NP>(at(t, 64 + j), 8 * TOK, m, v);
      auto act = [](float x, float y) { return __fdividef(x, 1.0f + __expf(-x)) * y; };
#pragma unroll
      for (int i = 0; i < NP; ++i)
        if (i < m)
          store_bf16x4(static_cast<__nv_bfloat16*>(ep.out) + (size_t)(tok0 + t + 8 * i) * ep.ldo + u * 64 + j,
                       act(g[i].x, v[i].x), act(g[i].y, v[i].y), act(g[i].z, v[i].z), act(g[i].w, v[i].w));
    }
  } else if (n0 >= ep.rope_cols && ep.vdst) {
    // v leaves transposed, in fp16 holding the bf16 values: four channels x four tokens per
    // thread, positions contiguous.  (Groups of 32 rows are consecutive positions of one
    // sequence from a multiple of 32, and a CTA's tokens a multiple of 4: 8-byte stores.)
    const int r = 4 * (et & 31);
    if (n0 + r >= a.N) return;
#pragma unroll 1
    for (int t = t0 + 4 * (et >> 5); t < t1; t += 16) {
      float4 x[4];
      cluster_sums<S, 4>(at(t, r), TOK, 4, x);
      auto h = [](float f) { return __bfloat162float(__float2bfloat16_rn(f)); };
      __half* o = ep.vdst + ((size_t)seq_s[t] * ep.G * ep.head_dim + (n0 + r - ep.rope_cols)) * ep.Tp + pos_s[t];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        auto f = [&](int i) { return h(c == 0 ? x[i].x : c == 1 ? x[i].y : c == 2 ? x[i].z : x[i].w); };
        *reinterpret_cast<uint2*>(o + (size_t)c * ep.Tp) = make_uint2(pack_f16x2(f(0), f(1)), pack_f16x2(f(2), f(3)));
      }
    }
  } else {  // q, k (and v without a store of its own): components j .. j + 3 and j + head_dim / 2 .. of a head
    const int half = ep.head_dim >> 1, jj = 4 * (et & 15), j = jj & (half - 1);
    const int r0 = jj + (jj & ~(half - 1)), r1 = r0 + half;
    if (n0 + r1 >= a.N) return;
    const bool rope = n0 < ep.rope_cols, to_k = rope && ep.kdst && n0 >= ep.k_col0;
    constexpr int NQ = S >= 4 ? 1 : 2;
#pragma unroll 1
    for (int t = t0 + (et >> 4); t < t1; t += 8 * NQ) {
      float4 x[NQ], y[NQ], c[NQ], d[NQ];  // c: {cos, sin} of j, j + 1; d: of j + 2, j + 3
      const int m = (t1 - t + 7) >> 3;
#pragma unroll
      for (int i = 0; i < NQ; ++i) {
        c[i] = d[i] = make_float4(1.f, 0.f, 1.f, 0.f);
        if (rope && i < m) {
          const float4* cs = reinterpret_cast<const float4*>(ep.rope + (size_t)pos_s[t + 8 * i] * half + j);
          c[i] = __ldg(cs);
          d[i] = __ldg(cs + 1);
        }
      }
      cluster_sums<S, NQ>(at(t, r0), 8 * TOK, m, x);
      cluster_sums<S, NQ>(at(t, r1), 8 * TOK, m, y);
#pragma unroll
      for (int i = 0; i < NQ; ++i) {
        if (i >= m) continue;
        const int tt = t + 8 * i;
        __nv_bfloat16* o = to_k ? ep.kdst + ((size_t)seq_s[tt] * ep.T + pos_s[tt]) * ep.G * ep.head_dim + (n0 - ep.k_col0)
                                : static_cast<__nv_bfloat16*>(ep.out) + (size_t)(tok0 + tt) * ep.ldo + n0;
        store_bf16x4(o + r0, x[i].x * c[i].x - y[i].x * c[i].y, x[i].y * c[i].z - y[i].y * c[i].w,
                     x[i].z * d[i].x - y[i].z * d[i].y, x[i].w * d[i].z - y[i].w * d[i].w);
        store_bf16x4(o + r1, y[i].x * c[i].x + x[i].x * c[i].y, y[i].y * c[i].z + x[i].y * c[i].w,
                     y[i].z * d[i].x + x[i].z * d[i].y, y[i].w * d[i].z + x[i].w * d[i].w);
      }
    }
  }
}

}  // namespace
}  // namespace dcl
