// What the hook kernels do with a row: small pieces, and a row of a small batch as part of the front kernel's launch.
#pragma once

#include "mix_internal.h"
#include "row_lookup.cuh"

namespace mix {

__device__ __forceinline__ void unpack8(const uint4& q, float* f) {
  const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&q);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float2 t = __bfloat1622float2(p[i]);
    f[2 * i] = t.x;
    f[2 * i + 1] = t.y;
  }
}

__device__ __forceinline__ uint4 pack8(const float* f) {
  uint4 q;
  __nv_bfloat162* p = reinterpret_cast<__nv_bfloat162*>(&q);
#pragma unroll
  for (int i = 0; i < 4; ++i) p[i] = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
  return q;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Four sums over the warp with 6 exchanges instead of 20; lanes 8c .. 8c + 7 return that of v[c].  (The same additions as in
// warp_sum, hence the same bits.)
__device__ __forceinline__ float warp_sum4(const float (&v)[4], int lane) {
  const bool b16 = lane & 16, b8 = lane & 8;
  const float a0 = (b16 ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, b16 ? v[0] : v[2], 16);
  const float a1 = (b16 ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, b16 ? v[1] : v[3], 16);
  float z = (b8 ? a1 : a0) + __shfl_xor_sync(0xffffffffu, b8 ? a0 : a1, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
  return z;
}

// 1 / (1 + e^-z) with the hardware exponential and reciprocal: a few instructions instead of the two library
// routines' hundred on the one-warp tail of a decode step (0.28 us of a 3 us step); the relative error stays
// below 1e-5 for |z| < 80, two orders under the 1e-3 the scores are held to.
__device__ __forceinline__ float fast_sigmoid(float z) { return __frcp_rn(1.f + __expf(-z)); }

// Logits (bias included) of one row in `logit` -> scores.  One warp; C <= 64.
__device__ __forceinline__ void finish_probe(const float* logit, int C, int act, float* __restrict__ out, int lane) {
  if (C == 1) {                                  // the decode step's case: one lane, no cross-lane work
    if (lane == 0) {
      const float z = logit[0];
      out[0] = act == MIX_ACT_NONE ? z : (act == MIX_ACT_SOFTMAX ? 1.f : fast_sigmoid(z));
    }
    return;
  }
  float z0 = lane < C ? logit[lane] : -INFINITY;
  float z1 = lane + 32 < C ? logit[lane + 32] : -INFINITY;
  if (act == MIX_ACT_SOFTMAX) {
    float m = fmaxf(z0, z1);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    const float e0 = lane < C ? expf(z0 - m) : 0.f;
    const float e1 = lane + 32 < C ? expf(z1 - m) : 0.f;
    const float sum = warp_sum(e0 + e1);
    z0 = e0 / sum;
    z1 = e1 / sum;
  } else if (act == MIX_ACT_SIGMOID) {
    z0 = fast_sigmoid(z0);
    z1 = fast_sigmoid(z1);
  }
  if (lane < C) out[lane] = z0;
  if (lane + 32 < C) out[lane + 32] = z1;
}

// Eight warps: with sixteen, which leaves each thread half as much, the sums over the warps cost more than that saves (187 rows
// of a three-app chain, d = 5120: 38 us for four layers against 33).
constexpr int kHookWarps = 8;
constexpr int kMostVec = 4;     // kHookWarps * 32 * kMostVec * 8 >= d_model: 8192 columns

// The app of a row of a small batch, by a CTA of kHookWarps warps that holds the row (hq) and, where the app has one, its single
// vector (vq) in registers.  Behind the programmatic wait; control flow is uniform across the CTA.
template <int NV>
__device__ __forceinline__ void row_app(const RowApp& a, const RowGate& gate, const uint4 (&hq)[NV], const uint4 (&vq)[NV], uint4* __restrict__ hrow,
                                        int nvec, float* __restrict__ scores, float (*s_part)[kMaxClasses]) {
  constexpr int NW = kHookWarps, NT = NW * 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float score = 0.f;
  if (a.gated) score = ld_score(gate.score);     // (requested with the row)
  // A one-class probe's bias came with the entry (registration put it into the `alpha` word); the biases of a
  // wider probe are requested as soon as the entry is here, not after the dot products they are added to.
  float bias_lo = 0.f, bias_hi = 0.f;
  if (a.kind == MIX_PROBE && warp == 0) {
    if (a.C == 1) {
      bias_lo = a.alpha;
    } else if (a.b != nullptr) {
      if (lane < a.C) bias_lo = __ldg(a.b + lane);
      if (lane + 32 < a.C) bias_hi = __ldg(a.b + lane + 32);
    }
  }
  if (a.gated && !gate_passes(gate, score)) return;       // gate closed: the row passes through
  if (a.kind == MIX_STEER) {
    if (a.alpha == 0.f) return;                  // identity; the row stays bit-exact
#pragma unroll
    for (int u = 0; u < NV; ++u) {
      const int v = threadIdx.x + u * NT;
      if (v < nvec) {
        float x[8], y[8];
        unpack8(hq[u], x);
        unpack8(vq[u], y);
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] = fmaf(a.alpha, y[e], x[e]);
        __stcs(hrow + v, pack8(x));
      }
    }
    return;
  }
  if (a.kind == MIX_PROJECT) {                 // h - beta (h . r) r
    if (a.alpha == 0.f) return;
    float dot = 0.f;
#pragma unroll
    for (int u = 0; u < NV; ++u) {
      const int v = threadIdx.x + u * NT;
      if (v < nvec) {
        float x[8], y[8];
        unpack8(hq[u], x);
        unpack8(vq[u], y);
#pragma unroll
        for (int e = 0; e < 8; ++e) dot = fmaf(x[e], y[e], dot);
      }
    }
    dot = warp_sum(dot);
    if (lane == 0) s_part[warp][0] = dot;
    __syncthreads();
    float total = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) total += s_part[w][0];
    const float coef = -a.alpha * total;
#pragma unroll
    for (int u = 0; u < NV; ++u) {
      const int v = threadIdx.x + u * NT;
      if (v < nvec) {
        float x[8], y[8];
        unpack8(hq[u], x);
        unpack8(vq[u], y);
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] = fmaf(coef, y[e], x[e]);
        __stcs(hrow + v, pack8(x));
      }
    }
    return;
  }
  if (a.kind != MIX_PROBE || scores == nullptr) return;
  if (a.C == 1) {                              // the probe vector is already here
    float acc = 0.f;
#pragma unroll
    for (int u = 0; u < NV; ++u) {
      const int v = threadIdx.x + u * NT;
      if (v < nvec) {
        float x[8], y[8];
        unpack8(hq[u], x);
        unpack8(vq[u], y);
#pragma unroll
        for (int e = 0; e < 8; ++e) acc = fmaf(x[e], y[e], acc);
      }
    }
    acc = warp_sum(acc);
    if (lane == 0) s_part[warp][0] = acc;
  }
  for (int c0 = 0; c0 < (a.C == 1 ? 0 : a.C); c0 += 4) {
    const int nc = min(4, a.C - c0);
    uint4 wq[4][NV];
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int u = 0; u < NV; ++u) {
        const int v = threadIdx.x + u * NT;
        if (c < nc && v < nvec) wq[c][u] = __ldg(a.W + (size_t)(c0 + c) * nvec + v);
      }
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int u = 0; u < NV; ++u) {
      const int v = threadIdx.x + u * NT;
      if (v < nvec) {
        float x[8];
        unpack8(hq[u], x);
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (c < nc) {
            float y[8];
            unpack8(wq[c][u], y);
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[c] = fmaf(x[e], y[e], acc[c]);
          }
      }
    }
    const float z = warp_sum4(acc, lane);
    if ((lane & 7) == 0 && (lane >> 3) < nc) s_part[warp][c0 + (lane >> 3)] = z;
  }
  __syncthreads();
  if (warp == 0) {
    for (int c = lane; c < a.C; c += 32) {
      float z = c < 32 ? bias_lo : bias_hi;
#pragma unroll
      for (int w = 0; w < NW; ++w) z += s_part[w][c];
      s_part[0][c] = z;            // only this lane reads or writes column c from here on
    }
    __syncwarp();
    finish_probe(s_part[0], a.C, a.act, scores, lane);
  }
}

// A row of a small batch of a context with weight sets: as probe_steer_team_kernel does it, but most rows may be another kernel's, so
// nothing is requested before the entry says that the row is this one's (1000 SAE rows of d = 2304: 6.2 -> 4.5 us).  What the
// library owns is read ahead of the programmatic wait, the rest behind it.
template <int NV>
__device__ __forceinline__ void late_row(int first_cta, const int* __restrict__ token_slot, int T,
                                         const AppEntry* __restrict__ apps, const GateEntry* __restrict__ gates, int n_slots,
                                         __nv_bfloat16* __restrict__ hidden, int d, float* __restrict__ scores, int C_max,
                                         unsigned* __restrict__ status, const uint4* __restrict__ vec_arena,
                                         float (*s_part)[kMaxClasses]) {
  const int t = (int)blockIdx.x - first_cta;     // < T_max: the slot map has an entry for every row
  const int slot = __ldg(token_slot + t);
  if (t >= T || slot == -1) {
    pdl_wait();
    return;
  }
  const int nvec = d >> 3;
  uint4* hrow = reinterpret_cast<uint4*>(hidden + (size_t)t * d);
  uint4 hq[NV], vq[NV];
  const RowApp a = lookup(slot, t, apps, gates, n_slots, status, threadIdx.x == 0, /*eval_gate=*/false);
  RowGate gate;
  if (a.gated) gate = load_gate(gates, slot, t);
  pdl_wait();
  if (a.kind == 0 || a.kind == MIX_SAE || a.kind == MIX_ROUTER) return;
#pragma unroll
  for (int u = 0; u < NV; ++u) {
    const int v = threadIdx.x + u * kHookWarps * 32;
    if (v < nvec) {
      vq[u] = __ldg(vec_arena + (size_t)slot * nvec + v);
      hq[u] = __ldcs(hrow + v);
    }
  }
  row_app<NV>(a, gate, hq, vq, hrow, nvec, scores == nullptr ? nullptr : scores + (size_t)t * C_max, s_part);
}

}  // namespace mix
