// Slot -> app lookup shared by the kernels that read the slot map: the 48-byte app entry in three
// 16-byte loads, the slot's gate, and the status bit for bad slot ids.
#pragma once

#include "mix_internal.h"

namespace mix {

struct RowApp {
  bool gated;           // the slot has a gate (whether or not it let this row through)
  bool chained;         // another app follows on the same row (set even when the gate is closed)
  int raw_kind;         // the slot's kind even when the gate is closed (0: no valid app)
  int kind, C, act;     // kind 0: nothing to do
  float alpha;
  const uint4* W;
  const float* b;
};

// A row's gate: the entry, which the library owns, and -- a second step -- the score, which the caller owns.
struct RowGate {
  const float* score;
  int cmp;
  float thr;
};
__device__ __forceinline__ RowGate load_gate(const GateEntry* __restrict__ gates, int s, int t) {
  const int4 g0 = __ldg(reinterpret_cast<const int4*>(gates + s));        // scores ptr, stride, col
  const int4 g1 = __ldg(reinterpret_cast<const int4*>(gates + s) + 1);    // cmp, thr
  RowGate r;
  r.score = reinterpret_cast<const float*>(((unsigned long long)(unsigned)g0.y << 32) | (unsigned)g0.x) + (size_t)t * g0.z + g0.w;
  r.cmp = g1.x;
  r.thr = __int_as_float(g1.y);
  return r;
}
// The score, by an ordinary load of the GPU's memory: the read-only path (__ldg) is for what nobody writes while the kernel runs, and the
// kernel in front, which a programmatic launch overlaps, or an earlier probe of the same chain writes scores.  A kernel that starts
// before the chain kernel in front of it has ended may find rows next to its own in an L1 that this one filled ahead of their probes.
__device__ __forceinline__ float ld_score(const float* p) {
  float v;
  asm volatile("ld.relaxed.gpu.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}
// Does a row with this score pass?  (NaN fails both comparisons.)
__device__ __forceinline__ bool gate_passes(const RowGate& g, float score) { return g.cmp == MIX_GATE_GE ? score >= g.thr : score < g.thr; }
__device__ __forceinline__ bool gate_open(const GateEntry* __restrict__ gates, int s, int t) {
  const RowGate g = load_gate(gates, s, t);
  return gate_passes(g, ld_score(g.score));
}

// Slot -> app for row t; flags bad slot ids; applies the slot's gate.  `leader` is the one
// thread that may raise status.
__device__ __forceinline__ RowApp lookup(int s, int t, const AppEntry* __restrict__ apps,
                                         const GateEntry* __restrict__ gates, int n_slots,
                                         unsigned* __restrict__ status, bool leader, bool eval_gate = true) {
  RowApp r;
  r.kind = 0;
  r.raw_kind = 0;
  r.C = 0;
  r.gated = false;
  r.chained = false;
  if (s == -1) return r;
  if (s < -1 || s >= n_slots) {
    if (leader) atomicOr(status, MIX_STATUS_BAD_SLOT);
    return r;
  }
  // the whole 48-byte entry in three independent 16-byte loads (one round trip)
  const int4* e = reinterpret_cast<const int4*>(apps + s);
  const int4 q0 = __ldg(e), q1 = __ldg(e + 1), q2 = __ldg(e + 2);
  if (!q0.x) {                                   // valid
    if (leader) atomicOr(status, MIX_STATUS_BAD_SLOT);
    return r;
  }
  r.gated = (q0.y & kKindGated) != 0;
  r.chained = (q0.y & kKindChained) != 0;
  r.raw_kind = q0.y & kKindMask;
  r.C = q0.z;
  if (eval_gate && r.gated && !gate_open(gates, s, t)) return r;  // gate closed: the row passes through
  r.kind = q0.y & kKindMask;
  r.act = q0.w;
  r.alpha = __int_as_float(q1.x);
  r.W = reinterpret_cast<const uint4*>(((unsigned long long)(unsigned)q2.y << 32) | (unsigned)q2.x);
  r.b = reinterpret_cast<const float*>(((unsigned long long)(unsigned)q2.w << 32) | (unsigned)q2.z);
  return r;
}

}  // namespace mix
