// The read (probe) and write (steering) primitives of the hook, and the small kernels around the slot map.
//
// probe_steer_kernel is the bandwidth kernel of the hook: one warp per token row, 16-byte
// loads, fp32 FMA, shuffle reductions.  A row whose slot is -1 costs one 4-byte load.
#include <string.h>

#include <type_traits>

#include "mix_internal.h"
#include "hook_row.cuh"
#include "row_lookup.cuh"

namespace mix {

namespace {

// h + alpha v for one row; nvec = d / 8 16-byte vectors.  The `stride` threads that share the
// row start at `first` (a warp: lane, 32; a CTA team: threadIdx.x, blockDim.x).
__device__ __forceinline__ void steer_row(uint4* __restrict__ h, const uint4* __restrict__ v, float alpha,
                                          int nvec, int first, int stride) {
  constexpr int U = 4;
  int i = first;
  for (; i + (U - 1) * stride < nvec; i += U * stride) {
    uint4 hq[U], vq[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      hq[u] = __ldcs(h + i + u * stride);
      vq[u] = __ldg(v + i + u * stride);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      float a[8], b[8];
      unpack8(hq[u], a);
      unpack8(vq[u], b);
#pragma unroll
      for (int e = 0; e < 8; ++e) a[e] = fmaf(alpha, b[e], a[e]);
      __stcs(h + i + u * stride, pack8(a));
    }
  }
  for (; i < nvec; i += stride) {
    float a[8], b[8];
    unpack8(__ldcs(h + i), a);
    unpack8(__ldg(v + i), b);
#pragma unroll
    for (int e = 0; e < 8; ++e) a[e] = fmaf(alpha, b[e], a[e]);
    __stcs(h + i, pack8(a));
  }
}

// Partial logits of RB rows against NC consecutive probe rows over this thread's share of the
// columns; warp-reduced, so every lane of a warp returns the warp's sums.
template <int RB, int NC>
__device__ __forceinline__ void probe_dots(const uint4* const* __restrict__ h, const uint4* __restrict__ W, int nvec,
                                           int nc, int first, int stride, float (*out)[NC]) {
  float acc[RB][NC];
#pragma unroll
  for (int r = 0; r < RB; ++r)
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[r][c] = 0.f;
  constexpr int U = (NC == 1 && RB == 1) ? 4 : 1;
  int i = first;
  for (; i + (U - 1) * stride < nvec; i += U * stride) {
    uint4 hq[U][RB];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int r = 0; r < RB; ++r) hq[u][r] = __ldg(h[r] + i + u * stride);
    uint4 wq[U][NC];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int c = 0; c < NC; ++c)
        if (c < nc) wq[u][c] = __ldg(W + (size_t)c * nvec + i + u * stride);
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll
      for (int c = 0; c < NC; ++c)
        if (c < nc) {
          float b[8];
          unpack8(wq[u][c], b);
#pragma unroll
          for (int r = 0; r < RB; ++r) {
            float a[8];
            unpack8(hq[u][r], a);
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[r][c] = fmaf(a[e], b[e], acc[r][c]);
          }
        }
    }
  }
  if (U > 1) {
    for (; i < nvec; i += stride) {
      float a[8], b[8];
      unpack8(__ldg(h[0] + i), a);
      unpack8(__ldg(W + i), b);
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[0][0] = fmaf(a[e], b[e], acc[0][0]);
    }
  }
#pragma unroll
  for (int r = 0; r < RB; ++r)
#pragma unroll
    for (int c = 0; c < NC; ++c) out[r][c] = warp_sum(acc[r][c]);
}

constexpr int kCoopMaxClasses = 32;    // widest probe the cooperative tensor-core pass takes

// One row, one warp: steer, single-class probe, or multi-class probe.
__device__ __forceinline__ void warp_row(const RowApp& a, __nv_bfloat16* __restrict__ hidden, int t, int d,
                                         float* __restrict__ scores, int C_max, float* s_logit, int lane) {
  const int nvec = d >> 3;
  uint4* hrow = reinterpret_cast<uint4*>(hidden + (size_t)t * d);
  if (a.kind == MIX_STEER) {
    if (a.alpha != 0.f) steer_row(hrow, a.W, a.alpha, nvec, lane, 32);   // alpha = 0: row stays bit-exact
    return;
  }
  const uint4* h1[1] = {hrow};
  if (a.kind == MIX_PROJECT) {                 // h - beta (h . r) r: one pass for the dot, one for the update
    if (a.alpha == 0.f) return;
    float z[1][1];
    probe_dots<1, 1>(h1, a.W, nvec, 1, lane, 32, z);
    steer_row(hrow, a.W, -a.alpha * z[0][0], nvec, lane, 32);
    return;
  }
  if (a.kind != MIX_PROBE || scores == nullptr) return;
  float* out = scores + (size_t)t * C_max;
  if (a.C == 1) {
    float z[1][1];
    probe_dots<1, 1>(h1, a.W, nvec, 1, lane, 32, z);
    if (lane == 0) {
      const float zz = z[0][0] + (a.b ? __ldg(a.b) : 0.f);
      // one class: raw logit, sigmoid, or a softmax over a single entry (= 1)
      out[0] = a.act == MIX_ACT_NONE ? zz : (a.act == MIX_ACT_SOFTMAX ? 1.f : fast_sigmoid(zz));
    }
    return;
  }
  for (int c0 = 0; c0 < a.C; c0 += 4) {
    float z[1][4];
    const int nc = min(4, a.C - c0);
    probe_dots<1, 4>(h1, a.W + (size_t)c0 * nvec, nvec, nc, lane, 32, z);
    if (lane == 0) {
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (c < nc) s_logit[c0 + c] = z[0][c] + (a.b ? __ldg(a.b + c0 + c) : 0.f);
    }
  }
  __syncwarp();
  finish_probe(s_logit, a.C, a.act, out, lane);
}

// Large batches: a CTA owns kWarps consecutive rows, one warp per row: streaming work (steering,
// single-class probes).  Multi-class probes up to kCoopMaxClasses classes are left to
// probe_tc_kernel (probe_tc.cu) when `multiclass_elsewhere` is set.
// Bound by the bytes in flight.  Small CTAs, as many warps as 56 registers let an SM hold (11111 rows of d = 5120, steering,
// one-class probes and projections: 37.2 us with eight-warp CTAs at 66 registers, 35.3 so) -- except beside the
// tensor-core kernel, which leaves room for eight warps at a time.
template <int kWarps, int kMinCtas>
__global__ void __launch_bounds__(kWarps * 32, kMinCtas)
probe_steer_kernel(const int* __restrict__ token_slot, int T,
                   const AppEntry* __restrict__ apps, const GateEntry* __restrict__ gates, int n_slots,
                   __nv_bfloat16* __restrict__ hidden, int d,
                   float* __restrict__ scores, int C_max, unsigned* __restrict__ status, int multiclass_elsewhere) {
  __shared__ float s_logit[kWarps][kMaxClasses];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = blockIdx.x * kWarps + warp;
  if (t >= T) return;
  const int slot = __ldg(token_slot + t);
  const RowApp a = lookup(slot, t, apps, gates, n_slots, status, lane == 0);
  if (a.kind == 0) return;
  if (multiclass_elsewhere && a.kind == MIX_PROBE && a.C > 1 && a.C <= kCoopMaxClasses) return;
  warp_row(a, hidden, t, d, scores, C_max, s_logit[warp], lane);
}

// 16-byte read-only load that the compiler may not sink below later volatile statements: keeps
// all loads of a batch in flight before the first MMA that consumes them.
__device__ __forceinline__ uint4 ldg128_early(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

constexpr int kMcRows = 16;            // rows per CTA of probe_multiclass_kernel (one m16 MMA tile)
constexpr int kMcWarps = 8;            // warps per CTA: they split d between them

// One warp's share of the contraction of 16 rows against one probe matrix on the warp-level
// tensor-core MMA (m16n8k16, bf16 -> fp32): every kMcWarps-th 32-column chunk of d, UB chunks in flight,
// KCT 8-class tiles.  Fragments come straight from global memory, 16 contiguous bytes per lane:
// lane (g, q) takes columns 8q..8q+7 of the chunk for rows g and g + 8 and for class g of each
// 8-class tile.  Which columns a fragment slot holds is immaterial as long as A and B agree,
// because the sum runs over all of them.  Partial logits go to part[row][class].
template <int KCT, int UB>
__device__ __forceinline__ void mc_contract(const uint4* __restrict__ h_lo, const uint4* __restrict__ h_hi,
                                            const uint4* __restrict__ W, int C, int n_chunks, int row_vecs,
                                            float (*part)[kCoopMaxClasses]) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, q = lane & 3;
  float acc[KCT][4];
#pragma unroll
  for (int ct = 0; ct < KCT; ++ct) acc[ct][0] = acc[ct][1] = acc[ct][2] = acc[ct][3] = 0.f;
  for (int ch0 = warp; ch0 < n_chunks; ch0 += kMcWarps * UB) {
    uint4 lo[UB], hi[UB], wq[UB][KCT];
#pragma unroll
    for (int u = 0; u < UB; ++u) {
      const int ch = ch0 + u * kMcWarps;
      const bool in = ch < n_chunks;
      lo[u] = in ? ldg128_early(h_lo + ch * 4 + q) : make_uint4(0u, 0u, 0u, 0u);
      hi[u] = in ? ldg128_early(h_hi + ch * 4 + q) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
      for (int ct = 0; ct < KCT; ++ct) {
        const int cls = ct * 8 + g;
        wq[u][ct] = (in && cls < C) ? ldg128_early(W + (size_t)cls * row_vecs + ch * 4 + q) : make_uint4(0u, 0u, 0u, 0u);
      }
    }
#pragma unroll
    for (int u = 0; u < UB; ++u) {
#pragma unroll
      for (int ct = 0; ct < KCT; ++ct) {
        asm volatile(
            "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
            "{%0, %1, %2, %3};"
            : "+f"(acc[ct][0]), "+f"(acc[ct][1]), "+f"(acc[ct][2]), "+f"(acc[ct][3])
            : "r"(lo[u].x), "r"(hi[u].x), "r"(lo[u].y), "r"(hi[u].y), "r"(wq[u][ct].x), "r"(wq[u][ct].y));
        asm volatile(
            "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
            "{%0, %1, %2, %3};"
            : "+f"(acc[ct][0]), "+f"(acc[ct][1]), "+f"(acc[ct][2]), "+f"(acc[ct][3])
            : "r"(lo[u].z), "r"(hi[u].z), "r"(lo[u].w), "r"(hi[u].w), "r"(wq[u][ct].z), "r"(wq[u][ct].w));
      }
    }
  }
  // lane (g, q): rows g (acc 0, 1) and g + 8 (acc 2, 3), classes 8 ct + 2q and + 1
#pragma unroll
  for (int ct = 0; ct < KCT; ++ct) {
    if (ct * 8 < C) {
      part[g][ct * 8 + 2 * q] = acc[ct][0];
      part[g][ct * 8 + 2 * q + 1] = acc[ct][1];
      part[g + 8][ct * 8 + 2 * q] = acc[ct][2];
      part[g + 8][ct * 8 + 2 * q + 1] = acc[ct][3];
    }
  }
}

// What the CTA knows about each of its rows.
struct McRow {
  const uint4* W;
  const float* b;
  int C, act;
  int slot;      // slot id if the row is a multi-class probe this kernel takes and its gate is open, else -1
};

// Multi-class probes of large batches.  16 rows x C classes x d is a skinny dense contraction;
// consecutive rows usually belong to one request and share the probe.  For every distinct
// multi-class probe among the CTA's 16 rows, the warps split d between them and contract ALL
// 16 rows against that probe's matrix, which is therefore streamed from L2 once per 16 rows;
// only the rows that belong to the probe keep their result.
__global__ void __launch_bounds__(kMcWarps * 32, 2)
probe_multiclass_kernel(const int* __restrict__ token_slot, int T,
                        const AppEntry* __restrict__ apps, const GateEntry* __restrict__ gates, int n_slots,
                        const __nv_bfloat16* __restrict__ hidden, int d, float* __restrict__ scores, int C_max,
                        const McCensus* __restrict__ census) {
  __shared__ float s_part[kMcWarps][kMcRows][kCoopMaxClasses];   // [warp][row][class]
  __shared__ float s_logit[kMcWarps][kCoopMaxClasses];
  __shared__ McRow s_row[kMcRows];
  __shared__ int s_any;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t0 = blockIdx.x * kMcRows;
  if (t0 >= T || scores == nullptr) return;
  if (census != nullptr && census->use_tc) return;          // this call's batch is probe_tc_kernel's
  if (threadIdx.x == 0) s_any = 0;
  __syncthreads();
  if (threadIdx.x < kMcRows) {           // one thread per row: slot -> entry -> gate
    const int t = t0 + threadIdx.x;
    McRow r;
    r.slot = -1;
    if (t < T) {
      const int s = __ldg(token_slot + t);
      const RowApp a = lookup(s, t, apps, gates, n_slots, nullptr, false);   // bad slots are flagged by probe_steer_kernel
      if (a.kind == MIX_PROBE && a.C > 1 && a.C <= kCoopMaxClasses) {
        r.W = a.W;
        r.b = a.b;
        r.C = a.C;
        r.act = a.act;
        r.slot = s;
        s_any = 1;
      }
    }
    s_row[threadIdx.x] = r;
  }
  __syncthreads();
  if (!s_any) return;                    // CTA-uniform
  const int g = lane >> 2;
  const uint4* h_lo = reinterpret_cast<const uint4*>(hidden + (size_t)min(t0 + g, T - 1) * d);
  const uint4* h_hi = reinterpret_cast<const uint4*>(hidden + (size_t)min(t0 + g + 8, T - 1) * d);
  const int n_chunks = d >> 5, row_vecs = d >> 3;
  for (int r = 0; r < kMcRows; ++r) {
    const McRow ci = s_row[r];
    if (ci.slot < 0) continue;
    bool first = true;
    for (int r2 = 0; r2 < r; ++r2) first = first && s_row[r2].slot != ci.slot;
    if (!first) continue;
    if (ci.C <= 16)
      mc_contract<2, 4>(h_lo, h_hi, ci.W, ci.C, n_chunks, row_vecs, s_part[warp]);
    else
      mc_contract<kCoopMaxClasses / 8, 2>(h_lo, h_hi, ci.W, ci.C, n_chunks, row_vecs, s_part[warp]);
    __syncthreads();
#pragma unroll 1
    for (int rr = warp; rr < kMcRows; rr += kMcWarps) {     // warp w finishes row w
      if (s_row[rr].slot != ci.slot) continue;
      for (int c = lane; c < ci.C; c += 32) {
        float z = ci.b ? __ldg(ci.b + c) : 0.f;
#pragma unroll
        for (int w = 0; w < kMcWarps; ++w) z += s_part[w][rr][c];
        s_logit[warp][c] = z;
      }
      __syncwarp();
      finish_probe(s_logit[warp], ci.C, ci.act, scores + (size_t)(t0 + rr) * C_max, lane);
      __syncwarp();
    }
    __syncthreads();                     // s_part is reused by the next probe
  }
}

// Small batches (decode): one CTA per row, the row held in registers (NV 16-byte vectors per thread, a kernel for each width:
// 52 ... 72 registers up to d = 4096 where one for all widths had 126, i.e. three or four CTAs on an SM instead of two, so that the
// kernels of a step's next layers are there, their look-ups done, when the present one ends; held to 64, i.e. four CTAs, the form of
// two vectors was no faster there, 148 us for 32 layers, and slower where probes are wide: 22 rows, 16 classes, three layers 28.0 us
// against 26.0).  The row's loads are issued as soon as the slot id is known to be
// >= 0, in parallel with the app-table lookup, so a cold row costs two dependent round trips
// (slot, then entry + data) instead of three.  Control flow is uniform across the CTA.
enum TeamForm { kTeamPlain, kTeamMapAhead };   // (forms of their own: as flags they cost the plain step 2.81 -> 2.86 us)

template <int NV, TeamForm kForm>
__global__ void __launch_bounds__(kHookWarps * 32, NV == 1 ? 4 : (NV == 2 ? 3 : 2))
probe_steer_team_kernel(const int* __restrict__ token_slot, int T,
                        const AppEntry* __restrict__ apps, const GateEntry* __restrict__ gates, int n_slots,
                        __nv_bfloat16* __restrict__ hidden, int d, float* __restrict__ scores, int C_max,
                        unsigned* __restrict__ status, const uint4* __restrict__ vec_arena, int pdl) {
  __shared__ float s_part[kHookWarps][kMaxClasses];
  constexpr int NT = kHookWarps * 32;
  const int t = blockIdx.x;                      // < T_max: the slot map has an entry for every row
  // Programmatic dependent launch (`pdl`: the launch asked for it): everything up to pdl_wait() reads only
  // tables the LIBRARY owns -- slot map, app entry, vector arena; copies write them, which are complete before a kernel
  // behind them starts, and, the map alone, kernels (see below) -- so it
  // may run while the kernel in front of this one in the stream (the layer that produces `hidden`, or the
  // previous hook) is still running.  Memory the caller owns (`hidden`, multi-class probe weights, gate scores)
  // is read after the wait only, and every thread waits before it leaves, so that this grid cannot end -- and
  // release ITS successor -- before its predecessor has.  Launched the ordinary way, nothing has to wait: the
  // row is then requested together with the vector and the app entry, one round trip earlier.  Behind a map that a
  // kernel installed (kPdlMapAhead) the wait comes first, and only then the trigger: a successor that reads the map
  // early must not start before the map is there.
  if (kForm == kTeamMapAhead) {
    pdl_wait();
    pdl_launch_dependents();
    pdl = 0;
  }
  if (pdl) pdl_launch_dependents();
  const int slot = __ldg(token_slot + t);
  if (t >= T || slot == -1) {
    if (pdl) pdl_wait();
    return;
  }
  const int nvec = d >> 3;
  uint4* hrow = reinterpret_cast<uint4*>(hidden + (size_t)t * d);
  // Single-vector weights (steering, projection, one-class probe) were copied at registration
  // into row `slot` of the context's vector arena, so their address follows from the slot id
  // alone: the row AND its vector are requested together, before the app entry is known.
  uint4 hq[NV], vq[NV];
  const bool slot_ok = slot >= 0 && slot < n_slots;
  if (slot_ok) {
#pragma unroll
    for (int u = 0; u < NV; ++u) {
      const int v = threadIdx.x + u * NT;
      if (v < nvec) vq[u] = __ldg(vec_arena + (size_t)slot * nvec + v);
    }
  }
  if (!pdl && slot_ok) {
#pragma unroll
    for (int u = 0; u < NV; ++u) {
      const int v = threadIdx.x + u * NT;
      if (v < nvec) hq[u] = __ldcs(hrow + v);
    }
  }
  // (A hint, so it may come before the wait: what the predecessor still writes of the row, it writes to this L2.  For a step
  // whose hidden states no longer lie there: 32 layers of 256 rows, d = 4096: 2.25 -> 1.9 us a layer.)
  if (pdl && slot_ok && threadIdx.x * 8 < nvec) asm volatile("prefetch.global.L2 [%0];" ::"l"(hrow + threadIdx.x * 8));
  RowApp a = lookup(slot, t, apps, gates, n_slots, status, threadIdx.x == 0, /*eval_gate=*/false);
  RowGate gate;
  if (a.gated) gate = load_gate(gates, slot, t);
  if (pdl) pdl_wait();
  if (pdl && slot_ok) {
#pragma unroll
    for (int u = 0; u < NV; ++u) {
      const int v = threadIdx.x + u * NT;
      if (v < nvec) hq[u] = __ldcs(hrow + v);
    }
  }
  row_app<NV>(a, gate, hq, vq, hrow, nvec, scores == nullptr ? nullptr : scores + (size_t)t * C_max, s_part);
}

// Contexts with weight sets, where these rows are not part of the front kernel's launch (see apply_impl); never launched programmatically.
template <int NV>
__global__ void __launch_bounds__(kHookWarps * 32, NV == 1 ? 4 : (NV == 2 ? 3 : 2))
probe_steer_late_kernel(const int* __restrict__ token_slot, int T,
                        const AppEntry* __restrict__ apps, const GateEntry* __restrict__ gates, int n_slots,
                        __nv_bfloat16* __restrict__ hidden, int d, float* __restrict__ scores, int C_max,
                        unsigned* __restrict__ status, const uint4* __restrict__ vec_arena, int) {
  __shared__ float s_part[kHookWarps][kMaxClasses];
  late_row<NV>(0, token_slot, T, apps, gates, n_slots, hidden, d, scores, C_max, status, vec_arena, s_part);
}

// Contexts with slot chains: one CTA per row, the row held in registers while the apps of its chain
// are applied one after the other (probe / steering / projection; an SAE app at the end of a chain
// is left to the SAE kernels, which start after this one).  A write rounds the row to bf16 in
// registers, exactly as a store and reload would; the row goes back to memory once, at the end,
// if any app changed it.  The j-th probe of a chain writes its scores after those of the earlier
// ones.  Control flow is uniform across the CTA.
// Bound by the chain of dependent loads: link -> entry -> gate -> score -> vector, app after app.  All of it that the
// library owns -- links, entries, gate entries, single vectors (in the arena) -- is read ahead of the programmatic wait, into
// shared memory, while the layer or hook in front still runs; behind the wait everything the caller owns is requested together
// (row, gate scores, biases), and the probes' partial logits meet once, behind the last app -- unless a gate further down the
// chain looks at a score that an earlier probe of the chain writes: separate calls decide it on the new score, so the probes in
// front of it are finished before its turn.
constexpr int kChainStaged = 2;      // single vectors of a chain that are staged (later ones are loaded when their turn comes)

struct ChainStep {
  int kind;              // 0: nothing to do
  int C, act, col;       // col: the probe's first column in the row's scores
  float alpha;           // (of a one-class probe with its vector in the arena: the bias)
  int staged;            // place of the vector in shared memory, or -1
  const uint4* W;
  const float* b;
  RowGate gate;
};

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem) : "memory");
}

// NV: 16-byte vectors of the row per thread.  (The bounds hold the CTAs an SM takes to what the registers came to by themselves
// before a chain could stop half-way.  That, and the gates decided by one warp for all, costs the chains that do not stop 0.7 us over
// four layers of 187 rows, d = 5120: 30.9 -> 31.6 us, with the comparison of addresses in the walk and the turn back marked as the
// rare one; with the scores finished by a second copy of the code below it was 1.3 us more, with the comparison behind the wait 1.0.)
template <int NV>
__global__ void __launch_bounds__(kHookWarps * 32, NV == 1 ? 4 : (NV == 2 ? 3 : 2))
probe_steer_chain_kernel(const int* __restrict__ token_slot, int T,
                         const AppEntry* __restrict__ apps, const GateEntry* __restrict__ gates,
                         const int* __restrict__ chain_next, int n_slots, __nv_bfloat16* __restrict__ hidden, int d,
                         float* __restrict__ scores, int C_max, unsigned* __restrict__ status, int in_arena, int pdl) {
  extern __shared__ uint4 s_vec[];               // [kChainStaged][nvec]
  __shared__ float s_part[kHookWarps][kMaxClasses];   // partial logits of all the chain's probes, by column
  __shared__ float s_dot[kMaxChain][kHookWarps];
  __shared__ ChainStep s_step[kMaxChain];
  __shared__ int s_n;
  __shared__ unsigned s_free, s_gated, s_own;    // steps without a gate; with one; with one on a column of an earlier probe of this chain
  __shared__ unsigned s_passed;
  constexpr int NW = kHookWarps, NT = NW * 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = blockIdx.x;                      // < T_max: the slot map has an entry for every row
  // programmatic dependent launch, as in probe_steer_team_kernel: what the library owns may be read while the
  // predecessor still runs, unless a kernel has just installed the map; everything else comes after the wait, and every
  // thread waits before it leaves
  if (pdl == kPdlMapAhead) pdl_wait();
  pdl_launch_dependents();
  const int slot0 = __ldg(token_slot + t);
  if (t >= T || slot0 == -1) {
    pdl_wait();
    return;
  }
  const int nvec = d >> 3;
  float* const row_scores = scores + (size_t)t * C_max;
  if (warp == 0) {                               // the row's apps, in order (every lane reads the same)
    int slot = slot0, n = 0, col = 0, staged = 0;
    unsigned free_bits = 0u, gated_bits = 0u, own_bits = 0u;
    while (n < kMaxChain) {
      const int next = slot >= 0 && slot < n_slots ? __ldg(chain_next + slot) : -1;     // (requested with the entry)
      const RowApp a = lookup(slot, t, apps, gates, n_slots, status, lane == 0, /*eval_gate=*/false);
      ChainStep st;
      st.kind = a.kind;
      st.C = a.C;
      st.act = a.act;
      st.col = col;
      st.alpha = a.alpha;
      st.W = a.W;
      st.b = a.b;
      st.staged = -1;
      if (staged < kChainStaged && (a.kind == MIX_STEER || a.kind == MIX_PROJECT || (a.kind == MIX_PROBE && a.C == 1))) st.staged = staged++;
      // (Registration keeps a chain's columns within C_max.  A walk that a registration on another stream overtakes may meet the old
      // link and the new, wider probe: it must not leave the row's scores, or shared memory.)
      if (a.kind == MIX_SAE || (a.kind == MIX_PROBE && col + a.C > C_max)) st.kind = 0;     // (an SAE app: the front kernel's, gate and all)
      if (st.kind != 0 && a.gated) {
        st.gate = load_gate(gates, slot, t);
        if (scores != nullptr && st.gate.score >= row_scores && st.gate.score < row_scores + col) own_bits |= 1u << n;
        else gated_bits |= 1u << n;
      } else if (st.kind != 0) {
        free_bits |= 1u << n;
      }
      if (lane == 0) s_step[n] = st;
      ++n;
      if (!a.chained) break;
      if (a.raw_kind == MIX_PROBE) col += a.C;
      slot = next;                               // (slot was in range: lookup() found a valid entry)
      if (slot < 0) break;
    }
    if (lane == 0) s_n = n, s_free = free_bits, s_gated = gated_bits, s_own = own_bits;
  }
  __syncthreads();
  const int n = s_n;
  // a thread stages the vectors that it will use itself, so nobody else has to know when they have arrived
  auto stage = [&]() {
    for (int i = 0; i < n; ++i) {
      const int at = s_step[i].staged;
      if (at < 0) continue;
#pragma unroll
      for (int u = 0; u < NV; ++u) {
        const int v = threadIdx.x + u * NT;
        if (v < nvec) cp_async16(s_vec + at * nvec + v, s_step[i].W + v);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (in_arena) stage();
  pdl_wait();
  uint4* hrow = reinterpret_cast<uint4*>(hidden + (size_t)t * d);
  uint4 hq[NV];
#pragma unroll
  for (int u = 0; u < NV; ++u) {
    const int v = threadIdx.x + u * NT;
    hq[u] = make_uint4(0u, 0u, 0u, 0u);
    if (v < nvec) hq[u] = __ldcs(hrow + v);
  }
  if (!in_arena) stage();
  // Gates are decided once for the row, by the first warp, a lane each: a score may be one that another row of this call is just
  // writing, and threads that read it for themselves could part ways in front of the barriers below.
  const unsigned gated = s_gated;
  float score = 0.f;
  if (warp == 0 && ((gated >> lane) & 1u)) score = ld_score(s_step[lane].gate.score);
  float bias_lo = 0.f, bias_hi = 0.f;            // of the probe that this warp will finish
  if (warp < n && s_step[warp].kind == MIX_PROBE) {
    const ChainStep& st = s_step[warp];
    if (in_arena && st.C == 1) {
      bias_lo = st.alpha;
    } else if (st.b != nullptr) {
      if (lane < st.C) bias_lo = __ldg(st.b + lane);
      if (lane + 32 < st.C) bias_hi = __ldg(st.b + lane + 32);
    }
  }
  unsigned open = s_free;                        // (a closed gate skips its app, not the chain behind it)
  if (gated != 0u) {
    if (warp == 0) {
      const unsigned passed = __ballot_sync(0xffffffffu, ((gated >> lane) & 1u) && gate_passes(s_step[lane].gate, score));
      if (lane == 0) s_passed = passed;
    }
    __syncthreads();
    open |= s_passed;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  unsigned own = s_own, finished = 0u;
  bool dirty = false;
  int i = 0;
again:                                           // up to the next step that is gated on a score of this chain
  const int end = __builtin_expect(own != 0u, 0) ? __ffs(own) - 1 : n;
#pragma unroll 1
  for (; i < end; ++i) {
    if (!((open >> i) & 1u)) continue;
    const ChainStep& st = s_step[i];
    const int kind = st.kind;
    const bool single = kind == MIX_STEER || kind == MIX_PROJECT || (kind == MIX_PROBE && st.C == 1);
    if ((kind == MIX_STEER || kind == MIX_PROJECT) && st.alpha == 0.f) continue;     // identity, bit-exact
    if (kind == MIX_PROBE && scores == nullptr) continue;
    if (single) {
      uint4 vq[NV];
      const uint4* src = st.staged >= 0 ? s_vec + st.staged * nvec : st.W;
#pragma unroll
      for (int u = 0; u < NV; ++u) {
        const int v = threadIdx.x + u * NT;
        vq[u] = make_uint4(0u, 0u, 0u, 0u);
        if (v < nvec) vq[u] = src[v];
      }
      float coef = st.alpha;
      if (kind != MIX_STEER) {
        float dot = 0.f;
#pragma unroll
        for (int u = 0; u < NV; ++u) {
          float x[8], y[8];
          unpack8(hq[u], x);
          unpack8(vq[u], y);
#pragma unroll
          for (int e = 0; e < 8; ++e) dot = fmaf(x[e], y[e], dot);
        }
        dot = warp_sum(dot);
        if (kind == MIX_PROBE) {
          if (lane == 0) s_part[warp][st.col] = dot;
          continue;
        }
        if (lane == 0) s_dot[i][warp] = dot;     // h - beta (h . r) r
        __syncthreads();
        float total = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) total += s_dot[i][w];
        coef = -st.alpha * total;
      }
#pragma unroll
      for (int u = 0; u < NV; ++u) {
        float x[8], y[8];
        unpack8(hq[u], x);
        unpack8(vq[u], y);
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] = fmaf(coef, y[e], x[e]);
        hq[u] = pack8(x);
      }
      dirty = true;
    } else if (kind == MIX_PROBE) {
      const int C = st.C, col = st.col;
      const uint4* W = st.W;
#pragma unroll 1
      for (int c0 = 0; c0 < C; c0 += 4) {
        const int nc = min(4, C - c0);
        uint4 wq[4][NV];
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int u = 0; u < NV; ++u) {
            const int v = threadIdx.x + u * NT;
            if (c < nc && v < nvec) wq[c][u] = __ldg(W + (size_t)(c0 + c) * nvec + v);
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
        if ((lane & 7) == 0 && (lane >> 3) < nc) s_part[warp][col + c0 + (lane >> 3)] = z;
      }
    }
  }
  if (own == 0u && dirty) {
#pragma unroll
    for (int u = 0; u < NV; ++u) {
      const int v = threadIdx.x + u * NT;
      if (v < nvec) __stcs(hrow + v, hq[u]);
    }
  }
  __syncthreads();
  if (scores != nullptr && warp < end && (((open & ~finished) >> warp) & 1u) && s_step[warp].kind == MIX_PROBE) {       // a warp per probe
    const ChainStep& st = s_step[warp];
    for (int c = lane; c < st.C; c += 32) {
      float z = c < 32 ? bias_lo : bias_hi;
#pragma unroll
      for (int w = 0; w < NW; ++w) z += s_part[w][st.col + c];
      s_part[0][st.col + c] = z;     // only this lane reads or writes the column from here on
    }
    __syncwarp();
    finish_probe(&s_part[0][st.col], st.C, st.act, row_scores + st.col, lane);
  }
  if (__builtin_expect(own != 0u, 0)) {
    // The score that step `end` is gated on now stands where separate calls would leave it; if that probe's gate was closed, it is
    // what was there before.
    finished = (1u << end) - 1u;
    __syncthreads();
    open &= ~(1u << end);
    if (gate_passes(s_step[end].gate, ld_score(s_step[end].gate.score))) open |= 1u << end;
    own &= own - 1u;
    goto again;
  }
}

// Router-logit steering: one thread per (row, expert).
__global__ void __launch_bounds__(256)
router_kernel(const int* __restrict__ token_slot, int T,
              const AppEntry* __restrict__ apps, const GateEntry* __restrict__ gates, int n_slots,
              float* __restrict__ logits, int n_experts) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int t = (int)(i / n_experts), e = (int)(i - (long long)t * n_experts);
  if (t >= T) return;
  const RowApp a = lookup(__ldg(token_slot + t), t, apps, gates, n_slots, nullptr, false);
  if (a.kind != MIX_ROUTER || a.C != n_experts) return;
  logits[i] += __ldg(reinterpret_cast<const float*>(a.W) + e);
}

// The step's slot map.  Rows behind the live ones hold -1, so a step is one operation on the stream: a copy where the map
// or one of these kernels, which set rows up to `n_fill` -- live in the previous map -- to -1 along the way.  With a live
// count of its own the map was two copies, and two staging copies, a kernel and a copy in the two-level form, at 2 us
// and more each on the stream and on the host.
// Contexts without SAE weight sets, of which a step has one per layer, take a map in host memory by kernel too: read over
// PCIe where it lies if the device can address it (2.9 us of stream time against 4.0 for a copy), among the kernel's
// parameters if it is pageable and short (1.1 us).  Contexts with weight sets keep the copy up to 2048 rows: their long kernels
// leave the translation of the host page cold, and the same read takes 5.3 us.
// 32 maps of 256 rows and the replay of 32 layers behind them: 260 us with two copies a map, 204 with one, 160 with this.
// Launched programmatically: a kernel is scheduled while its predecessor ends, and waits for it before it touches
// anything (the predecessor may still read the old map, or write the source).
constexpr int kMapThreads = 256;

// token_slot[t] = src[t]
__global__ void __launch_bounds__(kMapThreads)
install_map_kernel(const int* __restrict__ src, int T_live, int n_fill, int* __restrict__ token_slot) {
  pdl_launch_dependents();
  pdl_wait();
  const int t = blockIdx.x * kMapThreads + threadIdx.x;
  if (t < T_live) token_slot[t] = src[t];
  else if (t < n_fill) token_slot[t] = -1;
}

// The same with the map among the kernel's parameters.
struct MapParams {
  int slot[kMapParamRows];
};
__global__ void __launch_bounds__(kMapThreads)
install_map_params_kernel(const __grid_constant__ MapParams src, int T_live, int n_fill, int* __restrict__ token_slot) {
  pdl_launch_dependents();
  pdl_wait();
  const int t = blockIdx.x * kMapThreads + threadIdx.x;
  if (t < T_live) token_slot[t] = src.slot[t];
  else if (t < n_fill) token_slot[t] = -1;
}

// Two-level form: token_slot[t] = req_slot[token_req[t]]
__global__ void __launch_bounds__(kMapThreads)
compose_map_kernel(const int* __restrict__ token_req, const int* __restrict__ req_slot, int T_live, int n_req, int n_fill,
                   int* __restrict__ token_slot) {
  pdl_launch_dependents();
  pdl_wait();
  const int t = blockIdx.x * kMapThreads + threadIdx.x;
  if (t < T_live) {
    const int r = token_req[t];
    token_slot[t] = (r >= 0 && r < n_req) ? req_slot[r] : -1;
  } else if (t < n_fill) {
    token_slot[t] = -1;
  }
}

// b_eff[j] = b_enc[j] - sum_i W_enc[j,i] * b_dec[i]   (one warp per feature; registration time)
__global__ void fold_bias_kernel(const __nv_bfloat16* __restrict__ W_enc, const float* __restrict__ b_enc,
                                 const float* __restrict__ b_dec, float* __restrict__ b_eff, long long d_sae, int d) {
  const long long j = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (j >= d_sae) return;
  float acc = 0.f;
  for (int i = lane; i < d; i += 32) acc = fmaf(__bfloat162float(W_enc[j * d + i]), b_dec[i], acc);
  acc = warp_sum(acc);
  if (lane == 0) b_eff[j] = b_enc[j] - acc;
}

// Census of the batch's multi-class probe rows (2..32 classes; gates are not looked at): a CTA takes 8 tiles of
// 128 rows, one per warp (four rows per lane, their loads in flight together), counts each tile's such rows and
// appends the tiles that have any to a list -- one reservation per CTA, so the shared counters see two additions
// per 1024 rows; the last CTA to finish publishes the totals and the choice between the two probe kernels, and
// puts the working counters back to zero for the next call.
// The tensor-core kernel streams whole tiles, the 16-row kernel reaches 38 % of the HBM rate against its 80 %:
// it takes the call when the listed tiles are, on average, at least half full of such rows.
constexpr int kCensusWarps = 8;
__global__ void __launch_bounds__(kCensusWarps * 32)
mc_census_kernel(const int* __restrict__ token_slot, int T,
                 const AppEntry* __restrict__ apps, int n_slots, McCensus* __restrict__ census, int* __restrict__ tiles,
                 int* __restrict__ part_done) {
  if (blockIdx.x == 0)                                   // the tensor-core kernel's counters of finished column parts
    for (int i = threadIdx.x; i < kPPartItems * 4; i += kCensusWarps * 32) part_done[i] = 0;
  __shared__ int s_cnt[kCensusWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tile = blockIdx.x * kCensusWarps + warp;
  int slot[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int t = tile * kTileM + i * 32 + lane;
    slot[i] = t < T ? __ldg(token_slot + t) : -1;
  }
  int4 q[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    q[i] = make_int4(0, 0, 0, 0);
    if (slot[i] >= 0 && slot[i] < n_slots) q[i] = __ldg(reinterpret_cast<const int4*>(apps + slot[i]));    // valid, kind, n_classes, act
  }
  int cnt = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const bool hit = q[i].x && (q[i].y & kKindMask) == MIX_PROBE && q[i].z > 1 && q[i].z <= 32;
    cnt += __popc(__ballot_sync(0xffffffffu, hit));
  }
  if (lane == 0) s_cnt[warp] = cnt;
  __syncthreads();
  if (threadIdx.x == 0) {
    int n_local = 0, rows = 0;
#pragma unroll
    for (int w = 0; w < kCensusWarps; ++w) {
      n_local += s_cnt[w] > 0;
      rows += s_cnt[w];
    }
    if (n_local > 0) {
      int pos = atomicAdd(&census->w_tiles, n_local);
#pragma unroll
      for (int w = 0; w < kCensusWarps; ++w)
        if (s_cnt[w] > 0) tiles[pos++] = blockIdx.x * kCensusWarps + w;
      atomicAdd(&census->w_rows, rows);
    }
    __threadfence();
    if (atomicAdd(&census->w_done, 1) == (int)gridDim.x - 1) {
      const int n_tiles = atomicAdd(&census->w_tiles, 0), n_rows = atomicAdd(&census->w_rows, 0);
      census->n_tiles = n_tiles;
      census->n_rows = n_rows;
      census->use_tc = n_tiles > 0 && 2 * n_rows >= n_tiles * kTileM;
      census->w_tiles = 0;
      census->w_rows = 0;
      census->w_done = 0;
    }
  }
}

}  // namespace


bool has_multiclass_stage(const Ctx* c) {
  return c->cfg.T_max > kTeamMaxRows && c->cfg.C_max > 1 && !(c->cfg.flags & MIX_FLAG_SLOT_CHAINS);
}

cudaError_t launch_mc_census(const Ctx* c, int T, cudaStream_t s) {
  const int rows_per_cta = kCensusWarps * kTileM;
  mc_census_kernel<<<(c->cfg.T_max + rows_per_cta - 1) / rows_per_cta, kCensusWarps * 32, 0, s>>>(c->d_token_slot, T, c->d_apps,
                                                                           c->cfg.n_slots_max, c->d_mc_census, c->d_mc_tiles, c->d_part_done);
  return cudaGetLastError();
}

// The tensor-core probe kernel holds a whole SM's shared memory, as the SAE encode does: beside an encode
// it could only wait, so contexts with SAE weight sets leave every batch to the 16-row kernel.
bool has_tc_probe_stage(const Ctx* c) { return has_multiclass_stage(c) && c->cfg.n_groups_max == 0; }

cudaError_t launch_probe_steer(const Ctx* c, __nv_bfloat16* hidden, int T, float* scores, cudaStream_t s, bool allow_pdl, bool map_ahead) {
  const int pdl = (allow_pdl && (pdl_mask() & kPdlHook)) ? (map_ahead ? kPdlMapAhead : 1) : 0;
  const int nvec = c->cfg.d_model / 8, n_vec = (nvec + kHookWarps * 32 - 1) / (kHookWarps * 32);     // n_vec: per thread
  if (c->cfg.flags & MIX_FLAG_SLOT_CHAINS) {
    auto run = [&](auto kernel) {
      return launch_pdl(allow_pdl ? kPdlHook : 0, kernel, dim3(c->cfg.T_max), dim3(kHookWarps * 32), (size_t)kChainStaged * nvec * sizeof(uint4), s,
                        c->d_token_slot, T, c->d_apps, c->d_gates, c->d_chain_next, c->cfg.n_slots_max, hidden,
                        c->cfg.d_model, scores, c->cfg.C_max, c->d_status, c->d_vec_arena != nullptr ? 1 : 0, pdl);
    };
    switch (n_vec) {
      case 1: return run(probe_steer_chain_kernel<1>);
      case 2: return run(probe_steer_chain_kernel<2>);
      case 3: return run(probe_steer_chain_kernel<3>);
      default: return run(probe_steer_chain_kernel<kMostVec>);
    }
  } else if (c->cfg.T_max <= kTeamMaxRows) {
    auto run = [&](auto kernel) {
      return launch_pdl(allow_pdl ? kPdlHook : 0, kernel, dim3(c->cfg.T_max), dim3(kHookWarps * 32), 0, s, c->d_token_slot, T, c->d_apps, c->d_gates,
                        c->cfg.n_slots_max, hidden, c->cfg.d_model, scores, c->cfg.C_max, c->d_status,
                        reinterpret_cast<const uint4*>(c->d_vec_arena), pdl);
    };
    auto of_width = [&](auto nv) {
      constexpr int NV = decltype(nv)::value;
      if (c->cfg.n_groups_max > 0) return run(probe_steer_late_kernel<NV>);
      return pdl == kPdlMapAhead ? run(probe_steer_team_kernel<NV, kTeamMapAhead>) : run(probe_steer_team_kernel<NV, kTeamPlain>);
    };
    switch (n_vec) {
      case 1: return of_width(std::integral_constant<int, 1>());
      case 2: return of_width(std::integral_constant<int, 2>());
      case 3: return of_width(std::integral_constant<int, 3>());
      default: return of_width(std::integral_constant<int, kMostVec>());
    }
  } else {
    auto run = [&](auto kernel, int warps) {
      kernel<<<(c->cfg.T_max + warps - 1) / warps, warps * 32, 0, s>>>(c->d_token_slot, T, c->d_apps, c->d_gates,
                                                                      c->cfg.n_slots_max, hidden, c->cfg.d_model, scores,
                                                                      c->cfg.C_max, c->d_status, has_multiclass_stage(c) ? 1 : 0);
    };
    if (has_tc_probe_stage(c)) run(probe_steer_kernel<8, 3>, 8);
    else run(probe_steer_kernel<4, 8>, 4);
  }
  return cudaGetLastError();
}

cudaError_t launch_probe_multiclass(const Ctx* c, const __nv_bfloat16* hidden, int T, float* scores, cudaStream_t s) {
  const int blocks = (c->cfg.T_max + kMcRows - 1) / kMcRows;
  probe_multiclass_kernel<<<blocks, kMcWarps * 32, 0, s>>>(c->d_token_slot, T, c->d_apps, c->d_gates,
                                                                 c->cfg.n_slots_max, hidden, c->cfg.d_model, scores,
                                                                 c->cfg.C_max, has_tc_probe_stage(c) ? c->d_mc_census : nullptr);
  return cudaGetLastError();
}

cudaError_t launch_router(const Ctx* c, float* logits, int n_experts, int T, cudaStream_t s) {
  const long long n = (long long)c->cfg.T_max * n_experts;
  router_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(c->d_token_slot, T, c->d_apps, c->d_gates,
                                                            c->cfg.n_slots_max, logits, n_experts);
  return cudaGetLastError();
}

cudaError_t launch_install_map(const Ctx* c, const int* src, int T_live, int n_fill, cudaStream_t s) {
  const int n = T_live > n_fill ? T_live : n_fill;
  if (n == 0) return cudaSuccess;
  return launch_pdl(kPdlHook, install_map_kernel, dim3((n + kMapThreads - 1) / kMapThreads), dim3(kMapThreads), 0, s, src, T_live, n_fill,
                    c->d_token_slot);
}

cudaError_t launch_install_map_params(const Ctx* c, const int* host_src, int T_live, int n_fill, cudaStream_t s) {
  MapParams p;
  memcpy(p.slot, host_src, (size_t)T_live * sizeof(int));
  const int n = T_live > n_fill ? T_live : n_fill;
  return launch_pdl(kPdlHook, install_map_params_kernel, dim3((n + kMapThreads - 1) / kMapThreads), dim3(kMapThreads), 0, s, p, T_live, n_fill,
                    c->d_token_slot);
}

cudaError_t launch_compose_map(const Ctx* c, const int* token_req, const int* req_slot, int T_live, int n_req, int n_fill, cudaStream_t s) {
  const int n = T_live > n_fill ? T_live : n_fill;
  if (n == 0) return cudaSuccess;
  return launch_pdl(kPdlHook, compose_map_kernel, dim3((n + kMapThreads - 1) / kMapThreads), dim3(kMapThreads), 0, s, token_req, req_slot,
                    T_live, n_req, n_fill, c->d_token_slot);
}

cudaError_t launch_fold_bias(const __nv_bfloat16* W_enc, const float* b_enc, const float* b_dec, float* b_eff,
                             long long d_sae, int d, cudaStream_t s) {
  const unsigned blocks = (unsigned)((d_sae + 7) / 8);
  fold_bias_kernel<<<blocks, 256, 0, s>>>(W_enc, b_enc, b_dec, b_eff, d_sae, d);
  return cudaGetLastError();
}

}  // namespace mix
