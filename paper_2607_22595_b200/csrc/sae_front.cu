// Front of the SAE chain: slot routing and the row pack in ONE launch.
//
// Routing is integer work on the slot map: which rows carry an SAE app, of which weight set, and where each of
// them goes in the packed panel (weight set by weight set, ascending token order inside a set, every set
// starting on a 128-row tile).  Calls of up to kFrontLocal chunks of 256 token rows route without an exchange: every CTA
// classifies all rows for itself.  Longer ones do it as a chunked scan inside one grid -- every CTA classifies 256
// token rows and publishes their counts, every CTA then reads the small count table.  Either way the rows are packed right
// after, each CTA the eight panel rows it owns, found through its own classification or the published per-row records.
// The only waiting between CTAs is a bounded wait for the published chunks; see front_kernel.
//
// Pack forms: the bf16 row as it is; with an 8-bit encoder the row as E4M3 codes with a power-of-two row
// scale -- quantised (MIX_FLAG_FP8_ACT), or split exactly into two E4M3 operands hi + lo.
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <type_traits>

#include "hook_row.cuh"
#include "mix_internal.h"
#include "row_lookup.cuh"

namespace mix {

namespace {

constexpr int kFrontThreads = 256;        // = token rows a CTA classifies
constexpr int kFrontWarps = kFrontThreads / 32;   // = panel rows a CTA packs

// bf16 row -> panel row, or zeros for the padding rows of a tile.  (Nothing reads what comes of those; but zeros cost the tensor
// cores less power than rows that a longer call left there.  Batches of up to 2048 ragged rows over eight sets of d = 8192, 131072
// features, another map every call: median 1.60 ms with what was there, 1.51 with zeros.)
__device__ __forceinline__ void pack_row_bf16(const __nv_bfloat16* __restrict__ hidden, int t, __nv_bfloat16* __restrict__ panel,
                                              size_t p, int d, int lane) {
  uint4* dst = reinterpret_cast<uint4*>(panel + p * d);
  const int nvec = d >> 3;
  if (t < 0) {
    for (int i = lane; i < nvec; i += 32) dst[i] = make_uint4(0u, 0u, 0u, 0u);
    return;
  }
  const uint4* src = reinterpret_cast<const uint4*>(hidden + (size_t)t * d);
  for (int i = lane; i < nvec; i += 256) {               // eight loads in flight per lane, the ragged end included
    uint4 q[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (i + 32 * u < nvec) q[u] = __ldg(src + i + 32 * u);
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (i + 32 * u < nvec) dst[i + 32 * u] = q[u];
  }
}

// 8-bit encoder: the row goes into the panel as E4M3 codes with a power-of-two row scale.
// s = the smallest power of two with max|h_i| / s <= 448 (never below 2^-100; 1 for a row of zeros); h_i / s is
// exact in fp32, the conversion rounds to nearest even.  A first pass finds the largest magnitude, a second
// one (the row is in L1 by then) writes the codes.
//   kSplit = false (MIX_FLAG_FP8_ACT): code_i = E4M3 nearest to h_i / s -- the encoder's input IS quantised.
//   kSplit = true  (MIX_FLAG_FP8_W_ENC alone): the bf16 row is kept, as the sum of two E4M3 operands with the same
//     scale: hi_i = E4M3 nearest to x = h_i / s, lo_i = E4M3 nearest to x - hi_i (exact subtraction).  A bf16 value
//     has 8 significant bits, hi takes the leading 4 and the remainder has at most 4, so hi + lo = x exactly
//     unless bits of x lie below 2^-9 (the subnormal step of E4M3), i.e. the error per element is at most
//     2^-10 s <= 4.4e-6 max|h_i| and zero for |h_i| >= 2^-2 s.  The lo codes go to rows [lo_row0 + p] of the panel.
template <bool kSplit>
__device__ __forceinline__ void pack_row_e4m3(const __nv_bfloat16* __restrict__ hidden, int t, unsigned char* __restrict__ panel,
                                              float* __restrict__ act_scale, size_t p, int d, int lo_row0, int lane) {
  uint2* dst = reinterpret_cast<uint2*>(panel + p * d);
  uint2* dst_lo = reinterpret_cast<uint2*>(panel + ((size_t)lo_row0 + p) * d);
  const int nvec = d >> 3;
  if (t < 0) {
    for (int i = lane; i < nvec; i += 32) {
      dst[i] = make_uint2(0u, 0u);
      if (kSplit) dst_lo[i] = make_uint2(0u, 0u);
    }
    return;
  }
  const uint4* src = reinterpret_cast<const uint4*>(hidden + (size_t)t * d);
  unsigned m2 = 0u;                                     // two 15-bit magnitudes, compared as integers
  for (int i = lane; i < nvec; i += 32) {
    const uint4 q = __ldg(src + i);
    m2 = __vmaxu2(m2, __vmaxu2(__vmaxu2(q.x & 0x7fff7fffu, q.y & 0x7fff7fffu), __vmaxu2(q.z & 0x7fff7fffu, q.w & 0x7fff7fffu)));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m2 = __vmaxu2(m2, __shfl_xor_sync(0xffffffffu, m2, o));
  const unsigned a = max(m2 & 0xffffu, m2 >> 16);       // bf16 bits of max|h_i|: (1 + frac / 128) * 2^(E - 127)
  int e = 0;
  if (a != 0u) {
    const int E = (int)(a >> 7) - 127, frac = (int)(a & 0x7fu);
    e = max(E - (frac <= 96 ? 8 : 7), -100);            // 448 = 1.75 * 2^8, and 1.75 = 1 + 96 / 128
  }
  const float inv = __uint_as_float((unsigned)(127 - e) << 23);
  if (lane == 0) act_scale[p] = __uint_as_float((unsigned)(127 + e) << 23);
  for (int i = lane; i < nvec; i += 32) {
    const uint4 q = __ldg(src + i);
    const unsigned w[4] = {q.x, q.y, q.z, q.w};
    unsigned short c[4], cl[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float lo = __uint_as_float(w[u] << 16) * inv, hi = __uint_as_float(w[u] & 0xffff0000u) * inv;
      c[u] = __nv_cvt_float2_to_fp8x2(make_float2(lo, hi), __NV_SATFINITE, __NV_E4M3);
      if (kSplit) {
        const float2 back = __half22float2(__half2(__nv_cvt_fp8x2_to_halfraw2(c[u], __NV_E4M3)));   // exact: E4M3 fits fp16
        cl[u] = __nv_cvt_float2_to_fp8x2(make_float2(lo - back.x, hi - back.y), __NV_SATFINITE, __NV_E4M3);
      }
    }
    dst[i] = make_uint2((unsigned)c[0] | ((unsigned)c[1] << 16), (unsigned)c[2] | ((unsigned)c[3] << 16));
    if (kSplit) dst_lo[i] = make_uint2((unsigned)cl[0] | ((unsigned)cl[1] << 16), (unsigned)cl[2] | ((unsigned)cl[3] << 16));
  }
}

struct FrontArgs {
  // slot map and tables (read)
  const int* token_slot;
  int T;
  const AppEntry* apps;
  const GateEntry* gates;
  int n_slots;
  const GroupEntry* groups;
  int n_groups;
  const int* chain_next;
  int edit_only;
  // exchange between the CTAs of one launch
  int2* row_meta;          // [T_max] per token row: (weight set + 1) | edit count << 8 | error-term flag << 16 (0: not an SAE row), slot
  int* counts;             // [chunks][n_groups + 1] SAE rows per weight set in each chunk of 256 token rows; last column: delta-role rows
  int* sync;               // [0] chunks published so far in this call, [1] CTAs of this call that are done (both back to 0 when the call ends)
  // routing results (written)
  int* panel_row;
  RowRec* row_rec;
  int panel_cap;
  int* mtile_group;
  RouteState* rs;
  unsigned* status;
  int* row_flag;
  int* mtile_flag;
  int* n_flagged;
  cudaGraphConditionalHandle cond;
  int use_cond;
  // pack
  const __nv_bfloat16* hidden;
  void* panel;
  float* act_scale;
  int d;
  unsigned* tau_slots;
  unsigned* tau_min;
  int lo_row0;
  unsigned long long* clk;   // profiling aid or null
  int n_sms;
  int cand_tiles;
  // the rows of the other apps, where they are part of this launch
  __nv_bfloat16* rows;
  float* scores;
  int C_max;
  const uint4* vec_arena;
  int pdl;                   // as the hook kernel is told
  int n_front;               // CTAs of the routing and the pack; those behind them take a row each
  int pair_mode;             // 0: the encode runs on single CTAs, 1: on CTA pairs, 2: decided here from the routing result
};

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

constexpr long long kFrontWaitCycles = 2000000000ll;   // ~1 s: cap of the wait for the other CTAs' chunks

constexpr int kFrontLocal = 4;            // chunks (of 256 token rows) up to which every CTA routes the whole call for itself

// What the slot map says about one token row.
struct RowClass {
  int meta;        // (weight set + 1) | edit count << 8 | error-term flag << 16; 0: not an SAE row
  int slot;
  bool delta;      // a row of the tail kernel's delta role
};

// Slot and the part of the app entry that routing needs, requested together.
struct RowEntry {
  int slot;
  int2 q0;         // valid, kind
  int g, n_edit, add_error;
};
__device__ __forceinline__ RowEntry load_entry(const FrontArgs& a, int slot) {
  RowEntry r;
  r.slot = slot;
  r.q0 = make_int2(0, 0);
  r.g = -1;
  r.n_edit = r.add_error = 0;
  if (slot >= 0) {
    const AppEntry* e = a.apps + slot;
    r.q0 = __ldg(reinterpret_cast<const int2*>(e));
    r.g = __ldg(&e->group);
    const int2 ne = __ldg(reinterpret_cast<const int2*>(&e->n_edit));
    r.n_edit = ne.x;
    r.add_error = ne.y != 0;
  }
  return r;
}

__device__ __forceinline__ RowClass classify(const FrontArgs& a, RowEntry r, int t, const int* s_gact, const int* s_gtiles) {
  // a row whose slot starts a chain is an SAE row if the chain ends in an SAE app: follow the links
  if (r.q0.x && (r.q0.y & kKindChained) && (r.q0.y & kKindMask) != MIX_SAE) {
    int s2 = r.slot;
    int2 h2 = r.q0;
    for (int depth = 1; depth < kMaxChain && s2 >= 0; ++depth) {
      s2 = (h2.y & kKindChained) ? __ldg(a.chain_next + s2) : -1;
      if (s2 < 0 || s2 >= a.n_slots) { s2 = -1; break; }
      h2 = __ldg(reinterpret_cast<const int2*>(a.apps + s2));
      if (!h2.x) { s2 = -1; break; }
      if ((h2.y & kKindMask) == MIX_SAE) break;
    }
    if (s2 >= 0 && (h2.y & kKindMask) != MIX_SAE) s2 = -1;
    r = load_entry(a, s2);
  }
  RowClass c;
  c.meta = 0;
  c.slot = r.slot;
  c.delta = false;
  if (r.q0.x && (r.q0.y & kKindMask) == MIX_SAE) {
    if (r.g < 0 || r.g >= a.n_groups || s_gtiles[r.g] == 0) {
      atomicOr(a.status, MIX_STATUS_BAD_GROUP);
    } else if (a.edit_only && r.add_error && s_gact[r.g] != MIX_SAE_TOPK) {
      // handled by sae_edit_only_kernel: with the error term on, a ReLU / JumpReLU row needs
      // only the pre-activations of its edited features, not the whole encode
    } else if (!(r.q0.y & kKindGated) || gate_open(a.gates, r.slot, t)) {
      c.meta = (r.g + 1) | (r.n_edit << 8) | (r.add_error << 16);
      c.delta = r.add_error && r.n_edit > 0 && s_gact[r.g] != MIX_SAE_TOPK;
    }
  }
  return c;
}

__device__ __forceinline__ int warp_scan(int v, int lane) {      // inclusive
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}
__device__ __forceinline__ long long warp_sum64(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// What exists once per call, written by one warp (lane q: weight set q): the routing result the encode and the tail read,
// and which encode kernel takes which weight set.
__device__ __forceinline__ void write_route(const FrontArgs& a, int total, int nt, bool topk, int mt0, int mt, int n_delta, int lane) {
  const bool live = total > 0;
  const int m_tiles = (total + kTileM - 1) / kTileM;
  const int my_tiles = live ? m_tiles * nt : 0;
  const int tiles_incl = warp_scan(my_tiles, lane);
  const int tiles = __shfl_sync(0xffffffffu, tiles_incl, 31);
  a.rs->group_count[lane] = total;                  // (lanes of sets that do not exist: no rows)
  a.rs->group_mtile0[lane] = mt0;
  a.rs->group_tile0[lane] = tiles_incl - my_tiles;
  const int rows = __reduce_add_sync(0xffffffffu, total);
  const int topk_rows = __reduce_add_sync(0xffffffffu, topk ? total : 0);
  const int nt_most = max(1, __reduce_max_sync(0xffffffffu, live ? nt : 0));
  // per feature tile, in units of 1/40 of the time the W_enc tile takes to stream from HBM (measured on one
  // weight set with 64 ... 1024 rows): single CTAs stream at the full rate for one row tile, and from two row
  // tiles on every further tile costs 25 -- each of them fetches the W_enc tile again, from L2; a pair costs 46
  // per 256-row tile whether its second half has rows or not, streaming at a slightly lower rate
  const long long cs = live ? (long long)(m_tiles == 1 ? 40 : 25 * m_tiles) * nt : 0;
  const long long cp = live ? (long long)(46 * ((m_tiles + 1) / 2)) * nt : 0;
  const long long cost_single = warp_sum64(cs), cost_pair = warp_sum64(cp), cost_split = warp_sum64(min(cs, cp));
  const int live_mask = (int)__ballot_sync(0xffffffffu, live);
  const int split_mask = (int)__ballot_sync(0xffffffffu, live && cp < cs);
  const bool odd3 = __ballot_sync(0xffffffffu, live && cp >= cs && m_tiles >= 3) != 0u;
  // Pairs win where a weight set has an even number of row tiles (two tiles share one fetch of W_enc, and the
  // pair's instruction fills less shared memory per flop) and lose where half of a pair would repeat the other
  // half's work: one row tile, or three.  Each weight set may go to the form that is cheaper for it -- the two
  // encode kernels then both work, one after the other, which costs a second ramp-up and drain (about 25 us:
  // in the units above 25 x 40 / (time to stream one tile of 512 d bytes at 6.3 TB/s) = 1.23e7 / d).
  // Measured on config 4's replays, the split pays when two or more sets go to the pairs, or when a set of
  // three or more row tiles stays with the single CTAs; ONE two-tile set among one-tile sets does not: inside
  // the single-CTA kernel its second fetch of each W_enc tile and its tensor time hide behind the other sets'
  // streams (1.67 ms all single against 1.71-1.74 ms split for sets of 1, 1, 1, 1, 2 tiles), so such a call
  // stays with one form.
  int mask = a.pair_mode == 1 ? live_mask : 0;
  if (a.pair_mode == 2) {
    const bool both = split_mask != 0 && split_mask != live_mask;
    const long long split_total = cost_split + (both ? 12300000ll / max(a.d, 1) : 0ll);
    const bool split_pays = !both || __popc(split_mask) >= 2 || odd3;
    if (split_pays && split_total <= min(cost_single, cost_pair)) mask = split_mask;
    else mask = cost_pair < cost_single ? live_mask : 0;
  }
  // (Pairs give way to narrow tiles only where single CTAs can go down to 64 features: at 128 both forms bring the same
  // bytes into an SM per k-block.)
  if (a.pair_mode != 1 && 4 * tiles <= a.n_sms) mask = 0;
  if (lane == 0) {
    a.rs->group_mtile0[kMaxGroups] = mt;
    a.rs->group_tile0[kMaxGroups] = tiles;
    a.rs->n_panel_rows = mt * kTileM;
    a.rs->n_mtiles = mt;
    a.rs->n_sae_rows = rows;
    a.rs->total_tiles = tiles;
    a.rs->n_topk_rows = topk_rows;
    a.rs->n_delta_rows = n_delta;
    a.rs->tile_n = mask == 0 ? tile_width(tiles, nt_most, a.n_sms, a.cand_tiles) : kTileN;
    a.rs->pair_mask = mask;
    a.rs->use_pair = mask != 0;
    if (a.n_flagged) *a.n_flagged = 0;       // fallback-selection flags of the fused TopK path start clear every call
    // graph-conditional form: the rest of the SAE chain sits in the body of an IF node that runs only when a row needs it
    if (a.use_cond) cudaGraphSetConditional(a.cond, rows > 0 ? 1u : 0u);
  }
}

// Routing and row pack in one launch.
//   Calls of up to 1024 rows: every CTA classifies ALL token rows -- slot -> app entry -> SAE row of which weight set, four
//      rows a thread, their loads in flight together -- and so knows every row's place in the panel; the eight rows that
//      fall to the CTA are noted along the way.  No CTA waits for another.  (91 rows behind a 16384-feature encode: 8.2 us
//      with the exchange below, 4.7 without.)
//   Longer calls, where that would cost T rows times a CTA for every eight: CTA c < chunks classifies token rows
//      [256 c, 256 c + 256) and PUBLISHES the chunk -- per-row records, per-set counts, then one more on the call's counter
//      of published chunks.  Every CTA waits (one thread polls, bounded) until the counter says all chunks are there, reads
//      the small count table and scans it.  The publishing CTAs never wait before they publish, and CTAs are dispatched in
//      index order, so whoever waits, waits for work that is already running.  The rows of a CTA are found through the
//      scan and the published records.
// Launched programmatically behind the caller's work, or the hook kernel, of a small context: what is read before the wait is the slot map and the
// tables, as in that kernel; gates, `hidden` and everything that is written come after it.
// Then CTA b packs panel rows [8 b, 8 b + 8), one per warp.  The last CTA -- whose panel rows a call seldom needs -- writes
// what exists once (routing result, tile -> weight-set map, conditional handle), beside the others' packing.  The last CTA
// of the launch to leave puts the two counters back to zero for the next call.
// kPack: 0 the bf16 row, 1 E4M3 hi + lo (exact split), 2 E4M3 quantised.
// NV > 0 (contexts of up to 2048 rows, without chains): the rows of probes, steering vectors and projections, which no other
// part of the call touches, go with this launch, a CTA each behind the others, NV vectors of the row a thread.  As a kernel in front
// of this one they were a launch for the host and 1 ... 4 us on the stream: 64 rows called eagerly, d = 512, 34.4 -> 33.5 us; 1000 SAE
// rows of d = 2304, 206 -> 203.8; 91 of d = 4096 in a graph, 60.5 -> 60.1.
template <int kPack, int NV>
__global__ void __launch_bounds__(kFrontThreads, NV == 0 ? 1 : (NV <= 2 ? 3 : 2))
front_kernel(const FrontArgs a) {
  extern __shared__ int s_tab[];                      // [chunks][n_groups + 1]: counts, then exclusive prefixes over the chunks
  __shared__ int s_total[kMaxGroups + 1];
  __shared__ int s_gact[kMaxGroups], s_gtiles[kMaxGroups];   // per weight set: activation, feature tiles (0: not registered)
  __shared__ const __nv_bfloat16* s_gwdec[kMaxGroups];
  __shared__ const float* s_gtheta[kMaxGroups];
  __shared__ int s_wcnt[kFrontLocal * kFrontWarps][kMaxGroups + 1];   // rows per (chunk, warp) and weight set; then what comes before them
  __shared__ int s_row[kFrontWarps][3];                // this CTA's panel rows: token row, record, slot
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cta = blockIdx.x;
  const bool first_cta = cta == 0, route_cta = cta == a.n_front - 1;
  if (a.pdl == kPdlMapAhead) pdl_wait();               // (the slot map is read ahead of the waits below)
  if constexpr (NV > 0) {
    static_assert(kHookWarps * 32 == kFrontThreads, "a CTA per row");
    if (cta >= a.n_front) {
      __shared__ float s_part[kHookWarps][kMaxClasses];
      late_row<NV>(a.n_front, a.token_slot, a.T, a.apps, a.gates, a.n_slots, a.rows, a.d, a.scores, a.C_max, a.status, a.vec_arena, s_part);
      return;
    }
  }
  const int n_groups = a.n_groups, n_slots = a.n_slots, ncol = n_groups + 1;
  const int n_chunks = (a.T + kFrontThreads - 1) / kFrontThreads;     // the same in every CTA: who publishes is fixed by the launch
  const bool local = n_chunks <= kFrontLocal;
  phase_stamp(a.clk, 0, first_cta && tid == 0);
  if (tid < n_groups) {                                // requested now, needed after the first barrier
    const bool valid = __ldg(&a.groups[tid].valid) != 0;
    s_gact[tid] = __ldg(&a.groups[tid].act);
    s_gtiles[tid] = valid ? (int)(__ldg(&a.groups[tid].d_sae) / kTileN) : 0;
    s_gwdec[tid] = a.groups[tid].W_dec;
    s_gtheta[tid] = a.groups[tid].theta;
  }
  auto slot_of = [&](int t) {
    const int slot = t < a.T ? __ldg(a.token_slot + t) : -1;
    return slot < n_slots ? slot : -1;
  };
  int rank[kFrontLocal], grp[kFrontLocal];             // local: this thread's rows -- weight set or -1, place among the warp's rows of the set
  RowClass row[kFrontLocal];
  bool ok = true;
  if (local) {
    RowEntry e[kFrontLocal];
#pragma unroll
    for (int u = 0; u < kFrontLocal; ++u) e[u].slot = u < n_chunks ? slot_of(u * kFrontThreads + tid) : -1;
#pragma unroll
    for (int u = 0; u < kFrontLocal; ++u) e[u] = load_entry(a, e[u].slot);
    pdl_wait();
    for (int i = tid; i < n_chunks * kFrontWarps * ncol; i += kFrontThreads) s_wcnt[i / ncol][i % ncol] = 0;
    if (tid < kFrontWarps) s_row[tid][0] = -1;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kFrontLocal; ++u) {
      grp[u] = -1;
      rank[u] = 0;
      if (u < n_chunks) {
        row[u] = classify(a, e[u], u * kFrontThreads + tid, s_gact, s_gtiles);
        grp[u] = (row[u].meta & 0xff) - 1;
        const unsigned same = __match_any_sync(0xffffffffu, grp[u]);
        rank[u] = __popc(same & ((1u << lane) - 1u));
        if (grp[u] >= 0 && rank[u] == 0) s_wcnt[u * kFrontWarps + warp][grp[u]] = __popc(same);
        const unsigned dm = __ballot_sync(0xffffffffu, row[u].delta);
        if (lane == 0) s_wcnt[u * kFrontWarps + warp][n_groups] = __popc(dm);
      }
    }
    phase_stamp(a.clk, 1, first_cta && tid == 0);
    __syncthreads();
    for (int q = warp; q < ncol; q += kFrontWarps) {   // exclusive scan over (chunk, warp), one column per warp
      const int v = lane < n_chunks * kFrontWarps ? s_wcnt[lane][q] : 0;
      const int incl = warp_scan(v, lane);
      if (lane < n_chunks * kFrontWarps) s_wcnt[lane][q] = incl - v;
      if (lane == 31) s_total[q] = incl;
    }
  } else {
    if (cta < n_chunks) {                              // classify and publish one chunk
      const int t = cta * kFrontThreads + tid;
      const RowEntry e = load_entry(a, slot_of(t));
      pdl_wait();
      __syncthreads();                                 // the weight-set table is in shared memory
      const RowClass c = classify(a, e, t, s_gact, s_gtiles);
      if (t < a.T) a.row_meta[t] = make_int2(c.meta, c.slot);
      const int g = (c.meta & 0xff) - 1;
      for (int q = 0; q < n_groups; ++q) {
        const unsigned m = __ballot_sync(0xffffffffu, g == q);
        if (lane == 0) s_wcnt[warp][q] = __popc(m);
      }
      const unsigned m = __ballot_sync(0xffffffffu, c.delta);
      if (lane == 0) s_wcnt[warp][n_groups] = __popc(m);
      __syncthreads();
      if (tid < ncol) {
        int sum = 0;
#pragma unroll
        for (int w = 0; w < kFrontWarps; ++w) sum += s_wcnt[w][tid];
        a.counts[cta * ncol + tid] = sum;
      }
      __threadfence();
      __syncthreads();
      if (tid == 0) atomicAdd(a.sync, 1);              // (fence above + this: the chunk is published)
    } else {
      pdl_wait();
      __syncthreads();                                 // (the weight-set table)
    }
    phase_stamp(a.clk, 1, first_cta && tid == 0);
    // wait for every chunk, scan the counts
    if (tid == 0 && ld_acquire(a.sync) < n_chunks) {   // one polling thread per CTA, backing off: a thousand CTAs ask about one word
      const long long t0 = clock64();
      unsigned ns = 32;
      while (ld_acquire(a.sync) < n_chunks) {
        if (clock64() - t0 > kFrontWaitCycles) { ok = false; break; }
        __nanosleep(ns);
        if (ns < 256) ns *= 2;
      }
    }
    ok = __syncthreads_and(ok) != 0;
    if (ok) {
      for (int i = tid; i < n_chunks * ncol; i += kFrontThreads) s_tab[i] = __ldcg(a.counts + i);   // (never through L1: written by other SMs)
      __syncthreads();
      for (int q = warp; q < ncol; q += kFrontWarps) { // exclusive scan over the chunks, one column per warp
        int carry = 0;
        for (int c0 = 0; c0 < n_chunks; c0 += 32) {
          const int c = c0 + lane;
          const int v = c < n_chunks ? s_tab[c * ncol + q] : 0;
          const int incl = warp_scan(v, lane);
          if (c < n_chunks) s_tab[c * ncol + q] = carry + incl - v;
          carry += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0) s_total[q] = carry;
      }
    }
  }
  if (ok) {
    __syncthreads();
    phase_stamp(a.clk, 2, first_cta && tid == 0);
    // every warp works out where the weight sets' rows start (lane q: set q)
    const int my_total = lane < n_groups ? s_total[lane] : 0;
    const int my_mt = (my_total + kTileM - 1) / kTileM;
    const int mt_incl = warp_scan(my_mt, lane);
    const int n_mtiles = __shfl_sync(0xffffffffu, mt_incl, 31), n_panel_rows = n_mtiles * kTileM;
    const int my_base = (mt_incl - my_mt) * kTileM;
    int t = -1, meta = 0, slot = -1;
    const int p = cta * kFrontWarps + warp;
    if (local) {
#pragma unroll
      for (int u = 0; u < kFrontLocal; ++u) {
        if (u >= n_chunks) break;
        const int base = __shfl_sync(0xffffffffu, my_base, grp[u] & 31);
        if (grp[u] >= 0) {
          const int pp = base + s_wcnt[u * kFrontWarps + warp][grp[u]] + rank[u];
          if (pp / kFrontWarps == cta) {
            int* r = s_row[pp % kFrontWarps];
            r[0] = u * kFrontThreads + tid;
            r[1] = row[u].meta;
            r[2] = row[u].slot;
          }
        }
      }
      __syncthreads();
      t = s_row[warp][0];
      if (t >= 0) {
        meta = s_row[warp][1];
        slot = s_row[warp][2];
      }
    } else if (p < n_panel_rows) {
      // the set is the last one that starts at or before p; the row's rank within it follows
      const int g = 31 - __clz(__ballot_sync(0xffffffffu, lane < n_groups && my_mt > 0 && my_base <= p));
      const int r = p - __shfl_sync(0xffffffffu, my_base, g);
      if (r < __shfl_sync(0xffffffffu, my_total, g)) {
        // the chunk that holds rank r: the last one whose first rank is <= r
        int c_hit = 0;
        for (int c0 = 0; c0 < n_chunks; c0 += 32) {
          const int c = c0 + lane;
          const unsigned m = __ballot_sync(0xffffffffu, c < n_chunks && s_tab[c * ncol + g] <= r);
          if (m) c_hit = c0 + 31 - __clz(m);
        }
        int left = r - s_tab[c_hit * ncol + g];        // rank inside the chunk
        int2 mm[kFrontThreads / 32];
#pragma unroll
        for (int i = 0; i < kFrontThreads / 32; ++i) {
          const int tt = c_hit * kFrontThreads + i * 32 + lane;
          mm[i] = tt < a.T ? __ldcg(a.row_meta + tt) : make_int2(0, -1);
        }
        bool found = false;
#pragma unroll
        for (int i = 0; i < kFrontThreads / 32; ++i) {
          const unsigned m = __ballot_sync(0xffffffffu, (mm[i].x & 0xff) - 1 == g);
          const int cnt = __popc(m);
          if (!found) {
            if (left < cnt) {
              const int src = __fns(m, 0, left + 1);
              t = c_hit * kFrontThreads + i * 32 + src;
              meta = __shfl_sync(0xffffffffu, mm[i].x, src);
              slot = __shfl_sync(0xffffffffu, mm[i].y, src);
              found = true;
            } else {
              left -= cnt;
            }
          }
        }
      }
    }
    phase_stamp(a.clk, 3, first_cta && tid == 0);
    if (route_cta) {
      if (warp == 0) {
        const bool topk = lane < n_groups && s_gact[lane] == MIX_SAE_TOPK;
        write_route(a, my_total, lane < n_groups ? s_gtiles[lane] : 0, topk, mt_incl - my_mt, n_mtiles, s_total[n_groups], lane);
      } else {
        for (int m0 = (warp - 1) * 32; m0 < a.panel_cap / kTileM; m0 += (kFrontWarps - 1) * 32) {
          const int m = m0 + lane;
          int g = -1;
          for (int q = 0; q < n_groups; ++q) {         // (whole warps: the shuffles)
            const int first = __shfl_sync(0xffffffffu, mt_incl - my_mt, q), n = __shfl_sync(0xffffffffu, my_mt, q);
            if (m >= first && m < first + n) g = q;
          }
          if (m < a.panel_cap / kTileM) {
            a.mtile_group[m] = g;
            if (a.mtile_flag) a.mtile_flag[m] = 0;
          }
        }
      }
    }
    // this CTA's panel rows, one per warp
    if (p < a.panel_cap) {
      if (p < n_panel_rows) {
        if (a.tau_slots && t >= 0) {                     // the encode's TopK bound starts empty
          reinterpret_cast<uint4*>(a.tau_slots + (size_t)p * kTauSlots)[lane] = make_uint4(0u, 0u, 0u, 0u);
          if (lane == 0) a.tau_min[p] = 0u;
        }
        if (kPack == 0)
          pack_row_bf16(a.hidden, t, static_cast<__nv_bfloat16*>(a.panel), (size_t)p, a.d, lane);
        else
          pack_row_e4m3<kPack == 1>(a.hidden, t, static_cast<unsigned char*>(a.panel), a.act_scale, (size_t)p, a.d, a.lo_row0, lane);
      }
      if (lane == 0) {
        RowRec rec;
        const int g = (meta & 0xff) - 1;
        rec.t = t;
        rec.slot = t >= 0 ? slot : -1;
        rec.n_edit = (meta >> 8) & 0xff;
        rec.group_flags = t >= 0 ? (g | ((meta >> 16) & 1 ? kRecAddError : 0) | (s_gact[g] << kRecActShift)) : 0;
        rec.W_dec = t >= 0 ? s_gwdec[g] : nullptr;
        rec.theta = t >= 0 ? s_gtheta[g] : nullptr;
        a.row_rec[p] = rec;
        a.panel_row[p] = t;
        if (a.row_flag) a.row_flag[p] = 0;
      }
    }
  } else if (tid == 0) {
    atomicOr(a.status, MIX_STATUS_WAIT_TIMEOUT);
  }
  phase_stamp(a.clk, 4, first_cta && tid == 0);
  // Only now may the encode's CTAs be scheduled (where it is launched programmatically): they take most of an SM's
  // registers and shared memory, and resident any earlier they would crowd out the CTAs that still have rows to pack.
  pdl_launch_dependents();
  // the last CTA to leave closes the call: both counters are zero again when the next launch starts
  if (!local) {
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      if (atomicAdd(a.sync + 1, 1) == a.n_front - 1) {
        a.sync[0] = 0;
        a.sync[1] = 0;
      }
    }
  }
}

}  // namespace

int front_chunks(int T_max) { return (T_max + kFrontThreads - 1) / kFrontThreads; }

cudaError_t launch_front(const Ctx* c, __nv_bfloat16* hidden, int T, cudaStream_t s, bool pdl, unsigned long long cond, int use_cond,
                         const HookRows* rows) {
  FrontArgs a;
  a.token_slot = c->d_token_slot;
  a.T = T;
  a.apps = c->d_apps;
  a.gates = c->d_gates;
  a.n_slots = c->cfg.n_slots_max;
  a.groups = c->d_groups;
  a.n_groups = c->cfg.n_groups_max;
  a.chain_next = c->d_chain_next;
  a.edit_only = (c->cfg.flags & MIX_FLAG_SAE_EDIT_ONLY) ? 1 : 0;
  a.row_meta = c->d_row_meta;
  a.counts = c->d_front_counts;
  a.sync = c->d_front_sync;
  a.panel_row = c->d_panel_row;
  a.row_rec = c->d_row_rec;
  a.panel_cap = c->panel_rows_cap;
  a.mtile_group = c->d_mtile_group;
  a.rs = c->d_route;
  a.status = c->d_status;
  a.row_flag = c->d_row_flag;
  a.mtile_flag = c->d_mtile_flag;
  a.n_flagged = c->d_n_flagged;
  a.cond = static_cast<cudaGraphConditionalHandle>(cond);
  a.use_cond = use_cond;
  a.hidden = hidden;
  a.panel = c->d_panel;
  a.act_scale = c->d_act_scale;
  a.d = c->cfg.d_model;
  a.tau_slots = c->d_tau;
  a.tau_min = c->d_tau_min;
  a.lo_row0 = c->panel_rows_cap;
  a.clk = c->d_phase_clk;
  a.n_sms = c->n_sms;
  a.cand_tiles = c->cand_tiles;
  a.pair_mode = ((c->cfg.flags & MIX_FLAG_ENCODE_SIMT) || !encode_pair_possible(c)) ? 0 : encode_pair_mode(-1);
  const int chunks = front_chunks(T);
  const size_t smem = (size_t)front_chunks(c->cfg.T_max) * (c->cfg.n_groups_max + 1) * sizeof(int);
  const int pack_ctas = (c->panel_rows_cap + kFrontWarps - 1) / kFrontWarps;
  a.n_front = chunks > pack_ctas ? chunks : pack_ctas;
  a.rows = hidden;
  a.scores = rows ? rows->scores : nullptr;
  a.C_max = c->cfg.C_max;
  a.vec_arena = reinterpret_cast<const uint4*>(c->d_vec_arena);
  a.pdl = rows ? rows->pdl : 0;
  const dim3 grid(a.n_front + (rows ? c->cfg.T_max : 0));
  const int which = !pdl ? 0 : (rows ? kPdlHook : kPdlPack);
  auto with = [&](auto pack) -> cudaError_t {
    constexpr int kPack = decltype(pack)::value;
    auto run = [&](auto kernel) { return launch_pdl(which, kernel, grid, dim3(kFrontThreads), smem, s, a); };
    if (!rows) return run(front_kernel<kPack, 0>);
    switch ((c->cfg.d_model / 8 + kFrontThreads - 1) / kFrontThreads) {
      case 1: return run(front_kernel<kPack, 1>);
      case 2: return run(front_kernel<kPack, 2>);
      case 3: return run(front_kernel<kPack, 3>);
      default: return run(front_kernel<kPack, kMostVec>);
    }
  };
  if (c->cfg.flags & MIX_FLAG_FP8_ACT) return with(std::integral_constant<int, 2>());
  // (MIX_FLAG_FP8_W_ENC alone: hi codes in rows [0, P), lo codes in rows [P, 2P) of the same buffer)
  if (c->cfg.flags & MIX_FLAG_FP8_W_ENC) return with(std::integral_constant<int, 1>());
  return with(std::integral_constant<int, 0>());
}

}  // namespace mix
