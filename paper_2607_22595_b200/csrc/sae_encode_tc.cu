// SAE encode on the 5th-generation tensor cores (sm_100a only).
//
//   Z[p, j] = sum_i panel[p, i] * W_enc[j, i] + b_eff[j]        bf16 x bf16 -> fp32
//
// One persistent CTA per SM walks a device-built tile schedule (group, feature tile, row tile).
// Warp roles:  warp 0 and the last two = TMA producers, each with every third k-block (panel tile 128x64 and W_enc tile 256x64
// -- or 128x64, 64x64 where a call has few tiles -- into a ring of 128-byte-swizzled shared memory: TcCfg::kStages of
// full-width tiles, up to kMaxStages of narrower ones), warp 1 = MMA issuer (tcgen05.mma 128x256x16, fp32 accumulators in tensor
// memory, double buffered so the epilogue of one tile overlaps the main loop of the next), warps 2..9 = epilogue, two per
// tensor-memory lane quarter with 128 columns of the tile each (tcgen05.ld, + bias, which came with the tile
// -- then either the fp32 pre-activations to the Z
// scratch, or -- for TopK weight sets -- only the tile's 8 largest values per row plus its 9th, which the tail
// kernel turns into the exact TopK; the two warps of a quarter put their lists together through shared memory).
// Producers and issuer run their loops as whole warps and elect a lane for the instructions (elect_one says why).
// A second form (kPair) runs on clusters of two CTAs that share a 256-row tile through
// tcgen05.mma.cta_group::2; which form works on a call is decided on the device (see TcCfg).
// No TMA multicast in either form.  Every wait is bounded: on expiry the CTA raises
// MIX_STATUS_WAIT_TIMEOUT, lets its copies land, frees its tensor memory and returns.
//
// 8-bit encoder (kEnc != 0): W_enc is E4M3 codes with one fp32 scale per feature, and the contraction is
// tcgen05.mma kind::f8f6f4 (both operands E4M3), 128 x 256 x 32 per instruction.  A k-block is 128 elements
// (the same 128-byte swizzled rows: 16 KiB of panel, 32 KiB of W_enc, four instructions), so the kernel is the
// bf16 kernel with half as many k-blocks; the epilogue multiplies the accumulator by row scale x feature scale.
//   kEnc == 2 (8-bit input): the panel holds the row quantised to E4M3 with a power-of-two scale.
//   kEnc == 1 (the hidden state stays bf16): the pack step split each row EXACTLY (down to 2^-10 of the scale)
//     into two E4M3 operands hi + lo with one common power-of-two scale; a stage carries both panel tiles
//     (16 + 16 + 32 KiB, three stages) and the eight instructions of a k-block accumulate hi W and lo W into
//     the same accumulator.  Per element of K that is the tensor time of the bf16 kernel with half the W_enc
//     bytes: as fast as kEnc == 2 where the stream of W_enc is the bound, as fast as bf16 where the tensor
//     pipe is.
#include <stdlib.h>

#include "mix_internal.h"
#include "tc_common.cuh"

namespace mix {

namespace {

constexpr int kMaxStages = 16;
constexpr int kABytes = kTileM * kTileK * 2;   // 16 KiB: 128 rows of 128 bytes
constexpr int kBBytes = kTileN * kTileK * 2;   // 32 KiB: 256 rows of 128 bytes
constexpr int kCopyWarps = 3;                   // producers, each with every third k-block
constexpr int kSharedBytes = 1280;               // room for TcShared
constexpr int kVecs = 4;                        // tiles whose bias and scale are in shared memory
// An epilogue warp's list of a TopK tile: up to 8 values a row and a place for what is one too many, [entry][lane], then their
// columns.  The lists that are handed over are followed by three words a row: 9th value, number of entries, bound.
constexpr int kListRows = kCandPerTile + 1, kListBytes = kListRows * 32 * 5, kXchgListBytes = kListBytes + 3 * 32 * 4;
// kEnc: 0 = bf16 encoder and input; 1 = 8-bit encoder, bf16 input as two E4M3 operands; 2 = 8-bit encoder and 8-bit input
// kPair: two CTAs (a cluster) share one 256-row x 256-feature tile: each loads its own 128 panel rows and HALF of the
//        W_enc tile, and one tcgen05.mma.cta_group::2 instruction feeds both SMs' tensor cores -- a third less
//        shared-memory fill per SM and flop than a CTA working alone (32 instead of 48 KiB per k-block).
template <int kEnc, int kEpi, bool kPair> struct TcCfg {
  static_assert(kEpi == 4 || kEpi == 8, "epilogue warps");
  static constexpr bool kSplit = kEnc == 1;            // two panel tiles (hi, lo) per stage
  static constexpr int kBBytesCta = kPair ? kBBytes / 2 : kBBytes;
  static constexpr int kARingBytes = (kSplit ? 2 : 1) * kABytes;      // a stage's panel rows
  static constexpr int kStageBytes = kARingBytes + kBBytesCta;        // (of a full-width tile; narrower tiles leave room for more stages)
  static constexpr int kStages = kPair ? (kSplit ? 4 : 6) : (kSplit ? 3 : 4);
  static constexpr int kRingBytes = kStages * kStageBytes;
  static_assert(kStages >= kCopyWarps, "the producers' turns");
  // epilogue warps: 4 (one per tensor-memory lane quarter, all 256 columns) or 8 (two per quarter, 128 columns
  // each; the two top-9 lists of a row meet in shared memory).  One warp per scheduler runs the epilogue's
  // dependent compare/select chains at a fraction of the issue rate; two interleave.
  static constexpr int kEpiWarps = kEpi;
  static constexpr int kXchgBytes = kEpiWarps == 8 ? 2 * 4 * kXchgListBytes : 0;   // [acc][quarter]: the upper-half warps' lists
  static constexpr int kThreads = (kCopyWarps + 1 + kEpiWarps) * 32;      // (and the issuer)
  // The bias (and, for codes, the feature scale) of a tile's columns comes with the tile: the producer copies it into one of
  // kVecs places.  bf16 kernels keep the thresholds of each epilogue warp's columns behind them.
  static constexpr int kVecBytes = (kEnc != 0 ? 2 : 1) * kTileN * 4;
  static constexpr int kEpiVecBytes = 2 * 4 * kTileN * 4;
  static_assert(kVecs * kVecBytes + (kEnc == 0 ? 4 * kTileN * 4 : 0) <= kEpiVecBytes, "the tiles' vectors");
  static constexpr int kPickBytes = kEpiWarps == 8 ? 4 * kListBytes : 0;                 // the lower-half warps' lists
  static constexpr int kSmemBytes = kRingBytes + 1024 /* alignment slack */ + kSharedBytes + kXchgBytes + kEpiVecBytes + kPickBytes;
  static_assert(kSmemBytes <= 227 * 1024, "shared memory per CTA");
};
constexpr int kTmemCols = 512;                 // two 128 x 256 fp32 accumulators
constexpr long long kWaitCycles = 4000000000ll;   // ~2 s at 2 GHz
constexpr long long kWaitCyclesTest = 2000000ll;  // ~1 ms: the cap under MIX_FLAG_TEST_STALL_ENCODE

struct __align__(8) TcShared {
  unsigned long long full[kMaxStages];      // (a pair's leader: filled by both CTAs' copies)
  unsigned long long empty[kMaxStages];
  unsigned long long tmem_full[2];
  unsigned long long tmem_empty[2];
  unsigned long long vec_full[kVecs], vec_empty[kVecs];   // a tile's bias and scale
  unsigned long long top_full[2][4];      // [half][quarter]: that warp's 8 largest values are where the other one looks for them
  unsigned long long xchg_full[2][4];     // 8 epilogue warps: the upper-half warp's list of (accumulator, quarter) is in shared memory
  unsigned tmem_base;
  volatile int abort_flag;
  long long wait_cycles;      // cap of every bounded wait in this launch
  RouteState rs;
  // The weight sets of this call that are THIS kernel's (single CTAs or pairs, as the front kernel dealt them; all
  // of them in the pass over flagged row tiles), numbered through: first unit -- a 128-row tile, or a pair of
  // them -- and first tile of each set, totals in entry [n_groups]; sets of the other kernel have no units here
  short unit0[kMaxGroups + 1];
  int utile0[kMaxGroups + 1];
};
static_assert(sizeof(TcShared) <= kSharedBytes, "TcShared must fit the space reserved for it");

using namespace tc;

// Bounded wait on this kernel's shared state.
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, TcShared* sh, unsigned* status) {
  return mbar_wait_bounded(bar, parity, &sh->abort_flag, &sh->wait_cycles, status);
}

__device__ __forceinline__ bool mbar_wait_warp(unsigned bar, unsigned parity, TcShared* sh, unsigned* status) {
  return mbar_wait_bounded_warp(bar, parity, &sh->abort_flag, &sh->wait_cycles, status);
}

constexpr unsigned kIdescPair = idesc_f16(2 * kTileM, kTileN);     // the pair's instruction: M = 256
constexpr unsigned kIdescE4Pair = idesc_e4m3(2 * kTileM, kTileN);

struct Tile {
  int group, n_tile, m_tile_global, rows_valid;      // n_tile: in tiles of this call's width
  int m_tile_peer;      // CTA pairs: the row tile the other CTA of the pair works on (the same one when the weight set has an odd tile left over)
};

// Number of feature tiles per unit if it is the same for every weight set of this kernel that has rows (the
// usual case: one SAE width per context), else 0.
__device__ __forceinline__ int uniform_feature_tiles(const TcShared& sh, int n_groups) {
  int nt = -1;
  for (int g = 0; g < n_groups; ++g) {
    const int units = sh.unit0[g + 1] - sh.unit0[g];
    if (units == 0) continue;
    const int nt_g = (sh.utile0[g + 1] - sh.utile0[g]) / units;
    if (nt >= 0 && nt_g != nt) return 0;
    nt = nt_g;
  }
  return nt > 0 ? nt : 0;
}

// Linear tile id of this kernel -> (weight set, feature tile, unit of the set) and, for the CTA of rank `rank` of a
// pair, its own row tile.  With one SAE width the order is feature tile by feature tile over ALL units, so every
// row sees its first feature tiles finished early in the launch (the TopK epilogue's running bound needs that);
// otherwise weight set by weight set.  A weight set with an odd number of row tiles leaves its last pair half
// empty: the CTA without a tile of its own repeats the other one's loads and keeps nothing (rows_valid = 0).
template <bool kPair>
__device__ __forceinline__ Tile decode_tile(const TcShared& sh, int n_groups, int tile, int uniform_nt, int rank) {
  const RouteState& rs = sh.rs;
  Tile t;
  int g = 0, ul;
  if (uniform_nt > 0) {
    const int n_units = sh.unit0[n_groups];
    t.n_tile = tile / n_units;
    const int u = tile - t.n_tile * n_units;
    while (g + 1 < n_groups && u >= sh.unit0[g + 1]) ++g;
    ul = u - sh.unit0[g];
  } else {
    while (g + 1 < n_groups && tile >= sh.utile0[g + 1]) ++g;
    const int local = tile - sh.utile0[g];
    const int units = sh.unit0[g + 1] - sh.unit0[g];
    t.n_tile = local / units;
    ul = local - t.n_tile * units;
  }
  t.group = g;
  if (kPair) {
    const int mt = rs.group_mtile0[g + 1] - rs.group_mtile0[g];
    const int m_own = 2 * ul + rank, m_peer = 2 * ul + (1 - rank);
    t.m_tile_global = rs.group_mtile0[g] + min(m_own, mt - 1);
    t.m_tile_peer = rs.group_mtile0[g] + min(m_peer, mt - 1);
    t.rows_valid = m_own < mt ? min(kTileM, rs.group_count[g] - m_own * kTileM) : 0;
  } else {
    t.m_tile_global = rs.group_mtile0[g] + ul;
    t.m_tile_peer = t.m_tile_global;
    t.rows_valid = min(kTileM, rs.group_count[g] - ul * kTileM);
  }
  return t;
}

// mode 0: every tile; TopK weight sets emit candidates, the others write Z.
// mode 1: only row tiles flagged by the tail kernel (TopK sets), written to Z for the exact
//         fallback selection; returns at once when nothing is flagged.
__device__ __forceinline__ bool tile_wanted(const Tile& t, const GroupEntry* __restrict__ groups, int mode,
                                            const int* __restrict__ mtile_flag) {
  if (mode == 0) return true;
  return groups[t.group].act == MIX_SAE_TOPK && (mtile_flag[t.m_tile_global] | mtile_flag[t.m_tile_peer]) != 0;   // same answer in both CTAs of a pair
}

// Insert (x, c) into the descending list tv[0..8] if it beats the 9th entry.  Equal values keep
// the earlier (lower) column in front, which is the tie rule of the selection: the new element goes
// in front of the first entry it strictly beats, and everything from there on moves down one place.
__device__ __forceinline__ void top9_insert(float (&tv)[kCandPerTile + 1], int (&ti)[kCandPerTile + 1], float x, int c) {
  if (!(x > tv[kCandPerTile])) return;
  bool moving = false;
#pragma unroll
  for (int s = 0; s <= kCandPerTile; ++s) {
    moving = moving || x > tv[s];
    const float t = tv[s];
    const int u = ti[s];
    tv[s] = moving ? x : t;
    ti[s] = moving ? c : u;
    x = moving ? t : x;
    c = moving ? u : c;
  }
}

// Compare-exchange, larger value first; an 8-element sort (19 of them), and the merge of a bitonic sequence of 8 (12).
__device__ __forceinline__ void cmpx(float& a, float& b) {
  const float hi = fmaxf(a, b);
  b = fminf(a, b);
  a = hi;
}
__device__ __forceinline__ void sort8_desc(float (&b)[8]) {
  cmpx(b[0], b[1]); cmpx(b[2], b[3]); cmpx(b[4], b[5]); cmpx(b[6], b[7]);
  cmpx(b[0], b[2]); cmpx(b[1], b[3]); cmpx(b[4], b[6]); cmpx(b[5], b[7]);
  cmpx(b[1], b[2]); cmpx(b[5], b[6]);
  cmpx(b[0], b[4]); cmpx(b[1], b[5]); cmpx(b[2], b[6]); cmpx(b[3], b[7]);
  cmpx(b[2], b[4]); cmpx(b[3], b[5]);
  cmpx(b[1], b[2]); cmpx(b[3], b[4]); cmpx(b[5], b[6]);
}
__device__ __forceinline__ void merge8_desc(float (&b)[8]) {
  cmpx(b[0], b[4]); cmpx(b[1], b[5]); cmpx(b[2], b[6]); cmpx(b[3], b[7]);
  cmpx(b[0], b[2]); cmpx(b[1], b[3]); cmpx(b[4], b[6]); cmpx(b[5], b[7]);
  cmpx(b[0], b[1]); cmpx(b[2], b[3]); cmpx(b[4], b[5]); cmpx(b[6], b[7]);
}

// The same on (value, column) pairs: the larger value first, of equal ones the lower column.
__device__ __forceinline__ void cmpx(float& a, int& ca, float& b, int& cb) {
  const bool swap = b > a || (b == a && cb < ca);
  const float x = swap ? b : a, y = swap ? a : b;
  const int cx = swap ? cb : ca, cy = swap ? ca : cb;
  a = x; b = y; ca = cx; cb = cy;
}
#define MIX_CX(i, j) cmpx(v[i], c[i], v[j], c[j])
__device__ __forceinline__ void sort8_pairs(float (&v)[kCandPerTile + 1], int (&c)[kCandPerTile + 1]) {
  MIX_CX(0, 1); MIX_CX(2, 3); MIX_CX(4, 5); MIX_CX(6, 7);
  MIX_CX(0, 2); MIX_CX(1, 3); MIX_CX(4, 6); MIX_CX(5, 7);
  MIX_CX(1, 2); MIX_CX(5, 6);
  MIX_CX(0, 4); MIX_CX(1, 5); MIX_CX(2, 6); MIX_CX(3, 7);
  MIX_CX(2, 4); MIX_CX(3, 5);
  MIX_CX(1, 2); MIX_CX(3, 4); MIX_CX(5, 6);
}
// Merges a second sorted list of 9 (columns all higher) into the first: the 8 largest of both, sorted, and the 9th value.
template <class Get>
__device__ __forceinline__ void merge_lists(float (&v)[kCandPerTile + 1], int (&c)[kCandPerTile + 1], float ninth2, Get&& second) {
  float ninth = fmaxf(v[kCandPerTile], ninth2);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float x;
    int cx;
    second(7 - i, x, cx);
    ninth = fmaxf(ninth, fminf(v[i], x));
    c[i] = x > v[i] ? cx : c[i];
    v[i] = fmaxf(v[i], x);
  }
  MIX_CX(0, 4); MIX_CX(1, 5); MIX_CX(2, 6); MIX_CX(3, 7);
  MIX_CX(0, 2); MIX_CX(1, 3); MIX_CX(4, 6); MIX_CX(5, 7);
  MIX_CX(0, 1); MIX_CX(2, 3); MIX_CX(4, 5); MIX_CX(6, 7);
  v[kCandPerTile] = ninth;
}
#undef MIX_CX

template <int kEnc, int kEpi, bool kPair>
__global__ void __launch_bounds__(TcCfg<kEnc, kEpi, kPair>::kThreads, 1)
encode_tc_kernel(const __grid_constant__ PanelMaps tmap_panel, const __grid_constant__ CUtensorMap tmap_w_one, const CUtensorMap* __restrict__ tmap_w, const RouteState* __restrict__ rs_g, const GroupEntry* __restrict__ groups, int n_groups,
                 float* __restrict__ Z, long long ldz, int d, unsigned* __restrict__ status, int mode,
                 const int* __restrict__ mtile_flag, const int* __restrict__ n_flagged, float* __restrict__ cand_val,
                 int* __restrict__ cand_idx, float* __restrict__ cand_ninth, int cand_tiles, int w_tiled, int test_stall,
                 const float* __restrict__ act_scale, unsigned* __restrict__ tau_slots, unsigned* __restrict__ tau_min,
                 int lo_row0, const RowRec* __restrict__ row_rec, const int* __restrict__ edit_idx, int r_max, int all_z,
                 unsigned long long* __restrict__ clk) {
  constexpr bool kE4 = kEnc != 0;                      // E4M3 x E4M3 contraction
  constexpr bool kSplit = kEnc == 1;                   // the panel row is hi + lo: two operand tiles per k-block
  constexpr int kBlockK = kE4 ? 2 * kTileK : kTileK;   // elements per 128-byte row of either operand
  using Cfg = TcCfg<kEnc, kEpi, kPair>;
  constexpr int kTcThreads = Cfg::kThreads;
  constexpr int kEpiWarps = Cfg::kEpiWarps;
  constexpr int kEpiColsMax = kTileN / (kEpiWarps / 4);
  extern __shared__ unsigned char smem_raw[];
  // 1024-byte alignment: required by the 128-byte swizzle atoms
  unsigned char* tiles = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  TcShared* sh = reinterpret_cast<TcShared*>(tiles + Cfg::kRingBytes);
  unsigned char* xchg = reinterpret_cast<unsigned char*>(sh) + kSharedBytes;
  float* epi_vec = reinterpret_cast<float*>(xchg + Cfg::kXchgBytes);
  unsigned char* pick = reinterpret_cast<unsigned char*>(epi_vec) + Cfg::kEpiVecBytes;
  const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  // CTA pairs: rank 0 leads (it issues the pair's tensor-core instructions and owns the barriers both CTAs' copies
  // complete on); `worker` numbers the units that walk the tile list -- pairs, or single CTAs
  const int rank = kPair ? (int)cluster_ctarank() : 0;
  const bool leader = rank == 0;
  const int worker = kPair ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
  const int n_workers = kPair ? (int)(gridDim.x >> 1) : (int)gridDim.x;

  // what does not depend on the routing is done before the wait
  if (threadIdx.x == 0) {
    for (int s = 0; s < kMaxStages; ++s) {
      mbar_init(smem_u32(&sh->full[s]), 1);
      mbar_init(smem_u32(&sh->empty[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&sh->tmem_full[a]), 1);
      mbar_init(smem_u32(&sh->tmem_empty[a]), kPair ? 2 * kEpiWarps : kEpiWarps);   // a pair's leader hears from both CTAs' epilogues
      for (int q = 0; q < 4; ++q) {
        mbar_init(smem_u32(&sh->xchg_full[a][q]), 1);
        mbar_init(smem_u32(&sh->top_full[a][q]), 1);
      }
    }
    for (int v = 0; v < kVecs; ++v) {
      mbar_init(smem_u32(&sh->vec_full[v]), 1);
      mbar_init(smem_u32(&sh->vec_empty[v]), kEpiWarps);
    }
    sh->abort_flag = 0;
    sh->wait_cycles = test_stall ? kWaitCyclesTest : kWaitCycles;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  pdl_wait();
  pdl_launch_dependents();
  const bool stamp = clk != nullptr && blockIdx.x == 0 && threadIdx.x == 0 && mode == 0 && !kPair;
  phase_stamp(clk, 26, stamp);
  if (mode == 1 && *n_flagged == 0) return;
  for (int i = threadIdx.x; i < (int)(sizeof(RouteState) / sizeof(int)); i += kTcThreads)
    reinterpret_cast<int*>(&sh->rs)[i] = reinterpret_cast<const int*>(rs_g)[i];
  __syncthreads();
  // Feature width of this call's tiles: 256, or 128 / 64 where full-width tiles would leave half of the SMs or more without
  // one (decided by the front kernel).  A narrower tile makes a shorter stage, so the ring holds more of them.
  const int tile_n = kPair ? kTileN : uniform(sh->rs.tile_n);
  const int n_sub = kTileN / tile_n;                   // tiles per 256 features
  const int epi_cols = tile_n / (kEpiWarps / 4);       // columns of a tile per epilogue warp
  if (warp < 2) {
    // this kernel's weight sets (lane g: set g): units (row tiles, or pairs of them) and tiles, numbered through.  The full
    // pass has two kernels, single CTAs and CTA pairs, and the front kernel dealt this call's weight sets between them.
    static_assert(kMaxGroups == 32, "a lane per weight set");
    const int mt = lane < n_groups ? sh->rs.group_mtile0[lane + 1] - sh->rs.group_mtile0[lane] : 0;
    const int nt = mt > 0 ? (sh->rs.group_tile0[lane + 1] - sh->rs.group_tile0[lane]) / mt * n_sub : 0;
    const bool mine = mode != 0 || (((sh->rs.pair_mask >> lane) & 1) != 0) == kPair;
    const int units = !mine ? 0 : (kPair ? (mt + 1) / 2 : mt);
    if (warp == 0) {
      int nu = units, ut = units * nt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, nu, o), z = __shfl_up_sync(0xffffffffu, ut, o);
        if (lane >= o) {
          nu += y;
          ut += z;
        }
      }
      sh->unit0[lane + 1] = (short)nu;
      sh->utile0[lane + 1] = ut;
      if (lane == 0) {
        sh->unit0[0] = 0;
        sh->utile0[0] = 0;
      }
    } else if (__any_sync(0xffffffffu, units * nt != 0)) {     // (nothing for this kernel: no tensor memory is taken)
      if (kPair) tmem_alloc_pair(smem_u32(&sh->tmem_base), kTmemCols);
      else tmem_alloc(smem_u32(&sh->tmem_base), kTmemCols);
    }
  }
  tc_fence_before();
  __syncthreads();
  const int total_tiles = uniform(sh->utile0[n_groups]);
  if (total_tiles == 0) return;            // (both CTAs of a pair see the same)
  if (kPair) cluster_sync_all();           // the peer's barriers are initialised before anything is sent to them
  tc_fence_after();
  const unsigned tmem_base = (unsigned)uniform((int)sh->tmem_base);
  phase_stamp(clk, 27, stamp);
  // (the interleaved order serves the TopK epilogue's running bound; without TopK rows the plain order is a little faster)
  const int uniform_nt = sh->rs.n_topk_rows > 0 ? uniform_feature_tiles(*sh, n_groups) : 0;
  const int num_kb = d / kBlockK;
  auto tile_of = [&](int tile) { return decode_tile<kPair>(*sh, n_groups, tile, uniform_nt, rank); };
  // The ring.  Where tiles are narrow a CTA has one at most, and its stages hold the panel rows which that one has: smaller
  // stages, hence more of them, and of the stream of W_enc, which bounds such a call, more is under way (what a tile's
  // instructions read behind those rows is the stage's own W_enc or the next stage, and the accumulator's rows that come of it
  // nobody reads; all of it lies inside the CTA's shared memory).
  int box = kPanelBoxes - 1;                           // panel box: panel_box_rows(box) rows
  if (!kPair && n_sub > 1 && worker < total_tiles) {
    const int rows = uniform(tile_of(worker).rows_valid);
    while (box > 0 && panel_box_rows(box - 1) >= rows) --box;
  }
  const int a_bytes = panel_box_rows(box) * (kTileK * 2), a_ring = (kSplit ? 2 : 1) * a_bytes;
  const int stage_bytes = a_ring + (kPair ? Cfg::kBBytesCta : tile_n * (kTileK * 2));
  const int n_stages = min(kMaxStages, Cfg::kRingBytes / stage_bytes);

  if (warp == 0 || warp >= 2 + kEpiWarps) {
    // The producers, warp 0 and the last ones, take the k-blocks in turn.  What a k-block costs one warp is the latency of the
    // forty instructions around its two copies, 400 cycles, whatever the copies bring; one warp for all of them bounded the
    // calls with a narrow tile per SM (91 rows, d = 4096, 8192 features: 64 k-blocks in 15.8 us, 12.7 so; 9 rows 15.8 and 11.5).
    // Turns go on through the tiles: a warp's next k-block is always kCopyWarps further, so that when it looks at a stage of the
    // ring, which is at least as long, the k-block two rounds before is known to have been consumed -- the parity that it waits
    // for means one thing only.
    int first = warp == 0 ? 0 : warp - (1 + kEpiWarps);        // this warp's first k-block of the tile
    int stage0 = 0, vec = 0;                                   // stage and phase of the tile's first k-block
    unsigned phase0 = 0, vec_phase = 0;
    bool ok = true;
    const unsigned long long stream = l2_evict_first();
    for (int tile = worker; tile < total_tiles && ok; tile += n_workers) {
      const Tile t = tile_of(tile);
      if (!tile_wanted(t, groups, mode, mtile_flag)) continue;
      const int group = uniform(t.group), n_tile = uniform(t.n_tile), row0 = uniform(t.m_tile_global) * kTileM;
      const CUtensorMap* tp = &tmap_panel.box[box];
      // (boxes of as many W_enc rows as this kernel's tile has: a map array per width)
      // (no array: a single weight set whose map came with the launch, at the width the front kernel arrives at too)
      const CUtensorMap* tw = tmap_w == nullptr ? &tmap_w_one : tmap_w + (kPair || n_sub == 2 ? n_groups : (n_sub == 4 ? 2 * n_groups : 0)) + group;
      const int n256 = n_tile / n_sub, row_in_256 = kPair ? rank * (kTileN / 2) : (n_tile - n256 * n_sub) * tile_n;
      // A W_enc tile that one worker alone reads goes through L2 as the first to be evicted: otherwise the stream leaves
      // nothing of what the short kernels around it live on -- their code, the tables, the rows -- and each of them starts
      // with a chain of DRAM round trips (91 rows, d = 4096, 16384 features: front 12.3 -> 8.5 us, tail 19.4 -> 15.6).
      // Tiles that several row tiles share must stay (the mixed batch's encode 441 -> 480 us with the hint).
      const bool once = uniform(sh->unit0[group + 1] - sh->unit0[group]) == 1;
      // W_enc tile: rows n_tile * tile_n .. of the row-major matrix, or -- when the weights were re-laid out at
      // registration (always, for codes) -- rows of block (n256, kb) of the tile-contiguous copy
      // [S/256][d/kBlockK][256][kBlockK]
      const bool w_blocks = kE4 || w_tiled;
      const int wy0 = (w_blocks ? n256 * num_kb : n256) * kTileN + row_in_256;
      int stage = stage0 + first;
      unsigned phase = phase0;
      while (stage >= n_stages) { stage -= n_stages; phase ^= 1u; }
      unsigned ready = 0u;                                     // the present stage is free, as of one k-block ago
      for (int kb = first; kb < num_kb; kb += kCopyWarps) {
        if (!__all_sync(0xffffffffu, ready) && !mbar_wait_warp(smem_u32(&sh->empty[stage]), phase ^ 1u, sh, status)) { ok = false; break; }
        // Test hook (MIX_FLAG_TEST_STALL_ENCODE): the producers never fill a stage, so the consumer's
        // bounded wait runs out and the whole CTA leaves through the time-out path.
        if (test_stall) { ok = false; break; }
        int next = stage + kCopyWarps;
        unsigned next_phase = phase;
        if (next >= n_stages) { next -= n_stages; next_phase ^= 1u; }      // (n_stages >= kCopyWarps)
        ready = mbar_test(smem_u32(&sh->empty[next]), next_phase ^ 1u);
        const unsigned bar = smem_u32(&sh->full[stage]), sa = smem_u32(tiles + stage * stage_bytes), sw = sa + a_ring, on = elect_one();
        const int wx = w_blocks ? 0 : kb * kTileK, wy = w_blocks ? wy0 + kb * kTileN : wy0;
        if (kPair) {
          // both CTAs' copies complete on the LEADER's barrier, which expects the bytes of both; this CTA
          // fetches its own 128 panel rows and its half (128 features) of the W_enc tile
          if (leader) mbar_expect_tx(bar, 2 * stage_bytes, on);
          const unsigned bar_c = mapa_cluster(bar, 0);
          tma_load_2d_pair(sa, tp, kb * kBlockK, row0, bar_c, on);
          if (kSplit) tma_load_2d_pair(sa + a_bytes, tp, kb * kBlockK, lo_row0 + row0, bar_c, on);
          if (once) tma_load_2d_pair_hint(sw, tw, wx, wy, bar_c, stream, on);
          else tma_load_2d_pair(sw, tw, wx, wy, bar_c, on);
        } else {
          mbar_expect_tx(bar, stage_bytes, on);
          tma_load_2d(sa, tp, kb * kBlockK, row0, bar, on);
          if (kSplit) tma_load_2d(sa + a_bytes, tp, kb * kBlockK, lo_row0 + row0, bar, on);   // the lo codes
          if (once) tma_load_2d_hint(sw, tw, wx, wy, bar, stream, on);
          else tma_load_2d(sw, tw, wx, wy, bar, on);
        }
        stage = next;
        phase = next_phase;
      }
      if (warp == 0 && ok) {               // the tile's bias and scale, which nothing waits for before its end
        if (!mbar_wait_warp(smem_u32(&sh->vec_empty[vec]), vec_phase ^ 1u, sh, status)) break;
        const unsigned bar = smem_u32(&sh->vec_full[vec]), dst = smem_u32(epi_vec) + vec * Cfg::kVecBytes;
        const float* b_eff = groups[group].b_eff + (size_t)n_tile * tile_n;
        const float* w_scale = groups[group].w_scale + (size_t)n_tile * tile_n;
        if (elect_one()) {
          mbar_expect_tx(bar, (kE4 ? 2 : 1) * tile_n * 4);
          bulk_load(dst, b_eff, tile_n * 4, bar);
          if (kE4) bulk_load(dst + kTileN * 4, w_scale, tile_n * 4, bar);
        }
        if (++vec == kVecs) { vec = 0; vec_phase ^= 1u; }
      }
      first = (first + kCopyWarps - num_kb % kCopyWarps) % kCopyWarps;
      const int laps = (stage0 + num_kb) / n_stages;
      stage0 += num_kb - laps * n_stages;
      phase0 ^= (unsigned)(laps & 1);
    }
    if (warp == 0) phase_stamp(clk, 28, stamp);          // the last copy of this CTA has been issued (if it is this warp's)
  } else if (warp == 1) {
    if (leader) {
      const unsigned idesc = kE4 ? idesc_e4m3(kTileM, tile_n) : idesc_f16(kTileM, tile_n);   // D fp32, operands K-major
      int stage = 0;
      unsigned phase = 0, acc = 0, acc_phase = 0, ready = 0u;
      bool ok = true;
      for (int tile = worker; tile < total_tiles && ok; tile += n_workers) {
        if (mode != 0 && !tile_wanted(tile_of(tile), groups, mode, mtile_flag)) continue;
        if (!mbar_wait_warp(smem_u32(&sh->tmem_empty[acc]), acc_phase ^ 1u, sh, status)) break;
        tc_fence_after();
        const unsigned d_tmem = tmem_base + acc * kTileN;
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!__all_sync(0xffffffffu, ready) && !mbar_wait_warp(smem_u32(&sh->full[stage]), phase, sh, status)) { ok = false; break; }
          tc_fence_after();
          const unsigned sa = smem_u32(tiles + stage * stage_bytes);
          const unsigned sb = sa + a_ring;
          const unsigned long long da = umma_desc(sa), db = umma_desc(sb);
          const unsigned on = elect_one();
          const int next = stage + 1 == n_stages ? 0 : stage + 1;
          const unsigned next_phase = next == 0 ? phase ^ 1u : phase;
          ready = mbar_test(smem_u32(&sh->full[next]), next_phase);
#pragma unroll
          for (int k = 0; k < 4; ++k) {   // 16 bf16 or 32 codes = 32 bytes = 2 descriptor units per step
            const unsigned accum = (unsigned)((kb | k) != 0);
            if (kPair) {
              if (kE4) umma_e4m3_pair(d_tmem, da + 2ull * k, db + 2ull * k, kIdescE4Pair, accum, on);
              else umma_f16_pair(d_tmem, da + 2ull * k, db + 2ull * k, kIdescPair, accum, on);
            } else {
              if (kE4) umma_e4m3(d_tmem, da + 2ull * k, db + 2ull * k, idesc, accum, on);
              else umma_f16(d_tmem, da + 2ull * k, db + 2ull * k, idesc, accum, on);
            }
          }
          if (kSplit) {                   // + lo W into the same accumulator
            const unsigned long long dl = umma_desc(sa + a_bytes);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              if (kPair) umma_e4m3_pair(d_tmem, dl + 2ull * k, db + 2ull * k, kIdescE4Pair, 1u, on);
              else umma_e4m3(d_tmem, dl + 2ull * k, db + 2ull * k, idesc, 1u, on);
            }
          }
          // the stage is free again -- in both CTAs of a pair
          if (kPair) umma_commit_pair(smem_u32(&sh->empty[stage]), on);
          else umma_commit(smem_u32(&sh->empty[stage]), on);
          stage = next;
          phase = next_phase;
        }
        if (!ok) break;
        if (kPair) umma_commit_pair(smem_u32(&sh->tmem_full[acc]), elect_one());
        else umma_commit(smem_u32(&sh->tmem_full[acc]), elect_one());
        acc ^= 1u;
        if (acc == 0) acc_phase ^= 1u;
      }
    }
  } else {
    const int q = warp & 3;                  // tensor-memory lane quarter this warp may read
    const int half = (warp - 2) >> 2;        // 8 epilogue warps: which 128 columns of the tile
    const int c_lo = half * epi_cols;
    unsigned acc = 0, acc_phase = 0, vec = 0, vec_phase = 0;
    unsigned top_phase = 0;
    unsigned xchg_phase = 0;                 // bit a: phase of the next hand-over through xchg_full[a][q] (TopK tiles only)
    for (int tile = worker; tile < total_tiles; tile += n_workers) {
      const Tile t = tile_of(tile);
      if (!tile_wanted(t, groups, mode, mtile_flag)) continue;
      const int row_local = q * 32 + lane;
      const bool valid = row_local < t.rows_valid;
      const size_t p = (size_t)t.m_tile_global * kTileM + row_local;
      // TopK tiles: a lower bound on the row's k-th largest pre-activation, from what every CTA has seen of the
      // row so far in this call.  The row's k slots each hold the largest of a disjoint share of the values that
      // tiles already finished published (distinct elements of the row), so once no slot is empty there are k
      // elements >= the smallest slot: nothing below it can be in the TopK, and nearly everything is below it
      // after the first tiles.  Read before the wait for the accumulator; a stale value is merely a lower bound.
      const bool topk_tile = mode == 0 && groups[t.group].act == MIX_SAE_TOPK;
      const int k_row = groups[t.group].k;
      const bool use_tau = topk_tile && valid && tau_slots != nullptr && k_row <= kTauSlots;
      // (tiles of the launch's last wave publish nothing: no tile that starts later is left to read it)
      const bool publish_tau = use_tau && tile + n_workers < total_tiles;
      unsigned tau_key = 0u;                   // 0: no bound yet
      if (use_tau) tau_key = __ldcg(tau_min + p);     // the smallest slot, as of the last time a publisher looked
      constexpr bool kScaled = kEnc != 0;      // the accumulator is in units of the codes
      // This warp's columns of the bias and the feature scale, which the producer has copied.  (Read from global memory between
      // the tensor-memory loads they were four exposed round trips a tile; copied by each warp for itself ahead of its wait for
      // the accumulator, a trip that 8-bit tiles, which the epilogue sets the pace of, had no time for.)
      const float* wb = epi_vec + vec * (Cfg::kVecBytes / 4) + c_lo;
      const float* ws = wb + kTileN;
      const float* theta_t = nullptr;
      float* wt = kScaled ? nullptr : epi_vec + kVecs * kTileN + (warp - 2) * kEpiColsMax;
      bool want_bits = false, any_bits = false, jump = false, only_edits = false, any_full = false;
      unsigned edited = 0u;
      if (!topk_tile) {
        // For rows that are rebuilt from their active features, which of the tile's are active goes beside Z, a bit each:
        // the tail kernel then reads 3 KiB per row of 24576 features, and of Z what is active, instead of 100 KiB of Z and
        // as much of theta; and of Z only the groups of four with an active feature are written -- all of it (98 MB for 1000
        // rows) pushed W_dec out of L2 ahead of the gather.  1000 rows of d = 2304: the call 244 -> 219 us.  (Lists of the active
        // values instead of bits took this epilogue from 11 us a tile to 20.)
        const bool add_error = valid && (row_rec[p].group_flags & kRecAddError);
        want_bits = mode == 0 && valid && !add_error;
        any_bits = __any_sync(0xffffffffu, want_bits);
        // Of a row that keeps the error term only the edited features are needed (unless its active count is read out): the
        // groups of four that hold one, for any row of the warp, are written, and where that was, in the place of the bits --
        // the tail does not take Z's word for an edit that arrived on another stream after this kernel had looked.
        // 8192 rows, d = 5120, 23 % of them edited in two sets of 32768: the call 670 -> 630 us; d = 2304, 16384: 212 -> 186.  (Looked
        // up here, before the wait: behind it, the look-up showed in calls of one wave, 42 -> 44 us for 64 rows.)
        only_edits = mode == 0 && add_error && all_z == 0;
        any_full = __any_sync(0xffffffffu, valid && !want_bits && !only_edits);
        // (`edited`: lane w: the edited features among columns [32 w, 32 w + 32).)
        if (__any_sync(0xffffffffu, only_edits)) {
          const int n_edit = only_edits ? min(row_rec[p].n_edit, r_max) : 0;
          const int* list = edit_idx + (only_edits ? (size_t)row_rec[p].slot * r_max : 0);
          const int n_most = __reduce_max_sync(0xffffffffu, n_edit);
          for (int e0 = 0; e0 < n_most; e0 += 8) {
            int rel[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) rel[u] = e0 + u < n_edit ? list[e0 + u] - t.n_tile * tile_n : -1;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const bool in = (unsigned)rel[u] < (unsigned)tile_n;
              for (unsigned b = __ballot_sync(0xffffffffu, in); b != 0u;) {
                const int x = __shfl_sync(0xffffffffu, rel[u], __ffs(b) - 1);
                if (lane == (x >> 5)) edited |= 1u << (x & 31);
                b &= ~__ballot_sync(0xffffffffu, in && rel[u] == x);
              }
            }
          }
        }
        jump = any_bits && groups[t.group].act == MIX_SAE_JUMPRELU;
        if (jump) theta_t = groups[t.group].theta + (size_t)t.n_tile * tile_n + c_lo;
        if (jump && wt != nullptr) {
          for (int j = lane; j < epi_cols; j += 32) wt[j] = __ldg(theta_t + j);      // (theta need not be aligned)
          __syncwarp();
        }
      }
      // warp-uniform decision: tcgen05.ld below needs the whole warp
      if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&sh->vec_full[vec]), vec_phase, sh, status) &&
                                       mbar_wait(smem_u32(&sh->tmem_full[acc]), acc_phase, sh, status))) break;
      tc_fence_after();
      const float ars = kE4 ? (valid ? __ldg(act_scale + p) : 0.f) : 1.f;     // power of two: the products below are exact
      const unsigned taddr = tmem_base + ((unsigned)(q * 32) << 16) + acc * kTileN;
      if (topk_tile) {
        // `below`: what is not collected is at most that; the places of a list that nothing was collected for hold it
        const float tau = tau_key > 1u ? key2f(tau_key) : -INFINITY;
        float below = tau_key > 1u ? key2f(tau_key - 1u) : -INFINITY;
        auto to_z = [&](float v, float b, float s) { return kScaled ? fmaf(v, s * ars, b) : v + b; };
        // f(first column, 8 pre-activations) over this warp's columns, 32 of them a load: what a trip of eight costs beside the
        // work is the load's latency, also with the next load under way (eight a load 2.5 us for the networks of 64 columns and
        // 2.5 for what is collected, 32 a load 2.3 and 1.9).  A loop still: this code runs once or a few times per call, and what
        // is unrolled has to be fetched before it has an effect.
        auto columns = [&](auto&& f) {
#pragma unroll 1
          for (int c = c_lo; c < c_lo + epi_cols; c += 32) {
            float v[32];
            tmem_ld32(taddr + c, v);
#pragma unroll
            for (int g = 0; g < 32; g += 8) {
              float z[8];
#pragma unroll
              for (int i = 0; i < 8; i += 4) {
                const float4 b4 = *reinterpret_cast<const float4*>(wb + (c - c_lo) + g + i);
                float4 s4 = make_float4(1.f, 1.f, 1.f, 1.f);
                if (kScaled) s4 = *reinterpret_cast<const float4*>(ws + (c - c_lo) + g + i);
                z[i] = to_z(v[g + i], b4.x, s4.x);
                z[i + 1] = to_z(v[g + i + 1], b4.y, s4.y);
                z[i + 2] = to_z(v[g + i + 2], b4.z, s4.z);
                z[i + 3] = to_z(v[g + i + 3], b4.w, s4.w);
              }
              f(c + g, z);
            }
          }
        };
        // This warp's list: columns ascending, or sorted.  (Either way equal values stand in the order of their columns, which is
        // all that the selection asks of it.)
        auto handed = [&](unsigned a) { return xchg + (a * 4 + q) * kXchgListBytes; };
        unsigned char* list = half == 1 ? handed(acc) : pick + q * kListBytes;
        float* list_v = reinterpret_cast<float*>(list) + lane;
        unsigned char* list_c = list + kListRows * 32 * 4 + lane;
        float tv[kCandPerTile + 1];
        int ti[kCandPerTile + 1];
        int n = 0;                              // entries of the list
        bool listed = false, sorted = false;    // sorted: the list is in tv / ti, in descending order
        if (kEpiWarps == 8) {
          float least = tau;                    // what is collected: this and above
          tv[kCandPerTile] = below;
          // With a bound in force few columns pass it.  Without one -- the row's feature tiles that finished a wave ago cannot
          // have filled its k slots -- the 8 largest VALUES of the tile and the 9th are found first, by min / max networks in
          // which all lanes take part (11 instructions a column); the two warps of a quarter show each other theirs, and the 8th
          // of both is the bound, so that together they collect 8 and nobody sorts.  (Each warp collecting its own 8, sorting
          // them and merging: 6.5 us for a tile of 128 features and 4.2 for one of 64, where this takes 5.0 and 3.4.  Both warps
          // must come to the same answer here, so it does not hang on what either has read of the bound.)
          const int first_wave = n_workers / (uniform_nt > 0 ? sh->unit0[n_groups] : sh->unit0[t.group + 1] - sh->unit0[t.group]) + 1;
          const bool network = __any_sync(0xffffffffu, valid) &&
                               (tau_slots == nullptr || k_row > kTauSlots || (t.n_tile - first_wave) * kCandPerTile < k_row);
          if (network) {
            float top[8], ninth = -INFINITY;
#pragma unroll
            for (int s = 0; s < 8; ++s) top[s] = -INFINITY;
            columns([&](int, float (&b)[8]) {
#pragma unroll
              for (int s = 0; s < 8; ++s) b[s] = fmaxf(b[s], -INFINITY);          // (a NaN is never selected)
              sort8_desc(b);
#pragma unroll
              for (int s = 0; s < 8; ++s) {                                       // the 8 largest of both, and the largest of the rest
                const float lo = fminf(top[s], b[7 - s]);
                top[s] = fmaxf(top[s], b[7 - s]);
                ninth = fmaxf(ninth, lo);
              }
              merge8_desc(top);
            });
            // The lower-half warp leaves its values in the other accumulator's hand-over place, which it was the last to read;
            // the upper-half warp answers in the lower one's list, which that does not touch before it has read the answer.
            float* to = reinterpret_cast<float*>(half == 0 ? handed(acc ^ 1u) : pick + q * kListBytes) + lane;
            const float* from = reinterpret_cast<const float*>(half == 0 ? pick + q * kListBytes : handed(acc ^ 1u)) + lane;
            if (half == 1 && !__all_sync(0xffffffffu, mbar_wait(smem_u32(&sh->top_full[0][q]), top_phase, sh, status))) break;
            float other[8], ninth2 = 0.f;
            if (half == 1) {
#pragma unroll
              for (int s = 0; s < 8; ++s) other[s] = from[s * 32];
              ninth2 = from[8 * 32];
            }
#pragma unroll
            for (int s = 0; s < 8; ++s) to[s * 32] = top[s];
            to[8 * 32] = ninth;
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sh->top_full[half][q]));
            if (half == 0) {
              if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&sh->top_full[1][q]), top_phase, sh, status))) break;
#pragma unroll
              for (int s = 0; s < 8; ++s) other[s] = from[s * 32];
              ninth2 = from[8 * 32];
              __syncwarp();                     // (every lane has read before one writes its list there)
            }
            top_phase ^= 1u;
            least = INFINITY;
            ninth = fmaxf(ninth, ninth2);
#pragma unroll
            for (int s = 0; s < 8; ++s) {
              least = fminf(least, fmaxf(top[s], other[7 - s]));
              ninth = fmaxf(ninth, fminf(top[s], other[7 - s]));
            }
            below = -INFINITY;
            tv[kCandPerTile] = ninth;
          }
          if (!valid) least = NAN;
          columns([&](int c, float (&z)[8]) {
            float m = z[0];
#pragma unroll
            for (int i = 1; i < 8; ++i) m = fmaxf(m, z[i]);
            if (!__any_sync(0xffffffffu, m >= least)) return;
            // (stored whether they pass or not, the next one over what did not: a branch around each of them, taken for some
            // lane nearly every time, cost 86 cycles a column)
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const int at = min(n, kListRows - 1) * 32;
              list_v[at] = z[i];
              list_c[at] = (unsigned char)(c - c_lo + i);
              n += z[i] >= least;
            }
          });
          listed = __all_sync(0xffffffffu, n <= kCandPerTile);
          if (listed && half == 0) {
#pragma unroll
            for (int s = 0; s < kCandPerTile; ++s) {
              tv[s] = s < n ? list_v[s * 32] : below;
              ti[s] = c_lo + (s < n ? (int)list_c[s * 32] : 0);
            }
          }
        }
        if (!listed) {
          // More than 8 above the bound, or equal values at the 8th: a sorted list of 9, by insertion (kEpiWarps == 4, contexts
          // that had no TopK set when this was launched: always).
          below = tau_key > 1u ? key2f(tau_key - 1u) : -INFINITY;
#pragma unroll
          for (int s = 0; s <= kCandPerTile; ++s) {
            tv[s] = below;
            ti[s] = c_lo;
          }
          if (__any_sync(0xffffffffu, valid)) {
#pragma unroll 1
            for (int c = c_lo; c < c_lo + epi_cols; c += 8) {
              float v[8];
              tmem_ld8(taddr + c, v);
#pragma unroll
              for (int i = 0; i < 8; ++i) top9_insert(tv, ti, to_z(v[i], wb[c - c_lo + i], kScaled ? ws[c - c_lo + i] : 1.f), c + i);
            }
          }
          n = kCandPerTile;
          sorted = true;
        }
        bool writer = true;
        unsigned tau_pub = tau_key;
        if (kEpiWarps == 8) {
          // the upper-half warp's list is where the lower-half warp finds it; that one writes the tile's candidates: both lists
          // one behind the other where they fit (its columns come first), else the 8 largest of both
          unsigned char* up = handed(acc);
          float* xv = reinterpret_cast<float*>(up) + lane;
          unsigned char* xc = up + kListRows * 32 * 4 + lane;
          int* xw = reinterpret_cast<int*>(up + kListBytes) + lane;
          if (half == 1) {
            if (sorted) {
#pragma unroll
              for (int s = 0; s < kCandPerTile; ++s) {
                xv[s * 32] = tv[s];
                xc[s * 32] = (unsigned char)(ti[s] - c_lo);
              }
            }
            xw[0] = __float_as_int(tv[kCandPerTile]);
            xw[32] = n | (sorted ? 0x100 : 0);
            xw[64] = (int)tau_key;
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sh->xchg_full[acc][q]));
            writer = false;
          } else {
            if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&sh->xchg_full[acc][q]), (xchg_phase >> acc) & 1u, sh, status))) break;
            const int n2 = xw[32] & 0xff;
            const bool sorted2 = (xw[32] & 0x100) != 0;
            const float ninth2 = __int_as_float(xw[0]);
            if (__all_sync(0xffffffffu, n + n2 <= kCandPerTile)) {
#pragma unroll
              for (int s = 0; s < kCandPerTile; ++s) {
                if (s >= n && s < n + n2) {
                  tv[s] = xv[(s - n) * 32];
                  ti[s] = epi_cols + (int)xc[(s - n) * 32];
                }
              }
              tv[kCandPerTile] = fmaxf(tv[kCandPerTile], ninth2);
            } else {
              float v2[kCandPerTile + 1];
              int c2[kCandPerTile + 1];
#pragma unroll
              for (int s = 0; s < kCandPerTile; ++s) {
                v2[s] = s < n2 ? xv[s * 32] : -INFINITY;
                c2[s] = epi_cols + (s < n2 ? (int)xc[s * 32] : 0);
              }
              if (!sorted) sort8_pairs(tv, ti);
              if (!sorted2) sort8_pairs(v2, c2);
              merge_lists(tv, ti, ninth2, [&](int s, float& x, int& cx) { x = v2[s]; cx = c2[s]; });
            }
            // the two warps may have read the bound at different times: what is at or above the larger one is a
            // real element of the row (each warp's fillers lie below its own bound)
            tau_pub = max(tau_key, (unsigned)xw[64]);
          }
        }
        xchg_phase ^= 1u << acc;
        if (valid && writer) {
          const size_t slot = p * (size_t)cand_tiles + (size_t)t.n_tile;
          float4* cv = reinterpret_cast<float4*>(cand_val + slot * kCandPerTile);
          int4* ci = reinterpret_cast<int4*>(cand_idx + slot * kCandPerTile);
          const int j0 = t.n_tile * tile_n;
          cv[0] = make_float4(tv[0], tv[1], tv[2], tv[3]);
          cv[1] = make_float4(tv[4], tv[5], tv[6], tv[7]);
          ci[0] = make_int4(j0 + ti[0], j0 + ti[1], j0 + ti[2], j0 + ti[3]);
          ci[1] = make_int4(j0 + ti[4], j0 + ti[5], j0 + ti[6], j0 + ti[7]);
          cand_ninth[slot] = tv[kCandPerTile];
          if (publish_tau) {
            // this tile's r-th candidate goes to slot (n_tile + r k/8) mod k: no two (tile, rank) pairs are the same
            // element, eight consecutive feature tiles fill every slot, and every slot sees all places over time
            unsigned* sp = tau_slots + p * kTauSlots;
            bool raised_min = false;
            const int rank_step = max(k_row / kCandPerTile, 1);
            int slot_r = t.n_tile % k_row;
#pragma unroll
            for (int r = 0; r < kCandPerTile; ++r) {
              const unsigned key = f2key(tv[r]);
              if (key >= tau_pub && tv[r] > -INFINITY) {
                const unsigned old = atomicMax(sp + slot_r, key);
                raised_min = raised_min || old < key;      // the smallest slot may have moved up
              }
              slot_r += rank_step;
              if (slot_r >= k_row) slot_r -= k_row;
            }
            if (raised_min) {
              unsigned m = 0xffffffffu;
              for (int j = 0; j < k_row; j += 4) {
                const uint4 w = __ldcg(reinterpret_cast<const uint4*>(sp) + (j >> 2));
                m = min(m, w.x);
                if (j + 1 < k_row) m = min(m, w.y);
                if (j + 2 < k_row) m = min(m, w.z);
                if (j + 3 < k_row) m = min(m, w.w);
              }
              if (m > tau_pub) atomicMax(tau_min + p, m);
            }
          }
        }
      } else {
        float* out = Z + p * (size_t)ldz + (size_t)t.n_tile * tile_n;
        unsigned* bits = reinterpret_cast<unsigned*>(cand_idx) + p * (size_t)cand_tiles * kCandPerTile + t.n_tile * (tile_n / 32);
#pragma unroll 1
        for (int c = c_lo; c < c_lo + epi_cols; c += 32) {
          const unsigned here = __shfl_sync(0xffffffffu, edited, c >> 5);
          if (only_edits) bits[c >> 5] = here;
          if (!any_full && !any_bits && here == 0u) continue;
          float v[32];
          tmem_ld32(taddr + c, v);
          if (valid) {
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
              const float4 b4 = *reinterpret_cast<const float4*>(wb + (c - c_lo) + i);
              float4 s4 = make_float4(1.f, 1.f, 1.f, 1.f);
              if (kScaled) s4 = *reinterpret_cast<const float4*>(ws + (c - c_lo) + i);
              if (kE4) { s4.x *= ars; s4.y *= ars; s4.z *= ars; s4.w *= ars; }
              float4 o;
              o.x = kScaled ? fmaf(v[i], s4.x, b4.x) : v[i] + b4.x;
              o.y = kScaled ? fmaf(v[i + 1], s4.y, b4.y) : v[i + 1] + b4.y;
              o.z = kScaled ? fmaf(v[i + 2], s4.z, b4.z) : v[i + 2] + b4.z;
              o.w = kScaled ? fmaf(v[i + 3], s4.w, b4.w) : v[i + 3] + b4.w;
              if (!want_bits && (!only_edits || ((here >> i) & 15u))) *reinterpret_cast<float4*>(out + c + i) = o;
              v[i] = o.x; v[i + 1] = o.y; v[i + 2] = o.z; v[i + 3] = o.w;
            }
          }
          if (any_bits) {
            unsigned m = 0u;
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
              float4 t4 = make_float4(0.f, 0.f, 0.f, 0.f);
              if (jump) {
                const float* th = theta_t + (c - c_lo) + i;
                t4 = wt != nullptr ? *reinterpret_cast<const float4*>(wt + (c - c_lo) + i)
                                   : make_float4(__ldg(th), __ldg(th + 1), __ldg(th + 2), __ldg(th + 3));
              }
              if (v[i] > t4.x && v[i] != 0.f) m |= 1u << i;
              if (v[i + 1] > t4.y && v[i + 1] != 0.f) m |= 2u << i;
              if (v[i + 2] > t4.z && v[i + 2] != 0.f) m |= 4u << i;
              if (v[i + 3] > t4.w && v[i + 3] != 0.f) m |= 8u << i;
            }
            if (want_bits) {
              bits[c >> 5] = m;
#pragma unroll
              for (int i = 0; i < 32; i += 4)
                if ((m >> i) & 15u) *reinterpret_cast<float4*>(out + c + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {     // the accumulator is free: tell the CTA that issues the instructions
        if (kPair && !leader) mbar_arrive_cluster(mapa_cluster(smem_u32(&sh->tmem_empty[acc]), 0));
        else mbar_arrive(smem_u32(&sh->tmem_empty[acc]));
        mbar_arrive(smem_u32(&sh->vec_empty[vec]));
      }
      if (++vec == kVecs) { vec = 0; vec_phase ^= 1u; }
      acc ^= 1u;
      if (acc == 0) acc_phase ^= 1u;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (sh->abort_flag) {
    // give copies that are still in flight time to land before shared memory is released
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000ll) __nanosleep(1000);
  }
  // a pair leaves together: neither CTA's barriers or tensor memory go away while the other may still reach them
  if (kPair) cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    if (kPair) tmem_dealloc_pair(tmem_base, kTmemCols);
    else tmem_dealloc(tmem_base, kTmemCols);
  }
  phase_stamp(clk, 29, stamp);
}

// Registration-time copy of W_enc [S, d] into [S/256][d/64][256][64]: one thread per 16 bytes.
__global__ void retile_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst, long long d_sae, int d) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;      // index of a 16-byte piece of dst
  const int num_kb = d / kTileK;
  const long long total = d_sae * (long long)d / 8;
  if (i >= total) return;
  const int piece = (int)(i & 7);                       // 8 pieces per 64-column row
  const long long row_in_all = i >> 3;                  // row of the [.., 256, 64] blocks
  const int r = (int)(row_in_all % kTileN);
  const long long blk = row_in_all / kTileN;
  const int kb = (int)(blk % num_kb);
  const long long n_tile = blk / num_kb;
  dst[i] = src[((n_tile * kTileN + r) * (long long)d + (long long)kb * kTileK) / 8 + piece];
}

// The same for 8-bit codes: [S, d] bytes -> [S/256][d/kb_bytes][256][kb_bytes] bytes (kb_bytes = 64 for the
// widening kernel, 128 for the 8-bit contraction), one thread per 16 bytes.
__global__ void retile_fp8_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst, long long d_sae, int d, int kb_bytes) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int num_kb = d / kb_bytes;
  const int ppr = kb_bytes / 16;                        // 16-byte pieces per block row
  const long long total = d_sae * (long long)d / 16;
  if (i >= total) return;
  const int piece = (int)(i % ppr);
  const long long row_in_all = i / ppr;
  const int r = (int)(row_in_all % kTileN);
  const long long blk = row_in_all / kTileN;
  const int kb = (int)(blk % num_kb);
  const long long n_tile = blk / num_kb;
  dst[i] = src[((n_tile * kTileN + r) * (long long)d + (long long)kb * kb_bytes) / 16 + piece];
}

}  // namespace

cudaError_t launch_retile_fp8(const unsigned char* W_enc, unsigned char* W_tiled, long long d_sae, int d, int kb_bytes,
                              cudaStream_t s) {
  const long long total = d_sae * (long long)d / 16;
  retile_fp8_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(reinterpret_cast<const uint4*>(W_enc),
                                                                    reinterpret_cast<uint4*>(W_tiled), d_sae, d, kb_bytes);
  return cudaGetLastError();
}

cudaError_t launch_retile(const __nv_bfloat16* W_enc, __nv_bfloat16* W_tiled, long long d_sae, int d, cudaStream_t s) {
  const long long total = d_sae * (long long)d / 8;
  retile_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(reinterpret_cast<const uint4*>(W_enc),
                                                                reinterpret_cast<uint4*>(W_tiled), d_sae, d);
  return cudaGetLastError();
}

template <int kEnc, int kEpi, bool kPair>
static cudaError_t encode_tc_prepare_as() {
  return cudaFuncSetAttribute(encode_tc_kernel<kEnc, kEpi, kPair>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              TcCfg<kEnc, kEpi, kPair>::kSmemBytes);
}

cudaError_t encode_tc_prepare() {
  cudaError_t e = encode_tc_prepare_as<0, 4, false>();
  if (e == cudaSuccess) e = encode_tc_prepare_as<0, 8, false>();
  if (e == cudaSuccess) e = encode_tc_prepare_as<1, 4, false>();
  if (e == cudaSuccess) e = encode_tc_prepare_as<1, 8, false>();
  if (e == cudaSuccess) e = encode_tc_prepare_as<2, 4, false>();
  if (e == cudaSuccess) e = encode_tc_prepare_as<2, 8, false>();
  if (e == cudaSuccess) e = encode_tc_prepare_as<0, 4, true>();
  if (e == cudaSuccess) e = encode_tc_prepare_as<0, 8, true>();
  if (e == cudaSuccess) e = encode_tc_prepare_as<1, 4, true>();
  if (e == cudaSuccess) e = encode_tc_prepare_as<1, 8, true>();
  if (e == cudaSuccess) e = encode_tc_prepare_as<2, 4, true>();
  if (e == cudaSuccess) e = encode_tc_prepare_as<2, 8, true>();
  return e;
}

// CTA pairs or single CTAs: MIX_ENCODE_PAIR in the environment (0 / 1), read once; set by mix_set_encode_pair for A/B timing.
static int g_encode_pair = -1;
int encode_pair_mode(int set) {
  if (g_encode_pair < 0) {
    const int v = getenv("MIX_ENCODE_PAIR") ? atoi(getenv("MIX_ENCODE_PAIR")) : kEncodePairDefault;
    g_encode_pair = v == 0 || v == 1 ? v : 2;
  }
  const int old = g_encode_pair;
  if (set >= 0) g_encode_pair = set == 0 || set == 1 ? set : 2;
  return old;
}

template <int kEnc, int kEpi, bool kPair>
static cudaError_t launch_encode_tc_as(const Ctx* c, int mode, cudaStream_t s) {
  using Cfg = TcCfg<kEnc, kEpi, kPair>;
  const int w_tiled = (c->cfg.flags & MIX_FLAG_RETILE_W_ENC) ? 1 : 0;
  const int stall = (c->cfg.flags & MIX_FLAG_TEST_STALL_ENCODE) ? 1 : 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kPair ? (c->n_sms & ~1) : c->n_sms);
  cfg.blockDim = dim3(Cfg::kThreads);
  cfg.dynamicSmemBytes = Cfg::kSmemBytes;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  int n_at = 0;
  if (kPair) {
    at[n_at].id = cudaLaunchAttributeClusterDimension;
    at[n_at].val.clusterDim.x = 2;
    at[n_at].val.clusterDim.y = 1;
    at[n_at].val.clusterDim.z = 1;
    ++n_at;
  }
  if (pdl_mask() & (mode == 0 ? kPdlEncode : kPdlTail)) {
    at[n_at].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[n_at].val.programmaticStreamSerializationAllowed = 1;
    ++n_at;
  }
  cfg.attrs = at;
  cfg.numAttrs = n_at;
  return cudaLaunchKernelEx(&cfg, encode_tc_kernel<kEnc, kEpi, kPair>, c->tmap_panel, c->tmap_w_one,
                            static_cast<const CUtensorMap*>(c->d_tmap_w),
                            static_cast<const RouteState*>(c->d_route), static_cast<const GroupEntry*>(c->d_groups),
                            c->cfg.n_groups_max, c->d_z, (long long)c->cfg.d_sae_max, c->cfg.d_model, c->d_status, mode,
                            static_cast<const int*>(c->d_mtile_flag), static_cast<const int*>(c->d_n_flagged), c->d_cand_val,
                            c->d_cand_idx, c->d_cand_ninth, c->cand_tiles, w_tiled, stall,
                            static_cast<const float*>(c->d_act_scale), c->d_tau, c->d_tau_min, c->panel_rows_cap,
                            static_cast<const RowRec*>(c->d_row_rec), static_cast<const int*>(c->d_edit_idx), c->cfg.r_max,
                            c->out_n_active != nullptr ? 1 : 0, c->d_phase_clk);
}

// Eight epilogue warps pay off for the TopK epilogue (selection work per element); the plain store of the
// pre-activations is a little faster with four.  Either form is correct for any mix of weight sets; the choice
// is made from the sets registered when the call is enqueued (or captured).
// pair: the CTA-pair kernel (256-row tiles) or the single-CTA kernel; a full pass (mode 0) launches both, and
// the one the front kernel did not choose for this call returns at once.
cudaError_t launch_encode_tc(const Ctx* c, int mode, bool pair, cudaStream_t s) {
  bool topk = false;
  for (int g = 0; g < c->cfg.n_groups_max; ++g) topk = topk || (c->h_groups[g].valid && c->h_groups[g].act == MIX_SAE_TOPK);
  if (pair) {
    if (c->cfg.flags & MIX_FLAG_FP8_ACT) return topk ? launch_encode_tc_as<2, 8, true>(c, mode, s) : launch_encode_tc_as<2, 4, true>(c, mode, s);
    if (c->cfg.flags & MIX_FLAG_FP8_W_ENC) return topk ? launch_encode_tc_as<1, 8, true>(c, mode, s) : launch_encode_tc_as<1, 4, true>(c, mode, s);
    return topk ? launch_encode_tc_as<0, 8, true>(c, mode, s) : launch_encode_tc_as<0, 4, true>(c, mode, s);
  }
  if (c->cfg.flags & MIX_FLAG_FP8_ACT) return topk ? launch_encode_tc_as<2, 8, false>(c, mode, s) : launch_encode_tc_as<2, 4, false>(c, mode, s);
  if (c->cfg.flags & MIX_FLAG_FP8_W_ENC) return topk ? launch_encode_tc_as<1, 8, false>(c, mode, s) : launch_encode_tc_as<1, 4, false>(c, mode, s);
  return topk ? launch_encode_tc_as<0, 8, false>(c, mode, s) : launch_encode_tc_as<0, 4, false>(c, mode, s);
}

bool encode_pair_possible(const Ctx* c) { return encode_pair_mode(-1) != 0 && c->cfg.T_max > kTileM; }

}  // namespace mix
