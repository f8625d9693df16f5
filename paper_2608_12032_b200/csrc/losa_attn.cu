// Attention kernels of liblosa for sm_100a: dense attention, block-sparse attention over a
// frozen CSR pattern (Eq. 4), the exact block-mass pass (Eq. 1) and the fused construction step.
// They run in losa_tile_kernel (losa_attn_tile.cuh, included below), one warp-specialised persistent kernel: one
// query tile and three S buffers per CTA, on pairs of CTAs at head dimension 128.  Here is what surrounds it: the
// work units and their tile lists, the merge of units that were cut, tensor maps and launches.
//
// A work item is a pair of consecutive query tiles of one (batch, head) - of one problem, in a
// batched launch.  At head dimension 128 the key blocks the pair visits are the union of the index lists of its query
// blocks (two lists, four when R = 64), so that a K/V tile needed by both tiles is loaded once; at head
// dimension 64 each of the two tiles has a list of its own.  The items of the last, partly filled wave of the
// persistent grid are cut into parts of their lists, merged behind (merge_parts_kernel) or, where all of a call is one
// wave, by the clusters that they share (merge_in_cluster).
//
// Every wait is bounded; a wait that expires raises the CTA's abort flag, records
// LOSA_ERR_TIMEOUT, and all roles leave through the common teardown that frees TMEM.
#include <cuda.h>
#include <cuda_bf16.h>
#include <limits.h>
#include <math.h>

#include <algorithm>
#include <atomic>
#include <cstddef>
#include <type_traits>

#include "losa_common.cuh"
#include "losa_ptx.cuh"

namespace losa {
namespace {

std::atomic<uint32_t> g_stall_polls{0u};  // > 0: the next attention launch is a diagnostic one

// Thread layout.  Warps 0-3 are the utility warpgroup (TMA, 2 MMA issuers, scheduler); the 16 softmax
// warps follow, two threads per query row of a K/V tile, each of which holds 64 columns.  A warp's ex2 instructions
// occupy it for 8 issue cycles each and its other instructions do not overlap them (measured on the loop alone: 1301
// cycles per 128-column row with one warp per scheduler partition, 1130 with two), so a query tile's
// softmax needs two warps per partition to keep the special-function unit busy; the two warps
// never talk to each other on the common path (see the softmax role).
struct Lay {
  static constexpr int kSoftmaxWarps = 16;
  static constexpr int kThreads = 128 + 32 * kSoftmaxWarps;
  static constexpr int kRegsSoftmax = 104;
  static constexpr int kRegsUtility = 64;
  static constexpr int kRegsAtLaunch = 96;
  // setmaxnreg only moves registers inside the CTA's launch allocation: the increase waits until
  // the decrease has released enough, so the totals must balance or the increase never returns.
  static_assert(128 * kRegsUtility + 32 * kSoftmaxWarps * kRegsSoftmax <= kThreads * kRegsAtLaunch,
                "register reallocation exceeds the CTA's launch allocation");
  static_assert(kThreads * kRegsAtLaunch <= 65536, "launch allocation exceeds the register file");
};
// The utility warps take the LOWEST warp ids.  When several warps of a scheduler partition are
// ready, the hardware favours the lower (older) ids; a softmax warp in an arithmetic-dense
// stretch is ready every cycle, and with the MMA issuer behind it in that order each of the
// issuer's instructions waited ~10x longer (measured), which put the issuer on the critical path.
constexpr int kProducerWarp = 0, kIssuerWarp = 1, kSchedulerWarp = 3;  // issuers: warps 1 and 2
constexpr int kTmemCols = 512;
constexpr size_t kCounterBytes = 256;  // head of the workspace: the launch's counters
constexpr int kCounters = 2;  // work items drawn, units run again
constexpr size_t kPartMlBytes = (size_t)kMaxPersistentCtas * 2 * 128 * sizeof(float2);  // [slot][2][128] float2
constexpr int kTlChunks = 4;  // of the tile list ring in shared memory
constexpr uint32_t kTlItem = 1u << 28, kTlEnd = 2u << 28, kTlSkip = 3u << 28;  // entry type in bits 31:28 (0 = tile)
// An item header carries the work item in bits 23:0 and, for a unit that covers only part of the
// item's key range, the part index in bits 26:24 and a flag in bit 27.
constexpr uint32_t kTlItemMask = 0x00ffffffu, kTlPartial = 1u << 27;
// A K/V tile is a group of 128 / C consecutive tile entries (key block index in bits 15:0,
// membership bits from bit 16); the last group of an item is padded with this entry: no member,
// and a block index whose rows lie past the end of the tensor (the copy engine fills zeros).
constexpr uint32_t kTlPad = 0xffffu;
constexpr uint32_t kTlRagged = 1u << 20;  // tile entry: the sequence ends inside this key block
// What is said of a unit's tile list: how many K/V tiles, which query tiles list any (kHdrHas << query
// tile), and whether query tile 1 lists its first in the second K/V tile
// (a unit that is one query tile: bit kHdrHas alone, and which of the item's two it is, kHdrOdd)
constexpr uint32_t kHdrSetShift = 24;  // (of a unit that is run again)
constexpr uint32_t kHdrTiles = 0x00ffffffu, kHdrMax = 1u << 26, kHdrRedo = 1u << 27, kHdrOdd = 1u << 28, kHdrLate = 1u << 29, kHdrHas = 1u << 30;
// Tile lists per work unit: one for its pair of query tiles, or (head dimension 64, where a CTA works on
// one query tile at a time) one for each.
__host__ __device__ constexpr int tile_lists_per_unit(int D) { return D == 64 ? 2 : 1; }
constexpr int kMaxParts = 8;
constexpr int kMaxClusterCtas = 2 * kMaxParts;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
// a tile's half-row sum (or, where it comes out of the product with V, a unit's row sum) beyond
// 2^60 or NaN has the work unit computed again
constexpr float kSplitSafeSum = 1.152921504606846976e18f;

// One entry per problem of a batched launch (several layers or requests of one shape in one
// persistent launch): the problem's tensor maps, its output and its own CSR pattern.  The table
// lives in the workspace and is written by write_problems_kernel before the launch.
struct alignas(128) ProblemEntry {
  CUtensorMap map_q, map_k, map_v;
  CUtensorMap map_kh;  // K with boxes of at most 64 keys (the CTA-pair kernel copies half a K tile per CTA)
  // boxes that span several key blocks, for K/V tiles whose key blocks are consecutive (C < 128)
  CUtensorMap map_k64, map_k128, map_v128;
  void* o;
  const int32_t* offsets;
  const int32_t* kv_idx;
};

struct Params {
  int B, H, N, C, nQb, nKb, nQt, nPairs, nWork;
  // Batched launch: work items run over nProb problems, item w belongs to problem
  // w / (B * H * nPairs); `problems` is null for a single problem, whose maps are kernel
  // parameters and whose o / offsets / kv_idx are the fields below.
  int nProb;
  const ProblemEntry* problems;
  // Work units: items [0, split_first) whole, items [split_first, nWork) in split_parts parts of
  // their key-block lists each (the last, partly filled wave of the persistent grid is cut finer).
  int nUnits, split_first, split_parts;
  Divisor by_parts, by_pairs, by_heads, by_problem;  // split_parts, nPairs, H, B * H
  // Sparse mode: the merged tile lists of all units, built by build_tile_lists_kernel before the
  // attention kernel: unit u owns tl_entries[u * tl_cap ...], tl_count[u] of them (padded to whole tiles).
  uint32_t* tl_entries;
  int32_t* tl_count;  // (kHdrTiles, kHdrHas, kHdrLate)
  int tl_cap;
  float* part_o;    // [slot][2][128][D] unnormalised O of a partial unit, slot = (item - split_first) * parts + part
  float2* part_ml;  // [slot][2][128] (reference max, row sum) of a partial unit
  const int32_t* offsets;
  const int32_t* kv_idx;
  void* o;
  int o_f32;
  int64_t sb, sh, sn;
  float* mass;
  float* lse;
  int* work_counter;  // zeroed before the launch; CTAs draw work items from it
  float2* table;  // mass modes: [grid][2][nKb][128], sums of exponentials per row and key block (losa_attn_tile.cuh)
  float scale_log2;
  int* status;
  // How many work units were run again because their scores outgrew the reference, and a flag for each, so that one
  // is counted once.  Where units are neither drawn nor merged nobody counts them.
  int* redo_count;
  int* redo_flag;  // [nUnits], or a word per tile list (one_wave, where items are cut)
  // No more work units than work slots: each slot takes the one at its position, and needs
  // nothing prepared for it (counters, flags, tile lists), which saves a launch: the CTAs make their unit's
  // tile list themselves, and each list's flag says whether its unit was run again (where parts are merged).
  int one_wave;
  // ... and the parts of an item run in one cluster, whose CTAs merge them through each other's shared memory
  int in_cluster;
  // extents of the buffers the kernels index into (elements), for the checked build
  long long cap_part_rows, cap_table_floats, cap_mass, cap_lse, cap_units;
  uint32_t wait_polls;  // bound of every device-side wait, in polls (ptx::kWaitPolls)
  int stall;            // diagnostic launch: the scheduler publishes nothing, so that every wait runs out
};

// Checked build (-DLOSA_CHECKED=1, a substitute for a memory checker): every index the kernels
// compute into the workspace, the masses or the log-sum-exp is compared with the extent of its
// buffer; one that falls outside is recorded as LOSA_ERR_INTERNAL and the access is skipped (or
// redirected to element 0 of the same buffer).  The ordinary build compiles the checks away.
#ifndef LOSA_CHECKED
#define LOSA_CHECKED 0
#endif
#if LOSA_CHECKED
#define LOSA_IN_RANGE(idx, extent) \
  (((unsigned long long)(idx) < (unsigned long long)(extent)) || (report_error(p.status, LOSA_ERR_INTERNAL), false))
#else
#define LOSA_IN_RANGE(idx, extent) true
#endif

#define LOSA_WAIT_RELAXED(bar, parity)                                   \
  do {                                                                   \
    if (!ptx::mbar_wait_relaxed((bar), (parity), &ctl->abort_flag, p.wait_polls)) {    \
      ctl->abort_flag = 1;                                               \
      report_error(p.status, LOSA_ERR_TIMEOUT);                          \
      goto teardown;                                                     \
    }                                                                    \
  } while (0)

#define LOSA_WAIT(bar, parity)                                   \
  do {                                                           \
    if (!ptx::mbar_wait((bar), (parity), &ctl->abort_flag, p.wait_polls)) {    \
      ctl->abort_flag = 1;                                       \
      report_error(p.status, LOSA_ERR_TIMEOUT);                  \
      goto teardown;                                             \
    }                                                            \
  } while (0)

// An item's place: the problem of a batched launch, the head (b * H + h) in it and the pair of query tiles.
__device__ __forceinline__ void item_place(const Params& p, int w, int& problem, int& bh, int& pr) {
  problem = p.by_problem.divmod(p.by_pairs.divmod(w, pr), bh);
}

// ---- merge of the partial units: for every row of the split items, combine the parts' unnormalised
// O, reference maximum and row sum (the usual log-sum-exp merge) and write the attention output.
// (slot0: of part 0; part s of the row lies 256 s slots further.  Lanes are the columns.)
template <int D>
__device__ __forceinline__ void load_part_row(const Params& p, int64_t slot, int lane, float* v) {
  const float* src = p.part_o + slot * D + lane * (D / 32);
  if constexpr (D == 128) {
    const float4 x = __ldcg(reinterpret_cast<const float4*>(src));
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
  } else {
    const float2 x = __ldcg(reinterpret_cast<const float2*>(src));
    v[0] = x.x; v[1] = x.y;
  }
}
template <int D>
__device__ __forceinline__ void store_merged_row(const Params& p, int problem, int bh, int grow, int lane, const float* acc, float inv) {
  void* const o_base = (p.problems != nullptr) ? p.problems[problem].o : p.o;
  int h;
  const int b = p.by_heads.divmod(bh, h);
  const int64_t off = (int64_t)b * p.sb + (int64_t)h * p.sh + (int64_t)grow * p.sn + lane * (D / 32);
  if (p.o_f32) {
    float* dst = static_cast<float*>(o_base) + off;
    if constexpr (D == 128)
      *reinterpret_cast<float4*>(dst) = make_float4(acc[0] * inv, acc[1] * inv, acc[2] * inv, acc[3] * inv);
    else
      *reinterpret_cast<float2*>(dst) = make_float2(acc[0] * inv, acc[1] * inv);
  } else {
    __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(o_base) + off;
    if constexpr (D == 128)
      *reinterpret_cast<uint2*>(dst) = make_uint2(ptx::pack_bf16x2(acc[0] * inv, acc[1] * inv),
                                                  ptx::pack_bf16x2(acc[2] * inv, acc[3] * inv));
    else
      *reinterpret_cast<uint32_t*>(dst) = ptx::pack_bf16x2(acc[0] * inv, acc[1] * inv);
  }
}

// A warp per row; all
// parts of a row are read at once, whatever their weights turn out to be, because the merge is nothing
// but the latency of its loads (as a kernel of its own that read the statistics, then part after part, it
// took 14 us at D = 64 and 20 us at D = 128 for 8 parts; the attention kernel before it 21 us on a
// 2048-token layer).
template <int D>
__device__ __forceinline__ void merge_parts(const Params& p, int cta, int ctas) {
  constexpr int kCols = D / 32;
  const int warps = blockDim.x >> 5, lane = threadIdx.x & 31;
  const int parts = p.split_parts;
  if (parts <= 1) return;
  const int rows = (p.nWork - p.split_first) * 256;
  for (int i = cta * warps + (threadIdx.x >> 5); i < rows; i += ctas * warps) {
    const int r = i >> 8, qt = (i >> 7) & 1, row = i & 127;
    int problem, bh, pr;
    item_place(p, p.split_first + r, problem, bh, pr);
    const int T = 2 * pr + qt, grow = T * 128 + row;
    if (grow >= p.N) continue;
    const int64_t slot0 = ((int64_t)r * parts * 2 + qt) * 128 + row;
    float2 ml = make_float2(0.f, 0.f);
    if (lane < parts) ml = __ldcg(p.part_ml + slot0 + lane * 256);
    float v[kMaxParts][kCols];
#pragma unroll
    for (int s = 0; s < kMaxParts; ++s)
      if (s < parts) load_part_row<D>(p, slot0 + s * 256, lane, v[s]);
    // (a part without keys of the row has the sum 0; one that met NaN has the sum NaN, and so has the row)
    float m = (ml.y != 0.f) ? ml.x : -INFINITY;
#pragma unroll
    for (int d = kMaxParts / 2; d > 0; d >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, d));
    const float mine = (ml.y != 0.f) ? ptx::ex2_approx(ml.x - m) : 0.f;
    float L = 0.f, acc[kCols];
#pragma unroll
    for (int c = 0; c < kCols; ++c) acc[c] = 0.f;
#pragma unroll
    for (int s = 0; s < kMaxParts; ++s) {
      if (s < parts) {
        const float sc = __shfl_sync(0xffffffffu, mine, s);
        L += __shfl_sync(0xffffffffu, ml.y, s) * sc;
        if (sc != 0.f) {
#pragma unroll
          for (int c = 0; c < kCols; ++c) acc[c] += v[s][c] * sc;
        }
      }
    }
    store_merged_row<D>(p, problem, bh, grow, lane, acc, (L != 0.f) ? 1.f / L : 0.f);
  }
}

// Sparse mode, before the attention kernel: one warp per work unit merges the index lists of the
// unit's query blocks into its tile list (entry = key block index | membership bits << 16,
// padded to whole K/V tiles of G entries; for the order see below).  Every list becomes a bitmap in shared
// memory (coalesced reads, one atomicOr per index), the union's set bits are enumerated 32 words
// at a time with a warp scan.  Doing this ahead of the launch keeps the in-kernel scheduler warp,
// which shares a scheduler partition with two softmax warps and is favoured over them, nearly
// idle.  A unit that is a part of an item takes the same share, by position, of every list, so
// each (query block, key block) pair belongs to exactly one part.  Indices out of range are
// reported and skipped; an unsorted list still gives a valid tile list.
//
// One warp per list fills its bitmap (a list of a small layer is nothing but the latency of its two
// dependent loads), then the first warp writes the tile list.  The first CTA also zeroes the
// launch's counters, and every CTA its unit's flag.
// PER_TILE: a list is that of one query tile of the unit (its NB query blocks), in ascending order.

// A list's unit as (item, part of it).
__device__ __forceinline__ void unit_item(const Params& p, int unit, int& w, int& part, int& parts) {
  w = unit;
  part = 0;
  parts = 1;
  if (unit >= p.split_first) {
    parts = p.split_parts;
    w = p.split_first + p.by_parts.divmod(unit - p.split_first, part);
  }
}

// Bitmap of the n-th query block of a list (whole warp).
template <int NB, bool PER_TILE>
__device__ __forceinline__ void fill_tile_bitmap(const Params& p, int list, int n, int lane, uint32_t* bm) {
  const int bit0 = PER_TILE ? (list & 1) * NB : 0;  // membership bit of the first query block
  int w, part, parts;
  unit_item(p, PER_TILE ? list >> 1 : list, w, part, parts);
  int problem, bh, pr;
  item_place(p, w, problem, bh, pr);
  const int32_t* offsets = p.offsets;
  const int32_t* kv_idx = p.kv_idx;
  if (p.problems != nullptr) {
    const ProblemEntry* pe = p.problems + problem;
    offsets = pe->offsets;
    kv_idx = pe->kv_idx;
  }
  const int W = (p.nKb + 31) >> 5;
  uint32_t* const mine = bm + n * W;
  const int g = pr * (PER_TILE ? 2 * NB : NB) + bit0 + n;
  int b = 0, e = 0;
  if (g < p.nQb) {
    const int64_t row = (int64_t)bh * p.nQb + g;
    const int32_t nnz = __ldg(offsets + (int64_t)p.B * p.H * p.nQb);
    b = __ldg(offsets + row);
    e = __ldg(offsets + row + 1);
    if (b < 0 || e < b || e > nnz || e - b > p.nKb) {
      report_error(p.status, LOSA_ERR_BAD_INDEX);
      b = e = 0;
    }
  }
  for (int i = lane; i < W; i += 32) mine[i] = 0u;
  __syncwarp();
  {
    // (a list has fewer than 2^16 entries and is cut into kMaxParts parts at most)
    const int b2 = (parts == 1) ? b : b + p.by_parts.div((e - b) * part);
    const int e2 = (parts == 1) ? e : b + p.by_parts.div((e - b) * (part + 1));
#pragma unroll 4
    for (int i = b2 + lane; i < e2; i += 32) {
      const int v = __ldg(kv_idx + i);
      if ((unsigned)v < (unsigned)p.nKb) atomicOr(&mine[v >> 5], 1u << (v & 31));
      else report_error(p.status, LOSA_ERR_BAD_INDEX);  // skipped, never used as an address
    }
  }
}

// The tile list from its query blocks' bitmaps (whole warp).
// Returns what goes into tl_count; `copy`, if not null, receives the entries as well.
template <int NB, int G, bool PER_TILE>
__device__ __forceinline__ uint32_t emit_tile_list(const Params& p, int list, int lane, const uint32_t* bm,
                                                   uint32_t* copy) {
  const int W = (p.nKb + 31) >> 5;
  const int bit0 = PER_TILE ? (list & 1) * NB : 0;
  // Order of the entries.  A key block that only ONE of the unit's two query tiles lists is
  // processed by that tile alone, at half the CTA's rate; two such blocks, one of each tile, can
  // be in flight at the same time (the tiles' chains are independent).  So the list holds first
  // the blocks both tiles list, then the single-tile blocks of tile 0 and tile 1 in alternation
  // (K/V tile by K/V tile; a class that does not fill its last K/V tile pads it), then what is
  // left of the longer class.  Within a class the blocks ascend.  Correctness does not depend on
  // the order of the key blocks.
  uint32_t* dst = p.tl_entries + (int64_t)list * p.tl_cap;
  auto put = [&](int pos, uint32_t e) {
    dst[pos] = e;
    if (copy != nullptr) copy[pos] = e;
  };
  int nb = 0, na = 0, nbb = 0;  // both, tile 0 only, tile 1 only
  for (int w0 = 0; w0 < W; w0 += 32) {
    const int wi = w0 + lane;
    uint32_t ta = 0, tb = 0;
#pragma unroll
    for (int n = 0; n < NB; ++n) {
      const uint32_t m = (wi < W) ? bm[n * W + wi] : 0u;
      if (PER_TILE) ta |= m, tb |= m;
      else if (n < NB / 2) ta |= m;
      else tb |= m;
    }
    nb += __popc(ta & tb);
    na += __popc(ta & ~tb);
    nbb += __popc(tb & ~ta);
  }
  nb = __reduce_add_sync(0xffffffffu, nb);
  na = PER_TILE ? 0 : __reduce_add_sync(0xffffffffu, na);  // (a query tile's own list has one class)
  nbb = PER_TILE ? 0 : __reduce_add_sync(0xffffffffu, nbb);
  const int s1 = (nb + G - 1) / G * G;                       // entries of the first section
  const int tA = (na + G - 1) / G, tB = (nbb + G - 1) / G;   // K/V tiles of the single-tile classes
  const int tmin = min(tA, tB);
  const int total = min(s1 + (tA + tB) * G, p.tl_cap);
  // padding: the ends of the last K/V tile of each class
  auto slot_of = [&](int k, int r) {  // position of entry r of class k (1: tile 0 only, 2: tile 1 only)
    const int t = r / G;
    return s1 + ((t < tmin) ? 2 * t + (k - 1) : 2 * tmin + (t - tmin)) * G + r % G;
  };
  if (lane < G) {
    if (nb + lane < s1 && nb + lane < total) put(nb + lane, kTlPad);
    if (na + lane < tA * G && slot_of(1, na + lane) < total) put(slot_of(1, na + lane), kTlPad);
    if (nbb + lane < tB * G && slot_of(2, nbb + lane) < total) put(slot_of(2, nbb + lane), kTlPad);
  }
  const int ragged = (p.N % p.C != 0) ? p.nKb - 1 : -1;  // the key block in which the sequence ends
  int rb = 0, ra = 0, rbb = 0;  // entries of each class emitted by earlier words (windows)
  // Up to 16 words a lane per bit and word by word (about 40 instructions each); longer ones a lane per word and
  // bit by bit (up to 32 times 25 for 32 words).  With one word, 32 blocks, the latter is a single lane's work: 1.5 us of
  // a 20 us call.
  if (W <= 16) {
    for (int wi = 0; wi < W; ++wi) {
      uint32_t memb = 0, ta = 0, tb = 0;
#pragma unroll
      for (int n = 0; n < NB; ++n) {
        const uint32_t m = bm[n * W + wi];
        if (PER_TILE) ta |= m, tb |= m;
        else if (n < NB / 2) ta |= m;
        else tb |= m;
        memb |= ((m >> lane) & 1u) << (bit0 + n);
      }
      const uint32_t both = ta & tb, a = ta & ~tb, b = tb & ~ta, below = (1u << lane) - 1u;
      if (memb != 0u) {
        const int pos = ((both >> lane) & 1u) ? rb + __popc(both & below)
                        : ((a >> lane) & 1u)  ? slot_of(1, ra + __popc(a & below))
                                              : slot_of(2, rbb + __popc(b & below));
        const int j = wi * 32 + lane;
        if (pos < p.tl_cap) put(pos, (uint32_t)j | (memb << 16) | (j == ragged ? kTlRagged : 0u));
      }
      rb += __popc(both);
      ra += __popc(a);
      rbb += __popc(b);
    }
  }
  for (int w0 = 0; W > 16 && w0 < W; w0 += 32) {
    const int wi = w0 + lane;
    uint32_t m[NB], ta = 0, tb = 0;
#pragma unroll
    for (int n = 0; n < NB; ++n) {
      m[n] = (wi < W) ? bm[n * W + wi] : 0u;
      if (PER_TILE) ta |= m[n], tb |= m[n];
      else if (n < NB / 2) ta |= m[n];
      else tb |= m[n];
    }
    uint32_t cls[3] = {ta & tb, ta & ~tb, tb & ~ta};
    int incl[3], tot[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      incl[k] = __popc(cls[k]);
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl[k], d);
        if (lane >= d) incl[k] += t;
      }
      tot[k] = __shfl_sync(0xffffffffu, incl[k], 31);
    }
    const int base[3] = {rb, ra, rbb};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      uint32_t u = cls[k];
      int r = base[k] + incl[k] - __popc(u);  // rank of this lane's first entry within its class
      while (u) {
        const int bit = __ffs(u) - 1;
        u &= u - 1;
        uint32_t memb = 0;
#pragma unroll
        for (int n = 0; n < NB; ++n) memb |= ((m[n] >> bit) & 1u) << (bit0 + n);
        const int pos = (k == 0) ? r : slot_of(k, r);
        const int j = wi * 32 + bit;
        if (pos < p.tl_cap) put(pos, (uint32_t)j | (memb << 16) | (j == ragged ? kTlRagged : 0u));
        ++r;
      }
    }
    rb += tot[0];
    ra += tot[1];
    rbb += tot[2];
  }
  const uint32_t word = (uint32_t)(total / G) | ((nb + na > 0) ? kHdrHas : 0u) | ((nb + nbb > 0) ? 2u * kHdrHas : 0u) |
                        ((nb == 0 && tmin > 0) ? kHdrLate : 0u);
  if (lane == 0) p.tl_count[list] = (int32_t)word;
  return word;
}

template <int NB, int G, bool PER_TILE>
__global__ void __launch_bounds__(32 * NB) build_tile_lists_kernel(const Params p) {
  extern __shared__ uint32_t bm[];  // [NB][W] bitmaps
  ptx::grid_launch_dependents();
  ptx::grid_dependency_wait();
  const int lane = threadIdx.x & 31, n = threadIdx.x >> 5;
  const int list = blockIdx.x, unit = PER_TILE ? list >> 1 : list;
  if (list == 0 && threadIdx.x < kCounters) p.work_counter[threadIdx.x] = 0;
  fill_tile_bitmap<NB, PER_TILE>(p, list, n, lane, bm);
  __syncthreads();
  if (n != 0) return;
  emit_tile_list<NB, G, PER_TILE>(p, list, lane, bm, nullptr);
  if (lane == 0) p.redo_flag[unit] = 0;
}

// Tensor maps of a batched launch were written to the workspace by a kernel, over those of an earlier call: those that
// the tile kernel uses, a lane each (whole warp).
template <int D, int C_, bool HAS_V>
__device__ __forceinline__ void acquire_tile_maps(const ProblemEntry* pe, int lane) {
  const CUtensorMap* m = &pe->map_q;
  if (lane == 1) m = (D == 128) ? &pe->map_kh : &pe->map_k;
  if (lane == 2) m = (D == 128) ? &pe->map_k64 : &pe->map_k128;  // (equal to map_k where there is no such box)
  if (lane == 3) m = &pe->map_v;
  if (lane == 4) m = &pe->map_v128;
  if (lane < (HAS_V ? 5 : 3)) ptx::tensormap_acquire(m);
}

#include "losa_attn_tile.cuh"

#undef LOSA_WAIT_RELAXED
#undef LOSA_WAIT

// ---------------------------------------------------------------------------- host side

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* sym = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(sym);
  }
  return fn;
}

// bf16 [B,H,N,D] tensor, box = [box_rows][64] with 128-byte swizzle; rows >= N read as zero.
int make_map(CUtensorMap* m, const void* base, const Geometry& g, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) {
    set_cuda_error(cudaErrorUnknown, "cuTensorMapEncodeTiled entry point");
    return LOSA_ERR_CUDA;
  }
  const cuuint64_t dims[4] = {(cuuint64_t)g.D, (cuuint64_t)g.N, (cuuint64_t)g.H, (cuuint64_t)g.B};
  const cuuint64_t strides[3] = {(cuuint64_t)g.sn * 2, (cuuint64_t)g.sh * 2, (cuuint64_t)g.sb * 2};
  const cuuint32_t box[4] = {64, (cuuint32_t)box_rows, 1, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims,
                        strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_cuda_error(cudaErrorInvalidValue, "cuTensorMapEncodeTiled");
    return LOSA_ERR_CUDA;
  }
  return LOSA_OK;
}

// The tensor maps of one problem.  Boxes: the key blocks (kh: at most 64 keys, half a K/V tile), and
// for smaller blocks than a tile, which is copied whole where its blocks are consecutive, 64 and 128
// keys (k64 with 32-key blocks only, k128 at head dimension 64 only).  v null: the mass pass, which has none.
int make_maps(ProblemEntry* e, const Geometry& g, const void* q, const void* k, const void* v) {
  int rc;
  if ((rc = make_map(&e->map_q, q, g, 128)) != LOSA_OK) return rc;
  if ((rc = make_map(&e->map_k, k, g, g.C)) != LOSA_OK) return rc;
  e->map_v = e->map_k;
  if (v && (rc = make_map(&e->map_v, v, g, g.C)) != LOSA_OK) return rc;
  e->map_kh = e->map_k64 = e->map_k128 = e->map_k;
  e->map_v128 = e->map_v;
  if (g.C > 64 && (rc = make_map(&e->map_kh, k, g, 64)) != LOSA_OK) return rc;
  if (g.C < 64 && (rc = make_map(&e->map_k64, k, g, 64)) != LOSA_OK) return rc;
  if (g.C < 128 && g.D == 64 && (rc = make_map(&e->map_k128, k, g, 128)) != LOSA_OK) return rc;
  if (g.C < 128 && v && (rc = make_map(&e->map_v128, v, g, 128)) != LOSA_OK) return rc;
  return LOSA_OK;
}

// The merge of the partial units, a launch of its own behind the tile kernel (3.5 us).
constexpr int kMergeThreads = 128;
template <int D>
__global__ void __launch_bounds__(kMergeThreads) merge_parts_kernel(const Params p) {
  ptx::grid_dependency_wait();
  merge_parts<D>(p, blockIdx.x, gridDim.x);
  if (p.one_wave && blockIdx.x == 0 && threadIdx.x < 32) {
    // (how many units were recomputed: elsewhere the tile kernel counts them)
    constexpr int kLists = tile_lists_per_unit(D);
    int n = 0;
    for (int u = threadIdx.x; u < p.nUnits; u += 32)
      n += (p.redo_flag[u * kLists] | p.redo_flag[u * kLists + kLists - 1]) != 0 ? 1 : 0;
    n = __reduce_add_sync(0xffffffffu, n);
    if (threadIdx.x == 0) *p.redo_count = n;
  }
}

// Zeroes the counters and the units' flags of a launch that no other kernel precedes (a kernel and
// not a memset, so that the attention kernel can be launched as its dependent: 3 us of that kernel's
// set-up overlap).
constexpr int kInitThreads = 256;
__global__ void __launch_bounds__(kInitThreads) init_counters_kernel(int* counters, int* flags, int n) {
  ptx::grid_launch_dependents();
  ptx::grid_dependency_wait();  // (the stream's call before may still use the workspace)
  if (blockIdx.x == 0 && threadIdx.x < kCounters) counters[threadIdx.x] = 0;
  for (int64_t i = (int64_t)blockIdx.x * kInitThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kInitThreads)
    flags[i] = 0;
}

// Part of a batched launch's table, carried in the kernel's parameters: the call reads its host
// arguments before it returns, without a copy from pageable memory (which staged and waited, 20 us).
constexpr int kTableChunk = 8;
struct ProblemChunk {
  ProblemEntry e[kTableChunk];
};
__global__ void __launch_bounds__(256)
write_problems_kernel(const __grid_constant__ ProblemChunk chunk, ProblemEntry* table, int n) {
  ptx::grid_launch_dependents();
  ptx::grid_dependency_wait();
  const uint4* src = reinterpret_cast<const uint4*>(&chunk);
  uint4* dst = reinterpret_cast<uint4*>(table);
  for (int i = threadIdx.x; i < n * (int)(sizeof(ProblemEntry) / sizeof(uint4)); i += blockDim.x) dst[i] = src[i];
}

// Configures the tile kernel on the current device (once) and says how many clusters - pairs of CTAs, or (PAIR =
// false) CTAs - a call may have at work there.
// `ctas`: of a cluster.
template <int D, int R, int C_, int MODE, bool PAIR, bool ONE>
int configure_tile(const DeviceState& on, int ctas, int* clusters, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr) {
  using L = Lay;
  constexpr size_t smem = (size_t)tile_nq(D, MODE) * 256 * D + (size_t)(tile_nk(MODE) + tile_nv(MODE)) * kTileStage +
                          (D == 64 ? kTileOnes : 0) + sizeof(TileControl);
  static_assert(smem <= 227 * 1024, "shared memory of one CTA");
  auto kern = losa_tile_kernel<D, R, C_, MODE, PAIR, ONE>;
  // how many clusters of so many CTAs the device holds at once
  static std::atomic<int> max_on[kMaxDevices][kMaxClusterCtas + 1];
  const int dev = on.ordinal, sms = on.sm_count;
  *cfg = {};
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = ctas;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg->blockDim = dim3(L::kThreads, 1, 1);
  cfg->dynamicSmemBytes = smem;
  cfg->attrs = attr;
  cfg->numAttrs = ctas > 1 ? 2 : 1;
  if (max_on[dev][ctas].load(std::memory_order_acquire) == 0) {
    // the in-kernel register reallocation must fit the registers the CTA is launched with
    cudaFuncAttributes fa;
    LOSA_CUDA_TRY(cudaFuncGetAttributes(&fa, kern));
    if (fa.numRegs * L::kThreads < 128 * L::kRegsUtility + 32 * L::kSoftmaxWarps * L::kRegsSoftmax) {
      set_cuda_error(cudaErrorLaunchOutOfResources, "register budget of losa_tile_kernel");
      return LOSA_ERR_UNSUPPORTED;
    }
    LOSA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int n = sms;
    if (ctas > 1) {
      LOSA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
      cudaLaunchConfig_t ask = *cfg;
      ask.gridDim = dim3(ctas * kMaxPersistentCtas, 1, 1);
      ask.attrs = attr + 1;
      ask.numAttrs = 1;
      LOSA_CUDA_TRY(cudaOccupancyMaxActiveClusters(&n, kern, &ask));
    }
    max_on[dev][ctas].store(n < 1 ? -1 : n, std::memory_order_release);
  }
  const int n = max_on[dev][ctas].load(std::memory_order_acquire);
  *clusters = min(min(sms / ctas, n), kMaxPersistentCtas);
  if (n >= 1) return LOSA_OK;
  set_cuda_error(cudaErrorLaunchOutOfResources, "no resident cluster of losa_tile_kernel");
  return LOSA_ERR_UNSUPPORTED;
}

// Work slots of a call: pairs of CTAs, one for the two query tiles of a work item together (head dimension 128, on a
// cluster) or one CTA for each (head dimension 64).  Head dimension 128 with 64-row query blocks, 9600 tokens, 12 heads,
// against two query tiles on one CTA: dense 557 -> 487 us, sparse 457 -> 419, masses 474 -> 359, construction step 703 -> 538.
template <int D, int R, int C_, int MODE>
int work_slots(const DeviceState& dev, int* slots) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  int n = 0;
  const int rc = configure_tile<D, R, C_, MODE, D == 128, false>(dev, D == 128 ? 2 : 1, &n, &cfg, attr);
  *slots = (D == 128) ? n : max(1, n / 2);
  return rc;
}

// How a call's work items are spread over the slots.
struct Waves {
  int slots, units, split_first, parts;
  int ctas;  // of a cluster
  bool one_wave, in_cluster;
  // kernels: the tile kernel, ahead of it what prepares several waves, behind it the merge of parts that share no cluster
  int launches() const { return 1 + (one_wave ? 0 : 1) + (parts > 1 && !in_cluster ? 1 : 0); }
};

template <int D, int R, int C_, int MODE>
int plan_waves(int items, int nKb, const DeviceState& dev, Waves* waves) {
  constexpr bool kPair = D == 128;
  constexpr int kTileCtas = kPair ? 2 : 1;
  int rc, slots;
  if ((rc = work_slots<D, R, C_, MODE>(dev, &slots)) != LOSA_OK) return rc;
  Waves w = {slots, items, items, 1, kTileCtas, false, false};
  // The items of the last, partly filled wave of the persistent grid (all items, if there are
  // fewer than slots) are cut into parts of the key range, so that the wave ends after 1/parts of
  // an item; their partial results are merged by their clusters or by a launch behind.  Attention output
  // only: the mass epilogue needs a row's final statistics inside the kernel.
  constexpr bool kAttnOnly = (MODE == kDense || MODE == kSparse);
  if (kAttnOnly) {
    const int rest = (items < slots) ? items : items % slots;
    int parts = rest > 0 ? slots / rest : 1;
    parts = min(min(parts, kMaxParts), nKb);
    if (parts >= 2 && rest == items) {
      // A single wave: the parts of an item in one cluster (at head dimension 64 of each of its query tiles), where the
      // device holds all of them at once - of 16 CTAs 7, of 8 15, of 6 22, of 4 33, of 3 45.  Elsewhere a launch behind
      // merges them: with fewer parts, which would fit, calls were up to 30 % faster, but a part's largest weights round to
      // themselves, and the error against 64 bits grew (264 tokens, 4 heads, D = 64, 8 parts / 7: 1.7e-3 / 1.8e-3).
      int n = 0;
      cudaLaunchConfig_t cfg;
      cudaLaunchAttribute attr[2];
      rc = configure_tile<D, R, C_, MODE, kPair, true>(dev, kTileCtas * parts, &n, &cfg, attr);
      if (rc == LOSA_ERR_CUDA) (void)cudaGetLastError();  // (a device that cannot say how many it holds: none)
      if (rc == LOSA_OK && n >= rest * (kPair ? 1 : 2)) {
        w.in_cluster = true;
        w.ctas = kTileCtas * parts;
      }
    }
    if (parts >= 2) {
      w.split_first = items - rest;
      w.parts = parts;
      w.units = w.split_first + rest * parts;
    }
  }
  w.one_wave = w.units <= slots;
  *waves = w;
  return LOSA_OK;
}

template <int D, int R, int C_, int MODE>
int launch_t(const Geometry& g, const void* q, const void* k, const void* v, Params prm,
             const DeviceState& dev, cudaStream_t st) {
  constexpr bool kPair = D == 128;
  ProblemEntry maps;
  Waves w;
  int rc;
  if ((rc = make_maps(&maps, g, q, k, MODE != kMass ? v : nullptr)) != LOSA_OK) return rc;
  if ((rc = plan_waves<D, R, C_, MODE>(prm.nWork, prm.nKb, dev, &w)) != LOSA_OK) return rc;
  const int slots = w.slots;
  prm.nUnits = w.units;
  prm.split_first = w.split_first;
  prm.split_parts = w.parts;
  prm.in_cluster = w.in_cluster ? 1 : 0;
  prm.one_wave = w.one_wave ? 1 : 0;
  prm.by_parts = Divisor(prm.split_parts);
  prm.by_pairs = Divisor(prm.nPairs);
  prm.by_heads = Divisor(prm.H);
  prm.by_problem = Divisor(prm.B * prm.H);
  // Every kernel is launched as a dependent of the one before.
  if (prm.one_wave) {
    rc = LOSA_OK;
  } else if (MODE == kSparse) {
    constexpr int kLists = tile_lists_per_unit(D);
    constexpr int kBlocks = 256 / R / kLists;  // query blocks of a list
    const size_t bm_bytes = (size_t)kBlocks * ((prm.nKb + 31) / 32) * sizeof(uint32_t);  // <= 32 KB
    rc = launch(build_tile_lists_kernel<kBlocks, 128 / C_, kLists == 2>, dim3(prm.nUnits * kLists), 32 * kBlocks, bm_bytes,
                st, true, prm);
  } else {
    rc = launch(init_counters_kernel, dim3(min(slots, (prm.nUnits + 4 * kInitThreads - 1) / (4 * kInitThreads))),
                kInitThreads, 0, st, true, prm.work_counter, prm.redo_flag, prm.nUnits);
  }
  if (rc != LOSA_OK) return rc;
  auto launch_tile = [&](auto one) -> int {
    int n = 0;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    const int rc = configure_tile<D, R, C_, MODE, kPair, decltype(one)::value>(dev, w.ctas, &n, &cfg, attr);
    if (rc != LOSA_OK) return rc;
    cfg.gridDim = dim3(2 * min(slots, prm.nUnits), 1, 1);
    cfg.stream = st;
    LOSA_CUDA_TRY(cudaLaunchKernelEx(&cfg, losa_tile_kernel<D, R, C_, MODE, kPair, decltype(one)::value>, maps.map_q,
                                     kPair ? maps.map_kh : maps.map_k, maps.map_v, kPair ? maps.map_k64 : maps.map_k128,
                                     maps.map_v128, prm));
    return LOSA_OK;
  };
  if ((rc = prm.one_wave ? launch_tile(std::true_type()) : launch_tile(std::false_type())) != LOSA_OK) return rc;
  if (prm.stall || prm.split_parts == 1 || prm.in_cluster) return LOSA_OK;
  constexpr int kRows = kMergeThreads / 32;  // a warp per row
  return launch(merge_parts_kernel<D>, dim3((prm.nWork - prm.split_first) * (256 / kRows)), kMergeThreads, 0, st, true, prm);
}

// (128 x 32: the paper's own block geometry)
#define LOSA_GEOMETRIES(X) \
  X(128, 128, 128) X(64, 64, 64) X(128, 128, 32) X(64, 128, 32) X(128, 64, 64) X(64, 128, 128) X(128, 128, 64) X(64, 128, 64)

template <int MODE>
int dispatch(const Geometry& g, const void* q, const void* k, const void* v, const Params& prm,
             const DeviceState& dev, cudaStream_t st) {
#define LOSA_CASE(d, r, c) \
  if (g.D == d && g.R == r && g.C == c) return launch_t<d, r, c, MODE>(g, q, k, v, prm, dev, st);
  LOSA_GEOMETRIES(LOSA_CASE)
#undef LOSA_CASE
  return LOSA_ERR_UNSUPPORTED;
}

template <int MODE>
int plan_of(const Geometry& g, int items, const DeviceState& dev, Waves* w) {
#define LOSA_CASE(d, r, c) \
  if (g.D == d && g.R == r && g.C == c) return plan_waves<d, r, c, MODE>(items, g.nKb, dev, w);
  LOSA_GEOMETRIES(LOSA_CASE)
#undef LOSA_CASE
  return LOSA_ERR_UNSUPPORTED;
}

int plan_of(AttnMode mode, const Geometry& g, const DeviceState& dev, Waves* w) {
  // (calls of more items than the mask holds are refused)
  const int items = (int)std::min<int64_t>((int64_t)g.B * g.H * g.nPairs, kTlItemMask);
  switch (mode) {
    case kDense: return plan_of<kDense>(g, items, dev, w);
    case kSparse: return plan_of<kSparse>(g, items, dev, w);
    case kMass: return plan_of<kMass>(g, items, dev, w);
    case kFused: return plan_of<kFused>(g, items, dev, w);
  }
  return LOSA_ERR_UNSUPPORTED;
}

}  // namespace


namespace {
size_t part_o_bytes(const Geometry& g) {
  return (size_t)kMaxPersistentCtas * 2 * 128 * (size_t)g.D * sizeof(float);
}
// the last wave's items are cut into at most one unit per CTA
int64_t max_units(const Geometry& g, int n_prob) {
  return (int64_t)n_prob * g.B * g.H * g.nPairs + kMaxPersistentCtas;
}
int tile_list_cap(const Geometry& g) { return (g.nKb + 16 + 31) / 32 * 32; }  // union <= nKb, + padding of three sections
int64_t max_lists(const Geometry& g, int n_prob) { return max_units(g, n_prob) * tile_lists_per_unit(g.D); }
size_t redo_flag_bytes(const Geometry& g, int n_prob) {  // (one wave: a word per tile list, two per slot at most)
  return ((size_t)max_units(g, n_prob) * sizeof(int32_t) + 255) / 256 * 256;
}
size_t tl_count_bytes(const Geometry& g, int n_prob) {
  return ((size_t)max_lists(g, n_prob) * sizeof(int32_t) + 255) / 256 * 256;
}
size_t tl_entries_bytes(const Geometry& g, int n_prob) {
  return ((size_t)max_lists(g, n_prob) * tile_list_cap(g) * sizeof(uint32_t) + 255) / 256 * 256;
}
}  // namespace

void arm_stalled_launch(uint32_t polls) { g_stall_polls.store(polls); }

// Work slots that a call of this kind occupies on the current device, for callers that
// want to know how the work items are spread (which of them the last wave cuts into parts); 0 where it cannot run.
int attn_work_slots(AttnMode mode, const Geometry& g, const DeviceState& dev) {
  Waves w;
  return plan_of(mode, g, dev, &w) == LOSA_OK ? w.slots : 0;
}

// Kernels that such a call launches; 0 where it cannot run.
int attn_launches(AttnMode mode, const Geometry& g, const DeviceState& dev) {
  Waves w;
  if ((int64_t)g.B * g.H * g.nPairs > (int64_t)kTlItemMask) return 0;
  return plan_of(mode, g, dev, &w) == LOSA_OK ? w.launches() : 0;
}

size_t attn_workspace_bytes(AttnMode mode, const Geometry& g, int n_prob) {
  // attention output: counter, then one slot per partial unit (at most one per CTA) holding the
  // rows' (max, sum) and unnormalised O of both query tiles
  if (mode == kDense || mode == kSparse) {
    size_t bytes = kCounterBytes + kPartMlBytes + part_o_bytes(g);
    // sparse: the units' merged tile lists (count per unit, then tl_cap entries per unit)
    if (mode == kSparse) bytes += tl_count_bytes(g, n_prob) + tl_entries_bytes(g, n_prob);
    // batched launch: the table of the problems' tensor maps and pointers
    if (n_prob > 1) bytes += (size_t)n_prob * sizeof(ProblemEntry);
    // the work units' (or their tile lists') flags
    bytes += redo_flag_bytes(g, n_prob);
    return bytes;
  }
  // counter, per-CTA table of sums per row and key block (of both query tiles of an item), the units' flags
  return kCounterBytes + (size_t)kMaxPersistentCtas * 2 * (size_t)g.nKb * 128 * sizeof(float2) + redo_flag_bytes(g, 1);
}

// Batched launch (n_prob > 1, attention-only modes): `layers` is a host array of n_prob problems of
// the geometry g; q, k, v, offsets, kv_idx and o are then ignored.
int launch_attn(AttnMode mode, const Geometry& g, const void* q, const void* k, const void* v,
                const int32_t* offsets, const int32_t* kv_idx, void* o, int o_dtype, float* mass,
                float* lse, void* ws, cudaStream_t st, int n_prob, const losa_layer_t* layers) {
  Params prm;
  prm.B = g.B;
  prm.H = g.H;
  prm.N = g.N;
  prm.C = g.C;
  prm.nQb = g.nQb;
  prm.nKb = g.nKb;
  prm.nQt = g.nQt;
  prm.nPairs = g.nPairs;
  if ((int64_t)n_prob * g.B * g.H * g.nPairs > (int64_t)kTlItemMask)
    return LOSA_ERR_UNSUPPORTED;  // the tile list's item headers hold 24 bits
  prm.nWork = n_prob * g.B * g.H * g.nPairs;
  prm.nProb = n_prob;
  prm.problems = nullptr;
  prm.offsets = offsets;
  prm.kv_idx = kv_idx;
  prm.o = o;
  prm.o_f32 = (o_dtype == LOSA_DTYPE_F32) ? 1 : 0;
  prm.sb = g.sb;
  prm.sh = g.sh;
  prm.sn = g.sn;
  prm.mass = mass;
  prm.lse = lse;
  // workspace: [0, 256) counters, then (mass modes) per-CTA tables
  prm.work_counter = static_cast<int*>(ws);
  prm.table = reinterpret_cast<float2*>(static_cast<char*>(ws) + kCounterBytes);
  prm.part_ml = reinterpret_cast<float2*>(static_cast<char*>(ws) + kCounterBytes);
  prm.part_o = reinterpret_cast<float*>(static_cast<char*>(ws) + kCounterBytes + kPartMlBytes);
  {
    char* tl = static_cast<char*>(ws) + kCounterBytes + kPartMlBytes + part_o_bytes(g);
    prm.tl_count = reinterpret_cast<int32_t*>(tl);
    prm.tl_entries = reinterpret_cast<uint32_t*>(tl + tl_count_bytes(g, n_prob));
    prm.tl_cap = tile_list_cap(g);
    if (n_prob > 1) {
      // the problems' table, behind the tile lists (dense mode has none), written before the launch
      char* tab = tl + (mode == kSparse ? tl_count_bytes(g, n_prob) + tl_entries_bytes(g, n_prob) : 0);
      ProblemChunk chunk;
      for (int i0 = 0; i0 < n_prob; i0 += kTableChunk) {
        const int n = min(kTableChunk, n_prob - i0);
        for (int i = 0; i < n; ++i) {
          const losa_layer_t& l = layers[i0 + i];
          const int rc = make_maps(&chunk.e[i], g, l.q, l.k, l.v);
          if (rc != LOSA_OK) return rc;
          chunk.e[i].o = l.o;
          chunk.e[i].offsets = l.offsets;
          chunk.e[i].kv_idx = l.kv_idx;
        }
        const int rc = launch(write_problems_kernel, dim3(1), 256, 0, st, true, chunk,
                              reinterpret_cast<ProblemEntry*>(tab) + i0, n);
        if (rc != LOSA_OK) return rc;
      }
      prm.problems = reinterpret_cast<const ProblemEntry*>(tab);
      q = layers[0].q;  // the kernel's parameter maps are unused but must be valid
      k = layers[0].k;
      v = layers[0].v;
    }
    prm.redo_count = prm.work_counter + 1;
    prm.redo_flag = reinterpret_cast<int*>(
        tl + (mode == kSparse ? tl_count_bytes(g, n_prob) + tl_entries_bytes(g, n_prob) : 0) +
        (n_prob > 1 ? (size_t)n_prob * sizeof(ProblemEntry) : 0));
    if (mode == kFused || mode == kMass)  // behind the table
      prm.redo_flag = reinterpret_cast<int*>(reinterpret_cast<char*>(prm.table) +
                                             (size_t)kMaxPersistentCtas * 2 * (size_t)g.nKb * 128 * sizeof(float2));
  }
  prm.cap_part_rows = (long long)kMaxPersistentCtas * 2 * 128;
  prm.cap_table_floats = (long long)g.nKb * 256;
  prm.cap_mass = (long long)g.B * g.H * g.nQb * g.nKb;
  prm.cap_lse = (long long)g.B * g.H * g.N;
  prm.cap_units = (long long)max_lists(g, n_prob);
  prm.scale_log2 = g.scale * kLog2e;
  int rc = LOSA_OK;
  const DeviceState* dev = device_state(&rc);
  if (!dev) return rc;
  prm.status = dev->status_dev;
  // one-shot diagnostic armed by losa_debug_stall_next_launch()
  const uint32_t stall_polls = g_stall_polls.exchange(0u);
  prm.stall = stall_polls > 0u ? 1 : 0;
  prm.wait_polls = stall_polls > 0u ? stall_polls : ptx::kWaitPolls;
  switch (mode) {
    case kDense: return dispatch<kDense>(g, q, k, v, prm, *dev, st);
    case kSparse: return dispatch<kSparse>(g, q, k, v, prm, *dev, st);
    case kMass: return dispatch<kMass>(g, q, k, v, prm, *dev, st);
    case kFused: return dispatch<kFused>(g, q, k, v, prm, *dev, st);
  }
  return LOSA_ERR_INVALID_ARG;
}

}  // namespace losa
