// The tile kernel: one query tile per CTA, for dense and block-sparse forward (Eq. 4), the fused
// construction step (dense forward plus the block masses of Eq. 1) and the mass pass.  Included by
// losa_attn.cu, inside its namespace.
//
// Each CTA's tensor memory holds one O and THREE S buffers used in turn, so that the chain
// S -> softmax -> O += P V of one key tile overlaps the chains of the next two.
//
// Head dimension 128 (PAIR): a work item is a pair of consecutive query
// tiles, run by a PAIR of CTAs (a cluster of two, one SM each) that own one of the two tiles each and
// multiply together: every MMA is a tcgen05.mma.cta_group::2 over 256 rows (128 per CTA), issued by one
// thread of the first CTA, whose B operand is split between the two CTAs' shared memories - for
// S = Q K^T each CTA loads 64 of the tile's 128 keys, for O += P V each loads the 64 head-dimension
// columns of V that it accumulates into.  A K/V tile is thus fetched once for both query tiles, each
// SM reads 96 B per clock from shared memory instead of 128 (the limit), and half as many MMAs are
// issued.  A key tile that only one of the two query tiles lists is multiplied for both and masked to
// P = 0 for the other.
//
// Head dimension 64: the two query tiles of an item are two units, drawn one by one by single CTAs.
// K and V stages are 16 KB there too (128 keys of 64 columns), L2 delivers the second copy of each, and
// a query tile's list holds only what its own query blocks list.  Against two query tiles per CTA with
// rotating score buffers (every warp walking one list, 3344 cycles per key tile and two query tiles
// against 2048 of the special-function unit): 17776 tokens, 8 heads 893 -> 736 us dense, 1118 -> 887 us
// with the masses, 833 -> 761 us masses alone.
//
// Per CTA: warp 0 copies (its query tile, its share of every K and V tile), warp 3 of the (first) CTA
// publishes the work, warps 1 and 2 of the first CTA issue every S = Q K^T and every O += P V, and 16 softmax warps turn S into P: two threads per query
// row (64 columns each), key tiles taken alternately by two groups of eight warps, so that each
// group has two tile periods for one tile.  The exponentials are taken against a reference that
// never moves within a work unit (the row maximum over the first key tile the row attends to,
// handed from the group that meets that tile to the other); a unit whose scores outgrow it is run again
// by the same CTAs, against the logarithm of the row sums if these are still finite (scores up to about 80 nats above
// the first tile's) - no row's maximum is above that, nor further below than the logarithm of its keys - and else
// first for its rows' maxima and then against these.  (A launch of its own for such units
// cost every call 4 - 6 us and a launch; 2048 tokens, 4 heads, D = 64: 26.9 -> 21.5 us with the launch of the lists
// gone as well.  16384 tokens, 12 heads, every unit 60 nats above its first tiles from the third on, us with that launch /
// with a pass for the maxima / without: D = 128 dense 2600 / 3090 / 2390, masses 2040 / 2490 / 1760; D = 64 dense
// 2130 / 2220 / 1730, masses 2575 / 2140 / 1640.)
//
// Barriers that both CTAs feed (operands landed, P written, O read out, tile-list chunk consumed)
// live in the first CTA; barriers that the MMAs' completion feeds in both CTAs are reached with a
// commit to both.  Every wait is bounded; on the way out both CTAs meet at the cluster's barrier,
// so that neither leaves while the other may still signal into its shared memory.

constexpr int kTileMaxNK = 8, kTileNV = 7;   // K and V stages of 16 KB per CTA, at most
// Query tiles in shared memory: two where there is room, so that the next unit's keys and its first scores need not
// wait for this one's last.  The mass pass has no V: two query tiles at head dimension 128 too, and more K stages.
// (Two query tiles and five V stages in the other modes there: within the noise, the construction step 1 % slower.)
__host__ __device__ constexpr int tile_nq(int D, int mode) { return (D == 64 || mode == kMass) ? 2 : 1; }
__host__ __device__ constexpr int tile_nk(int mode) { return mode == kMass ? 8 : 4; }
__host__ __device__ constexpr int tile_nv(int mode) { return mode == kMass ? 0 : kTileNV; }
constexpr int kTileStage = 16384;
// Head dimension 64: one K step (16 keys) of 64 more columns of V, all ones, behind the V stages.  Every
// O += P V reads 16 of these columns, so that the row sums of P come out of it as columns of O: 64 x 80
// instead of 64 x 64 per K step on the tensor cores, which are idle half of the time, and 96 warp instructions per 64
// scores fewer on the softmax warps (64 adds and the moves that they need, of 405).  At head dimension 128 tensor
// memory has no columns left.
constexpr int kTileOnes = 2048;
#ifndef LOSA_POLY_OF
#define LOSA_POLY_OF 8
#endif
#ifndef LOSA_POLY_OF_MASS
#define LOSA_POLY_OF_MASS 4
#endif
constexpr float kTileSafeLow = 8.6736173798840355e-19f;  // 2^-60
// A row sum in this range says how high the row's scores go.  (A score that left the exponential's own range counts as
// infinite or 2^127; one that fell below it as zero.)
constexpr float kTileKnownLow = 7.8886090522101181e-31f, kTileKnownHigh = 1.3292279957849159e+36f;  // 2^-100, 2^120

struct TileControl {
  uint64_t q_full[2], q_empty[2];
  uint64_t k_full[kTileMaxNK], k_empty[kTileMaxNK];
  uint64_t v_full[kTileNV], v_empty[kTileNV];
  uint64_t s_full[3], p_ready[3], pv_done[3];  // per score buffer
  uint64_t o_done[4], o_free;
  uint64_t hdr_full[2], hdr_empty[2], hdr_next;
  uint64_t tl_full[kTlChunks], tl_empty[kTlChunks];
  uint64_t pair_bar[8];    // per (group, lane quarter): the two halves of a row
  uint64_t ref_full[2][2], ref_empty[2][2];  // [set][query block of the query tile]
  uint64_t item_bar;       // all softmax warps of the CTA, at the end of an item
  uint64_t l_full[4];      // the group that is done with a unit first has left its rows' partial sums
  uint64_t fold_bar;       // ... and after the fused step's masses are folded out of the table
  uint64_t drain;
  alignas(16) uint32_t hdr[4][12];  // (TILE_HDR_PUT)
  alignas(16) uint32_t tl[kTlChunks * 32];  // (read in groups of up to four entries with one vector load)
  uint32_t redo_mark[4];   // per unit (of four in turn): 1 + the tile list of one that outgrew its reference
  uint32_t redo_need[4];   // ... whether its rows' maxima have to be taken first (directly behind the marks)
  uint32_t cluster_marked; // one_wave: a unit of this cluster has to be run again
  uint32_t redo_queue[4];  // the scheduler's: units to be run again (kRedoList ...), and (1 + the one whose maxima were
  alignas(16) uint32_t redo_state[4];  // taken last; head and tail of the queue; whether there ever was one)
  uint8_t seen[4][16];     // a warp met keys that its rows attend to
  uint8_t max_uses[16];    // a warp's uses of item_bar, where only units that are run again use it
  float redo_ref[4][128];  // per unit (of four in turn): what its rows are run again against
  float half_max[2][2][128];  // ... over each half of the tile it is taken from
  float ref[2][128];       // the rows' reference, from the group that met the first tile to the other
  float xch[2][8][128];    // the rows' partial sums at the end of an item (two sets, used in turn):
                           // four of the rounded weights, four of the unrounded exponentials (fused step)
  uint32_t tmem_base;
  int abort_flag;
};

// Key blocks of a unit in the dense modes.
__device__ __forceinline__ void tile_key_range(const Params& p, uint32_t ent, int& jlo, int& jhi) {
  const int part = (int)((ent >> 24) & 7u);
  jlo = (ent & kTlPartial) ? p.by_parts.div(p.nKb * part) : 0;
  jhi = (ent & kTlPartial) ? p.by_parts.div(p.nKb * (part + 1)) : p.nKb;
}

// (a barrier whose data the other CTA of a pair may have written)
#define TILE_WAIT(bar, parity)                                                             \
  do {                                                                                     \
    if (!(PAIR ? ptx::mbar_wait_cluster((bar), (parity), &ctl->abort_flag, p.wait_polls)   \
               : ptx::mbar_wait((bar), (parity), &ctl->abort_flag, p.wait_polls))) {       \
      ctl->abort_flag = 1;                                                                 \
      report_error(p.status, LOSA_ERR_TIMEOUT);                                            \
      goto teardown;                                                                       \
    }                                                                                      \
  } while (0)

// What the roles are told.  Per work unit the scheduler of the first CTA publishes a header in both
// CTAs: the item, and a word with the number of K/V tiles (kHdrTiles), which of the two query tiles
// lists any (kHdrHas), and whether query tile 1 lists its first one in the unit's second tile instead
// of its first (kHdrLate).  The dense modes need no more than the unit's share of the key range, which
// is in the header as well (worked out by every warp with two 64-bit divisions, a unit of 4 K/V tiles
// took 0.5 us longer: 37 heads of 512 tokens, D = 64, 10.1 -> 9.5 us; of 2048 55.2 -> 53.1, D = 128 83.4 -> 80.5).
// In the sparse mode the unit's tile list follows in chunks of 32 entries - GROUPS of
// kG = 128 / C, one per K/V tile, a unit beginning with a chunk of its own - which only the producers
// and the softmax warps read, the latter only the tiles they work on.  (When every warp walked one
// list of headers and tiles entry by entry, in the dense modes too, that took more instructions per
// tile than the exponentials: 529 warp instructions per 64 scores of a warp, 224 of them arithmetic.)
//
// A unit in the scheduler's queue: its tile list, which of redo_ref is its own, whether its rows' maxima are needed.
constexpr uint32_t kRedoList = 0x03ffffffu, kRedoSetShift = 28u, kRedoNeed = 1u << 30;
static_assert(2u * (kTlItemMask + 1u) - 1u <= kRedoList, "a tile list's number");

// Next header (whole warp); `nu` is the warp's unit counter.  N: how much of it the role reads, in groups of
// four words.
#define TILE_HDR_NEXT(hdr_, N)                                                             \
  do {                                                                                     \
    if (ONE && nu == 1u && unit_over()) goto teardown;                                     \
    const uint32_t s_ = nu & 1u;                                                           \
    TILE_WAIT(&ctl->hdr_full[s_], (nu >> 1) & 1u);                                         \
    _Pragma("unroll") for (int i_ = 0; i_ < (N); ++i_)                                     \
        ptx::ld_shared_volatile_vec<4>(&ctl->hdr[nu & 3u][4 * i_], (hdr_) + 4 * i_);       \
    __syncwarp();                                                                          \
    if (lane == 0) arrive0<PAIR>(hdr_empty0 + 8u * s_);                                    \
    ++nu;                                                                                  \
  } while (0)

// Chunk `nc` of the tile lists: wait for it, hand it back (whole warp).
#define TILE_CHUNK_WAIT() TILE_WAIT(&ctl->tl_full[nc & (kTlChunks - 1)], (nc / kTlChunks) & 1u)
#define TILE_CHUNK_DONE()                                                                  \
  do {                                                                                     \
    __syncwarp();                                                                          \
    if (lane == 0) arrive0<PAIR>(tl_empty0 + 8u * (nc & (kTlChunks - 1)));                 \
    ++nc;                                                                                  \
  } while (0)

// Scheduler of the first CTA: publish a header in both CTAs, a lane per word.  It says where the unit lies, so
// that not every warp has to divide the item's number up again (five divisions, between two units).  A header
// lies in one of four places in turn: it is there until its readers are done with the unit.
#define TILE_HDR_PUT(ent, word, jlo, jhi, pr, bh, b, h, o, problem)                        \
  do {                                                                                     \
    const uint32_t s_ = nu & 1u;                                                           \
    LOSA_WAIT_RELAXED(&ctl->hdr_empty[s_], ((nu >> 1) & 1u) ^ 1u);                         \
    const uint64_t o_ = (uint64_t)reinterpret_cast<uintptr_t>(o);                          \
    const uint32_t all_[11] = {(ent), (word), (uint32_t)(jlo), (uint32_t)(jhi), (uint32_t)(pr), (uint32_t)(bh), \
                               (uint32_t)(b), (uint32_t)(h), (uint32_t)o_, (uint32_t)(o_ >> 32), (uint32_t)(problem)}; \
    uint32_t mine_ = 0u;                                                                   \
    _Pragma("unroll") for (int i_ = 0; i_ < 11; ++i_) if (lane == i_) mine_ = all_[i_];    \
    if (lane < 11) {                                                                        \
      ctl->hdr[nu & 3u][lane] = mine_;                                                     \
      if (PAIR) {                                                                          \
        ptx::st_cluster_u32(hdr1 + 48u * (nu & 3u) + 4u * lane, mine_);                    \
        ptx::fence_acq_rel_cluster();                                                      \
      }                                                                                    \
    }                                                                                      \
    __syncwarp();                                                                          \
    if (lane == 0) {                                                                       \
      ptx::mbar_arrive(&ctl->hdr_full[s_]);                                                \
      if (PAIR) ptx::mbar_arrive_cluster(hdr_full1 + 8u * s_);                             \
    }                                                                                      \
    __syncwarp();                                                                          \
    ++nu;                                                                                  \
  } while (0)

// Arrivals on, and copies counted by, a barrier of the first CTA (of the only one, without pairs).
template <bool PAIR>
__device__ __forceinline__ void arrive0(uint32_t bar0) {
  if (PAIR) ptx::mbar_arrive_cluster(bar0);
  else ptx::mbar_arrive_u32(bar0);
}
template <bool PAIR>
__device__ __forceinline__ void expect0(uint32_t bar0, uint32_t bytes) {
  if (PAIR) ptx::mbar_arrive_expect_tx_cluster(bar0, bytes);
  else ptx::mbar_arrive_expect_tx_u32(bar0, bytes);
}
template <bool PAIR>
__device__ __forceinline__ void load0(uint32_t dst, const CUtensorMap* map, uint32_t bar0, int c0, int c1, int c2, int c3) {
  if (PAIR) ptx::tma_load_4d_pair(dst, map, bar0, c0, c1, c2, c3);
  else ptx::tma_load_4d_u32(dst, map, bar0, c0, c1, c2, c3);
}
// Signals a barrier when the MMAs issued so far are complete: in the first CTA, or in both.
template <bool PAIR>
__device__ __forceinline__ void commit0(uint64_t* bar) {
  if (PAIR) ptx::mma2_commit(bar);
  else ptx::mma_commit(bar);
}
template <bool PAIR>
__device__ __forceinline__ void commit_all(uint64_t* bar, uint32_t pair_ctas) {
  if (PAIR) ptx::mma2_commit_both(bar, pair_ctas);
  else ptx::mma_commit(bar);
}

// A lane holds N chunks of 16 bytes of a row of its own; afterwards lane j of a group of N holds chunk j of each of
// the group's rows, that of the group's i-th in place i (whole warp).
template <int N>
__device__ __forceinline__ void transpose_chunks(uint32_t* r, int lane) {
#pragma unroll
  for (int b = 1; b < N; b <<= 1) {
    const bool hi = (lane & b) != 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      if (i & b) continue;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        uint32_t &x = r[4 * i + e], &y = r[4 * (i | b) + e];
        const uint32_t other = __shfl_xor_sync(0xffffffffu, hi ? x : y, b);
        if (hi) x = other;
        else y = other;
      }
    }
  }
}

// The merge of an item's parts by the CTAs of their cluster, each of them its share of the query tile's rows: the
// launch of its own that merges parts elsewhere cost a call 4 us, all of it latency (8 heads of 1024 tokens, D = 64, dense
// 14.0 -> 10.3 us, D = 128 18.4 -> 13.6, with the headers written ahead and the shorter way out).  The same
// arithmetic as merge_parts.  first, step: the ranks of the CTAs with parts 0, 1, ... of this query tile.
template <int D>
__device__ __forceinline__ void merge_in_cluster(const Params& p, int unit, int tile, uint32_t first, uint32_t step,
                                                 uint32_t park_o, uint32_t park_ml, int warp, int lane) {
  constexpr int kLanes = D / 4, kRows = 32 / kLanes;  // lanes of a row, rows of a warp
  const int parts = p.split_parts;
  int part, problem, bh, pr, h;
  const int w = p.by_parts.divmod(unit, part);  // (all items are cut)
  item_place(p, w, problem, bh, pr);
  const int b = p.by_heads.divmod(bh, h);
  const int T = 2 * pr + tile, sub = lane / kLanes, col = lane % kLanes;
  if (T >= p.nQt) return;
  const int row0 = p.by_parts.div(128 * part), row1 = p.by_parts.div(128 * (part + 1));
  void* const o_base = (p.problems != nullptr) ? p.problems[problem].o : p.o;
  const int64_t place = (int64_t)b * p.sb + (int64_t)h * p.sh + (int64_t)T * 128 * p.sn + 4 * col;
  for (int r0 = row0 + warp * kRows; r0 < row1; r0 += 16 * kRows) {
    const int row = r0 + sub;
    const bool here = row < row1 && T * 128 + row < p.N;
    const uint32_t at = (uint32_t)(row * kLanes + ((col & ~7) | ((col ^ row) & 7))) * 16u;
    float4 v[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
    auto fetch = [&](int s0) {
#pragma unroll
      for (int j = 0; j < 2; ++j)
        if (s0 + j < parts && here) v[j] = ptx::ld_cluster_f32x4(ptx::mapa(park_o + at, first + step * (s0 + j)));
    };
    float2 ml = make_float2(0.f, 0.f);
    if (here && col < parts) ml = ptx::ld_cluster_f32x2(ptx::mapa(park_ml + 8u * row, first + step * col));
    fetch(0);
    // (a part without keys of the row has the sum 0; one that met NaN has the sum NaN, and so has the row)
    float m = (ml.y != 0.f) ? ml.x : -INFINITY;
#pragma unroll
    for (int d = kMaxParts / 2; d > 0; d >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, d, kLanes));
    const float mine = (ml.y != 0.f) ? ptx::ex2_approx(ml.x - m) : 0.f;
    float L = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    // (two parts at a time, the first two ahead: unrolled over all eight, the code that a short call runs once and cold took
    // longer than its loads)
#pragma unroll 1
    for (int s0 = 0; s0 < parts; s0 += 2) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        if (s0 + j >= parts) break;
        const float sc = __shfl_sync(0xffffffffu, mine, s0 + j, kLanes);
        L += __shfl_sync(0xffffffffu, ml.y, s0 + j, kLanes) * sc;
        // (What was fetched is used, also where it weighs nothing: the last meeting waits for no reads, and the CTA that is
        // read from must not leave before they have come.  A zero adds nothing to a sum that is never -0.)
        const bool none = sc == 0.f;
        acc.x += (none ? 0.f : v[j].x) * sc;
        acc.y += (none ? 0.f : v[j].y) * sc;
        acc.z += (none ? 0.f : v[j].z) * sc;
        acc.w += (none ? 0.f : v[j].w) * sc;
      }
      fetch(s0 + 2);
    }
    if (!here) continue;
    const float inv = (L != 0.f) ? 1.f / L : 0.f;
    const int64_t off = place + (int64_t)row * p.sn;
    if (p.o_f32)
      *reinterpret_cast<float4*>(static_cast<float*>(o_base) + off) = make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
    else
      *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(o_base) + off) =
          make_uint2(ptx::pack_bf16x2(acc.x * inv, acc.y * inv), ptx::pack_bf16x2(acc.z * inv, acc.w * inv));
  }
}

template <int D, int R, int C_, int MODE, bool PAIR, bool ONE>
__global__ void __launch_bounds__(Lay::kThreads, 1)
losa_tile_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                 const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_kw,
                 const __grid_constant__ CUtensorMap map_vw, const Params p) {
  using L = Lay;
  static_assert(PAIR ? D == 128 : D == 64, "pairs at head dimension 128, one CTA at 64");
  constexpr int kQB = 128 / R;  // query blocks of the query tile
  constexpr int kC = C_, kG = 128 / C_, kW = 128;
  constexpr int kQBytes = 128 * D * 2;
  constexpr int kNQ = tile_nq(D, MODE), kNK = tile_nk(MODE), kNV = tile_nv(MODE);
  constexpr uint32_t kNVs = kNV > 0 ? kNV : 1;
  constexpr int kKRows = PAIR ? 64 : 128;             // keys of a K tile that this CTA copies
  constexpr int kKBox = (C_ < kKRows) ? C_ : kKRows;  // ... per copy
  constexpr int kKCopies = kKRows / kKBox;            // ... and copies per 64-column slab
  constexpr int kSlabs = D / 64;                      // slabs of a K tile
  constexpr uint32_t kIdescQK = ptx::idesc_bf16_f32(PAIR ? 256 : 128, 128, false, false);
  constexpr uint32_t kIdescPV =
      ptx::idesc_bf16_f32(PAIR ? 256 : 128, (D == 64 && MODE != kMass) ? D + 16 : D, false, true);
  // Head dimension 64: a key tile needs 1024 cycles of the special-function unit against 512 of the
  // tensor cores, so one group of four scores in every kPolyOf takes its exponentials from a
  // polynomial on the FMA pipe.  17776 tokens, 8 heads: dense 735 us with one in 8, 742 in 16, 763 in 6,
  // 805 in 4.  The mass pass (no P to pack and to sum) takes one in 4: 735 us, 759 in 8, 786 in 6; at head
  // dimension 128 (32760 tokens, 12 heads, 128-key blocks, unit normal q and k) 3463 us, 3639 in 8, 3924
  // without (against 64 bits its masses err by 1 % more with it than without, 2e-7).
  constexpr int kPolyOf = (MODE == kMass) ? LOSA_POLY_OF_MASS : (D == 64) ? LOSA_POLY_OF : 0;
  using Ctl = TileControl;
  // The row sums of P come out of O += P V (see kTileOnes).  The second 32 of a thread's scores are then
  // fetched while the first are worked on, and P is stored 32 scores at a time: without the sums' chains the
  // compiler spread the exponentials so far that it spilled.  17776 tokens, 48 heads, against sums in the softmax
  // warps: dense 4757 us, 4727 with the sums as columns, 4512 with the late fetch, 4470 with the early store as well;
  // sparse (coverage 0.85) 4510, 4247, 4187, 4157.  A share of 1 in 8 for the polynomial stays the best one (dense
  // 4531 us without, 4543 in 16, 4564 in 7, 4788 in 4).
  constexpr bool kSumCol = (D == 64 && MODE != kMass);
  // Who writes O out (and ends the unit): see the end of an item.
  constexpr bool kOneGroup = (MODE == kDense || MODE == kSparse);
  constexpr bool kWantMass = (MODE == kFused || MODE == kMass);  // the block masses (Eq. 1) are wanted
  // the mass pass alone has no V, no P and no O: its score buffers go back as soon as they are read
  constexpr bool kHasV = (MODE != kMass);
  // When a unit's place is read from its header: at its end, but in those mass passes that came out faster with it in
  // registers from the unit's start; and which four of 16 scores the mass pass takes from the polynomial.  That is the
  // compiler's ordering of the exponentials, so the lines lie where they were measured, and have to be measured again when
  // the loop changes (masses, 16384 tokens, 12 heads, us: at the start / at the end, and with the second four instead of the
  // first: D = 64, C = 32 908 / 917, 920 / 929, C = 64 826 / 854, 886 / 826, C = 128 851 / 843, 818 / 843; D = 128, C = 32
  // 1059 / 992, 1023 / 1054, C = 64 963 / 948, 965 / 945, C = 128 946 / 961, 918 / 956).
  constexpr bool kInfoEarly = MODE == kMass && (D == 64 || C_ == 128);
  constexpr int kPolyAt = (MODE == kMass && C_ == 128) ? 1 : 0;
  constexpr int kChunkTiles = (MODE == kSparse) ? 32 / kG : (1 << 28);  // K/V tiles per chunk of the list
  static_assert(offsetof(TileControl, tl) % 16 == 0, "the tile list is read with 16-byte loads");
  static_assert(offsetof(TileControl, redo_need) == offsetof(TileControl, redo_mark) + 16, "reached from the marks");

  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* const sQ = smem_raw;
  uint8_t* const sK = sQ + kNQ * kQBytes;
  uint8_t* const sV = sK + kNK * kTileStage;
  uint8_t* const sOnes = sV + kNV * kTileStage;
  Ctl* const ctl = reinterpret_cast<Ctl*>(sOnes + (D == 64 ? kTileOnes : 0));
  // what a part leaves for the others of its cluster, where its K tiles were: unnormalised O, 16 bytes at a time, and the
  // rows' reference and sum
  uint4* const park_o = reinterpret_cast<uint4*>(sK);
  float2* const park_ml = reinterpret_cast<float2*>(&ctl->half_max[0][0][0]);
  static_assert(!kOneGroup || kNK * kTileStage >= 128 * D * 4, "room for a part's O");

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // The parts of an item that a single wave is cut into may share a cluster (p.in_cluster): pairs of CTAs, or CTAs, in
  // the order of the parts.
  const bool in_cluster = ONE && kOneGroup && p.in_cluster;
  const uint32_t cta = PAIR ? ptx::cluster_ctarank() : 0u, cta0 = ONE ? cta & ~1u : 0u;
  const uint32_t rank = cta - cta0;  // 0: the CTA that issues the MMAs; also the query tile
  const uint32_t pair_ctas = 3u << cta0;
  // the tile list, which says the unit, that the CTA works on first
  auto first_list = [&]() {
    if (PAIR || !in_cluster) return (int)(PAIR ? blockIdx.x >> 1 : blockIdx.x);
    // (a cluster per query tile)
    int part;
    const int c = p.by_parts.divmod((int)blockIdx.x, part);
    return 2 * ((c >> 1) * p.split_parts + part) + (c & 1);
  };
  ptx::grid_launch_dependents();
  // (the swizzled tiles rely on the declared alignment of the dynamic shared memory)
  const bool misaligned = (ptx::smem_u32(smem_raw) & 1023u) != 0;

  // shared::cluster addresses of the first CTA's barriers that both CTAs arrive on, and of the
  // second CTA's copy of the tile list (used by the first CTA's scheduler)
  auto at0 = [&](const void* x) { return PAIR ? ptx::mapa(ptx::smem_u32(x), cta0) : ptx::smem_u32(x); };
  auto at1 = [&](const void* x) { return PAIR ? ptx::mapa(ptx::smem_u32(x), cta0 + 1u) : 0u; };
  const uint32_t q_full0 = at0(&ctl->q_full[0]);
  const uint32_t k_full0 = at0(&ctl->k_full[0]);
  const uint32_t v_full0 = at0(&ctl->v_full[0]);
  const uint32_t p_ready0 = at0(&ctl->p_ready[0]);
  const uint32_t o_free0 = at0(&ctl->o_free);
  const uint32_t redo_mark0 = at0(&ctl->redo_mark[0]);
  const uint32_t tl_empty0 = at0(&ctl->tl_empty[0]);
  const uint32_t tl_full1 = at1(&ctl->tl_full[0]);
  const uint32_t hdr_empty0 = at0(&ctl->hdr_empty[0]);
  const uint32_t hdr_full1 = at1(&ctl->hdr_full[0]);
  const uint32_t hdr1 = at1(&ctl->hdr[0][0]);
  const uint32_t tl1 = at1(&ctl->tl[0]);
  const uint32_t abort_peer = PAIR ? ptx::mapa(ptx::smem_u32(&ctl->abort_flag), cta ^ 1u) : 0u;

  // One unit to a CTA, or pair of them (p.one_wave): where a warp is through with it, it meets the other warps of the
  // cluster, and where no unit of the cluster has to be run again all may leave.  (Asking the scheduler for the next unit
  // instead, and being told that there is none, took 1800 cycles of a 2048-token call's 26000.)
  int over = -1;
  auto unit_over = [&]() -> bool {
    ptx::tc_fence_before_sync();
    // What was stored into another CTA's shared memory - arrivals on a pair's barriers, the abort flag - has to be there
    // before that CTA may leave, and what is left for the other parts before they read it.  (Elsewhere a release would only
    // wait for O's way to memory.)
    if (PAIR || (in_cluster && warp >= 4)) {
      ptx::cluster_meet();
    } else {
      ptx::cluster_arrive_relaxed();
      ptx::cluster_wait();
    }
    over = *reinterpret_cast<volatile uint32_t*>(&ctl->cluster_marked) == 0u ? 1 : 0;
    return over != 0;
  };
  // (every CTA of the cluster is told)
  auto mark_cluster = [&]() {
    if (!ONE) return;
    const uint32_t ctas = (PAIR ? 2u : 1u) * (in_cluster ? (uint32_t)p.split_parts : 1u);
    for (uint32_t c = 0; c < ctas; ++c) ptx::st_cluster_u32(ptx::mapa(ptx::smem_u32(&ctl->cluster_marked), c), 1u);
    ptx::fence_acq_rel_cluster();
  };

  if (threadIdx.x == 0) {
    constexpr int kCtas = PAIR ? 2 : 1;
    for (int i = 0; i < 2; ++i) {
      ptx::mbar_init(&ctl->q_full[i], kCtas);   // one arrival (with its byte count) per CTA's producer
      ptx::mbar_init(&ctl->q_empty[i], 1);
    }
    for (int i = 0; i < 4; ++i) {
      ptx::mbar_init(&ctl->o_done[i], 1);
      ptx::mbar_init(&ctl->l_full[i], 8);
    }
    for (int i = 0; i < kNK; ++i) {
      ptx::mbar_init(&ctl->k_full[i], kCtas);
      ptx::mbar_init(&ctl->k_empty[i], 1);
    }
    for (int i = 0; i < kNV; ++i) {
      ptx::mbar_init(&ctl->v_full[i], kCtas);
      ptx::mbar_init(&ctl->v_empty[i], 1);
    }
    for (int i = 0; i < 3; ++i) {
      ptx::mbar_init(&ctl->s_full[i], 1);
      ptx::mbar_init(&ctl->p_ready[i], 8 * kCtas);  // the eight warps of a group, in both CTAs
      ptx::mbar_init(&ctl->pv_done[i], 1);
    }
    // every softmax warp of both CTAs reads a part of its rows' O, or every one of one group
    ptx::mbar_init(&ctl->o_free, (kOneGroup ? 8 : 16) * kCtas);
    for (int i = 0; i < kTlChunks; ++i) {
      ptx::mbar_init(&ctl->tl_full[i], 1);
      ptx::mbar_init(&ctl->tl_empty[i], 17 * kCtas);  // readers: each CTA's producer and 16 softmax warps
    }
    for (int i = 0; i < 2; ++i) {
      ptx::mbar_init(&ctl->hdr_full[i], 1);
      ptx::mbar_init(&ctl->hdr_empty[i], 17 * kCtas + 2);  // ... and the two issuers
    }
    ptx::mbar_init(&ctl->hdr_next, 1);  // the first CTA's producer, near the end of a unit
    for (int i = 0; i < 8; ++i) ptx::mbar_init(&ctl->pair_bar[i], 2);
    for (int i = 0; i < 2; ++i) {
      for (int q = 0; q < kQB; ++q) {
        ptx::mbar_init(&ctl->ref_full[i][q], 4 / kQB);   // the first halves' warps of the group that sets it
        ptx::mbar_init(&ctl->ref_empty[i][q], 8 / kQB);  // the warps of the other group
      }
    }
    ptx::mbar_init(&ctl->item_bar, 16);
    ptx::mbar_init(&ctl->fold_bar, 16);
    ptx::mbar_init(&ctl->drain, 2);
    for (int i = 0; i < 4; ++i) ctl->redo_mark[i] = ctl->redo_need[i] = ctl->redo_state[i] = 0u;
    ctl->cluster_marked = 0u;
    for (int i = 0; i < 16; ++i) ctl->max_uses[i] = 0;
    ctl->abort_flag = 0;
    ptx::fence_barrier_init();
  }
  // A call's first header says where the unit at this CTA's position lies, and is written ahead: in the dense modes it is
  // all there is to say, and where the CTA makes its own list all but what that says.  (Where the list comes from the
  // launch ahead, the header as well does: written here, that sparse kernel was up to 8 % slower in all of its units, the
  // compiler's doing.)
  const bool early = (ONE || MODE != kSparse) && p.problems == nullptr && !p.stall;
  if (warp == kSchedulerWarp && early) {
    int unit = first_list();
    const uint32_t odd = (!PAIR && (unit & 1)) ? kHdrOdd : 0u;
    if (!PAIR) unit >>= 1;
    int w, part, parts, problem, bh, pr, h, jlo, jhi;
    unit_item(p, unit, w, part, parts);
    const uint32_t ent = kTlItem | (parts > 1 ? kTlPartial | ((uint32_t)part << 24) : 0u) | (uint32_t)w;
    item_place(p, w, problem, bh, pr);
    const int b = p.by_heads.divmod(bh, h);
    tile_key_range(p, ent, jlo, jhi);
    const bool two = 2 * pr + 1 < p.nQt;  // the pair's second query tile exists
    const uint32_t tiles = (uint32_t)((jhi - jlo + kG - 1) / kG);
    const uint32_t word = PAIR ? (two ? 3u : 1u) * kHdrHas | tiles : odd | ((two || odd == 0u) ? kHdrHas | tiles : 0u);
    const uint64_t o = (uint64_t)reinterpret_cast<uintptr_t>(p.o);
    const uint32_t all[11] = {ent, word, (uint32_t)jlo, (uint32_t)jhi, (uint32_t)pr, (uint32_t)bh, (uint32_t)b, (uint32_t)h,
                              (uint32_t)o, (uint32_t)(o >> 32), 0u};
    uint32_t mine = 0u;
#pragma unroll
    for (int i = 0; i < 11; ++i) if (lane == i) mine = all[i];
    if (lane < 11) ctl->hdr[0][lane] = mine;
    __syncwarp();
  }
  if (kSumCol && threadIdx.x < kTileOnes / 16) {
    reinterpret_cast<uint4*>(sOnes)[threadIdx.x] = make_uint4(0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u);
    ptx::fence_proxy_async();
  }
  if (warp == kIssuerWarp) {
    // (one warp of each CTA of the pair)
    if (PAIR) {
      ptx::tmem_alloc2(&ctl->tmem_base, kTmemCols);
      ptx::tmem_relinquish_alloc_permit2();
    } else {
      ptx::tmem_alloc(&ctl->tmem_base, kTmemCols);
      ptx::tmem_relinquish_alloc_permit();
    }
  }
  if (warp == kProducerWarp && lane == 0) {
    ptx::prefetch_tensormap(&map_q);
    ptx::prefetch_tensormap(&map_k);
    ptx::prefetch_tensormap(&map_v);
    if (kG > 1) {
      ptx::prefetch_tensormap(&map_kw);
      ptx::prefetch_tensormap(&map_vw);
    }
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  if (MODE != kSparse && early && warp == kSchedulerWarp && lane == 0) ptx::mbar_arrive(&ctl->hdr_full[0]);
  if (PAIR || in_cluster) ptx::cluster_sync();  // both CTAs' barriers are initialised before either signals the other
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base = ctl->tmem_base;
  {
    // the MMAs address both CTAs' tensor memory with one address
    const uint32_t other =
        PAIR ? ptx::ld_cluster_u32(ptx::mapa(ptx::smem_u32(&ctl->tmem_base), cta ^ 1u)) : tmem_base;
    if (misaligned || other != tmem_base) {
      if (threadIdx.x == 0) {
        ctl->abort_flag = 1;
        report_error(p.status, LOSA_ERR_CUDA);
      }
    }
  }
  __syncthreads();
  // (the tile lists and the counters come from the kernel before; everything up to here overlaps it)
  ptx::grid_dependency_wait();
  // (its entries, of which there are few where a slot has 256 tokens or more, are read from shared memory the first
  // time; they lie behind what the first unit's end uses of that place)
  constexpr int kListAt = 512;
  static_assert(2 * kQB * ((256 / C_ * (kMaxPersistentCtas / 2) + 31) / 32) <= kListAt, "room for the bitmaps");
  static_assert(sizeof(TileControl::xch) >= 4 * (kListAt + 256 / C_ * (kMaxPersistentCtas / 2) + 48), "room for a list");
  constexpr bool kPerTile = tile_lists_per_unit(D) == 2;
  constexpr int kListBlocks = (kPerTile ? 1 : 2) * kQB;  // query blocks of a list
  if (MODE == kSparse && ONE) {
    // ... or the tile list of this CTA's unit from here: the bitmaps of its query blocks, in a place not in use yet
    if (rank == 0 && warp < kListBlocks)
      fill_tile_bitmap<kListBlocks, kPerTile>(p, first_list(), warp, lane, reinterpret_cast<uint32_t*>(&ctl->xch[0][0][0]));
    __syncthreads();
  }

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(L::kRegsUtility));
    if (ctl->abort_flag) goto teardown;
    if (warp == kProducerWarp) {
      // ------------------------------------------------------------------ TMA producer (both CTAs)
      // One elected thread makes the copies: from a lane test the compiler cannot tell that there is only one.
      const bool leader = ptx::elect_one();
      const uint32_t sQ_a = ptx::smem_u32(sQ), sK_a = ptx::smem_u32(sK), sV_a = ptx::smem_u32(sV);
      const uint32_t k_empty_a = ptx::smem_u32(&ctl->k_empty[0]), v_empty_a = ptx::smem_u32(&ctl->v_empty[0]);
      const uint32_t tl_a = ptx::smem_u32(&ctl->tl[0]);
      uint32_t nq = 0, nk = 0, vs = 0, v_par = 1u, nu = 0, nc = 0, hdr[12];
      int problem = -1;  // batched launch: whose tensor maps this warp has acquired
      // One wave: every stage and score buffer is free again.  The tensor cores say so, in both CTAs of a pair, some time
      // after the MMAs were issued, and nobody else waits for the last of it: a CTA must not leave before.  A lane for each;
      // false: gave up.  (2048 tokens, 4 heads, D = 64 14.35 -> 14.38 us.  In the other kernels two headers lie between the
      // last of it and the end; waiting there as well made them 1 - 3 % slower at head dimension 128, the compiler's doing.)
      auto all_returned = [&]() -> bool {
        const int who = __ffs(__ballot_sync(0xffffffffu, leader)) - 1;  // (it alone has counted)
        const uint32_t k0 = __shfl_sync(0xffffffffu, nk, who), v0 = __shfl_sync(0xffffffffu, vs, who);
        const uint32_t v0_par = __shfl_sync(0xffffffffu, v_par, who);
        uint32_t bar = 0u, par = 0u;
        if (lane < kNQ) {
          const uint32_t i = nq + lane;
          bar = ptx::smem_u32(&ctl->q_empty[i % kNQ]);
          par = ((i / kNQ) & 1u) ^ 1u;
        } else if (lane < kNQ + kNK) {
          const uint32_t i = k0 + lane - kNQ;
          bar = k_empty_a + 8u * (i % kNK);
          par = ((i / kNK) & 1u) ^ 1u;
        } else if (lane < kNQ + kNK + kNV) {
          const uint32_t i = lane - kNQ - kNK;
          bar = v_empty_a + 8u * i;
          par = i >= v0 ? v0_par : v0_par ^ 1u;
        } else if (kHasV && rank == 0 && lane < kNQ + kNK + kNV + 3) {
          const uint32_t i = k0 + lane - kNQ - kNK - kNV;  // (a product for each K tile)
          bar = ptx::smem_u32(&ctl->pv_done[i % 3u]);
          par = ((i / 3u) & 1u) ^ 1u;
        }
        if (bar != 0u && !ptx::mbar_wait_relaxed_u32(bar, par, &ctl->abort_flag, p.wait_polls)) {
          ctl->abort_flag = 1;
          report_error(p.status, LOSA_ERR_TIMEOUT);
        }
        __syncwarp();
        return *reinterpret_cast<volatile int*>(&ctl->abort_flag) == 0;
      };
      for (;;) {
        if (ONE && nu == 1u && !all_returned()) goto teardown;
        TILE_HDR_NEXT(hdr, 3);
        const uint32_t ent = hdr[0], word = hdr[1];
        if (ent == kTlSkip) {
          if (rank == 0 && leader) ptx::mbar_arrive(&ctl->hdr_next);
          continue;
        }
        if ((ent >> 28) != 1) break;
        const int pr = (int)hdr[4], b = (int)hdr[6], h = (int)hdr[7];
        // (map_kw: K in boxes of 64 keys, map_vw: V in boxes of 128 keys, for consecutive key blocks)
        const CUtensorMap *mq = &map_q, *mk = &map_k, *mv = &map_v, *mkw = &map_kw, *mvw = &map_vw;
        if (p.problems != nullptr) {
          const ProblemEntry* pe = p.problems + hdr[10];
          mq = &pe->map_q;
          mk = PAIR ? &pe->map_kh : &pe->map_k;
          mv = &pe->map_v;
          mkw = PAIR ? &pe->map_k64 : &pe->map_k128;
          mvw = &pe->map_v128;
          if (PAIR && (int)hdr[10] != problem) {
            problem = (int)hdr[10];
            acquire_tile_maps<D, C_, kHasV>(pe, lane);
            __syncwarp();
          }
        }
        // this CTA's query tile (rows past the end of the sequence are filled with zeros)
        const int T = 2 * pr + (PAIR ? (int)rank : (int)((word & kHdrOdd) != 0u));
        const uint32_t qs = nq % kNQ;
        LOSA_WAIT_RELAXED(&ctl->q_empty[qs], ((nq / kNQ) & 1) ^ 1);
        if (leader) {
          expect0<PAIR>(q_full0 + 8u * qs, kQBytes);
#pragma unroll
          for (int s = 0; s < kSlabs; ++s)
            load0<PAIR>(sQ_a + qs * kQBytes + s * 16384, mq, q_full0 + 8u * qs, s * 64, T * 128, h, b);
        }
        ++nq;
        const int tiles = (int)(word & kHdrTiles);
        const int jlo = (int)hdr[2], jhi = (int)hdr[3];  // dense modes: the unit's key blocks
        // the scheduler draws the next unit when this one is 16 tiles from its end
        const int call_at = max(0, tiles - 16);
        if (tiles == 0 && rank == 0 && leader) ptx::mbar_arrive(&ctl->hdr_next);
        for (int base = 0; base < tiles; base += kChunkTiles) {
          if (MODE == kSparse) TILE_CHUNK_WAIT();
          const int end = min(tiles, base + kChunkTiles);
          if (leader) {
            bool in_time = true;
            for (int i = base; i < end; ++i) {
              if (i == call_at && rank == 0) ptx::mbar_arrive(&ctl->hdr_next);
              uint32_t grp[kG];
              if (MODE == kSparse) {
                ptx::ld_shared_volatile_vec_u32<kG>(tl_a + 4u * ((nc & (kTlChunks - 1)) * 32 + (i - base) * kG), grp);
#pragma unroll
                for (int g = 0; g < kG; ++g) grp[g] &= 0xffffu;
              } else {
#pragma unroll
                for (int g = 0; g < kG; ++g) grp[g] = (jlo + i * kG + g < jhi) ? (uint32_t)(jlo + i * kG + g) : kTlPad;
              }
              // K: a pair's CTAs keys 64 * rank ... + 63 of the tile each; all head-dimension columns, per slab of 64
              const uint32_t ks = nk % kNK;
              in_time = ptx::mbar_wait_relaxed_u32(k_empty_a + 8u * ks, ((nk / kNK) & 1) ^ 1, &ctl->abort_flag, p.wait_polls);
              if (!in_time) break;
              ++nk;
              expect0<PAIR>(k_full0 + 8u * ks, kTileStage);
              const uint32_t k_to = sK_a + ks * kTileStage;
              // several key blocks: this CTA's, if consecutive, are one copy per slab (every copy costs its thread
              // about 70 ns, and at head dimension 64 a tile takes 550)
              constexpr int kKBlocks = (kKRows / kC > 0) ? kKRows / kC : 1;  // key blocks of this CTA's rows
              uint32_t mine[kKBlocks];
              bool wide_k = kKBlocks > 1;
#pragma unroll
              for (int j = 0; j < kKBlocks; ++j) {
                mine[j] = (PAIR && kG > 1 && rank == 1) ? grp[(kG / 2 + j) % kG] : grp[j];
                if (j > 0) wide_k = wide_k && mine[j] == mine[0] + j;
              }
              if (wide_k) {
#pragma unroll
                for (int s = 0; s < kSlabs; ++s)
                  load0<PAIR>(k_to + s * (kKRows * 128), mkw, k_full0 + 8u * ks, s * 64, (int)mine[0] * kC, h, b);
              } else {
#pragma unroll
                for (int j = 0; j < kKCopies; ++j) {
                  const int inb = (PAIR && kG == 1) ? 64 * (int)rank : 0;  // (half of a 128-key block)
                  const int r0 = (mine[j] == kTlPad) ? p.nKb * kC : (int)mine[j] * kC + inb;
#pragma unroll
                  for (int s = 0; s < kSlabs; ++s)
                    load0<PAIR>(k_to + s * (kKRows * 128) + j * kKBox * 128, mk, k_full0 + 8u * ks, s * 64, r0, h, b);
                }
              }
              if (!kHasV || (word & kHdrMax)) continue;
              // V: all 128 keys of the tile, (a pair: of each CTA) 64 of the head-dimension columns, one slab
              in_time = ptx::mbar_wait_relaxed_u32(v_empty_a + 8u * vs, v_par, &ctl->abort_flag, p.wait_polls);
              if (!in_time) break;
              expect0<PAIR>(v_full0 + 8u * vs, kTileStage);
              const uint32_t v_to = sV_a + vs * kTileStage;
              bool wide_v = kG > 1;
#pragma unroll
              for (int g = 1; g < kG; ++g) wide_v = wide_v && grp[g] == grp[0] + g;
              if (wide_v) {
                load0<PAIR>(v_to, mvw, v_full0 + 8u * vs, (int)rank * 64, (int)grp[0] * kC, h, b);
              } else {
#pragma unroll
                for (int g = 0; g < kG; ++g)
                  load0<PAIR>(v_to + g * kC * 128, mv, v_full0 + 8u * vs, (int)rank * 64,
                              (grp[g] == kTlPad) ? p.nKb * kC : (int)grp[g] * kC, h, b);
              }
              if (++vs == (uint32_t)kNV) {
                vs = 0u;
                v_par ^= 1u;
              }
            }
            if (!in_time) {
              ctl->abort_flag = 1;
              report_error(p.status, LOSA_ERR_TIMEOUT);
            }
          }
          __syncwarp();
          if (*reinterpret_cast<volatile int*>(&ctl->abort_flag)) goto teardown;
          if (MODE == kSparse) TILE_CHUNK_DONE();
        }
      }
      if (ONE) all_returned();
    } else if (warp == kIssuerWarp && rank == 0) {
      // ------------------------------------------------------------------ S = Q K^T of the pair
      // Score k of the launch goes into buffer k % 3, which holds the P of score k - 3 until the
      // product that reads it has run (pv_done, from the other issuer).
      const bool leader = ptx::elect_one();
      constexpr uint32_t kDescHi = ptx::smem_desc_hi_sw128(1024);
      const uint32_t k_lo = ptx::smem_desc_lo(ptx::smem_u32(sK), 16);
      uint32_t qd[D / 16];
#pragma unroll
      for (int kk = 0; kk < D / 16; ++kk)
        qd[kk] = ptx::smem_desc_lo(ptx::smem_u32(sQ), 16) + (((kk >> 2) * 16384 + (kk & 3) * 32) >> 4);
      uint32_t nq = 0, nt = 0, nu = 0, hdr[4];
      for (;;) {
        TILE_HDR_NEXT(hdr, 1);
        const uint32_t ent = hdr[0], word = hdr[1];
        if (ent == kTlSkip) continue;
        if ((ent >> 28) != 1) break;
        bool q_ready = false;
        for (int i = (int)(word & kHdrTiles); i > 0; --i) {
          const uint32_t ks = nt % kNK;
          LOSA_WAIT(&ctl->k_full[ks], (nt / kNK) & 1);
          if (!q_ready) {
            LOSA_WAIT(&ctl->q_full[nq % kNQ], (nq / kNQ) & 1);
            q_ready = true;
          }
          const uint32_t bsel = nt % 3u;
          if (nt >= 3u) {
            // (mass pass: the softmax warps of both CTAs hand the buffer back once it is in registers)
            if (kHasV) LOSA_WAIT(&ctl->pv_done[bsel], (nt / 3u - 1u) & 1);
            else LOSA_WAIT(&ctl->p_ready[bsel], (nt / 3u - 1u) & 1);
          }
          ptx::tc_fence_after_sync();
          if (leader) {
            const uint32_t kd0 = k_lo + ks * (kTileStage >> 4), q0 = (nq % kNQ) * (kQBytes >> 4);
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk)
              if (PAIR)
                ptx::mma2_ss_lo(tmem_base + bsel * 128, qd[kk] + q0, kd0 + (((kk >> 2) * 8192 + (kk & 3) * 32) >> 4),
                                kDescHi, kIdescQK, kk > 0 ? 1u : 0u);
              else
                ptx::mma_ss_lo(tmem_base + bsel * 128, qd[kk] + q0, kd0 + (((kk & 3) * 32) >> 4), kDescHi, kIdescQK,
                               kk > 0 ? 1u : 0u);
            commit_all<PAIR>(&ctl->s_full[bsel], pair_ctas);
            commit_all<PAIR>(&ctl->k_empty[ks], pair_ctas);
          }
          ++nt;
        }
        if (!q_ready) {
          // a unit without key tiles: the query tiles were loaded all the same
          LOSA_WAIT(&ctl->q_full[nq % kNQ], (nq / kNQ) & 1);
        }
        if (leader) commit_all<PAIR>(&ctl->q_empty[nq % kNQ], pair_ctas);
        ++nq;
      }
    } else if (warp == kIssuerWarp + 1 && rank == 0) {
      // ------------------------------------------------------------------ O += P V of the pair
      const bool leader = ptx::elect_one();
      constexpr uint32_t kDescHi = ptx::smem_desc_hi_sw128(1024);
      // (without pairs of CTAs a product's columns from 64 on, which lie a leading byte offset behind its
      // first key's row, are the ones: the offset shrinks as the row advances)
      const uint32_t v_lo = ptx::smem_desc_lo(ptx::smem_u32(sV), kSumCol ? kNV * kTileStage : kTileStage);
      auto v_desc = [&](uint32_t bytes) { return v_lo + (bytes >> 4) - (kSumCol ? (bytes >> 4) << 16 : 0u); };
      const uint32_t tO = tmem_base + 384;
      uint32_t nof = 0, nt = 0, nv = 0, nu = 0, hdr[4];
      // one wave, no products to wait for: this thread's own arrivals, which are there before it meets the other warps, not
      // the tensor cores', which nobody waits for
      const uint32_t o_done1 = at1(&ctl->o_done[0]);
      auto no_products = [&](uint32_t od) {
        ptx::mbar_arrive(&ctl->o_done[od]);
        if (PAIR) ptx::mbar_arrive_cluster(o_done1 + 8u * od);
      };
      for (;;) {
        TILE_HDR_NEXT(hdr, 1);
        const uint32_t ent = hdr[0], word = hdr[1];
        if ((ent >> 28) == 2) break;
        const uint32_t od = (nu - 1u) & 3u;
        if (ent == kTlSkip || (kHasV && (word & kHdrMax))) {
          // (no P and no products: the score buffers go back as soon as they are read)
          for (int i = (int)(word & kHdrTiles); i > 0; --i, ++nt) {
            LOSA_WAIT(&ctl->p_ready[nt % 3u], (nt / 3u) & 1);
            if (leader) commit0<PAIR>(&ctl->pv_done[nt % 3u]);
          }
          if (leader) {
            if (ONE) no_products(od);
            else commit_all<PAIR>(&ctl->o_done[od], pair_ctas);
          }
          continue;
        }
        uint32_t pv_item = 0;
        for (int i = kHasV ? (int)(word & kHdrTiles) : 0; i > 0; --i) {  // (the mass pass has no products)
          const uint32_t vs = nv % kNVs;
          LOSA_WAIT(&ctl->v_full[vs], (nv / kNVs) & 1);
          const uint32_t bsel = nt % 3u;
          if (pv_item == 0 && nof > 0) LOSA_WAIT(&ctl->o_free, (nof - 1) & 1);
          LOSA_WAIT(&ctl->p_ready[bsel], (nt / 3u) & 1);
          ptx::tc_fence_after_sync();
          if (leader) {
            const uint32_t tP = tmem_base + bsel * 128;
            const uint32_t vd0 = v_desc(vs * kTileStage);
            // (each half of a row packs its P over the head of its own 64 score columns)
#pragma unroll
            for (int kk = 0; kk < kW / 16; ++kk)
              if (PAIR)
                ptx::mma2_ts_lo(tO, tP + (kk & 3) * 8 + (kk >> 2) * 64, vd0 + kk * (2048 >> 4), kDescHi, kIdescPV,
                                (kk > 0 || pv_item > 0) ? 1u : 0u);
              else
                ptx::mma_ts_lo(tO, tP + (kk & 3) * 8 + (kk >> 2) * 64,
                               vd0 + kk * (kSumCol ? (2048u >> 4) - (2048u << 12) : 2048u >> 4), kDescHi, kIdescPV,
                               (kk > 0 || pv_item > 0) ? 1u : 0u);
            commit0<PAIR>(&ctl->pv_done[bsel]);
            commit_all<PAIR>(&ctl->v_empty[vs], pair_ctas);
          }
          ++pv_item;
          ++nt;
          ++nv;
        }
        if (leader) {
          if (ONE && pv_item == 0) no_products(od);
          else commit_all<PAIR>(&ctl->o_done[od], pair_ctas);  // every product of the item is done
        }
        if (pv_item > 0) ++nof;
      }
    } else if (warp == kSchedulerWarp && rank == 0) {
      // ------------------------------------------------------------------ scheduler of the pair
      // A unit that outgrew its reference is run again: for its rows' maxima (kHdrMax), where these are needed, and
      // against what it left or these left in redo_ref (kHdrRedo; which of the four: kHdrSet).  Every warp marks it before it takes the next header but one, and header nu goes out
      // when all have taken header nu - 2: the mark of unit nu - 3 is final then.  Before the end comes a header
      // without work: when that one has been taken, so are the marks of the last two units.
      uint32_t nu = 0, nc = 0;
      int idle = 0;
      int acquired = -1;  // batched launch: whose tensor maps this warp has acquired
      bool first_item = true, drawn = false;
      uint32_t own_word = 0u;  // one_wave: what tl_count holds of the CTA's unit
      // (how many units were run again is for tests to read: where no launch behind adds their flags up, the flags say it)
      if (in_cluster && blockIdx.x == 0 && lane == 0) *p.redo_count = -1;
      if (MODE == kSparse && ONE) {
        uint32_t* const bm = reinterpret_cast<uint32_t*>(&ctl->xch[0][0][0]);
        own_word = emit_tile_list<kListBlocks, kG, kPerTile>(p, first_list(), lane, bm, bm + kListAt);
        __syncwarp();
      }
      // A unit's tile list, in chunks of 32 entries, to both CTAs; `own`: made by this CTA, in shared memory.  False: gave up.
      auto publish_list = [&](int list, int cnt, bool own) -> bool {
        const uint32_t* src = p.tl_entries + (int64_t)list * p.tl_cap;
        for (int base = 0; base < cnt; base += 32) {
          const uint32_t e = (base + lane >= cnt) ? 0u
                             : own ? reinterpret_cast<const uint32_t*>(&ctl->xch[0][0][0])[kListAt + base + lane]
                                   : __ldcg(src + base + lane);
          const uint32_t c = nc & (kTlChunks - 1);
          if (!ptx::mbar_wait_relaxed(&ctl->tl_empty[c], ((nc / kTlChunks) & 1u) ^ 1u, &ctl->abort_flag, p.wait_polls)) {
            ctl->abort_flag = 1;
            report_error(p.status, LOSA_ERR_TIMEOUT);
            return false;
          }
          ctl->tl[c * 32 + lane] = e;
          if (PAIR) {
            ptx::st_cluster_u32(tl1 + 4u * (c * 32 + lane), e);
            ptx::fence_acq_rel_cluster();
          }
          __syncwarp();
          if (lane == 0) {
            ptx::mbar_arrive(&ctl->tl_full[c]);
            if (PAIR) ptx::mbar_arrive_cluster(tl_full1 + 8u * c);
          }
          ++nc;
        }
        return true;
      };
      for (;;) {
        if (p.stall) break;  // diagnostic launch: nothing is published and every wait runs out
        if (nu == 0u && early) {
          // (the first unit's header is there: in the sparse mode without what its list says)
          first_item = false;
          if (MODE == kSparse) {
            const int list = first_list();
            const int cnt = min((int)(own_word & kHdrTiles) * kG, p.tl_cap);
            if (lane == 0) {
              const uint32_t word = (own_word & ~kHdrTiles) | ((!PAIR && (list & 1)) ? kHdrOdd : 0u) | (uint32_t)(cnt / kG);
              *reinterpret_cast<volatile uint32_t*>(&ctl->hdr[0][1]) = word;
              if (PAIR) {
                ptx::st_cluster_u32(hdr1 + 4u, word);
                ptx::fence_acq_rel_cluster();
              }
              ptx::mbar_arrive(&ctl->hdr_full[0]);
              if (PAIR) ptx::mbar_arrive_cluster(hdr_full1);
            }
            __syncwarp();
            if (!publish_list(list, cnt, true)) goto teardown;
          }
          ++nu;
          LOSA_WAIT_RELAXED(&ctl->hdr_next, 0u);
          continue;
        }
        if (ONE && nu == 1u && unit_over()) {
          if (p.split_parts > 1 && lane == 0) p.redo_flag[first_list()] = 0;
          goto teardown;
        }
        LOSA_WAIT_RELAXED(&ctl->hdr_empty[nu & 1u], ((nu >> 1) & 1u) ^ 1u);
        if (PAIR) ptx::fence_acq_rel_cluster();
        auto take_mark = [&](uint32_t unit_no) {
          volatile uint32_t* const at = &ctl->redo_mark[unit_no & 3u];
          const uint32_t mark = *at;
          if (mark == 0u) return false;
          const uint32_t need = *reinterpret_cast<volatile uint32_t*>(&ctl->redo_need[unit_no & 3u]);
          __syncwarp();
          if (lane == 0) {
            *at = 0u;
            ctl->redo_queue[ctl->redo_state[2]++ & 3u] =
                (mark - 1u) | ((unit_no & 3u) << kRedoSetShift) | (need != 0u ? kRedoNeed : 0u);
          }
          __syncwarp();
          return true;
        };
        if (nu >= 3u) take_mark(nu - 3u);
        if (lane == 0) ctl->redo_mark[nu & 3u] = ctl->redo_need[nu & 3u] = 0u;
        int w = 0;
        uint32_t mode = 0u;
        bool again = false;  // (a unit's first time again)
        uint32_t state[4];
        ptx::ld_shared_volatile_vec<4>(ctl->redo_state, state);
        if (state[0] != 0u) {
          w = (int)((state[0] - 1u) & kRedoList);
          mode = kHdrRedo | (((state[0] - 1u) >> kRedoSetShift & 3u) << kHdrSetShift);
          __syncwarp();
          if (lane == 0) ctl->redo_state[0] = 0u;
        } else if (state[1] != state[2]) {
          const uint32_t e = *reinterpret_cast<volatile uint32_t*>(&ctl->redo_queue[state[1] & 3u]);
          w = (int)(e & kRedoList);
          mode = ((e & kRedoNeed) ? kHdrMax : kHdrRedo) | ((e >> kRedoSetShift & 3u) << kHdrSetShift);
          again = true;
          __syncwarp();
          if (lane == 0) {
            if (e & kRedoNeed) ctl->redo_state[0] = e + 1u;
            ctl->redo_state[1] = state[1] + 1u;
            ctl->redo_state[3] = 1u;
          }
        } else if (!drawn) {
          // a first unit by position, then from the counter; without pairs of CTAs a unit's two query
          // tiles are drawn one by one
          w = first_list();
          if (!first_item) {
            if (ONE) {
              w = INT_MAX;
            } else {
              if (lane == 0) w = (int)(PAIR ? gridDim.x >> 1 : gridDim.x) + atomicAdd(p.work_counter, 1);
              w = __shfl_sync(0xffffffffu, w, 0);
            }
          }
          first_item = false;
          drawn = (PAIR ? w : w >> 1) >= p.nUnits;
        }
        if (drawn && mode == 0u) {
          if (idle == 1) {
            // (all have taken the header without work: the last unit's mark is final, too)
            LOSA_WAIT(&ctl->hdr_empty[(nu - 1u) & 1u], ((nu - 1u) >> 1) & 1u);
            if (PAIR) ptx::fence_acq_rel_cluster();
            if (nu < 2u || !take_mark(nu - 2u)) break;
            idle = 0;
            continue;
          }
          ++idle;
          TILE_HDR_PUT(kTlSkip, 0u, 0, 0, 0, 0, 0, 0, nullptr, 0);
          LOSA_WAIT_RELAXED(&ctl->hdr_next, (nu - 1u) & 1u);
          continue;
        }
        idle = 0;
        const int list = w;  // its tile list
        const uint32_t odd = ((!PAIR && (w & 1)) ? kHdrOdd : 0u) | mode;
        if (!PAIR) w >>= 1;
        if (again && !ONE && lane == 0 && atomicExch(p.redo_flag + w, 1) == 0) atomicAdd(p.redo_count, 1);
        uint32_t flags = 0;
        if (w >= p.split_first) {
          int part;
          w = p.split_first + p.by_parts.divmod(w - p.split_first, part);
          flags = kTlPartial | ((uint32_t)part << 24);
        }
        int pr, problem, bh, h;
        item_place(p, w, problem, bh, pr);
        const int b = p.by_heads.divmod(bh, h);
        void* o = p.o;
        if (p.problems != nullptr) {
          o = p.problems[problem].o;
          // (without pairs of CTAs the producer's maps, ahead of it: 1 us)
          if (!PAIR && problem != acquired) {
            acquired = problem;
            acquire_tile_maps<D, C_, kHasV>(p.problems + problem, lane);
            __syncwarp();
          }
        }
        if (MODE == kSparse) {
          const bool own = ONE && mode == 0u;  // (made by this CTA)
          const uint32_t word = own ? own_word : LOSA_IN_RANGE(list, p.cap_units) ? (uint32_t)__ldcg(p.tl_count + list) : 0u;
          const int cnt = min((int)(word & kHdrTiles) * kG, p.tl_cap);
          TILE_HDR_PUT(kTlItem | flags | (uint32_t)w, (word & ~kHdrTiles) | odd | (uint32_t)(cnt / kG), 0, 0, pr, bh, b, h, o, problem);
          if (!publish_list(list, cnt, own)) goto teardown;
        } else {
          const uint32_t ent = kTlItem | flags | (uint32_t)w;
          int jlo, jhi;
          tile_key_range(p, ent, jlo, jhi);
          const bool two = 2 * pr + 1 < p.nQt;  // the pair's second query tile exists
          if (PAIR) {
            TILE_HDR_PUT(ent, mode | (two ? 3u : 1u) * kHdrHas | (uint32_t)((jhi - jlo + kG - 1) / kG), jlo, jhi, pr, bh, b, h, o, problem);
          } else {
            // (a query tile that does not exist is a unit without tiles)
            TILE_HDR_PUT(ent, odd | ((two || !(odd & kHdrOdd)) ? kHdrHas | (uint32_t)((jhi - jlo + kG - 1) / kG) : 0u), jlo, jhi, pr, bh, b, h,
                         o, problem);
          }
        }
        LOSA_WAIT_RELAXED(&ctl->hdr_next, (nu - 1u) & 1u);
      }
      if (!p.stall) TILE_HDR_PUT(kTlEnd, 0u, 0, 0, 0, 0, 0, 0, nullptr, 0);
      if (ONE && p.split_parts > 1 && lane == 0)
        p.redo_flag[first_list()] = *reinterpret_cast<volatile int*>(&ctl->redo_state[3]);
    }
  } else {
    // ------------------------------------------------------------------ softmax warps (both CTAs)
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(L::kRegsSoftmax));
    if (ctl->abort_flag) goto teardown;
    const int sw = warp - 4;
    const int grpi = sw >> 3, half = (sw >> 2) & 1, wl = sw & 3;  // group: which key tiles (even / odd)
    const int row = wl * 32 + lane;
    const uint32_t lane_base = (uint32_t)(wl * 32) << 16;
    const uint32_t tO = tmem_base + lane_base + 384;
    const int sub = (R == 64) ? (wl >> 1) : 0;   // query block of the query tile
    constexpr int kHB = (kG >= 2) ? kG / 2 : 1;  // key blocks of a half (a half block when C = 128)
    constexpr int kBW = 64 / kHB;                // columns per such block
    uint64_t* const pair_bar = &ctl->pair_bar[grpi * 4 + wl];
    const int quarter = grpi * 2 + half;         // which 32 columns of O this thread writes out
    // (cnt: bit 0 the uses of pair_bar, above it the units with a reference)
    uint32_t kq = 0, cnt = 0, nitem = 0, nfold = 0, nu = 0, nc = 0, hdr[4];
    // fused step: this row's column of the CTA's table of per-block sums of the unrounded
    // exponentials (one float per row and 64-column half of a key tile when a key block fills the
    // tile, else one per row and key block)
    float* const tabf = kWantMass ? reinterpret_cast<float*>(p.table) +
                                        (int64_t)blockIdx.x * 2 * (int64_t)p.nKb * 256 + row
                                  : nullptr;

    for (;;) {
      TILE_HDR_NEXT(hdr, 1);
      const uint32_t ent = hdr[0], word = hdr[1];
      if ((ent >> 28) == 2) break;
      // Which of the groups is through with the unit first, and leaves its end to the other.
      constexpr bool kExchange = kOneGroup && (!kSumCol || (kQB > 1 && MODE == kSparse));
      if (kExchange && (ent == kTlSkip || (word & kHdrMax))) {
        // (nothing to leave: keeps the phases of these barriers in step with the headers)
        if (lane == 0 && grpi == 0) ptx::mbar_arrive(&ctl->l_full[(nu - 1u) & 3u]);
      }
      if (ent == kTlSkip) continue;
      const int tile = PAIR ? (int)rank : (int)((word & kHdrOdd) != 0u);  // of the item's two query tiles
      const int my_bit = tile * kQB + sub;
      // where the unit lies, and what else of its header only its end needs: read again then, not kept in registers
      uint32_t info[7];
      auto read_info = [&]() {
        ptx::ld_shared_volatile_vec<4>(&ctl->hdr[(nu - 1u) & 3u][4], info);
        ptx::ld_shared_volatile_vec<2>(&ctl->hdr[(nu - 1u) & 3u][8], info + 4);
        if (kOneGroup) ptx::ld_shared_volatile_vec<1>(&ctl->hdr[(nu - 1u) & 3u][0], info + 6);
      };
      if (kInfoEarly) read_info();
      float m_ref = 0.f, l = 0.f, le = 0.f;  // le: row sum of the unrounded exponentials (masses, LSE)
      bool ovf = false, seen = false;  // (seen: this warp met keys that its rows attend to)
      const int tiles = (int)(word & kHdrTiles);
      const uint32_t pv_item = (uint32_t)tiles;
      // does this query tile list any of the unit's tiles?
      const bool has = (word & (PAIR ? kHdrHas << tile : kHdrHas)) != 0;
      // dense modes: the unit's key blocks, the end of its keys
      const int jlo = (int)hdr[2], jhi = (int)hdr[3];
      const int kend = min(p.N, jhi * kC);
      // Score k of the launch (kq: of the unit's first tile) is worked on by group k % 2 and lies in
      // buffer k % 3, in that buffer's use k / 3.
      const int first = (grpi ^ (int)kq) & 1;
      uint32_t bsel = (kq + (uint32_t)first) % 3u, sph = ((kq + (uint32_t)first) / 3u) & 1u;
      if (word & kHdrMax) {
        // ---- the rows' maxima over all keys they attend to, for a unit that is run again
        if (kOneGroup) {
          nitem = ctl->max_uses[sw];
          __syncwarp();
        }
        float mx = -INFINITY;
        for (int base = 0; base < tiles; base += kChunkTiles) {
          if (MODE == kSparse) TILE_CHUNK_WAIT();
          const int end = min(tiles, base + kChunkTiles);
          for (int i = base + first; i < end; i += 2) {
            uint32_t own[kHB];
            if (MODE == kSparse)
              ptx::ld_shared_volatile_vec<kHB>(
                  &ctl->tl[(nc & (kTlChunks - 1)) * 32 + (i - base) * kG + ((kG >= 2) ? half * kHB : 0)], own);
            LOSA_WAIT(&ctl->s_full[bsel], sph);
            ptx::tc_fence_after_sync();
#pragma unroll
            for (int c0 = 0; c0 < 64; c0 += 32) {
              uint32_t r[32];
              ptx::tmem_ld32(tmem_base + lane_base + bsel * 128 + half * 64 + c0, r);
              ptx::tmem_wait_ld();
#pragma unroll
              for (int c = 0; c < 32; ++c) {
                const int j = (c0 + c) / kBW;
                int valid;  // of the block's columns
                if (MODE == kSparse)
                  valid = ((own[j] >> (16 + my_bit)) & 1u)
                              ? p.N - (int)(own[j] & 0xffffu) * kC - ((kG == 1) ? 64 * half : 0) : 0;
                else
                  valid = has ? kend - (jlo + i * kG) * kC - 64 * half - j * kBW : 0;
                if ((c0 + c) % kBW < valid) mx = fmaxf(mx, __uint_as_float(r[c]));
              }
            }
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) arrive0<PAIR>(p_ready0 + 8u * bsel);
            if (bsel == 0u) {
              bsel = 2u;
            } else {
              bsel -= 1u;
              sph ^= 1u;
            }
          }
          if (MODE == kSparse) TILE_CHUNK_DONE();
        }
        kq += (uint32_t)tiles;
        // (where the unit would leave its sums)
        float* const xset = kOneGroup ? &ctl->xch[0][0][0] + ((nu - 1u) & 3u) * 512 : &ctl->xch[nitem & 1][0][0];
        xset[quarter * 128 + row] = mx;
        if (kOneGroup) ctl->max_uses[sw] = (uint8_t)(nitem + 1u);
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&ctl->item_bar);
        LOSA_WAIT(&ctl->item_bar, nitem & 1);
        if (!kOneGroup) ++nitem;
        // (every thread of the row finds and leaves the same value)
        ctl->redo_ref[(word >> kHdrSetShift) & 3u][row] = fmaxf(fmaxf(xset[row], xset[128 + row]), fmaxf(xset[256 + row], xset[384 + row])) * p.scale_log2;
        continue;
      }
      // ---- the reference of the unit: the rows' maximum over the first key tile their query block
      // lists, from the group that works on that tile to the other.  Where the query tile is a query
      // block that tile is one of the unit's first two, the first of the group that works on it, and
      // the reference is exchanged here; with two query blocks (R = 64) and a list it may be any tile
      // and is exchanged when the loop below comes to it.
      constexpr bool kLazyRef = kQB > 1 && MODE == kSparse;
      const uint32_t rs = (cnt >> 1) & 1u;
      const bool redo = (word & kHdrRedo) != 0;  // against what the unit's rows are known to reach
      bool have_ref = !has || redo;
      if (redo) m_ref = ctl->redo_ref[(word >> kHdrSetShift) & 3u][row];
      int ref_tile = (PAIR && tile == 1 && (word & kHdrLate)) ? 1 : 0;
      bool listed_only = true;  // the maximum is over the keys the row attends to
      // The maximum of this half's 64 columns of tile i of the unit, whose group lies at `at` in the list's
      // chunk; the halves exchange theirs.  (Over all 128 columns by each half, column by column, it took a unit's
      // first softmax group 1.1 us, for which the other group waits.)
      auto half_max = [&](int i, uint32_t chunk, int at) {
        const uint32_t tSh = tmem_base + lane_base + bsel * 128 + half * 64;
        int hv[kHB];  // columns of each block that count
        bool whole = true;
        uint32_t e[kHB];
        if (MODE == kSparse)
          ptx::ld_shared_volatile_vec<kHB>(&ctl->tl[(chunk & (kTlChunks - 1)) * 32 + at + ((kG >= 2) ? half * kHB : 0)], e);
#pragma unroll
        for (int j = 0; j < kHB; ++j) {
          if (MODE == kSparse)
            hv[j] = (!listed_only || ((e[j] >> (16 + my_bit)) & 1u))
                        ? p.N - (int)(e[j] & 0xffffu) * kC - ((kG == 1) ? 64 * half : 0) : 0;
          else
            hv[j] = kend - (jlo + i * kG) * kC - 64 * half - j * kBW;
          whole = whole && hv[j] >= kBW;
        }
        uint32_t r[64];
        ptx::tmem_ld32(tSh, &r[0]);
        ptx::tmem_ld32(tSh + 32, &r[32]);
        ptx::tmem_wait_ld();
        if (!whole) {
#pragma unroll
          for (int c = 0; c < 64; ++c)
            if ((c % kBW) >= hv[c / kBW]) r[c] = 0xff800000u;
        }
        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int c = 0; c < 64; c += 2) mx[(c >> 1) & 3] = ptx::max3(mx[(c >> 1) & 3], __uint_as_float(r[c]), __uint_as_float(r[c + 1]));
        return fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * p.scale_log2;
      };
      // (m_ref of the group that has it)
#define TILE_REF_GIVE(half_mx)                                                                      \
  do {                                                                                              \
    const float mx_ = (half_mx);                                                                    \
    ctl->half_max[rs][half][row] = mx_;                                                             \
    __syncwarp();                                                                                   \
    if (lane == 0) ptx::mbar_arrive(pair_bar);                                                      \
    LOSA_WAIT(pair_bar, cnt & 1u);                                                                  \
    cnt ^= 1u;                                                                                      \
    m_ref = fmaxf(mx_, ctl->half_max[rs][half ^ 1][row]);                                           \
    if (half == 0) {                                                                                \
      /* (the slot's last readers, two units with a reference ago, are done with it) */             \
      if (cnt >= 4u) LOSA_WAIT(&ctl->ref_empty[rs][sub], ((cnt >> 2) - 1u) & 1);                    \
      ctl->ref[rs][row] = m_ref;                                                                    \
      __syncwarp();                                                                                 \
      if (lane == 0) ptx::mbar_arrive(&ctl->ref_full[rs][sub]);                                     \
    }                                                                                               \
  } while (0)
#define TILE_REF_TAKE()                                                                             \
  do {                                                                                              \
    LOSA_WAIT(&ctl->ref_full[rs][sub], (cnt >> 2) & 1);                                             \
    m_ref = ctl->ref[rs][row];                                                                      \
    __syncwarp();                                                                                   \
    if (lane == 0) ptx::mbar_arrive(&ctl->ref_empty[rs][sub]);                                      \
  } while (0)
      if (has && !redo) {
        if (kLazyRef) {
          // a query block that lists none of the first chunk's entries takes the maximum over all keys
          // of the first tile
          TILE_CHUNK_WAIT();
          const uint32_t e = *reinterpret_cast<volatile uint32_t*>(&ctl->tl[(nc & (kTlChunks - 1)) * 32 + lane]);
          const uint32_t mine = __ballot_sync(0xffffffffu, lane < tiles * kG && ((e >> (16 + my_bit)) & 1u));
          listed_only = mine != 0u;
          ref_tile = listed_only ? (__ffs(mine) - 1) / kG : 0;
        } else {
          if (first == ref_tile) {
            if (MODE == kSparse) TILE_CHUNK_WAIT();
            LOSA_WAIT(&ctl->s_full[bsel], sph);
            ptx::tc_fence_after_sync();
            TILE_REF_GIVE(half_max(first, nc, first * kG));
          } else {
            TILE_REF_TAKE();
          }
          have_ref = true;
        }
      }
      const float2 sc2 = make_float2(p.scale_log2, p.scale_log2);
      for (int base = 0; base < tiles; base += kChunkTiles) {
      if (MODE == kSparse) TILE_CHUNK_WAIT();
      const int end = min(tiles, base + kChunkTiles);
      for (int i = base + first; i < end; i += 2) {
        // the key blocks of this half of the tile: a half block (C = 128), one block, or two (C = 32)
        uint32_t own[kHB];
        bool mine, ragged;  // the row attends to some of the half's keys; not all of them exist
        if (MODE == kSparse) {
          const uint32_t* e = &ctl->tl[(nc & (kTlChunks - 1)) * 32 + (i - base) * kG + ((kG >= 2) ? half * kHB : 0)];
          ptx::ld_shared_volatile_vec<kHB>(e, own);
          uint32_t any = 0u;
#pragma unroll
          for (int j = 0; j < kHB; ++j) any |= ((own[j] >> (16 + my_bit)) & 1u) ? own[j] : 0u;
          ragged = (any & kTlRagged) != 0u;
          mine = any != 0u;
          if (kG == 1 && ragged) mine = p.N - (int)(own[0] & 0xffffu) * kC > 64 * half;
        } else {
          const int key0 = (jlo + i * kG) * kC + 64 * half;
          mine = has && key0 < kend;
          ragged = key0 + 64 > kend;
        }
        const uint32_t tS = tmem_base + lane_base + bsel * 128 + half * 64;
        LOSA_WAIT(&ctl->s_full[bsel], sph);
        ptx::tc_fence_after_sync();
        if (kLazyRef && !have_ref && i >= ref_tile) {
          if (i == ref_tile) {
            TILE_REF_GIVE(half_max(i, nc, (i - base) * kG));
          } else {
            TILE_REF_TAKE();
          }
          have_ref = true;
        }
        uint32_t sr[64];
        if (kQB > 1) seen = seen || mine;
        if (mine) {
          ptx::tmem_ld32(tS, &sr[0]);
          ptx::tmem_wait_ld();
          if (!kSumCol) ptx::tmem_ld32(tS + 32, &sr[32]);
          // keys that do not exist (>= N, in the sequence's last key block): -inf column by column
          auto cut_ragged = [&](int from, int to) {
            int hv[kHB];
#pragma unroll
            for (int j = 0; j < kHB; ++j) {
              if (MODE == kSparse) hv[j] = p.N - (int)(own[j] & 0xffffu) * kC - ((kG == 1) ? 64 * half : 0);
              else hv[j] = kend - (jlo + i * kG) * kC - 64 * half - j * kBW;
            }
#pragma unroll
            for (int c = 0; c < 64; ++c)
              if (c >= from && c < to && (c % kBW) >= hv[c / kBW]) sr[c] = 0xff800000u;
          };
          if (ragged) {
            if (!kSumCol) ptx::tmem_wait_ld();
            cut_ragged(0, kSumCol ? 32 : 64);
          }
          if (!kHasV) {
            // mass pass: the scores are in registers and nothing is packed over them
            ptx::tmem_wait_ld();
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) arrive0<PAIR>(p_ready0 + 8u * bsel);
          }
          // key blocks the row's query block does not list get -inf as the addend of the scaling FMA
          // (one block per half or less: the half would not be here)
          float2 nm2[kHB];
#pragma unroll
          for (int j = 0; j < kHB; ++j) {
            const bool listed = MODE != kSparse || kHB == 1 || ((own[j] >> (16 + my_bit)) & 1u);
            const float a = listed ? -m_ref : -INFINITY;
            nm2[j] = make_float2(a, a);
          }
          // The output is normalised by the sum of the weights the tensor core multiplies with V -
          // P as rounded to bf16 - so that o is a weighted mean of V whatever the rounding does.
          float2 racc[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
          float2 eacc[kHB];  // fused step: sums of the unrounded exponentials, per block of this half
#pragma unroll
          for (int j = 0; j < kHB; ++j) eacc[j] = make_float2(0.f, 0.f);
#pragma unroll
          for (int c = 0; c < 64; c += 4) {
            if (kSumCol && c == 24) ptx::tmem_ld32(tS + 32, &sr[32]);
            if (kSumCol && c == 32) ptx::tmem_st16(tS, &sr[0]);
            if (kHasV && c == 32) {
              ptx::tmem_wait_ld();
              if (kSumCol && ragged) cut_ragged(32, 64);
            }
            float2 x0 = ptx::fma2(make_float2(__uint_as_float(sr[c]), __uint_as_float(sr[c + 1])), sc2,
                                  nm2[c / kBW]);
            float2 x1 = ptx::fma2(make_float2(__uint_as_float(sr[c + 2]), __uint_as_float(sr[c + 3])), sc2,
                                  nm2[c / kBW]);
            // (at head dimension 128 a share of these on the FMA pipe measured -1 % at 12.5 % and +5 % at 25 %)
            if (kPolyOf > 0 && (c >> 2) % (kPolyOf > 0 ? kPolyOf : 1) == kPolyAt) {
              x0 = ptx::ex2_poly2(x0);
              x1 = ptx::ex2_poly2(x1);
            } else {
              x0.x = ptx::ex2_approx(x0.x);
              x0.y = ptx::ex2_approx(x0.y);
              x1.x = ptx::ex2_approx(x1.x);
              x1.y = ptx::ex2_approx(x1.y);
            }
            if (kHasV) {
              const uint32_t u0 = ptx::pack_bf16x2(x0.x, x0.y), u1 = ptx::pack_bf16x2(x1.x, x1.y);
              sr[c >> 1] = u0;
              sr[(c >> 1) + 1] = u1;
              if (!kSumCol) {
                ptx::add_bf16x2(racc[0], u0);
                ptx::add_bf16x2(racc[1], u1);
              }
            }
            if (kWantMass) eacc[c / kBW] = ptx::add2(eacc[c / kBW], ptx::add2(x0, x1));
          }
          float tsum = (racc[0].x + racc[0].y) + (racc[1].x + racc[1].y);
          if (!kHasV) {
#pragma unroll
            for (int j = 0; j < kHB; ++j) tsum += eacc[j].x + eacc[j].y;
          }
          // (in the mass pass l is le once more; without it, and with a vote over the whole sums at the unit's end, the
          // compiler ordered the exponentials worse: 1024 key blocks 4090 us against 4300)
          if (!kSumCol) {
            // (the same twice; which, is a matter of the order that the compiler finds: masses, 16384 tokens, 12 heads, D = 64
            // with 128-key blocks 872 / 836 us, with 64 825 / 856; D = 128 969 - 1043 / 957 - 1010)
            if (MODE == kMass && !(D == 64 && C_ == 64)) ovf = __any_sync(0xffffffffu, ovf || !(tsum <= kSplitSafeSum));
            else ovf = ovf || __any_sync(0xffffffffu, !(tsum <= kSplitSafeSum));
            l += tsum;
          }
          if (kSumCol) ptx::tmem_st16(tS + 16, &sr[16]);
          else if (kHasV) ptx::tmem_st32(tS, &sr[0]);
          if (kWantMass) {
#pragma unroll
            for (int j = 0; j < kHB; ++j) {
              const float es = eacc[j].x + eacc[j].y;
              le += es;
              // (kG = 1: entry of this half of the key block; else of the key block)
              const int sb = (kG >= 2) ? jlo + i * kG + half * kHB + j : (jlo + i) * 2 + half;
              const bool exists = kHB == 1 || sb < jhi;
              if (exists && LOSA_IN_RANGE((int64_t)sb * 128 + row, p.cap_table_floats)) tabf[(int64_t)sb * 128] = es;
            }
          }
        } else {
          // this half of the row lists none of the tile's keys: P = 0
          if (kHasV) {
            uint32_t z[32];
#pragma unroll
            for (int c = 0; c < 32; ++c) z[c] = 0u;
            ptx::tmem_st32(tS, z);
          } else {
            // mass pass: the buffer goes back untouched
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) arrive0<PAIR>(p_ready0 + 8u * bsel);
          }
          // (a key block that fills the tile but ends before this half: its entry of the table is 0)
          if (kWantMass && kG == 1 && has &&
              LOSA_IN_RANGE(((int64_t)(jlo + i) * 2 + half) * 128 + row, p.cap_table_floats))
            tabf[((int64_t)(jlo + i) * 2 + half) * 128] = 0.f;
        }
        if (kHasV) {
          ptx::tmem_wait_st();
          ptx::tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) arrive0<PAIR>(p_ready0 + 8u * bsel);
        }
        // two scores on: k + 2 lies in the buffer before k's, in that buffer's next use, or in the last one
        if (bsel == 0u) {
          bsel = 2u;
        } else {
          bsel -= 1u;
          sph ^= 1u;
        }
      }
      if (MODE == kSparse) TILE_CHUNK_DONE();
      }
      kq += (uint32_t)tiles;

      // ---- end of the item
      if (kLazyRef && !have_ref) TILE_REF_TAKE();  // (this group met no tile from the reference's on)
      if (has && !redo) cnt += 2u;
#undef TILE_REF_GIVE
#undef TILE_REF_TAKE
      if (!kInfoEarly) read_info();
      const uint32_t item = kOneGroup ? info[6] : ent;
      const int w = (int)(item & kTlItemMask);
      const bool partial = (item & kTlPartial) != 0;
      const int part = (int)((item >> 24) & 7u);
      const int pr = (int)info[0], bh = (int)info[1], b = (int)info[2], h = (int)info[3];
      void* const o_base = reinterpret_cast<void*>((uint64_t)info[4] | ((uint64_t)info[5] << 32));
      const int T = 2 * pr + tile;
      const int grow = T * 128 + row;
      auto hand_over = [&]() {
        mark_cluster();
        const int unit = partial ? p.split_first + (w - p.split_first) * p.split_parts + part : w;
        const uint32_t mark = 1u + (uint32_t)(PAIR ? unit : 2 * unit + tile);
        if (PAIR) {
          ptx::st_cluster_u32(redo_mark0 + 4u * ((nu - 1u) & 3u), mark);
          ptx::fence_acq_rel_cluster();
        } else {
          *reinterpret_cast<volatile uint32_t*>(&ctl->redo_mark[(nu - 1u) & 3u]) = mark;
        }
      };
      if (!kSumCol && ovf && !redo && lane == 0) hand_over();
      // What the row is run again against, should any of the unit's rows have outgrown its reference, from the row's
      // whole sum (one thread of a row).
      auto leave_ref = [&](float sum) {
        ctl->redo_ref[(nu - 1u) & 3u][row] = (sum > 0.f) ? m_ref + __log2f(sum) : m_ref;
        if (!(sum < kTileKnownHigh) || (kLazyRef && seen && sum < kTileKnownLow)) {
          if (PAIR) {
            ptx::st_cluster_u32(redo_mark0 + 16u + 4u * ((nu - 1u) & 3u), 1u);
            ptx::fence_acq_rel_cluster();
          } else {
            *reinterpret_cast<volatile uint32_t*>(&ctl->redo_need[(nu - 1u) & 3u]) = 1u;
          }
        }
      };
      // Columns c0 ... of the rows of O of this warp's 32 lanes, a row a lane, to `dst` (rows of `stride` elements of
      // 4 bytes, or of 2 and rounded); those from `rows` on do not exist.  Groups of lanes write a row's columns
      // together: with a row a lane every store of 16 bytes went to 32 lines, and the 2048 cycles that took held up
      // the copies, the next unit's reference and whatever else goes through shared memory.
      auto store_rows = [&](uint32_t* r, void* dst, int64_t stride, int rows, float by, bool f32, auto cols) {
        constexpr int kCols = decltype(cols)::value;
#pragma unroll
        for (int c = 0; c < kCols; ++c) r[c] = __float_as_uint(__uint_as_float(r[c]) * by);
        if (f32) {
#pragma unroll
          for (int c = 0; c < kCols; c += 16) {
            transpose_chunks<4>(r + c, lane);
            float* to = static_cast<float*>(dst) + (int64_t)(lane & ~3) * stride + c + 4 * (lane & 3);
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if ((lane & ~3) + i < rows)
                *reinterpret_cast<uint4*>(to + i * stride) = make_uint4(r[c + 4 * i], r[c + 4 * i + 1], r[c + 4 * i + 2], r[c + 4 * i + 3]);
          }
        } else {
          constexpr int kN = kCols / 8;  // chunks of a row
#pragma unroll
          for (int c = 0; c < kCols; c += 2) r[c >> 1] = ptx::pack_bf16x2(__uint_as_float(r[c]), __uint_as_float(r[c + 1]));
          transpose_chunks<kN>(r, lane);
          __nv_bfloat16* to = static_cast<__nv_bfloat16*>(dst) + (int64_t)(lane & ~(kN - 1)) * stride + 8 * (lane & (kN - 1));
#pragma unroll
          for (int i = 0; i < kN; ++i)
            if ((lane & ~(kN - 1)) + i < rows)
              *reinterpret_cast<uint4*>(to + i * stride) = make_uint4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
        }
      };
      const int row0 = T * 128 + wl * 32;  // of this warp
      const int rows = (T < p.nQt) ? p.N - row0 : 0;
      // the same to O
      auto store_o = [&](uint32_t* r, int c0, float inv, auto cols) {
        const int64_t off = (int64_t)b * p.sb + (int64_t)h * p.sh + (int64_t)row0 * p.sn + c0;
        store_rows(r, p.o_f32 ? static_cast<void*>(static_cast<float*>(o_base) + off)
                              : static_cast<void*>(static_cast<__nv_bfloat16*>(o_base) + off),
                   p.sn, rows, inv, p.o_f32 != 0, cols);
      };
      if constexpr (kOneGroup) {
        // The group that worked on the unit's last tile writes O out; the other, whose turn the next tile
        // is, goes on to the next unit, so that the special-function unit has work while the last product
        // runs and O is read.  It may be two units ahead before O is free: four sets of partial sums.
        const uint32_t set = (nu - 1u) & 3u, phase = ((nu - 1u) >> 2) & 1u;
        float* const xset = &ctl->xch[0][0][0] + set * 512;
        if (!kSumCol) xset[quarter * 128 + row] = l;
        if (kLazyRef && lane == 0) ctl->seen[set][sw] = seen ? 1 : 0;
        const bool last = grpi == (int)((kq - 1u) & 1u);
        if (kExchange) {
          __syncwarp();
          if (last) {
            if (lane == 0) ptx::mbar_arrive(pair_bar);
            LOSA_WAIT(pair_bar, cnt & 1u);
            cnt ^= 1u;
            LOSA_WAIT(&ctl->l_full[set], phase);
          } else if (lane == 0) {
            ptx::mbar_arrive(&ctl->l_full[set]);
          }
        }
        if (!last) continue;
        if (!kSumCol) l = (xset[row] + xset[128 + row]) + (xset[256 + row] + xset[384 + row]);
        if (kLazyRef) {
          const volatile uint8_t* met = ctl->seen[set];
          seen = (met[wl] | met[4 + wl] | met[8 + wl] | met[12 + wl]) != 0;
        }
        constexpr int kOC = D / 2;  // columns of this half
        float inv = 0.f;
        const int64_t pslot = ((((int64_t)(w - p.split_first) * p.split_parts + part) * 2 + tile) * 128 + row);
        if (pv_item > 0) {
          LOSA_WAIT(&ctl->o_done[set], phase);
          ptx::tc_fence_after_sync();
        }
#pragma unroll
        for (int c0 = 0; c0 < kOC; c0 += 32) {
          uint32_t r[32];
          if (pv_item > 0) {
            ptx::tmem_ld32(tO + half * kOC + c0, r);
            if (kSumCol && c0 == 0) l = __uint_as_float(ptx::tmem_ld1(tO + D));
            ptx::tmem_wait_ld();
            if (c0 + 32 == kOC) {
              // (O is in registers: the next item's first product may overwrite it)
              ptx::tc_fence_before_sync();
              __syncwarp();
              if (lane == 0) arrive0<PAIR>(o_free0);
            }
          } else {
#pragma unroll
            for (int c = 0; c < 32; ++c) r[c] = 0u;
          }
          if (c0 == 0) {
            // rows whose own keys lie 40 nats below a reference taken over other keys: their weights may
            // have lost their tail
            if (!redo && half == 0) leave_ref(l);
            const bool low = kLazyRef && seen && l < kTileSafeLow;
            if ((kLazyRef || kSumCol) && !redo &&
                __any_sync(0xffffffffu, low || (kSumCol && !(l <= kSplitSafeSum))) && lane == 0)
              hand_over();
            // (run again only rows that met a score that is not a number add up to that much)
            if (redo && !(l <= kSplitSafeSum)) l = __int_as_float(0x7fc00000);
            inv = (l == 0.f) ? 0.f : 1.f / l;
            if (in_cluster) {
              if (half == 0) park_ml[row] = make_float2(m_ref, l);
            } else if (partial && half == 0 && T < p.nQt && LOSA_IN_RANGE(pslot, p.cap_part_rows)) {
              p.part_ml[pslot] = make_float2(m_ref, l);
            }
          }
          if (in_cluster) {
            // (16 bytes of a row lie where eight lanes' stores meet no bank twice)
#pragma unroll
            for (int c = 0; c < 32; c += 4)
              park_o[row * (D / 4) + ((((half * kOC + c0 + c) >> 2) & ~7) | ((((half * kOC + c0 + c) >> 2) ^ row) & 7))] =
                  make_uint4(r[c], r[c + 1], r[c + 2], r[c + 3]);
            // (the copies of a unit that is run again come behind this)
            if (c0 + 32 == kOC) ptx::fence_proxy_async();
          } else if (partial) {
            const int64_t slot0 = pslot - lane;  // (of the warp's first row; 32 rows of it exist in any case)
            if (T < p.nQt)
              store_rows(r, p.part_o + (LOSA_IN_RANGE(pslot, p.cap_part_rows) ? slot0 : 0) * D + half * kOC + c0, D, 32,
                         1.f, true, std::integral_constant<int, 32>());
          } else {
            store_o(r, half * kOC + c0, inv, std::integral_constant<int, 32>());
          }
        }
        continue;
      }
      // the four partial sums of a row (two groups, two halves) meet in shared memory
      float* const xset = &ctl->xch[nitem & 1][0][0];
      if (!kSumCol) xset[quarter * 128 + row] = l;
      xset[(4 + quarter) * 128 + row] = le;
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&ctl->item_bar);
      LOSA_WAIT(&ctl->item_bar, nitem & 1);
      ++nitem;
      if (!kSumCol) l = (xset[row] + xset[128 + row]) + (xset[256 + row] + xset[384 + row]);
      // every thread writes out a quarter of its row of O
      constexpr int kOC = kHasV ? D / 4 : 1;
      const int c0 = quarter * kOC;
      uint32_t r[kOC];
      if (kHasV) {
        if (pv_item > 0) {
          LOSA_WAIT(&ctl->o_done[(nu - 1u) & 3u], ((nu - 1u) >> 2) & 1u);
          ptx::tc_fence_after_sync();
          if constexpr (kOC == 32) ptx::tmem_ld32(tO + c0, r);
          else if constexpr (kOC == 16) ptx::tmem_ld16(tO + c0, r);
          if (kSumCol) l = __uint_as_float(ptx::tmem_ld1(tO + D));
          ptx::tmem_wait_ld();
          // (O is in registers: the next item's first product may overwrite it)
          ptx::tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) arrive0<PAIR>(o_free0);
        } else {
#pragma unroll
          for (int c = 0; c < kOC; ++c) r[c] = 0u;
        }
        if (kSumCol && !redo && __any_sync(0xffffffffu, !(l <= kSplitSafeSum)) && lane == 0) hand_over();
        if (!redo && quarter == 0) leave_ref(l);
        // (run again only rows that met a score that is not a number add up to that much)
        if (redo && !(l <= kSplitSafeSum)) l = __int_as_float(0x7fc00000);
        store_o(r, c0, (l == 0.f) ? 0.f : 1.f / l, std::integral_constant<int, kOC>());
      }
      if (!kHasV && !redo && quarter == 0) leave_ref(l);
      if (kWantMass) {
        // ---- fused construction step: the block masses of this CTA's query tile (Eq. 1).  The
        // reference did not move during the item, so a row's weight is 1 / (its sum of unrounded
        // exponentials) and a mass is the mean over the query block's rows of weight x (the row's
        // sum over the key block).  The table was written by this CTA's softmax threads before the
        // item's barrier; all 16 warps fold it, key block by key block.
        if (quarter == 0 && T < p.nQt && grow < p.N && p.lse != nullptr &&
            LOSA_IN_RANGE((int64_t)bh * p.N + grow, p.cap_lse)) {
          const float le_row = (xset[512 + row] + xset[640 + row]) + (xset[768 + row] + xset[896 + row]);
          p.lse[(int64_t)bh * p.N + grow] =
              (!redo || le_row <= kSplitSafeSum) ? (m_ref + log2f(le_row)) * kLn2 : __int_as_float(0x7fc00000);
        }
        if (T < p.nQt) {
          const float* tb = reinterpret_cast<const float*>(p.table) + (int64_t)blockIdx.x * 2 * (int64_t)p.nKb * 256;
          // Lane l sums rows 4 l .. 4 l + 3 of four key blocks at a time: one 16-byte load per block (two
          // where the halves of a block have entries of their own) and four blocks in flight.  The fold is
          // the latency of these loads: one block at a time in four 4-byte loads, the mass pass took 4523 us
          // with 1024 key blocks (32760 tokens, 12 heads) and takes 4250.
          float iv[4];
#pragma unroll
          for (int rr = 0; rr < 4; ++rr) {
            const int r = 4 * lane + rr;
            const float le_r = (xset[512 + r] + xset[640 + r]) + (xset[768 + r] + xset[896 + r]);
            iv[rr] = (T * 128 + r < p.N && le_r > 0.f && (!redo || le_r <= kSplitSafeSum)) ? 1.f / le_r : 0.f;
          }
          constexpr int kFold = 4, kParts = (kG >= 2) ? 1 : 2;
          for (int u0 = sw; u0 < p.nKb; u0 += 16 * kFold) {
            float4 t[kFold][kParts];
#pragma unroll
            for (int j = 0; j < kFold; ++j) {
#pragma unroll
              for (int q = 0; q < kParts; ++q)
                t[j][q] = (u0 + 16 * j < p.nKb)
                              ? reinterpret_cast<const float4*>(tb)[((int64_t)(u0 + 16 * j) * kParts + q) * 32 + lane]
                              : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int j = 0; j < kFold; ++j) {
              const float4 a = t[j][0], b = t[j][kParts - 1];
              float acc = 0.f;
              acc += (iv[0] > 0.f) ? (kParts == 2 ? a.x + b.x : a.x) * iv[0] : 0.f;
              acc += (iv[1] > 0.f) ? (kParts == 2 ? a.y + b.y : a.y) * iv[1] : 0.f;
              acc += (iv[2] > 0.f) ? (kParts == 2 ? a.z + b.z : a.z) * iv[2] : 0.f;
              acc += (iv[3] > 0.f) ? (kParts == 2 ? a.w + b.w : a.w) * iv[3] : 0.f;
#pragma unroll
              for (int d = 16 / kQB; d > 0; d >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
              const int g = T * kQB + lane / (32 / kQB);  // query block of this lane's rows
              const int u = u0 + 16 * j;
              const int64_t mi = ((int64_t)bh * p.nQb + g) * p.nKb + u;
              if (lane % (32 / kQB) == 0 && u < p.nKb && g < p.nQb && LOSA_IN_RANGE(mi, p.cap_mass))
                p.mass[mi] = acc / (float)min(R, p.N - g * R);
            }
          }
        }
        // (the table is written again by the next item)
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&ctl->fold_bar);
        LOSA_WAIT(&ctl->fold_bar, nfold & 1);
        ++nfold;
      }
    }
  }

teardown:
  if (ctl->abort_flag) {
    // the other CTA's waits give up at their next look at the flag (where all have met already, none is left to be told,
    // and that CTA may be gone)
    if (PAIR && lane == 0 && !(ONE && over == 1)) ptx::st_cluster_u32(abort_peer, 1u);
    // give MMAs and bulk copies still in flight a bounded time to land before shared memory and
    // tensor memory are released
    if (rank == 0 && (warp == kIssuerWarp || warp == kIssuerWarp + 1) && ptx::elect_one()) {
      commit0<PAIR>(&ctl->drain);
      for (uint32_t it = 0; it < (1u << 16); ++it) {
        if (ptx::mbar_try_wait(&ctl->drain, 0)) break;
        __nanosleep(128);
      }
    }
    if (warp == kProducerWarp && lane == 0) {
      for (uint32_t it = 0; it < (1u << 10); ++it) __nanosleep(1024);
    }
  }
  // neither CTA leaves, or frees its tensor memory, while the other may still signal into it
  if (ONE && over < 0) unit_over();
  if (!ONE || over != 1) {
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (PAIR || in_cluster) ptx::cluster_sync();
  }
  if constexpr (ONE && kOneGroup) {
    if (in_cluster) {
      // (every part has left its rows; none leaves the cluster before they are read)
      if (warp >= 4 && !ctl->abort_flag) {
        const int list = first_list();
        merge_in_cluster<D>(p, PAIR ? list : list >> 1, PAIR ? (int)rank : list & 1, PAIR ? rank : 0u, PAIR ? 2u : 1u,
                            ptx::smem_u32(park_o), ptx::smem_u32(park_ml), warp - 4, lane);
      }
      __syncwarp();
      ptx::cluster_arrive_relaxed();
      ptx::cluster_wait();
    }
  }
  if (warp == kIssuerWarp) {
    ptx::tc_fence_after_sync();
    if (PAIR) ptx::tmem_dealloc2(tmem_base, kTmemCols);
    else ptx::tmem_dealloc(tmem_base, kTmemCols);
  }
}

#undef TILE_HDR_PUT
#undef TILE_HDR_NEXT
#undef TILE_CHUNK_WAIT
#undef TILE_CHUNK_DONE
#undef TILE_WAIT
