// losa_select: retained-mass selection (Eq. 3) and CSR validation.
//
// Two launches over a [rows, nKb] fp32 mass matrix:
//   1. select_rows_kernel   one warp per row of at most 1024 blocks, two, four or eight warps for
//                           longer rows; the row stays in registers, the threshold value is found
//                           with one histogram pass (no sort); the kept set is written as a bitmap
//                           over block indices plus its size.
//   2. expand_rows_kernel   every CTA adds up the sizes of the rows before its own (offsets) and
//                           turns its rows' bitmaps into ascending block indices.
// Few rows take one launch of one cluster instead (select_small_kernel).
// Each mass element is read once and each kept index written once; the bitmap adds 1/16
// of the mass bytes.  The result is deterministic (no floating-point atomics).
#include <limits.h>

#include <atomic>

#include "losa_common.cuh"
#include "losa_ptx.cuh"

namespace losa {
namespace {

// The kept set of Eq. 3 is "every block heavier than v*, plus the lowest-indexed blocks equal to v*
// until the sum reaches tau", where v* is the largest value v with sum(mass >= v) >= tau.
// Non-negative floats order like their bit patterns, so the row is split into bins by the leading
// bits: the exponent and four mantissa bits.  All values of a bin share their exponent, so a bin's
// sum is exact in two 32-bit integers - how many values, and the sum of their 19 low mantissa bits
// (8192 of them stay below 2^32) - which the warps gather with shared-memory integer atomics.  A
// scan over the bins from the heaviest down, in 2^-60 fixed point, gives the bin of v*; its few
// values are put into a list, and v* is found among them bit by bit.  Integer addition is exact and
// order-independent, so the result is deterministic and differs from a sequential fp64 sum by less
// than 1e-14 (masses below 2^-37 lose low bits).
//
// A bin with more values than the list holds (diffuse masses: nearly all of a row may lie within a
// sixteenth of a binade) is split by its values' next bits, with the same histogram and scan: by the
// nine after those that all of them share, and again where a bin of those is crowded still.  22296 rows of
// 3713 masses within 3 % of one another take 406 us (216 us where they spread over orders of magnitude), of
// 929 masses within 1e-4 163 us; searched bit by bit over the row they took 3014 and 1336 us, and before the
// histogram 6128 (sorted) and 415 us.
//
// The bins end at the mass limit 8 and begin kBins * 2^(1/16) steps below it (about 2^-35): lighter
// values share bin 0.  A threshold in bin 0 is searched bit by bit over the row instead (31 masked
// sums).  The fixed-ratio rule only counts: its bins take one mantissa bit and reach down to zero.
//
// What bounds it: instructions per value (1300 per warp of 29 blocks a lane; 69 % of the issue slots).
// 22296 rows of 3713 blocks take 155 us, and 67 us to expand; with a sort in shared memory, which
// moved every value about 70 times, both took 5.48 ms, and rows of up to 1024 blocks, searched bit by
// bit with 31 masked 64-bit sums, 0.33 ms at 929 blocks.
constexpr int kBins = 608;   // per lane of one warp 19, an odd number: the scan has no bank conflicts
constexpr int kTauShift = 19, kCountShift = 22;
constexpr uint32_t kMaxMassBits = 0x41000000u;       // the largest mass, 8.0
constexpr int kTopBin = kMaxMassBits >> kTauShift;
constexpr int kListCap = 256;
constexpr int kSplitBins = 512;  // ... of a bin with more values than the list holds
constexpr double kFixedOne = 1152921504606846976.0;  // 2^60

struct RowShared {
  uint32_t cnt[kBins], low[kBins];
  uint32_t list[kListCap];
  unsigned long long total[8];   // per warp of the row
  unsigned long long above;      // weight of the bins heavier than the one of v*
  double sum[8];
  int bin, list_len;
  uint32_t v;
  int need, eq_total;
  int part[8];
};

// (cap: see `tiny` below)
__device__ __forceinline__ unsigned long long fixed_weight(uint32_t bits, double scale, double cap) {
  return (unsigned long long)(fmin((double)__uint_as_float(bits), cap) * scale);
}

// warp sum of 64-bit values as three integer reductions of 22-bit limbs (one instruction each)
__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long a) {
  const unsigned r0 = __reduce_add_sync(0xffffffffu, (unsigned)(a & 0x3fffffull));
  const unsigned r1 = __reduce_add_sync(0xffffffffu, (unsigned)((a >> 22) & 0x3fffffull));
  const unsigned r2 = __reduce_add_sync(0xffffffffu, (unsigned)(a >> 44));
  return (unsigned long long)r0 + ((unsigned long long)r1 << 22) + ((unsigned long long)r2 << 44);
}

template <int W>  // warps per row
__device__ __forceinline__ void row_sync() {
  if (W == 1) __syncwarp();
  else __syncthreads();  // (the row has the CTA to itself)
}

// sum over the row's threads (W > 1: through shared memory; every thread gets the result)
template <int W>
__device__ __forceinline__ unsigned long long row_sum_u64(unsigned long long a, RowShared* rs, int warp, int lane) {
  a = warp_sum_u64(a);
  if (W == 1) return a;
  if (lane == 0) rs->total[warp] = a;
  __syncthreads();
  unsigned long long t = 0ull;
#pragma unroll
  for (int w = 0; w < W; ++w) t += rs->total[w];
  __syncthreads();
  return t;
}

// What a list of m values (low bits x) is searched for: the largest v with weight(values >= v) >= missing,
// and how many of the values equal to v are needed.  A value weighs lead + x, or 1 if COUNT.  Whole warp.
// A list of more than eight values is first split by its five leading bits, 32 bins again (in cnt and
// low), and the values of the threshold's bin are put into `few`.
template <bool COUNT>
__device__ __forceinline__ void search_list(const uint32_t* list, int m, int bits, uint32_t lead,
                                            unsigned long long missing, int lane, uint32_t* cnt, uint32_t* low,
                                            uint32_t* few, uint32_t* v_out, int* need_out, int* eq_out) {
  if (m > 8) {
    cnt[lane] = 0u;
    low[lane] = 0u;
    __syncwarp();
    const int shift = bits - 5;
    for (int i = lane; i < m; i += 32) {
      const uint32_t x = list[i];
      atomicAdd(&cnt[x >> shift], 1u);
      if (!COUNT) atomicAdd(&low[x >> shift], x);
    }
    __syncwarp();
    uint32_t n = cnt[31 - lane], l = low[31 - lane];  // heaviest first
    const uint32_t n0 = n, l0 = l;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t un = __shfl_up_sync(0xffffffffu, n, d), ul = __shfl_up_sync(0xffffffffu, l, d);
      if (lane >= d) {
        n += un;
        l += ul;
      }
    }
    const unsigned long long w = COUNT ? n : (unsigned long long)n * lead + l;
    const int at = __ffs(__ballot_sync(0xffffffffu, w >= missing)) - 1;
    const uint32_t n_before = __shfl_sync(0xffffffffu, n - n0, at), l_before = __shfl_sync(0xffffffffu, l - l0, at);
    missing -= COUNT ? n_before : (unsigned long long)n_before * lead + l_before;
    const uint32_t bin = 31u - (uint32_t)at;
    int len = 0;
    for (int i0 = 0; i0 < m; i0 += 32) {
      const uint32_t x = (i0 + lane < m) ? list[i0 + lane] : 0u;
      const bool in = i0 + lane < m && (x >> shift) == bin;
      const uint32_t mask = __ballot_sync(0xffffffffu, in);
      if (in) few[len + __popc(mask & ((1u << lane) - 1u))] = x;
      len += __popc(mask);
    }
    __syncwarp();
    list = few;
    m = len;
  }
  uint32_t v = 0u;
  int n_eq = 0;
  unsigned long long ge = 0ull;  // weight of the values >= v
  if (m <= 32) {
    // every lane adds up the values at or above its own
    const uint32_t x = (lane < m) ? list[lane] : 0u;
    uint32_t n = 0u, l = 0u;
    for (int j = 0; j < m; ++j) {
      const uint32_t y = __shfl_sync(0xffffffffu, x, j);
      if (y >= x) {
        n += 1u;
        l += y;
      }
    }
    const unsigned long long w = COUNT ? n : (unsigned long long)n * lead + l;
    const bool ok = lane < m && w >= missing;
    v = __reduce_max_sync(0xffffffffu, ok ? x : 0u);
    const uint32_t eq = __ballot_sync(0xffffffffu, lane < m && x == v);
    n_eq = __popc(eq);
    ge = __shfl_sync(0xffffffffu, w, __ffs(eq) - 1);
  } else {
    // (many nearly equal values) bit by bit
    auto measure = [&](uint32_t from, int* n_out) -> unsigned long long {
      uint32_t n = 0u, l = 0u;
      for (int i = lane; i < m; i += 32) {
        const uint32_t x = list[i];
        n += (x >= from) ? 1u : 0u;
        l += (x >= from) ? x : 0u;
      }
      n = __reduce_add_sync(0xffffffffu, n);
      *n_out = (int)n;
      if (COUNT) return n;
      l = __reduce_add_sync(0xffffffffu, l);
      return (unsigned long long)n * lead + l;
    };
    int n;
    for (int b = bits - 1; b >= 0; --b) {
      if (measure(v | (1u << b), &n) >= missing) v |= 1u << b;
    }
    int n_gt;
    ge = measure(v, &n);
    measure(v + 1u, &n_gt);
    n_eq = n - n_gt;
  }
  int need = n_eq;
  if (n_eq > 1) {
    const unsigned long long each = COUNT ? 1ull : (unsigned long long)lead + v;
    const unsigned long long gt = ge - (unsigned long long)n_eq * each;  // weight of the values > v
    need = (int)min((missing - gt + each - 1ull) / each, (unsigned long long)n_eq);
  }
  *v_out = v;
  *need_out = need;
  *eq_out = n_eq;
}

// The bin in which the bins' weights, added up from the heaviest (highest) down, reach `target`: rs->bin,
// and the weight of those above it in rs->above; both stay as they are if the sum never does.  Thread t
// of the row owns bins [hi - kPer + 1, hi].
template <int W, int BINS, typename F>
__device__ __forceinline__ void find_bin(RowShared* rs, unsigned long long target, int warp, int lane, F bin_weight) {
  constexpr int T = 32 * W, kPer = (BINS + T - 1) / T;
  const int hi = BINS - 1 - (warp * 32 + lane) * kPer;
  unsigned long long own = 0ull;
#pragma unroll
  for (int j = 0; j < kPer; ++j)
    if (hi - j >= 0) own += bin_weight(hi - j);
  unsigned long long incl = own;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned long long up = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += up;
  }
  if (W > 1) {
    if (lane == 31) rs->total[warp] = incl;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < W; ++w)
      if (w < warp) incl += rs->total[w];
  }
  unsigned long long acc = incl - own;
  if (acc < target && incl >= target) {  // exactly one thread, or none
    for (int b = hi; b > hi - kPer && b >= 0; --b) {
      const unsigned long long w = bin_weight(b);
      if (acc + w >= target) {
        rs->bin = b;
        rs->above = acc;
        break;
      }
      acc += w;
    }
  }
  row_sync<W>();
}

// What a row of at most 32 blocks keeps, a lane each: a block is kept if what comes before it - heavier blocks, and equal ones
// of lower index - does not reach the target yet.  All compared with all, 10 instructions for each block of the row; the
// histogram's bins alone are 38 for a lane (masses, selection and attention of 256 tokens, 8 rows of 4 blocks: 24.4 -> 22.5
// us a call; a row of 32 blocks as before).
template <bool COUNT, bool EARLY>
__device__ __forceinline__ uint32_t kept_word(const float* src, int nKb, int lane, double tau, int fixed_count, int* status) {
  const bool here = lane < nKb;
  uint32_t x = here ? __float_as_uint(EARLY ? __ldca(src) : __ldg(src)) : 0u;
  bool bad = false;
  if (x > kMaxMassBits) {
    bad = x != 0x80000000u;
    x = 0u;
  }
  double sum = (double)__uint_as_float(x);
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
  const bool too_heavy = sum > 8.0;  // (more than the fixed point holds: keeps every block)
  if (bad || (lane == 0 && too_heavy)) report_error(status, LOSA_ERR_BAD_MASS);
  const unsigned long long target = COUNT ? (unsigned long long)min(fixed_count, nKb)
                                          : (unsigned long long)(fmin(tau, 1.0) * kFixedOne);
  const unsigned long long mine = COUNT ? 1ull : (unsigned long long)((double)__uint_as_float(x) * kFixedOne);
  unsigned long long before = 0ull;
#pragma unroll 4
  for (int j = 0; j < nKb; ++j) {
    const uint32_t y = __shfl_sync(0xffffffffu, x, j);
    const unsigned long long w = COUNT ? 1ull : __shfl_sync(0xffffffffu, mine, j);
    if (y > x || (y == x && j < lane)) before += w;
  }
  const bool all = !COUNT && (tau >= 1.0 || too_heavy);
  return __ballot_sync(0xffffffffu, here && (all || before < target));
}

// What a row keeps.  W warps per row, K blocks per lane: warp w of the row owns blocks [w * 32 K, (w + 1) * 32 K), its
// lane l the blocks l, l + 32, ... of those, so that a ballot is a bitmap word; lane k gets word k of its warp's K.
// `src`: the lane's first block, `mine`: how many blocks of the warp exist (may be none).  COUNT: the fixed-ratio rule.
// PICK: see below.
template <int W, int K, bool COUNT, bool EARLY, bool PICK>
__device__ __forceinline__ uint32_t kept_words(RowShared* rs, const float* src, int mine, int warp, int lane, int nKb,
                                               double tau, int fixed_count, int* status) {
  constexpr int T = 32 * W;
  constexpr int kShift = COUNT ? kCountShift : kTauShift;
  constexpr int kBase = COUNT ? 0 : kTopBin - (kBins - 1);
  constexpr uint32_t kLowMask = (1u << kShift) - 1u;
  const int t = warp * 32 + lane;                       // thread of the row
  // EARLY: the kernel ahead may have written the masses while this one was starting, so that they are no read-only data.
  auto load = [](const float* at) { return EARLY ? __ldca(at) : __ldg(at); };
  // (blocks past the row's end weigh nothing; they are told apart by their index where they could count)
  uint32_t bits[K];
#pragma unroll
  for (int k = 0; k < K; ++k) bits[k] = 0u;
#pragma unroll
  for (int k = 0; k < K; ++k) if (k * 32 + lane < mine) bits[k] = __float_as_uint(load(src + k * 32));
  for (int i = t; i < kBins; i += T) {
    rs->cnt[i] = 0u;
    if (!COUNT) rs->low[i] = 0u;
  }
  if (t == 0) {
    rs->list_len = 0;
    rs->bin = -1;
  }
  row_sync<W>();
  // (what is no mass is looked for one by one only where there is any: 22296 rows of 3713, fixed ratio 258 -> 245 us, 3716 of
  // 929 18.4 -> 16.9; retained mass 211.3 -> 210.4, 2200 of 275 30.5 -> 29.9)
  bool bad = false;
  float sum = 0.0f;
  uint32_t top = 0u;
#pragma unroll
  for (int k = 0; k < K; ++k) top = max(top, bits[k]);
  if (__any_sync(0xffffffffu, top > kMaxMassBits)) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      if (bits[k] > kMaxMassBits) {  // negative, NaN, or far beyond any mass; -0 becomes +0
        bad |= bits[k] != 0x80000000u;
        bits[k] = 0u;
      }
    }
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    sum += __uint_as_float(bits[k]);
    // (a mass of zero changes no sum: only the fixed-ratio rule counts it)
    if (COUNT ? k * 32 + lane < mine : bits[k] != 0u) {
      const int bin = max((int)(bits[k] >> kShift) - kBase, 0);
      atomicAdd(&rs->cnt[bin], 1u);
      if (!COUNT) atomicAdd(&rs->low[bin], bits[k] & kLowMask);
    }
  }
  // The fixed-point sums hold at most 16: a row whose masses add up to more than 8 (a mass row sums
  // to 1) is reported, and keeps every block, instead of wrapping silently.  (The fixed-ratio rule adds
  // nothing up and keeps its k blocks; it reports such a row too.)
  double row_sum = (double)sum;
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) row_sum += __shfl_xor_sync(0xffffffffu, row_sum, d);
  if (W > 1 && lane == 0) rs->sum[warp] = row_sum;
  row_sync<W>();
  if (W > 1) {
    row_sum = 0.0;
#pragma unroll
    for (int w = 0; w < W; ++w) row_sum += rs->sum[w];
  }
  const bool too_heavy = row_sum > 8.0;
  if (bad || (t == 0 && too_heavy)) report_error(status, LOSA_ERR_BAD_MASS);

  // A tau far below any useful threshold would be lost in units of 2^-60: its rows are searched over
  // the registers in units of about 2^-50 tau, with every weight cut off at tau (a block of that mass
  // reaches the threshold alone), so that sums still fit.  (Every positive float is above 2^-200.)
  const bool tiny = !COUNT && tau < 0x1p-20;
  double scale = kFixedOne, cap = 8.0;
  if (tiny) {
    cap = fmax(tau, 0x1p-200);
    scale = __hiloint2double((1023 + 49 - (((__double2hiint(cap) >> 20) & 0x7ff) - 1023)) << 20, 0);
  }
  const unsigned long long target = COUNT ? (unsigned long long)min(fixed_count, nKb)
                                          : (unsigned long long)(fmin(tiny ? cap : tau, 1.0) * scale);
  bool all = !COUNT && (tau >= 1.0 || too_heavy);  // (too heavy: keeps every block)
  uint32_t v = 0u;   // kept: bits > v, and the first `need` (by index) with bits == v
  int need = 0, eq_total = 0;
  if (!all) {
    // ---- the bin of v*
    find_bin<W, kBins>(rs, target, warp, lane, [&](int b) -> unsigned long long {
      const uint32_t c = rs->cnt[b];
      if (COUNT) return c;
      const uint32_t lead = (uint32_t)(b + kBase);  // exponent and four mantissa bits
      const unsigned long long mant = (unsigned long long)c * ((16u | (lead & 15u)) << kTauShift) + rs->low[b];
      return (b == 0) ? 0ull : mant << ((lead >> 4) - 90u);  // the mantissa's unit is 2^(e - 150); e >= 92 here
    });
    // ---- v* within the bin
    const int bin = tiny ? -1 : rs->bin;
    if (bin >= 0) {
      uint32_t lead = (uint32_t)(bin + kBase);  // the leading bits of its values
      int rest = kShift;                        // ... and how many bits follow
      int m = (int)rs->cnt[bin];                // how many values
      // a value weighs `each` and its following bits, in units of the bin's mantissas
      uint32_t each = COUNT ? 1u : (16u | (lead & 15u)) << kTauShift;
      // what they have to add: rounded up, their sums are whole
      const uint32_t lift = COUNT ? 0u : (lead >> 4) - 90u;
      unsigned long long missing = (target - rs->above + ((1ull << lift) - 1ull)) >> lift;
      const int mine_k = (mine - lane + 31) >> 5;  // this lane's blocks that exist (fixed-ratio rule: zeros count)
      // More values than the list holds: split by the bits that follow, until it does or no bits are left
#pragma unroll 1
      while (m > kListCap && rest > 0) {
        // the bits that all of them share are skipped (equal values would queue up at one bin's counters)
        uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll
        for (int k = 0; k < K; ++k) {
          if ((bits[k] >> rest) == lead && (!COUNT || k < mine_k)) {
            lo = min(lo, bits[k]);
            hi = max(hi, bits[k]);
          }
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if (W > 1) {
          if (lane == 0) {
            rs->list[warp] = lo;
            rs->list[W + warp] = hi;
          }
          __syncthreads();
#pragma unroll
          for (int w = 0; w < W; ++w) {
            lo = min(lo, rs->list[w]);
            hi = max(hi, rs->list[W + w]);
          }
        }
        const int differ = (lo == hi) ? 0 : max(32 - __clz(lo ^ hi), 5);
        if (!COUNT) each += ((lo & ((1u << rest) - 1u)) >> differ) << differ;
        lead = lo >> differ;
        rest = differ;
        if (rest == 0) break;
        const int next = (rest == 5) ? 0 : max(rest - 9, 5);
        row_sync<W>();  // (the bins, and what was found, have been read)
        for (int i = t; i < kSplitBins; i += T) {
          rs->cnt[i] = 0u;
          if (!COUNT) rs->low[i] = 0u;
        }
        row_sync<W>();
#pragma unroll
        for (int k = 0; k < K; ++k) {
          if ((bits[k] >> rest) == lead && (!COUNT || k < mine_k)) {
            const uint32_t x = bits[k] & ((1u << rest) - 1u);
            atomicAdd(&rs->cnt[x >> next], 1u);
            if (!COUNT) atomicAdd(&rs->low[x >> next], x);
          }
        }
        row_sync<W>();
        find_bin<W, kSplitBins>(rs, missing, warp, lane, [&](int b) -> unsigned long long {
          return COUNT ? rs->cnt[b] : (unsigned long long)rs->cnt[b] * each + rs->low[b];
        });
        const uint32_t b = (uint32_t)rs->bin;
        m = (int)rs->cnt[b];
        missing -= rs->above;
        lead = (lead << (rest - next)) | b;
        if (!COUNT) each += b << next;
        rest = next;
      }
      if (rest == 0) {
        // (that many equal values)
        v = lead;
        eq_total = m;
        need = (int)min((missing + each - 1u) / each, (unsigned long long)m);
      } else {
        uint32_t in = 0u;  // bit k: this lane's block k is in the bin
#pragma unroll
        for (int k = 0; k < K; ++k) in |= ((bits[k] >> rest) == lead) ? 1u << k : 0u;
        if (COUNT) in &= (mine_k >= 32) ? 0xffffffffu : (1u << max(mine_k, 0)) - 1u;
        // (A lane has one or two of them: their values are read again instead of picked out of registers.  Where few warps
        // share an SM and the loads are not read-only ones, nothing hides these reads - 64 rows of 256 blocks, a third of
        // them, 7.6 us a call instead of 4.3 - and they are picked; of long rows among many that costs 10 - 14 %.)
        if (PICK) {
#pragma unroll
          for (int k = 0; k < K; ++k)
            if ((in >> k) & 1u) rs->list[atomicAdd(&rs->list_len, 1)] = bits[k] & ((1u << rest) - 1u);
          in = 0u;
        }
        while (in != 0u) {
          const int k = __ffs(in) - 1;
          in &= in - 1u;
          uint32_t x = __float_as_uint(load(src + k * 32));
          if (x > kMaxMassBits) x = 0u;
          rs->list[atomicAdd(&rs->list_len, 1)] = x & ((1u << rest) - 1u);
        }
        row_sync<W>();
        if (warp == 0) {
          search_list<COUNT>(rs->list, m, rest, each, missing, lane, rs->cnt, rs->low, rs->cnt + 32, &v, &need, &eq_total);
          v |= lead << rest;
          if (W > 1 && lane == 0) {
            rs->v = v;
            rs->need = need;
            rs->eq_total = eq_total;
          }
        }
        if (W > 1) {
          row_sync<W>();
          v = rs->v;
          need = rs->need;
          eq_total = rs->eq_total;
        }
      }
    } else if (!COUNT) {
      // ---- bit by bit over the row: masked sums of the blocks with bits >= v (read again, so that this
      // path takes no registers from the other)
      auto measure_ge = [&](uint32_t from) -> unsigned long long {
        unsigned long long a = 0ull;
#pragma unroll 1
        for (int k = 0; k * 32 + lane < mine; ++k) {
          uint32_t x = __float_as_uint(load(src + k * 32));
          if (x > kMaxMassBits) x = 0u;
          if (x >= from) a += fixed_weight(x, scale, cap);
        }
        __syncwarp();
        return row_sum_u64<W>(a, rs, warp, lane);
      };
      all = measure_ge(0u) < target;  // never reaches tau
      if (!all) {
        for (int b = 30; b >= 0; --b) {
          const uint32_t cand = v | (1u << b);
          if (measure_ge(cand) >= target) v = cand;
        }
        const unsigned long long gt = measure_ge(v + 1u);
        unsigned long long n = 0ull;
#pragma unroll
        for (int k = 0; k < K; ++k) n += (k * 32 + lane < mine && bits[k] == v) ? 1ull : 0ull;
        eq_total = (int)row_sum_u64<W>(n, rs, warp, lane);
        const unsigned long long fv = fixed_weight(v, scale, cap);
        const unsigned long long need64 = (fv == 0ull) ? (unsigned long long)eq_total : (target - gt + fv - 1ull) / fv;
        need = (int)min(need64, (unsigned long long)eq_total);
      }
    }
  }
  // ---- bitmap words
  uint32_t out = 0u;  // lane k: word k of this warp's K
  if (all || need >= eq_total) {
    // (all ties are kept: their order does not matter)
    const uint32_t from = all ? 0u : v;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const uint32_t word = __ballot_sync(0xffffffffu, bits[k] >= from);
      if (lane == k) out = word;
    }
  } else {
    // of the blocks equal to v the first `need` by index
    int seen = 0;  // ties at lower indices
    if (W > 1) {
      int n = 0;
#pragma unroll
      for (int k = 0; k < K; ++k) n += (k * 32 + lane < mine && bits[k] == v) ? 1 : 0;
      n = __reduce_add_sync(0xffffffffu, n);
      if (lane == 0) rs->part[warp] = n;
      __syncthreads();
#pragma unroll
      for (int w = 0; w < W; ++w)
        if (w < warp) seen += rs->part[w];
      __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const bool eq = k * 32 + lane < mine && bits[k] == v;
      const uint32_t eqm = __ballot_sync(0xffffffffu, eq);
      const uint32_t word =
          __ballot_sync(0xffffffffu, bits[k] > v || (eq && seen + __popc(eqm & ((1u << lane) - 1u)) < need));
      seen += __popc(eqm);
      if (lane == k) out = word;
    }
  }
  // (bits of blocks past the end of the row)
  const int valid = mine - lane * 32;
  if (lane >= K || valid <= 0) out = 0u;
  else if (valid < 32) out &= (1u << valid) - 1u;
  return out;
}

// One row per CTA, or four at W = 1.
template <int W, int K, bool COUNT>
__global__ void __launch_bounds__(W == 1 ? 128 : 32 * W, W == 1 ? 7 : 28 / W)
select_rows_kernel(const float* __restrict__ mass, int rows, int nKb, double tau, int fixed_count,
                   int32_t* __restrict__ counts, uint32_t* __restrict__ bitmaps, int* status) {
  constexpr int kRowsPerCta = (W == 1) ? 4 : 1;
  __shared__ RowShared shared[kRowsPerCta];
  const int lane = threadIdx.x & 31;
  const int warp = (W == 1) ? 0 : threadIdx.x >> 5;     // of the row
  RowShared* const rs = &shared[(W == 1) ? threadIdx.x >> 5 : 0];
  const int64_t row = (int64_t)blockIdx.x * kRowsPerCta + ((W == 1) ? threadIdx.x >> 5 : 0);
  ptx::grid_launch_dependents();
  ptx::grid_dependency_wait();
  if (row >= rows) return;
  const int words = (nKb + 31) >> 5;
  const int mine = min(32 * K, nKb - warp * 32 * K);
  const float* src = mass + row * nKb + warp * 32 * K + lane;
  const uint32_t out = kept_words<W, K, COUNT, !COUNT, false>(rs, src, mine, warp, lane, nKb, tau, fixed_count, status);
  if (lane < K && warp * K + lane < words) bitmaps[row * words + warp * K + lane] = out;
  int kept = __reduce_add_sync(0xffffffffu, __popc(out));
  if (W > 1) {
    if (lane == 0) rs->part[warp] = kept;
    __syncthreads();
    kept = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) kept += rs->part[w];
  }
  if (warp * 32 + lane == 0) counts[row] = kept;
}

// Few rows: one launch, of one cluster.  A warp per row, two rows at most, spread over the cluster's CTAs; the sizes of all
// rows meet in every CTA's shared memory, and each warp writes the indices of its own rows.  The two launches of the general
// way are all latency there (masses, selection and attention of 256 tokens, 27.8 -> 24.5 us; 4 x 32 rows of 32 blocks,
// calls in a row, 9.1 -> 6.1).
constexpr int kSmallWarps = 16, kSmallCtas = 8, kSmallRows = 2 * kSmallWarps * kSmallCtas;
// Which calls: those that the eight SMs get through about as fast as the general way gets through its two launches; us a
// call in a captured graph, that way / this one (from the host a call of either rule is 2 - 2.6 us shorter this way).
//   256 rows of 32 blocks, all compared with all   5.6 / 5.6 (retained mass), 5.4 / 4.9 (fixed ratio)
//   128 rows of 256 blocks, a row a warp           6.1 / 6.2, 6.4 / 5.0;  64 of 128 5.8 / 4.4, 5.9 / 3.9
//   128 of 512                                     6.6 - 10.5 / 7.4 - 8.2 by the masses (on average 8.4 / 7.7), 7.4 / 6.5
//   64 of 1024, half as many warps to an SM        8.0 - 11.7 / 7.0 - 8.0, 10.0 / 8.0;  128 7.8 - 12.5 / 9.8 - 10.9
//   256 of 64, two rows a warp                     5.8 / 9.5, 5.8 / 6.8;  of 128 5.8 / 9.7, 6.0 / 7.5;  of 256 6.1 / 10.5, 6.4 / 8.5
// Under the fixed-ratio rule two rows a warp are taken up to 128 blocks all the same: what they lose on the device is less
// than what they save on the host.
bool small_selection(int64_t rows, int nKb, bool fixed) {
  if (nKb <= (fixed ? 128 : 32)) return rows <= kSmallRows;
  return nKb <= 512 ? rows <= kSmallRows / 2 : nKb <= 1024 && rows <= kSmallRows / 4;
}
struct SmallShared {
  RowShared rows[kSmallWarps];
  int counts[kSmallRows];
};
template <int K, bool COUNT>
__global__ void __launch_bounds__(32 * kSmallWarps)
select_small_kernel(const float* __restrict__ mass, int rows, int nKb, double tau, int fixed_count,
                    int32_t* __restrict__ offsets, int32_t* __restrict__ kv_idx, int64_t kv_capacity, int* status) {
  extern __shared__ __align__(16) unsigned char small_raw[];
  SmallShared* const sh = reinterpret_cast<SmallShared*>(small_raw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, ctas = gridDim.x, warps = blockDim.x >> 5;
  ptx::grid_launch_dependents();
  ptx::cluster_sync();  // (the other CTAs' shared memory is there)
  ptx::grid_dependency_wait();
  uint32_t word[2] = {0u, 0u};
  int kept[2] = {0, 0};
#pragma unroll 1
  for (int i = 0; i < 2; ++i) {
    const int row = (i * ctas + (int)blockIdx.x) * warps + warp;
    if (row >= rows) break;
    const float* const src = mass + (int64_t)row * nKb + lane;
    uint32_t out;  // (lane k: word k)
    if (K == 8 && nKb <= 32 && (COUNT || tau >= 0x1p-20)) {  // (smaller ones are lost in units of 2^-60)
      out = kept_word<COUNT, true>(src, nKb, lane, tau, fixed_count, status);
      if (lane > 0) out = 0u;
    } else {
      out = kept_words<1, K, COUNT, true, true>(&sh->rows[warp], src, nKb, 0, lane, nKb, tau, fixed_count, status);
    }
    const int n = __reduce_add_sync(0xffffffffu, __popc(out));
    if (lane < ctas) ptx::st_cluster_u32(ptx::mapa(ptx::smem_u32(&sh->counts[row]), lane), (uint32_t)n);
    if (i == 0) word[0] = out, kept[0] = n;
    else word[1] = out, kept[1] = n;
    __syncwarp();
  }
  ptx::cluster_sync();
  const uint32_t bit = 1u << lane, below = bit - 1u;
  const int words = (nKb + 31) >> 5;
#pragma unroll 1
  for (int i = 0; i < 2; ++i) {
    const int row = (i * ctas + (int)blockIdx.x) * warps + warp;
    if (row >= rows) break;
    int at = 0;
    for (int r = lane; r < row; r += 32) at += sh->counts[r];
    at = __reduce_add_sync(0xffffffffu, at);
    const uint32_t mine = (i == 0) ? word[0] : word[1];
    const int n = (i == 0) ? kept[0] : kept[1];
    if (lane == 0) {
      offsets[row] = at;
      if (row == rows - 1) {
        offsets[rows] = at + n;
        if ((int64_t)at + n > kv_capacity) report_error(status, LOSA_ERR_CAPACITY);
      }
    }
    for (int w = 0; w < words; ++w) {
      const uint32_t x = __shfl_sync(0xffffffffu, mine, w);
      const int to = at + __popc(x & below);
      if ((x & bit) && to < kv_capacity) kv_idx[to] = w * 32 + lane;
      at += __popc(x);
    }
  }
}

// Bitmaps -> ascending indices, `per_cta` consecutive rows per CTA.  The CTA first adds up the sizes
// of all rows before its own: that is a read of at most 4 bytes per row from L2, and it replaces a
// launch that scanned the sizes with one CTA.  Then a warp per row, 32 indices at a time: lane b
// stands for bit b of a bitmap word, so the stores of a word are contiguous.  (One lane per word,
// each writing its word's indices one after the other, stored 32 separate sectors per instruction.)
constexpr int kExpandThreads = 512;

__global__ void __launch_bounds__(kExpandThreads)
expand_rows_kernel(const int32_t* __restrict__ counts, const uint32_t* __restrict__ bitmaps, int rows, int nKb,
                   int per_cta, int32_t* __restrict__ offsets, int32_t* __restrict__ kv_idx, int64_t kv_capacity,
                   int* status) {
  constexpr int kWarps = kExpandThreads / 32;
  __shared__ int warp_total[kWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int row0 = blockIdx.x * per_cta, row1 = min(rows, row0 + per_cta);
  const int words = (nKb + 31) >> 5;
  ptx::grid_dependency_wait();
  int before = 0;
  for (int i = threadIdx.x; i < (row0 >> 2); i += kExpandThreads) {
    const int4 c = __ldcg(reinterpret_cast<const int4*>(counts) + i);
    before += (c.x + c.y) + (c.z + c.w);
  }
  if (threadIdx.x < (row0 & 3)) before += __ldcg(counts + (row0 & ~3) + threadIdx.x);
  before = __reduce_add_sync(0xffffffffu, before);
  if (lane == 0) warp_total[warp] = before;
  __syncthreads();
  int pos = 0;  // first index of the row
#pragma unroll
  for (int w = 0; w < kWarps; ++w) pos += warp_total[w];
  for (int r0 = row0; r0 < row1; r0 += 32) {
    // 32 rows: every warp scans their sizes and expands its share of them
    const int r = r0 + lane;
    const int c = (r < row1) ? __ldcg(counts + r) : 0;
    int incl = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += up;
    }
    const int n = min(32, row1 - r0);
    if (warp == 0 && lane < n) offsets[r] = pos + incl - c;
    for (int j = warp; j < n; j += kWarps) {
      int at = pos + __shfl_sync(0xffffffffu, incl - c, j);
      const bool fits = (int64_t)at + __shfl_sync(0xffffffffu, c, j) <= kv_capacity;
      const uint32_t below = (1u << lane) - 1u, bit = 1u << lane;
      const uint32_t* bm = bitmaps + (int64_t)(r0 + j) * words;
      for (int w0 = 0; w0 < words; w0 += 32) {
        const uint32_t mine = (w0 + lane < words) ? __ldcg(bm + w0 + lane) : 0u;
        const int m = min(32, words - w0);
        if (fits) {
          int* to = kv_idx + at;
          int value = w0 * 32 + lane;
#pragma unroll 8
          for (int i = 0; i < m; ++i) {
            const uint32_t word = __shfl_sync(0xffffffffu, mine, i);
            if (word & bit) to[__popc(word & below)] = value;
            to += __popc(word);
            value += 32;
          }
          at = (int)(to - kv_idx);
        } else {
          for (int i = 0; i < m; ++i) {
            const uint32_t word = __shfl_sync(0xffffffffu, mine, i);
            const int to = at + __popc(word & below);
            if ((word & bit) && to < kv_capacity) kv_idx[to] = (w0 + i) * 32 + lane;
            at += __popc(word);
          }
        }
      }
    }
    pos += __shfl_sync(0xffffffffu, incl, 31);
  }
  if (row1 == rows && threadIdx.x == 0) {
    offsets[rows] = pos;
    if ((int64_t)pos > kv_capacity) report_error(status, LOSA_ERR_CAPACITY);
  }
}

__global__ void __launch_bounds__(256)
validate_csr_kernel(int rows, int nKb, const int32_t* __restrict__ offsets,
                    const int32_t* __restrict__ kv_idx, int* status) {
  const int lane = threadIdx.x & 31;
  const int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (row >= rows) return;
  const int32_t b = offsets[row], e = offsets[row + 1];
  const int32_t nnz = offsets[rows];  // every read below stays inside [0, nnz)
  bool bad = (row == 0 && b != 0) || e <= b || (e - b) > nKb || b < 0 || e > nnz;
  if (!bad) {
    for (int p = b + lane; p < e; p += 32) {
      const int32_t j = kv_idx[p];
      if (j < 0 || j >= nKb) bad = true;
      if (p > b && kv_idx[p - 1] >= j) bad = true;
    }
  }
  if (bad) report_error(status, LOSA_ERR_BAD_INDEX);
}

// Retained and total mass of every row under a CSR pattern (Eq. 2 before the outer sums): one
// warp per row, fp64 partial sums per lane, shuffle tree.
__global__ void __launch_bounds__(256)
row_recall_kernel(const float* __restrict__ mass, int rows, int nKb,
                  const int32_t* __restrict__ offsets, const int32_t* __restrict__ kv_idx,
                  double* __restrict__ retained, double* __restrict__ total, int* status) {
  const int lane = threadIdx.x & 31;
  const int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (row >= rows) return;
  const float* mrow = mass + row * nKb;
  double tot = 0.0, ret = 0.0;
  for (int j = lane; j < nKb; j += 32) tot += (double)mrow[j];
  const int32_t b = offsets[row], e = offsets[row + 1];
  bool bad = false;
  for (int p = b + lane; p < e; p += 32) {
    const int32_t j = kv_idx[p];
    if (j < 0 || j >= nKb) bad = true;  // skipped, never used as an address
    else ret += (double)mrow[j];
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    tot += __shfl_xor_sync(0xffffffffu, tot, d);
    ret += __shfl_xor_sync(0xffffffffu, ret, d);
  }
  if (bad) report_error(status, LOSA_ERR_BAD_INDEX);
  if (lane == 0) {
    retained[row] = ret;
    total[row] = tot;
  }
}

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

}  // namespace

size_t select_workspace_bytes(int64_t rows, int nKb) {
  const size_t words = (size_t)(nKb + 31) / 32;
  return align_up((size_t)rows * sizeof(int32_t), 256) + (size_t)rows * words * sizeof(uint32_t);
}

int select_launches(int64_t rows, int nKb, bool fixed) { return small_selection(rows, nKb, fixed) ? 1 : 2; }

template <int K, bool COUNT>
static int launch_small(int ctas, const float* mass, int rows, int nKb, double tau, int fixed_count, int32_t* offsets,
                        int32_t* kv_idx, int64_t kv_capacity, int* status, int dev, cudaStream_t st) {
  auto kern = select_small_kernel<K, COUNT>;
  static std::atomic<int> ready[kMaxDevices];
  if (!ready[dev].load(std::memory_order_acquire)) {
    LOSA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallShared)));
    ready[dev].store(1, std::memory_order_release);
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = ctas;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.gridDim = dim3(ctas, 1, 1);
  cfg.blockDim = dim3(32 * min(kSmallWarps, (rows + ctas - 1) / ctas), 1, 1);
  cfg.dynamicSmemBytes = sizeof(SmallShared);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  LOSA_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, mass, rows, nKb, tau, fixed_count, offsets, kv_idx, kv_capacity, status));
  return LOSA_OK;
}

int launch_select(int rows, int nKb, const float* mass, double tau, int fixed_count,
                  int32_t* offsets, int32_t* kv_idx, int64_t kv_capacity, void* ws, int* status, int dev,
                  cudaStream_t st) {
  int32_t* counts = static_cast<int32_t*>(ws);
  uint32_t* bitmaps = reinterpret_cast<uint32_t*>(static_cast<char*>(ws) +
                                                  align_up((size_t)rows * sizeof(int32_t), 256));
  if (small_selection(rows, nKb, fixed_count > 0)) {
    const int ctas = min(kSmallCtas, rows);
#define LOSA_SELECT_SMALL(k)                                                                                  \
  (fixed_count > 0 ? launch_small<k, true>(ctas, mass, rows, nKb, tau, fixed_count, offsets, kv_idx, kv_capacity, status, dev, st) \
                   : launch_small<k, false>(ctas, mass, rows, nKb, tau, 0, offsets, kv_idx, kv_capacity, status, dev, st))
    return nKb <= 256 ? LOSA_SELECT_SMALL(8) : nKb <= 512 ? LOSA_SELECT_SMALL(16) : LOSA_SELECT_SMALL(32);
#undef LOSA_SELECT_SMALL
  }
  // (registers hold 32 blocks per lane at most: longer rows take more warps.  Under the retained-mass rule the launch is a
  // dependent: 1024 key blocks of 1536 rows 14.3 -> 11.6 us, 928 of 3716 22.4 -> 19.8.  Under the fixed-ratio rule its
  // kernel is 13 - 17 % slower with loads that are not read-only ones, and waits for the kernel ahead.)
#define LOSA_SELECT_ROWS(w, k)                                                                                 \
  do {                                                                                                         \
    const int ctas = (w) == 1 ? (rows + 3) / 4 : rows, threads = (w) == 1 ? 128 : 32 * (w);                    \
    rc = fixed_count > 0 ? launch(select_rows_kernel<w, k, true>, dim3(ctas), threads, 0, st, false, mass, rows, nKb, tau,  \
                                  fixed_count, counts, bitmaps, status)                                        \
                         : launch(select_rows_kernel<w, k, false>, dim3(ctas), threads, 0, st, true, mass, rows, nKb, tau, \
                                  0, counts, bitmaps, status);                                                 \
  } while (0)
  int rc;
  if (nKb <= 256) LOSA_SELECT_ROWS(1, 8);
  else if (nKb <= 512) LOSA_SELECT_ROWS(1, 16);
  else if (nKb <= 1024) LOSA_SELECT_ROWS(1, 32);
  else if (nKb <= 2048) LOSA_SELECT_ROWS(2, 32);
  else if (nKb <= 4096) LOSA_SELECT_ROWS(4, 32);
  else LOSA_SELECT_ROWS(8, 32);
#undef LOSA_SELECT_ROWS
  // four CTAs per SM at most (but no fewer rows than warps): adding up the sizes of the rows before
  // costs every CTA the same, so more of them only read more
  const int per_cta = max(kExpandThreads / 32, (rows + 591) / 592);
  if (rc != LOSA_OK) return rc;
  return launch(expand_rows_kernel, dim3((rows + per_cta - 1) / per_cta), kExpandThreads, 0, st, true, counts, bitmaps, rows,
                nKb, per_cta, offsets, kv_idx, kv_capacity, status);
}

// ---- allocation-free variant ----------------------------------------------------------
// Scratch for losa_select_noalloc lives in the library image: one array per GPU that loads
// the library, held until the process exits.  The first 256 bytes hold the status word of
// the last call, the rest is the counts + bitmaps workspace.
constexpr size_t kStaticStatusBytes = 256;
static __device__ __align__(256) unsigned char g_select_scratch[LOSA_SELECT_NOALLOC_MAX_SCRATCH];

namespace {
unsigned char* g_scratch_addr[kMaxDevices] = {};  // device address of g_select_scratch, per device
}  // namespace

size_t select_noalloc_workspace_limit() {
  return (size_t)LOSA_SELECT_NOALLOC_MAX_SCRATCH - kStaticStatusBytes;
}

int launch_select_noalloc(int rows, int nKb, const float* mass, double tau, int32_t* offsets,
                          int32_t* kv_idx, int64_t kv_capacity, int32_t* device_status,
                          cudaStream_t st) {
  int dev = 0;
  LOSA_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return LOSA_ERR_UNSUPPORTED;
  if (!g_scratch_addr[dev]) {
    // In host code the array's name is only a handle; the device address must be asked for,
    // once per device, with that device current.
    unsigned char* ptr = nullptr;
    LOSA_CUDA_TRY(cudaGetSymbolAddress(reinterpret_cast<void**>(&ptr), g_select_scratch));
    g_scratch_addr[dev] = ptr;
  }
  unsigned char* base = g_scratch_addr[dev];
  int* status = reinterpret_cast<int*>(base);
  unsigned char* ws = base + kStaticStatusBytes;
  // the array keeps the previous call's contents: the status word must start at zero; counts
  // and bitmaps are fully rewritten by the first kernel before anything reads them
  LOSA_CUDA_TRY(cudaMemsetAsync(status, 0, sizeof(int), st));
  // the same kernels, dispatch and workspace layout as losa_select
  const int rc = launch_select(rows, nKb, mass, tau, 0, offsets, kv_idx, kv_capacity, ws, status, dev, st);
  if (rc != LOSA_OK) return rc;
  if (device_status)
    LOSA_CUDA_TRY(cudaMemcpyAsync(device_status, status, sizeof(int), cudaMemcpyDeviceToDevice, st));
  return LOSA_OK;
}

int launch_row_recall(int rows, int nKb, const float* mass, const int32_t* offsets,
                      const int32_t* kv_idx, double* retained, double* total, cudaStream_t st) {
  int rc = LOSA_OK;
  const DeviceState* dev = device_state(&rc);
  if (!dev) return rc;
  int* status = dev->status_dev;
  row_recall_kernel<<<(rows + 7) / 8, 256, 0, st>>>(mass, rows, nKb, offsets, kv_idx, retained,
                                                    total, status);
  LOSA_CUDA_TRY(cudaGetLastError());
  return LOSA_OK;
}

int launch_validate_csr(int rows, int nKb, const int32_t* offsets, const int32_t* kv_idx,
                        cudaStream_t st) {
  int rc = LOSA_OK;
  const DeviceState* dev = device_state(&rc);
  if (!dev) return rc;
  int* status = dev->status_dev;
  validate_csr_kernel<<<(rows + 7) / 8, 256, 0, st>>>(rows, nKb, offsets, kv_idx, status);
  LOSA_CUDA_TRY(cudaGetLastError());
  return LOSA_OK;
}

}  // namespace losa
