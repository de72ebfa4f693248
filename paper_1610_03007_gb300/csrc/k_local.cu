// Round 0's last step when the radix sort took only the top bits of the
// initial keys: every run of equal top bits (a bucket) that fits a tile is
// sorted, renamed, tested for uniqueness and compacted inside one block
// (Section 2.1, Algorithm 1's sort, Algorithm 2's CmpName, Algorithm 6's
// Unique and Algorithm 5's discarding in one pass over the keys).
//
// A least-significant-digit sort reads and writes every key once per digit.
// After the passes over the top bits alone a bucket of a large text holds a
// few to a few hundred keys, which differ in their next bits; so one pass
// that orders them in shared memory replaces the remaining digit passes and
// the rename:
//
//   - Tile t owns the buckets that start in positions [t W, (t + 1) W); the
//     last may run up to CAP - W items past the window. A bucket that does
//     not end there is left to the global path (k_gather_big, radix sort,
//     k_rename), and tiles inside it own nothing.
//   - A bucket of s items spreads them over up to s bins by its next key bits
//     (bins take the bucket's own range of slots), about one item per bin. An
//     item's place is its bin's start plus the number of smaller keys in the
//     bin (equal keys in input order, which is the stable sort's); the same
//     comparisons count its equal keys, so nothing is read back in sorted
//     order.
//   - A tile whose bins hold many items (skewed or repeated text) compares
//     the items of its large bins with their first one. A bin of one
//     repeated key is a run: its members keep their arrival order, the first
//     position in front. The others are spread again by their next key bits,
//     until every large bin is a run, or holds one key of which some are tail
//     suffixes: these (less than c0) move to a bin of their own before the rest.
//   - The tail rule and the unique test are k_rename's, but a group never
//     leaves its tile, so no offsets of earlier tiles are needed: one atomic
//     reserves the tile's survivors and groups (the next list needs each
//     group contiguous, in any order), and a group's final name is known at
//     once.
//   - SA of a unique suffix is written at its rank, and SA_NONE at every
//     other rank, so that k_isa_fill can take the unique suffixes' names
//     from the SA and no queue of them is written.
//
// Bound: HBM in principle, 12 bytes read and 4 written per item; in practice
// shared-memory latency and barriers of the steps above.
#include "launch.h"

namespace gbsa {

namespace {

// 512 threads with 6 items each, 2 blocks per SM (64 registers), windows of
// 5 rows. Measured at 2^28 DNA after three passes (16 items to a bucket) and
// Markov DNA after four: 3.61 and 6.47 ms; windows of 4 rows 3.67 and 6.70;
// 8 items, 3584-item windows 3.83 and 7.03; 256 x 8 3.60 and 8.59; 256 x 12
// 4.58 and 11.2; 384 x 8 3.76 and 8.15; 3 blocks per SM 3.55 and 7.05.
constexpr int LC_BLOCK = 512;
constexpr int LC_ITEMS = 6;
constexpr int LC_CAP = LC_BLOCK * LC_ITEMS;
constexpr int LC_W = LOCAL_TILE;
constexpr int LC_WARPS = LC_BLOCK / 32;
constexpr int LC_SEGS = LC_ITEMS * LC_WARPS;  // (row, warp) segments of 32 items
// Bins of at least LC_RUN_MIN items are spread again or found to be runs, in
// tiles that would make more than LC_AVG comparisons per item. (16 and 6, 16
// and 24, 64 and 48 against these: 8 M characters of prose 0.50, 0.48, 0.49
// and 0.46 ms, 2^25 Zipf bytes 0.575, 0.551, 0.559 and 0.551 ms.)
constexpr uint32_t LC_RUN_MIN = 32, LC_AVG = 12;
constexpr uint32_t LC_NO_ITEM = 0xFFFFFFFFu;
constexpr uint32_t LC_MIXED = 0x80000000u;  // bin flag: not one run of equal keys
constexpr uint32_t LC_PARTED = 64;  // in place of a bin's remaining key bits: tails apart
static_assert(LC_W % LC_BLOCK == 0 && LC_CAP > LC_W && LC_CAP < 0x8000, "window of whole rows");
static_assert(LC_CAP <= 2 * LC_W, "the flags take the place of the bucket starts");
static_assert(LC_SEGS % 32 == 0 && LC_SEGS <= LC_BLOCK, "one warp scans the segments");

struct LcSmem {
  uint64_t key[LC_CAP];       // bin order
  uint32_t val[LC_CAP];       // sorted order; before that each run's first (index, slot)
  uint32_t bin[LC_CAP + 1];   // counts, then starts; names of the groups at the end
  uint16_t idx[LC_CAP];       // input index | tail << 15 of key's slots
  // First item of each bucket, then the end; later LC_CAP flags of the sorted
  // positions.
  __align__(4) uint16_t start[LC_W + 2];
  uint32_t heads[LC_SEGS];    // bucket heads; later group heads in sorted order
  uint32_t surv[LC_SEGS];     // survivors in sorted order
  uint32_t pre[LC_SEGS];      // exclusive counts of the heads, then of survivors | heads << 16
  uint32_t tmp[LC_WARPS + 1];
  uint32_t sq;                // comparisons the tile would make
  uint32_t surv_base, grp_base, upd_base;
};

// The lane's arrival number in bin x (LC_NO_ITEM: none), counting it. Every
// lane of the warp calls it. In tiles with runs many lanes share a bin, whose
// atomics on one word would be served one by one: one atomic per distinct
// bin of the warp instead. (Elsewhere the plain atomics are faster: a check
// for a common bin there cost 5 % of the kernel on DNA.)
__device__ __forceinline__ uint32_t arrive_runs(uint32_t *bins, uint32_t x) {
  const uint32_t peers = __match_any_sync(0xffffffffu, x);
  const uint32_t before = peers & lanemask_lt();
  uint32_t base = 0;
  if (x != LC_NO_ITEM && before == 0) base = atomicAdd(&bins[x], (uint32_t)__popc(peers));
  return __shfl_sync(0xffffffffu, base, __ffs(peers) - 1) + __popc(before);
}

// S.bin from counts to exclusive starts (every thread of the block calls
// it; the counts are complete and synchronised before, the starts after).
// Adds the sum of the squared counts to S.sq.
__device__ __forceinline__ void scan_bins(LcSmem &S, uint32_t c) {
  const int tid = threadIdx.x, lane = tid & 31;
  uint32_t v[LC_ITEMS], sum = 0, sq = 0;
#pragma unroll
  for (int i = 0; i < LC_ITEMS; ++i) {
    v[i] = S.bin[tid * LC_ITEMS + i];
    sum += v[i];
    sq += v[i] * v[i];
  }
  sq = __reduce_add_sync(0xffffffffu, sq);
  if (lane == 0 && sq) atomicAdd(&S.sq, sq);
  uint32_t total;
  uint32_t run = block_exclusive<LC_BLOCK>(sum, OpAdd(), 0u, S.tmp, total);
#pragma unroll
  for (int i = 0; i < LC_ITEMS; ++i) {
    S.bin[tid * LC_ITEMS + i] = run;
    run += v[i];
  }
  if (tid == 0) S.bin[LC_CAP] = c;
  __syncthreads();
}

// Exclusive sums over the segments' packed counts by one warp.
__device__ __forceinline__ uint32_t scan_segments(uint32_t *v) {
  constexpr int PER = LC_SEGS / 32;
  const int lane = threadIdx.x & 31;
  uint32_t c[PER], s = 0;
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    c[i] = v[lane * PER + i];
    s += c[i];
  }
  const uint32_t incl = warp_inclusive(s, OpAdd());
  uint32_t run = incl - s;
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    v[lane * PER + i] = run;
    run += c[i];
  }
  return __shfl_sync(0xffffffffu, incl, 31);
}

// First set bit at or after item e in the segments' ballots, at most `end`.
__device__ __forceinline__ uint32_t next_head(const uint32_t *ballots, uint32_t e, uint32_t end) {
  uint32_t w = e >> 5;
  if (e >= end) return end;
  uint32_t b = ballots[w] & (0xFFFFFFFFu << (e & 31));
  while (!b) {
    if (++w * 32 >= end) return end;
    b = ballots[w];
  }
  const uint32_t x = w * 32 + __ffs(b) - 1;
  return x < end ? x : end;
}

}  // namespace

// One tile. Every thread of the block calls it; all returns are uniform.
__device__ __forceinline__ void local_tile(LcSmem &S, const LocalArgs &a) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint64_t *__restrict__ K = a.plan->kfinal;
  const uint32_t *__restrict__ V = a.plan->vfinal;
  const uint32_t w0 = blockIdx.x * (uint32_t)LC_W;
  const uint32_t left = a.m - w0;  // items from the window's start on
  const uint32_t win = min((uint32_t)LC_W, left);
  const uint32_t R = a.R;

  // Item e of the tile is row e / LC_BLOCK of thread e % LC_BLOCK. A bucket
  // head differs from the item before in the top bits; the end of the list
  // counts as one.
  uint64_t key[LC_ITEMS];
  uint32_t val[LC_ITEMS];
  auto load_row = [&](int k) {
    const uint32_t e = k * LC_BLOCK + tid;
    key[k] = e < left ? K[w0 + e] : 0ull;
    val[k] = e < left ? V[w0 + e] : 0u;
  };
  auto mark_row = [&](int k) -> bool {
    const uint32_t e = k * LC_BLOCK + tid;
    uint64_t prev = __shfl_up_sync(0xffffffffu, key[k], 1);
    if (lane == 0) prev = e < left && w0 + e > 0 ? K[w0 + e - 1] : 0ull;
    const bool head = e >= left || w0 + e == 0 || ((key[k] ^ prev) >> R) != 0ull;
    const uint32_t b = __ballot_sync(0xffffffffu, head);
    if (lane == 0) S.heads[k * LC_WARPS + warp] = b;
    return head;
  };
#pragma unroll
  for (int k = 0; k < LC_W / LC_BLOCK; ++k) load_row(k);
  if (tid == 0) S.sq = has_error(a.ctrl) ? 1u : 0u;
#pragma unroll
  for (int k = 0; k < LC_W / LC_BLOCK; ++k) mark_row(k);
  __syncthreads();
  if (S.sq) return;  // an earlier kernel failed
  const uint32_t first = next_head(S.heads, 0, win);
  if (first >= win) return;  // inside a bucket of an earlier tile
  // The end of the last bucket that starts in the window.
  uint32_t end = win;
  bool big = false;
  int rows = LC_W / LC_BLOCK;
  if (left > (uint32_t)LC_W) {
    big = true;
#pragma unroll
    for (int k = LC_W / LC_BLOCK; k < LC_ITEMS; ++k) {
      if (big) {  // block-uniform
        load_row(k);
        const bool head = mark_row(k);
        rows = k + 1;
        if (__syncthreads_or(head)) big = false;
      }
    }
    end = next_head(S.heads, LC_W, LC_CAP);
    if (end > left) end = left;
  }
  if (big) {
    // The last bucket runs past the tile: find its end (32 probes at a time)
    // and hand it to the global path.
    uint32_t p = win - 1;  // its start: the last head in the window
    while (!((S.heads[p >> 5] >> (p & 31)) & 1u)) {
      const uint32_t b = S.heads[p >> 5] & ((2u << (p & 31)) - 1u);
      p = b ? (p & ~31u) + 31 - __clz(b) : (p & ~31u) - 1;
    }
    end = p;
    if (warp == 0) {
      const uint64_t t = K[w0 + p] >> R;
      uint32_t lo = w0 + LC_CAP - 1, n = a.m - lo;  // lo is inside; the end is in (lo, lo + n]
      while (n > 1) {
        const uint32_t step = (n + 31) / 32;
        const uint64_t x = (uint64_t)lane * step;
        const bool in = x < n && (K[lo + x] >> R) == t;
        const uint32_t q = 31 - __clz(__ballot_sync(0xffffffffu, in));  // lane 0 is always in
        lo += q * step;
        n = min(step, n - q * step);
      }
      if (lane == 0) {
        const uint32_t start = w0 + p, size = lo + 1 - start;
        const unsigned long long old =
            atomicAdd(&a.ctrl->rc.large, (1ull << 32) | (unsigned long long)size);
        const uint32_t g = (uint32_t)(old >> 32), off = (uint32_t)old;
        if (g < a.max_large) {
          a.lg[g] = start;
          a.loff[g] = off;
          a.lbase[g] = start - off;
          a.lold[g] = NO_NAME;
        } else {  // never taken unless a logic error
          raise_error(a.ctrl, ERR_INTERNAL, 20);
        }
      }
    }
    if (end == first) return;
  }
  const uint32_t c = end - first;  // the tile's items: [first, end)
  const uint32_t rank0 = w0 + first;
  __syncthreads();

  // Buckets: their ordinals (heads at or before an item, less one) and
  // first items.
  if (tid < LC_SEGS) S.pre[tid] = tid < rows * LC_WARPS ? __popc(S.heads[tid]) : 0u;
  if (tid == 0) S.sq = 0u;
#pragma unroll
  for (int k = 0; k < LC_ITEMS; ++k) S.bin[k * LC_BLOCK + tid] = 0u;
  __syncthreads();
  if (warp == 0) scan_segments(S.pre);
  __syncthreads();
  const uint32_t le = lanemask_lt() | (1u << lane);
#pragma unroll
  for (int k = 0; k < LC_ITEMS; ++k) {
    const uint32_t e = k * LC_BLOCK + tid;
    if (k < rows && e < end) {
      const uint32_t h = S.heads[k * LC_WARPS + warp];
      if ((h >> lane) & 1u) S.start[S.pre[k * LC_WARPS + warp] + __popc(h & le) - 1u] = (uint16_t)e;
      if (e + 1 == end) S.start[S.pre[k * LC_WARPS + warp] + __popc(h & le)] = (uint16_t)end;
    }
  }
  __syncthreads();
  // A bucket of s items has 2^floor(log2 s) bins of its next bits, at its
  // own slots. bin: the item's bin | its key bits below the bin's << 16.
  uint32_t bin[LC_ITEMS], slot[LC_ITEMS];
#pragma unroll
  for (int k = 0; k < LC_ITEMS; ++k) {
    const uint32_t e = k * LC_BLOCK + tid;
    bin[k] = LC_NO_ITEM;
    uint32_t x = LC_NO_ITEM;
    if (k < rows && e >= first && e < end) {
      const uint32_t lb =
          S.pre[k * LC_WARPS + warp] + __popc(S.heads[k * LC_WARPS + warp] & le) - 1u;
      const uint32_t s0 = S.start[lb], size = S.start[lb + 1] - s0;
      const uint32_t d = min(31u - __clz(size), R);
      x = s0 - first + ((uint32_t)(key[k] >> (R - d)) & ((1u << d) - 1u));
      bin[k] = x | ((R - d) << 16);
    }
    slot[k] = x != LC_NO_ITEM ? atomicAdd(&S.bin[x], 1u) : 0u;
  }
  __syncthreads();
  uint8_t *flag = reinterpret_cast<uint8_t *>(S.start);  // of the sorted positions
  for (uint32_t x = tid; x < LC_CAP / 4; x += LC_BLOCK) reinterpret_cast<uint32_t *>(S.start)[x] = 0u;
  scan_bins(S, c);

  // Tail suffixes (fewer than c0 characters left in their text) are groups
  // of their own.
  uint32_t tails = 0;
#pragma unroll
  for (int k = 0; k < LC_ITEMS; ++k) {
    if (bin[k] == LC_NO_ITEM) continue;
    bool t;
    if (a.S <= 1) {
      t = a.N - val[k] < a.c0;
    } else {
      const uint32_t s = (uint32_t)(key[k] >> a.cb);
      t = __ldg(a.seg_off + s + 1) - (val[k] - s) < a.c0;  // text end - ungapped position
    }
    tails |= (uint32_t)t << k;
  }
  auto to_slots = [&]() {  // keys to their slots, from the arrival order in the bin
#pragma unroll
    for (int k = 0; k < LC_ITEMS; ++k) {
      if (bin[k] == LC_NO_ITEM) continue;
      slot[k] += S.bin[bin[k] & 0xFFFFu];
      S.key[slot[k]] = key[k];
      S.idx[slot[k]] = (uint16_t)((k * LC_BLOCK + tid) | (((tails >> k) & 1u) << 15));
    }
  };
  to_slots();
  const bool runs = S.sq > LC_AVG * c;
  __syncthreads();
  if (runs) {
    for (;;) {
      // Flag the large bins of more than one key (a tail counts as one, so
      // that a run has none).
#pragma unroll
      for (int k = 0; k < LC_ITEMS; ++k) {
        if (bin[k] == LC_NO_ITEM) continue;
        const uint32_t x = bin[k] & 0xFFFFu;
        const uint32_t lo = S.bin[x] & ~LC_MIXED, n = (S.bin[x + 1] & ~LC_MIXED) - lo;
        if (n >= LC_RUN_MIN && (S.key[lo] != key[k] || ((tails >> k) & 1u)))
          atomicOr(&S.bin[x], LC_MIXED);
      }
      __syncthreads();
      // Spread those again; every other bin keeps its slots. (A run of a text's
      // smallest character that ends the text has the key of its own tails:
      // compared all against all, 2500 of them in 2^20 characters of DNA
      // took a build 1.75 ms instead of 0.64.)
      uint32_t next[LC_ITEMS];
      bool more = false;
#pragma unroll
      for (int k = 0; k < LC_ITEMS; ++k) {
        next[k] = LC_NO_ITEM;
        if (bin[k] == LC_NO_ITEM) continue;
        const uint32_t x = bin[k] & 0xFFFFu, r = bin[k] >> 16;
        const uint32_t b0 = S.bin[x], lo = b0 & ~LC_MIXED, n = (S.bin[x + 1] & ~LC_MIXED) - lo;
        next[k] = lo | (r << 16);
        if ((b0 & LC_MIXED) && r != LC_PARTED) {
          const uint32_t d = min(31u - __clz(n), r);
          if (r > 0)
            next[k] = (lo + ((uint32_t)(key[k] >> (r - d)) & ((1u << d) - 1u))) | ((r - d) << 16);
          else  // one key: its tails, then the others
            next[k] = (lo + (((tails >> k) & 1u) ? 0u : 1u)) | (LC_PARTED << 16);
          more = true;
        }
      }
      if (!__syncthreads_or(more)) break;
#pragma unroll
      for (int k = 0; k < LC_ITEMS; ++k) S.bin[k * LC_BLOCK + tid] = 0u;
      __syncthreads();
#pragma unroll
      for (int k = 0; k < LC_ITEMS; ++k) {
        bin[k] = next[k];
        slot[k] = arrive_runs(S.bin, bin[k] == LC_NO_ITEM ? LC_NO_ITEM : bin[k] & 0xFFFFu);
      }
      __syncthreads();
      scan_bins(S, c);
      to_slots();
      __syncthreads();
    }
    // The first item of each run.
#pragma unroll
    for (int k = 0; k < LC_ITEMS; ++k) S.val[k * LC_BLOCK + tid] = 0xFFFFFFFFu;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < LC_ITEMS; ++k) {
      uint32_t x = LC_NO_ITEM;
      if (bin[k] != LC_NO_ITEM) {
        const uint32_t b0 = S.bin[bin[k] & 0xFFFFu];
        if (!(b0 & LC_MIXED) && (S.bin[(bin[k] & 0xFFFFu) + 1] & ~LC_MIXED) - b0 >= LC_RUN_MIN)
          x = bin[k] & 0xFFFFu;
      }
      const uint32_t mine = ((uint32_t)(k * LC_BLOCK + tid) << 16) | slot[k];
      const uint32_t x0 = __shfl_sync(0xffffffffu, x, 0);
      if (__all_sync(0xffffffffu, x == x0)) {  // the first lane holds the first item
        if (lane == 0 && x != LC_NO_ITEM) atomicMin(&S.val[x], mine);
      } else if (x != LC_NO_ITEM) {
        atomicMin(&S.val[x], mine);
      }
    }
    __syncthreads();
  }
  // slot becomes the item's sorted position; eq its equal keys (itself
  // included, tails apart) << 16 | those before it, 1 << 16 if unique.
  uint32_t eq[LC_ITEMS];
#pragma unroll
  for (int k = 0; k < LC_ITEMS; ++k) {
    eq[k] = 1u << 16;
    if (bin[k] == LC_NO_ITEM) continue;
    const uint32_t b0 = S.bin[bin[k] & 0xFFFFu], lo = b0 & ~LC_MIXED;
    const uint32_t hi = S.bin[(bin[k] & 0xFFFFu) + 1] & ~LC_MIXED, self = slot[k];
    if (hi - lo == 1) continue;  // alone in its bin
    const uint32_t e = k * LC_BLOCK + tid;
    if (runs && hi - lo >= LC_RUN_MIN && !(b0 & LC_MIXED)) {
      // One run: arrival order, with the first item in front.
      const uint32_t m = S.val[bin[k] & 0xFFFFu];
      if (m >> 16 == e)
        slot[k] = lo;
      else if (self == lo)
        slot[k] = m & 0xFFFFu;
      eq[k] = ((hi - lo) << 16) | (slot[k] - lo);
      continue;
    }
    uint32_t smaller = 0, equal = 0;
    for (uint32_t x = lo; x < hi; ++x) {
      const uint64_t o = S.key[x];
      smaller += o < key[k] ? 1u : 0u;
      equal += o == key[k] ? 1u : 0u;
    }
    slot[k] = lo + smaller;
    if (equal == 1) continue;
    const bool tail = (tails >> k) & 1u;
    uint32_t same = 0, before = 0, tail_before = 0;
    for (uint32_t x = lo; x < hi; ++x) {
      if (S.key[x] != key[k] || x == self) continue;
      const uint32_t id = S.idx[x];
      const uint32_t earlier = (id & 0x7FFFu) < e ? 1u : 0u;
      if (id >> 15) {
        tail_before += earlier;
      } else {
        ++same;
        before += earlier;
      }
    }
    // Tails precede the longer suffixes of the same key in input order.
    slot[k] += tail_before + before;
    if (!tail) eq[k] = ((same + 1) << 16) | before;
  }

  // Values in sorted order; survivors (1) and their groups' heads (3) flagged.
  if (runs) __syncthreads();  // the runs' first items are read
  bool any = false;
#pragma unroll
  for (int k = 0; k < LC_ITEMS; ++k) {
    if (bin[k] == LC_NO_ITEM) continue;
    uint32_t v = val[k];
    if (eq[k] != 1u << 16) {
      any = true;
      flag[slot[k]] = (eq[k] & 0xFFFFu) ? 1 : 3;
    } else if (a.S > 1) {  // final: the index local to the suffix's text
      const uint32_t s = (uint32_t)(key[k] >> a.cb);
      v -= __ldg(a.seg_off + s) + s;
    }
    S.val[slot[k]] = v;
  }
  if (!__syncthreads_or(any)) {  // every suffix is unique: SA at the ranks
#pragma unroll
    for (int k = 0; k < LC_ITEMS; ++k) {
      const uint32_t e = k * LC_BLOCK + tid;
      if (e < c) a.sa[rank0 + e] = S.val[e];
    }
    return;
  }
#pragma unroll
  for (int k = 0; k < LC_ITEMS; ++k) {
    const uint32_t f = flag[k * LC_BLOCK + tid];
    const uint32_t Sv = __ballot_sync(0xffffffffu, f != 0), H = __ballot_sync(0xffffffffu, f == 3);
    if (lane == 0) {
      S.surv[k * LC_WARPS + warp] = Sv;
      S.heads[k * LC_WARPS + warp] = H;
      S.pre[k * LC_WARPS + warp] = __popc(Sv) | (__popc(H) << 16);
    }
  }
  __syncthreads();
  if (warp == 0) {
    const uint32_t tot = scan_segments(S.pre);
    if (lane == 0) {
      const unsigned long long old =
          atomicAdd(reinterpret_cast<unsigned long long *>(&a.ctrl->rc.m_s),
                    ((unsigned long long)(tot >> 16) << 32) | (tot & 0xFFFFu));
      S.surv_base = (uint32_t)old;
      S.grp_base = (uint32_t)(old >> 32);
      S.upd_base = atomicAdd(&a.ctrl->rc.upd, tot & 0xFFFFu);
    }
  }
  __syncthreads();
  // Each group's head records its start in the next list, head rank and
  // name; the members take the name from shared memory.
  uint32_t *names = S.bin;  // every bin start is read
#pragma unroll
  for (int k = 0; k < LC_ITEMS; ++k) {
    if (bin[k] == LC_NO_ITEM || eq[k] == 1u << 16 || (eq[k] & 0xFFFFu)) continue;
    const uint32_t w = slot[k] >> 5, m = (1u << (slot[k] & 31)) - 1u;
    const uint32_t o = (S.pre[w] >> 16) + __popc(S.heads[w] & m);
    const uint32_t at = S.surv_base + (S.pre[w] & 0xFFFFu) + __popc(S.surv[w] & m);
    const uint32_t size = eq[k] >> 16, rank = rank0 + slot[k], g = S.grp_base + o;
    const uint32_t name = a.naming == NAMES_RETAIN ? rank + size / 2 : rank;
    names[o] = name;
    if (g >= a.max_groups) {  // never taken unless a logic error
      raise_error(a.ctrl, ERR_INTERNAL, 21);
      continue;
    }
    a.gstart_out[g] = at;
    a.gname_out[g] = name;
    a.ghead_out[g] = rank;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < LC_ITEMS; ++k) {
    const uint32_t e = k * LC_BLOCK + tid;
    if (e >= c) continue;
    const uint32_t w = k * LC_WARPS + warp, v = S.val[e];
    const bool surv = (S.surv[w] >> lane) & 1u;
    a.sa[rank0 + e] = surv ? SA_NONE : v;
    if (!surv) continue;
    const uint32_t i = (S.pre[w] & 0xFFFFu) + __popc(S.surv[w] & (le >> 1));
    const uint32_t o = (S.pre[w] >> 16) + __popc(S.heads[w] & le) - 1u;
    if (S.surv_base + i >= a.N || v >= a.isa_len) {  // never taken unless a logic error
      raise_error(a.ctrl, ERR_INTERNAL, 23);
      continue;
    }
    a.act_out[S.surv_base + i] = ((uint64_t)(S.grp_base + o) << 32) | v;
    a.upd[S.upd_base + i] = ((uint64_t)names[o] << 32) | v;
  }
}

__global__ void __launch_bounds__(LC_BLOCK, 2) k_local(LocalArgs a) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  LcSmem &S = *reinterpret_cast<LcSmem *>(smem_raw);
  local_tile(S, a);
  if (!a.host) return;
  // The last tile reports the counts and the error word to the host.
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence_system();  // the host may act on the report before the kernel ends
    S.sq = atomicAdd(&a.ctrl->done[1], 1u) + 1u == gridDim.x ? 1u : 0u;
  }
  __syncthreads();
  if (!S.sq) return;
  __threadfence();
  if (threadIdx.x < 16)
    a.host[threadIdx.x] = load_volatile_u32(reinterpret_cast<const uint32_t *>(a.ctrl) + threadIdx.x);
  report_to_host(a.host_flag);
}

cudaError_t launch_local(const LocalArgs &a, cudaStream_t stream) {
  if (a.m == 0) return cudaSuccess;
  if (a.R == 0 || a.R >= 64) return cudaErrorInvalidValue;
  const int smem = (int)sizeof(LcSmem);
  cudaError_t e = ensure_smem_attributes(reinterpret_cast<const void *>(&k_local), smem, true);
  if (e != cudaSuccess) return e;
  k_local<<<(a.m + LC_W - 1) / LC_W, LC_BLOCK, smem, stream>>>(a);
  return cudaGetLastError();
}

// The buckets left to the global path: their items, bucket by bucket, keyed
// by (bucket ordinal, low key bits). Ordinals fit the top bits they replace
// (there are no more buckets than values of those bits).
__global__ void __launch_bounds__(256) k_gather_big(GatherBigArgs a) {
  const uint64_t j64 = (uint64_t)blockIdx.x * 256 + threadIdx.x;
  if (j64 >= a.mL) return;
  const uint32_t j = (uint32_t)j64;
  uint32_t lo = 0, hi = a.GL - 1;  // the last bucket with loff <= j
  while (lo < hi) {
    const uint32_t mid = (lo + hi + 1) >> 1;
    if (__ldg(a.loff + mid) <= j)
      lo = mid;
    else
      hi = mid - 1;
  }
  const uint32_t src = __ldg(a.lg + lo) + (j - __ldg(a.loff + lo));
  if (src >= a.m) {  // never taken unless a logic error
    raise_error(a.ctrl, ERR_INTERNAL, 22);
    return;
  }
  a.keys[j] = ((uint64_t)lo << a.R) | (a.kin[src] & ((1ull << a.R) - 1ull));
  a.vals[j] = a.vin[src];
  a.sa[src] = SA_NONE;
}

cudaError_t launch_gather_big(const GatherBigArgs &a, cudaStream_t stream) {
  if (a.mL == 0) return cudaSuccess;
  k_gather_big<<<(unsigned)(((uint64_t)a.mL + 255) / 256), 256, 0, stream>>>(a);
  return cudaGetLastError();
}

}  // namespace gbsa
