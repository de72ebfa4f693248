// Round driver and C-ABI of gbsa: prefix doubling with discarding in
// inverse-suffix-array form (Section 2.1, Algorithms 1, 4 and 5).
//
// Round 0 (initial names, Algorithm 1's first lines):
//   byte histogram and a sample of prefixes -> alphabet and number of digits
//   (host, choose_split) -> packed keys -> radix sort of the top digits ->
//   sort/rename/unique/compact of the buckets of equal top bits tile by tile
//   (k_local.cu; buckets too large for a tile: radix sort of their other
//   digits and k_rename), or radix sort of all digits -> k_rename; then the
//   ISA entries of the suffixes already final that later rounds read
//   (k_isa.cu) and, in large texts, the groups in position order (k_reorder.cu).
// Round r >= 1 (one doubling step, h = c0 * 2^(r-1) characters resolved):
//   large groups: partner-name gather -> radix sort of (group, partner)
//   keys; small groups: tile-local refine (k_refine.cu); then the rename of
//   the large groups, the queued ISA updates and the classification of the
//   new groups.
// With sa_options.multiplier a = 3 or 4 (Section 2.1, Prefix Quadrupling) a
// round ranks the names of i, i + h, .., i + (a-1)h and h grows a-fold: the
// sorts become two stable sorts (later partners, then group and first
// partner) and the boundary tests compare the whole tuple.
// The loop ends when no suffix is active (every name unique; the paper's
// loop bound is one round short, so the count decides). SA is complete then:
// each suffix wrote SA[name] = i when its name became unique.
//
// Host <-> device per round: one 64-byte read of the control block (active
// and group counts of both producers, large-group counts, pass count, error
// word) at the end of the round. Round 0 reads the byte counts and the sample
// first and, from buckets, the control block before and after the large ones'
// rename; reports that a kernel writes to pinned memory are polled.
//
// Data layout in HBM (N characters in S texts, gapped positions N + S):
//   keys A/B u64[N], vals A/B u32[N] (radix sort of round 0 and of large
//   groups), active lists u64[N] x2 (g << 32 | i', current and next), queued
//   ISA updates u64[N], ISA u32[N + S + 1] (end slots hold 0xFFFFFFFF),
//   group starts, names and head ranks u32[N/2+1] x2 each, parent names
//   u32[N/2+1], large-group lists, the refine tile map, look-back status,
//   control block, plan, histograms: about 67 bytes per character.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <set>
#include <utility>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "../../include/gbsa.h"
#include "launch.h"
#include "segcopy.h"

#define GBSA_API extern "C" __attribute__((visibility("default")))

namespace gbsa {
namespace {

constexpr uint32_t DEFAULT_SPIN_LIMIT = 1u << 20;  // ~1 s with the 1 us back-off cap
// ISA writes are bucketed by position when this many may be pending (the
// default discard threshold; sa_options.bucket_min and the tuning table
// override it).
constexpr uint32_t BUCKET_MIN = 1u << 22;

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

// NVTX ranges (header-only NVTX 3: without a profiler attached a push or
// pop is a call through a pointer to a function that returns at once).
// A build is one range, each round a range inside it, each kernel launch
// a range named for its class, so a profiler's launch list attributes
// every kernel to its round and step.
const char *const KERNEL_RANGE[SA_K_CLASSES] = {
    "gbsa:byte_hist", "gbsa:pack",     "gbsa:digit_hist", "gbsa:plan",     "gbsa:onesweep",
    "gbsa:rename",    "gbsa:gather",   "gbsa:output",     "gbsa:refine",   "gbsa:scatter",
    "gbsa:classify",  "gbsa:apply",    "gbsa:bucket",     "gbsa:reorder"};

struct NvtxRange {
  bool open = true;
  explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
  void end() {
    if (open) nvtxRangePop();
    open = false;
  }
  ~NvtxRange() { end(); }
  NvtxRange(const NvtxRange &) = delete;
  NvtxRange &operator=(const NvtxRange &) = delete;
};

struct Layout {
  size_t ctrl, plan, hist, dbase, bytehist, code, segoff;
  size_t ka, kb, va, vb, act0, act1, upd, isa, gs0, gs1, gn0, gn1, gh0, gh1, gold;
  size_t lg, loff, lbase, lold, tfirst, bcount, pm1, need;
  size_t st_sort, st_ren, zeroed, total;
  uint32_t max_groups, max_large, max_tiles, need_words;
};

// Granules of the needed ISA entries (k_isa.cu): position >> need_shift.
uint32_t need_shift(uint64_t positions) {
  uint32_t s = 0;
  while (positions >> s >= (uint64_t)NEED_WORDS * 32) ++s;
  return s;
}
uint32_t need_words(uint64_t positions) {
  return (uint32_t)((positions >> need_shift(positions)) / 32 + 1);
}

Layout make_layout(uint64_t N, uint32_t S) {
  Layout L{};
  size_t o = 0;
  auto take = [&](size_t bytes) {
    size_t r = o;
    o += align256(bytes);
    return r;
  };
  const uint64_t Nm = N ? N : 1;
  // What starts at zero, in one piece: control block, histograms and the
  // look-back status words.
  L.ctrl = take(sizeof(Ctrl));
  L.hist = take(MAX_PASSES * RADIX * 4);
  L.bytehist = take(RADIX * 4 + sizeof(KeySample));
  const uint64_t ts = std::max<uint64_t>(1, (N + SORT_TILE_MIN - 1) / SORT_TILE_MIN);
  L.st_sort = take(ts * RADIX * 8);
  const uint64_t tr = std::max<uint64_t>(1, (N + RENAME_TILE - 1) / RENAME_TILE);
  L.st_ren = take(tr * 3 * 8);
  L.zeroed = o;
  L.plan = take(sizeof(SortPlan));
  L.dbase = take(MAX_PASSES * RADIX * 4);
  L.code = take(RADIX);
  L.segoff = take(((size_t)S + 1) * 4);
  // The key buffers also hold the group order's scan sums and marks, which
  // a batch of mostly empty texts needs more of than of keys.
  L.ka = take(std::max<uint64_t>(Nm * 8, rank_sums_words(N + S, Nm / 2) * 4));
  L.kb = take(std::max<uint64_t>(Nm * 8, rank_lines(N + S) * 32));
  L.va = take(Nm * 4);
  L.vb = take(Nm * 4);
  L.act0 = take(Nm * 8);
  L.act1 = take(Nm * 8);
  L.upd = take(Nm * 8);
  L.isa = take((N + S + 1) * 4);
  L.max_groups = (uint32_t)(Nm / 2 + 1);
  L.gs0 = take(((size_t)L.max_groups + 1) * 4);
  L.gs1 = take(((size_t)L.max_groups + 1) * 4);
  L.gn0 = take((size_t)L.max_groups * 4);
  L.gn1 = take((size_t)L.max_groups * 4);
  L.gh0 = take((size_t)L.max_groups * 4);
  L.gh1 = take((size_t)L.max_groups * 4);
  L.gold = take((size_t)L.max_groups * 4);
  L.max_large = (uint32_t)(Nm / (REFINE_MIN_NOMINAL + 1) + 1);
  L.lg = take((size_t)L.max_large * 4);
  L.loff = take((size_t)L.max_large * 4);
  L.lbase = take((size_t)L.max_large * 4);
  L.lold = take((size_t)L.max_large * 4);
  L.bcount = take((size_t)BUCKET_BLOCKS_MAX * RADIX * 4);
  L.pm1 = take(8);
  L.need_words = need_words(N + S);
  L.need = take(3 * (size_t)L.need_words * 4);
  L.max_tiles = (uint32_t)((Nm + REFINE_MIN_NOMINAL - 1) / REFINE_MIN_NOMINAL);
  L.tfirst = take(((size_t)L.max_tiles + 1) * 4);
  L.total = o;
  return L;
}

uint32_t bits_for(uint64_t v) {  // bits to hold values 0..v
  uint32_t b = 0;
  while (b < 64 && (v >> b) != 0) ++b;
  return b;
}

int sm_count() { return device_sm_count(); }

// Library-private stream-ordered pools, one per device (never trimmed, so
// repeated builds reuse their memory without touching the process-wide
// default pool).
std::mutex g_pool_mu;
std::map<int, cudaMemPool_t> g_pools;

cudaError_t pool_alloc(void **p, size_t bytes, cudaStream_t st) {
  std::mutex &mu = g_pool_mu;
  std::map<int, cudaMemPool_t> &pools = g_pools;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  cudaMemPool_t pool;
  {
    std::lock_guard<std::mutex> g(mu);
    auto it = pools.find(dev);
    if (it == pools.end()) {
      cudaMemPoolProps props{};
      props.allocType = cudaMemAllocationTypePinned;
      props.location.type = cudaMemLocationTypeDevice;
      props.location.id = dev;
      e = cudaMemPoolCreate(&pool, &props);
      if (e != cudaSuccess) return e;
      uint64_t thr = UINT64_MAX;
      cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr);
      pools[dev] = pool;
    } else {
      pool = it->second;
    }
  }
  return cudaMallocFromPoolAsync(p, bytes, pool, st);
}

struct PoolBuf {
  void *p = nullptr;
  cudaStream_t st = nullptr;
  ~PoolBuf() {
    if (p) cudaFreeAsync(p, st);
  }
};

#define CK(x)                                  \
  do {                                         \
    cudaError_t e_ = (x);                      \
    if (e_ != cudaSuccess) return SA_ERR_CUDA; \
  } while (0)

// Mirror of the first 64 bytes of Ctrl.
// Pinned host staging for the small readbacks of a build (control block,
// byte histogram): a kernel writes them into pinned host memory, so a
// readback does not wait on a copy engine behind the large copies of
// builds on other streams (a server's concurrent requests). Blocks are
// allocated once (mapped into every device's address space) and reused.
constexpr size_t STAGE_BYTES = 16 << 10;
std::mutex g_stage_mu;
std::vector<void *> g_stage_free;

struct PinnedStage {
  void *p = nullptr;
  cudaError_t get() {
    if (p) return cudaSuccess;
    {
      std::lock_guard<std::mutex> g(g_stage_mu);
      if (!g_stage_free.empty()) {
        p = g_stage_free.back();
        g_stage_free.pop_back();
        return cudaSuccess;
      }
    }
    const cudaError_t e = cudaHostAlloc(&p, STAGE_BYTES, cudaHostAllocMapped | cudaHostAllocPortable);
    if (e != cudaSuccess) p = nullptr;  // nothing to hand back to the free list
    return e;
  }
  ~PinnedStage() {
    if (!p) return;
    std::lock_guard<std::mutex> g(g_stage_mu);
    g_stage_free.push_back(p);
  }
};

// Costs of round 0's steps over all items in units of one radix pass, and
// a pass's time: a fixed part and 7 ps per item (choose_split). The tile
// pass costs LOCAL_COST, more for larger buckets (per doubling) and, in
// buckets of more than one item, for skewed digits (by the deviation of
// -log2 p over 8 bits). Measured against the model at 2^28: DNA after 3, 4, 5
// passes 1.92, 1.55, 1.40 (1.93, 1.45, 1.45), Markov DNA after 4 and 5 3.4
// and 2.7 (3.3, 2.1), Zipf bytes at 2^25 after 4 and 5 3.1 and 2.3 (3.2, 2.1).
constexpr double LOCAL_COST = 1.45, LOCAL_SIZE_COST = 0.06, LOCAL_SKEW_COST = 0.8;
constexpr double RENAME_COST = 1.5;
constexpr double PASS_FIXED_US = 9.0, PASS_ITEM_US = 7e-6;
constexpr uint32_t REFINE_HALF_MIN = 1u << 19;
constexpr uint64_t LOCAL_REPORT_MAX = 1ull << 22;
// log2 of the bucket size from which the model takes buckets to be too large
// for a tile. A tile takes one of s items with probability (3072 - s) / 2560,
// half of those of 2^10.8 and 71 % here. With 10.8 the choices for Zipf bytes,
// protein and random bytes of 2^20 to 2^30 characters are the same, but for two
// digits instead of three for random bytes of 2^26: 3.71 ms, 2.57.
constexpr double LOCAL_LARGE_LOG2 = 10.3;
// From the first length on, with at most a quarter of the suffixes active,
// the ISA gets only the entries that later rounds read (k_isa.cu), and from
// the second on they go through a list that can be bucketed by position (an
// ISA that the L2 holds is written directly).
constexpr uint64_t NEED_MIN_N = 1ull << 22, COLLECT_MIN_N = 1ull << 25;
// Texts at least this long wait for the gram histogram to model their
// prefixes by its statistics; shorter ones take the character counts.
constexpr uint64_t GRAM_MODEL_MIN = 1ull << 22;

// Texts at least this long are sampled (KeySample; the counting blocks take as
// long) by as many blocks as show a bucket size of 2^11 in 8 pairs or more up to
// 2^28 characters. Batches are sampled whatever their size and by more blocks:
// texts of few letters beside texts of many hide in the batch's counts, and of
// 16 batches of 48 such texts, in which 6 digits are best, 16 blocks chose 5
// for three, 64 for one (0.74 ms, 0.80).
constexpr uint64_t SAMPLE_MIN_N = 1ull << 22;
// Texts of at most this many bits per character are modelled by their grams and
// are left to them (8 characters are two digits of theirs).
constexpr uint32_t SAMPLE_MIN_BITS = 2;
// Characters in too large buckets from which the fixed costs of sorting these
// count in full, as a sample's tail of fewer may be the fit's alone. (Batches of
// 28 to 48 texts, half DNA, half Zipf bytes: from 2^10 characters on a digit too
// many, 0.746 ms instead of 0.742, from 2^16 on one too few, 0.80.)
constexpr double SAMPLE_CERTAIN = 32768.0;
uint32_t sample_blocks(uint64_t n, uint32_t texts) {
  if (n < SAMPLE_MIN_N && texts == 1) return 0;
  return n < (1ull << 28) && texts == 1 ? 16u : SAMPLE_BLOCKS_MAX;
}

// Share of n characters in buckets too large for a tile, by a sample of which
// `pairs` and `triples` agree in `chars` characters (1 to SAMPLE_CHARS): of the
// bucket sizes (over the characters) the pairs give the mean, the triples the
// mean square, and a lognormal distribution has these; between whole characters
// its parameters lie between theirs. A bucket of s items that starts anywhere
// in a tile's window does not fit with probability (s - 512) / 2560. Fewer than
// 8 pairs tell nothing.
double sampled_large_share(const KeySample &k, double chars, uint32_t blocks, uint64_t n) {
  const uint32_t c = (uint32_t)chars;
  if (k.pairs[c - 1] < 8) return 0.0;
  const double scale = (double)n / SAMPLE_KEYS, drawn = (double)blocks * SAMPLE_KEYS;
  auto fit = [&](uint32_t i, double &mu, double &sd) {  // of the logarithm of the size
    const double mean = 1.0 + 2.0 * std::max(0.5, (double)k.pairs[i]) / drawn * scale;
    const double square = 6.0 * (double)k.triples[i] / drawn * scale * scale;
    const double var = std::log(std::max(1.0, square / (mean * mean)));
    sd = std::sqrt(std::min(4.0, std::max(0.05, var)));
    mu = std::log(mean) - sd * sd / 2;
  };
  double mu, sd;
  fit(c - 1, mu, sd);
  if (chars > c) {
    double mu1, sd1;
    fit(c, mu1, sd1);
    mu += (chars - c) * (mu1 - mu);
    sd += (chars - c) * (sd1 - sd);
  }
  if (mu + 3.5 * sd <= std::log(512.0)) return 0.0;
  double share = 0, weight = 0;
  for (double z = -3.5; z <= 3.5; z += 0.5) {  // over the normal distribution
    const double w = std::exp(-z * z / 2);
    share += w * std::min(1.0, std::max(0.0, (std::exp(mu + sd * z) - 512.0) / 2560.0));
    weight += w;
  }
  return share / weight;
}

// How the probability of a k-character prefix is spread, as the normal
// distribution of its logarithm over the text's positions: mean and variance
// of -log2 p for the first g characters, then per further character (the
// last of a g-character gram given the others). For choosing a sort only.
struct PrefixModel {
  // (and the least -log2 p, that of the most frequent prefix)
  double g = 1, mean = 0, var = 0, mean1 = 0, var1 = 0, least = 0, least1 = 0;

  static void moments(const double *p, const double *q, int n, double &mean, double &var,
                      double &least) {
    // of -log2 q under p
    double s1 = 0, s2 = 0;
    least = 64;
    for (int i = 0; i < n; ++i)
      if (p[i] > 0) {
        const double x = -std::log2(q[i]);
        s1 += p[i] * x;
        s2 += p[i] * x * x;
        least = std::min(least, x);
      }
    mean = s1;
    var = std::max(0.0, s2 - s1 * s1);
  }

  static PrefixModel characters(const uint32_t *hist) {
    double p[RADIX], total = 0;
    for (int c = 0; c < RADIX; ++c) total += hist[c];
    for (int c = 0; c < RADIX; ++c) p[c] = hist[c] / total;
    PrefixModel m;
    moments(p, p, RADIX, m.mean, m.var, m.least);
    m.mean1 = m.mean;
    m.var1 = m.var;
    m.least1 = m.least;
    return m;
  }

  // From the counts of the 8-bit grams of 8 / b characters.
  static PrefixModel grams(const uint32_t *hist, uint32_t b) {
    double p[RADIX], q[RADIX], total = 0;
    for (int c = 0; c < RADIX; ++c) total += hist[c];
    for (int c = 0; c < RADIX; ++c) p[c] = hist[c] / total;
    const int last = 1 << b;
    for (int c = 0; c < RADIX; c += last) {
      double ctx = 0;
      for (int x = 0; x < last; ++x) ctx += p[c + x];
      for (int x = 0; x < last; ++x) q[c + x] = ctx > 0 ? p[c + x] / ctx : 0;
    }
    PrefixModel m;
    m.g = 8.0 / b;
    moments(p, p, RADIX, m.mean, m.var, m.least);
    moments(p, q, RADIX, m.mean1, m.var1, m.least1);
    return m;
  }

  // Mean and variance of -log2 p of a `chars`-character prefix, and its least.
  void prefix(double chars, double &mu, double &v, double &top) const {
    mu = mean * chars / g, v = var * chars / g, top = least * chars / g;
    if (chars > g) {
      mu = mean + (chars - g) * mean1;
      v = var + (chars - g) * var1;
      top = least + (chars - g) * least1;
    }
  }

  // Cost of the tile pass over buckets of `chars`-character prefixes of a text
  // of 2^log_len characters; digit_chars characters to 8 bits.
  double local_cost(double chars, double log_len, double digit_chars) const {
    double mu, v, top;
    prefix(chars, mu, v, top);
    const double size = log_len - mu, sd = std::sqrt(std::max(v, 0.05));
    const double shared = 0.5 * std::erfc(-size / (sd * std::sqrt(2.0)));
    return LOCAL_COST + LOCAL_SIZE_COST * std::max(0.0, size + 4.0) +
           LOCAL_SKEW_COST * std::sqrt(var1 * digit_chars) * shared;
  }

  // Share of a text of 2^log_len characters whose `chars`-character prefix
  // occurs more than 2^log_large times.
  double large_share(double chars, double log_len, double log_large) const {
    if (chars <= 0) return log_len > log_large ? 1.0 : 0.0;
    double mu, v, top;
    prefix(chars, mu, v, top);
    if (log_len - top < log_large - 1.0) return 0.0;
    const double z = (log_large - (log_len - mu)) / std::sqrt(2.0 * std::max(v, 0.05));
    return 0.5 * std::erfc(z);
  }
};

struct HostCtrl {
  uint32_t error, err_where, passes, pass_mask;
  uint32_t m_s, g_s, m_l, g_l, upd, mid;
  unsigned long long large;
  uint32_t zero[4];
  uint32_t m_next() const { return m_s + m_l; }
  uint32_t g_next() const { return g_s + g_l; }
  uint32_t m_large() const { return (uint32_t)large; }
  uint32_t g_large() const { return (uint32_t)(large >> 32); }
};
static_assert(sizeof(HostCtrl) == 64, "HostCtrl mirrors the head of Ctrl");

struct Build {
  PinnedStage stage;            // small readbacks (fetch)
  bool stage_readbacks = true;  // false: copy-engine readbacks (no host allocation)
  // inputs
  const uint8_t *text = nullptr;
  uint64_t N = 0;
  uint32_t S = 1;
  std::vector<uint32_t> off;  // S+1 ungapped offsets
  uint32_t *sa = nullptr;
  uint32_t *isa_out = nullptr;
  sa_options opt{};
  sa_stats *stats = nullptr;
  cudaStream_t st = nullptr;
  // workspace
  uint8_t *ws = nullptr;
  Layout L{};
  Ctrl *ctrl = nullptr;
  SortPlan *plan = nullptr;
  uint32_t *hist = nullptr, *dbase = nullptr, *bytehist = nullptr, *segoff = nullptr;
  uint8_t *code = nullptr;
  uint64_t *ka = nullptr, *kb = nullptr, *act[2] = {nullptr, nullptr}, *upd = nullptr;
  uint64_t *st_sort = nullptr, *st_ren = nullptr;
  uint32_t *va = nullptr, *vb = nullptr, *isa = nullptr;
  uint32_t *gstart[2] = {nullptr, nullptr}, *gname[2] = {nullptr, nullptr};
  uint32_t *ghead[2] = {nullptr, nullptr}, *gold = nullptr;
  uint32_t *lg = nullptr, *loff = nullptr, *lbase = nullptr, *lold = nullptr, *tfirst = nullptr;
  uint32_t *bcount = nullptr;  // position-bucketing counts (BUCKET_BLOCKS_MAX x 256)
  uint32_t *need = nullptr;    // granules: active, covered, missing (k_isa.cu)
  bool isa_cleared = false;
  bool need_filtered = false;  // only needed ISA entries are written
  uint32_t *pm1 = nullptr;     // (passes, pass mask) of the first sort of an a-tuple round
  // launch bookkeeping
  uint32_t epoch = 0, slot = 0;
  uint32_t spin = DEFAULT_SPIN_LIMIT;
  bool inject_pending = false;
  uint64_t bytes = 0;
  uint32_t launches = 0;
  uint32_t naming = NAMES_RETAIN;
  uint32_t shape = 0, nominal = 512, small = 512;  // refine tile shape, window, largest group
  uint32_t sort_items = SORT_ITEMS_DEFAULT;  // keys per thread of the radix pass
  uint32_t bucket_min = BUCKET_MIN;  // pending ISA writes that are bucketed first
  uint32_t mult = 2;  // a: names ranked per round (2: doubling, 4: quadrupling)
  // per-kernel profiling (events on the build's stream)
  struct Rec {
    int cls, pass;
    uint64_t bytes;
    cudaEvent_t a, b;
  };
  bool prof = false;
  // Launches whose byte counts wait for the round's control block.
  static constexpr uint64_t PENDING = ~0ull;
  struct Pending {
    uint32_t scatter = 0, apply = 0, bucket_upd = 0, bucket_surv = 0, classify = 0;
  } pend;
  std::vector<cudaEvent_t> evpool;
  size_t evused = 0;
  std::vector<Rec> recs;

  ~Build() {
    for (cudaEvent_t e : evpool) cudaEventDestroy(e);
  }

  template <class T>
  T *at(size_t off_) {
    return reinterpret_cast<T *>(ws + off_);
  }

  void carve() {
    ctrl = at<Ctrl>(L.ctrl);
    plan = at<SortPlan>(L.plan);
    hist = at<uint32_t>(L.hist);
    dbase = at<uint32_t>(L.dbase);
    bytehist = at<uint32_t>(L.bytehist);
    code = at<uint8_t>(L.code);
    segoff = at<uint32_t>(L.segoff);
    ka = at<uint64_t>(L.ka);
    kb = at<uint64_t>(L.kb);
    va = at<uint32_t>(L.va);
    vb = at<uint32_t>(L.vb);
    act[0] = at<uint64_t>(L.act0);
    act[1] = at<uint64_t>(L.act1);
    upd = at<uint64_t>(L.upd);
    isa = at<uint32_t>(L.isa);
    gstart[0] = at<uint32_t>(L.gs0);
    gstart[1] = at<uint32_t>(L.gs1);
    gname[0] = at<uint32_t>(L.gn0);
    gname[1] = at<uint32_t>(L.gn1);
    ghead[0] = at<uint32_t>(L.gh0);
    ghead[1] = at<uint32_t>(L.gh1);
    gold = at<uint32_t>(L.gold);
    lg = at<uint32_t>(L.lg);
    loff = at<uint32_t>(L.loff);
    lbase = at<uint32_t>(L.lbase);
    lold = at<uint32_t>(L.lold);
    bcount = at<uint32_t>(L.bcount);
    pm1 = at<uint32_t>(L.pm1);
    need = at<uint32_t>(L.need);
    tfirst = at<uint32_t>(L.tfirst);
    st_sort = at<uint64_t>(L.st_sort);
    st_ren = at<uint64_t>(L.st_ren);
  }

  cudaError_t event(cudaEvent_t &e) {
    if (evused == evpool.size()) {
      cudaEvent_t x;
      cudaError_t r = cudaEventCreate(&x);
      if (r != cudaSuccess) return r;
      evpool.push_back(x);
    }
    e = evpool[evused++];
    return cudaEventRecord(e, st);
  }

  // Issues one kernel launch; with profiling, brackets it with events.
  // `bytes` is the launch's algorithmic traffic (radix passes: counted only
  // if the device plan kept the pass; rename: settled at the round's sync).
  template <class F>
  sa_status launch(int cls, int pass, uint64_t nbytes, F f) {
    NvtxRange range(KERNEL_RANGE[cls]);
    ++launches;
    cudaEvent_t a = nullptr, b = nullptr;
    if (prof) CK(event(a));
    CK(f());
    if (prof) {
      CK(event(b));
      recs.push_back({cls, pass, nbytes, a, b});
    }
    return SA_OK;
  }

  // After a stream sync: fold the recorded launches into the statistics.
  sa_status flush(uint32_t pass_mask, uint64_t rename_bytes_now, uint32_t mask1 = 0) {
    if (!prof || !stats) {
      recs.clear();
      evused = 0;
      return SA_OK;
    }
    for (const Rec &r : recs) {
      if (r.cls == SA_K_ONESWEEP &&
          !(((r.pass >= 32 ? mask1 : pass_mask) >> (r.pass & 31)) & 1u))
        continue;
      float ms = 0.f;
      CK(cudaEventElapsedTime(&ms, r.a, r.b));
      stats->kernel_ms[r.cls] += ms;
      stats->kernel_launches[r.cls] += 1;
      stats->kernel_bytes[r.cls] += r.cls == SA_K_RENAME ? rename_bytes_now : r.bytes;
    }
    recs.clear();
    evused = 0;
    return SA_OK;
  }

  sa_status next_launch(uint32_t *&ctr, uint32_t &ep) {
    if (slot == (uint32_t)TILE_COUNTERS) {
      CK(cudaMemsetAsync(ctrl->tile_ctr, 0, sizeof(ctrl->tile_ctr), st));
      slot = 0;
    }
    ctr = &ctrl->tile_ctr[slot++];
    ep = ++epoch;
    return SA_OK;
  }

  // bytes of device memory into host memory, synchronising `st`: through
  // the pinned stage by a kernel (a multiple of 4 bytes, at most
  // STAGE_BYTES), else, or without a stage, on the copy engine.
  cudaError_t fetch(void *host, const void *dev, size_t bytes) {
    if (stage_readbacks && bytes <= STAGE_BYTES && bytes % 4 == 0 && stage.get() != cudaSuccess) {
      cudaGetLastError();  // no pinned block to be had: the copy engine instead
      stage_readbacks = false;
    }
    if (!stage_readbacks || bytes > STAGE_BYTES || bytes % 4) {
      cudaError_t e = cudaMemcpyAsync(host, dev, bytes, cudaMemcpyDeviceToHost, st);
      return e == cudaSuccess ? cudaStreamSynchronize(st) : e;
    }
    cudaError_t e = launch_copy_words(reinterpret_cast<uint32_t *>(stage.p),
                                      reinterpret_cast<const uint32_t *>(dev), bytes / 4, st);
    if (e == cudaSuccess) ++launches;
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess) memcpy(host, stage.p, bytes);
    return e;
  }

  // Reports: words that a kernel's last block writes into the stage, then a
  // flag of its own (in its own cache line), cleared here before the launch.
  uint32_t *stage_words() { return reinterpret_cast<uint32_t *>(stage.p); }
  uint32_t *report_flag(int k) {
    uint32_t *f = stage_words() + 2 * RADIX + 32 * k;
    __atomic_store_n(f, 0u, __ATOMIC_RELAXED);
    return f;
  }

  // Waits for a report: polls its flag for a while (a stream synchronisation
  // returns about 4 us after the flag is set), then synchronises the stream.
  // A kernel that fails sets no flag, and the synchronisation returns its
  // error. With per-launch events the stream is always synchronised.
  cudaError_t wait_report(const uint32_t *flag) {
    if (!prof) {
      const auto t0 = std::chrono::steady_clock::now();
      do {
        for (int i = 0; i < 64; ++i)
          if (__atomic_load_n(flag, __ATOMIC_ACQUIRE)) return cudaSuccess;
      } while (std::chrono::steady_clock::now() - t0 < std::chrono::microseconds(300));
    }
    return cudaStreamSynchronize(st);
  }

  sa_status read_ctrl(HostCtrl &hc) {
    CK(fetch(&hc, ctrl, sizeof(HostCtrl)));
    return ctrl_status(hc);
  }

  static sa_status ctrl_status(const HostCtrl &hc) {
    if (hc.error == ERR_TIMEOUT) return SA_ERR_TIMEOUT;
    if (hc.error != ERR_NONE) return SA_ERR_INTERNAL;
    return SA_OK;
  }

  // Radix sort of (ka, va)[0, m) by the digits of spec; result where the
  // device plan says (plan->kfinal / vfinal).
  // chain 1: the first of the two sorts of an a-tuple round (its kept
  // passes are copied to pm1 afterwards; profile records tag pass + 32).
  // from_text (round 0, one text): pass 0 builds the keys from the text
  // (the pack wrote only the histograms), so it is kept even if constant.
  // keep: further passes kept whatever their digits (launch_sort_plan).
  sa_status sort(uint32_t m, const DigitSpec &spec, bool hist_ready = false, int chain = 0,
                 const PackArgs *from_text = nullptr, uint32_t keep = 0,
                 const PackArgs *grams = nullptr) {
    sa_status s = SA_OK;
    if (!hist_ready) {
      CK(cudaMemsetAsync(hist, 0, (size_t)spec.P * RADIX * 4, st));
      s = launch(SA_K_DIGIT_HIST, 0, 8ull * m, [&] {
        return launch_digit_histogram(ka, m, spec, hist, sm_count(), st);
      });
      if (s != SA_OK) return s;
      bytes += 8ull * m;  // histogram read
    }
    s = launch(SA_K_PLAN, 0, (uint64_t)spec.P * RADIX * 8, [&] {
      return launch_sort_plan(hist, dbase, spec, m, ka, kb, va, vb, plan, ctrl, st, nullptr,
                              keep | (from_text ? 1u : 0u), grams);
    });
    if (s != SA_OK) return s;
    for (uint32_t p = 0; p < spec.P; ++p) {
      PassArgs pa{};
      pa.plan = plan;
      pa.p = (int)p;
      pa.shift = spec.shift[p];
      pa.bits = spec.bits[p];
      pa.digit_base = dbase + p * RADIX;
      pa.m = m;
      pa.status = st_sort;
      s = next_launch(pa.tile_ctr, pa.epoch);
      if (s != SA_OK) return s;
      pa.ctrl = ctrl;
      pa.spin_limit = spin;
      pa.inject = inject_pending ? 1u : 0u;
      pa.items = sort_items;
      uint64_t pass_bytes = 24ull * m;
      if (from_text && p == 0) {
        pa.text = from_text->text;
        pa.code = from_text->code;
        pa.b = from_text->b;
        pa.c0 = from_text->c0;
        pa.cb = from_text->cb;
        pa.tails = std::min(m, from_text->c0 - 1);
        pass_bytes = 13ull * m;  // the text read, the sorted keys and positions written
      }
      s = launch(SA_K_ONESWEEP, (int)p + 32 * chain, pass_bytes,
                 [&] { return launch_onesweep(pa, st); });
      if (s != SA_OK) return s;
    }
    inject_pending = false;
    if (chain == 1) CK(cudaMemcpyAsync(pm1, &ctrl->passes, 8, cudaMemcpyDeviceToDevice, st));
    return SA_OK;
  }

  // The top `digits` 8-bit digits of total_bits-bit keys.
  static DigitSpec top_spec(uint32_t total_bits, uint32_t digits) {
    DigitSpec s{};
    s.P = digits;
    for (uint32_t p = 0; p < digits; ++p) {
      s.shift[p] = (uint8_t)(total_bits - (digits - p) * RADIX_BITS);
      s.bits[p] = RADIX_BITS;
    }
    return s;
  }

  static DigitSpec spec_for(uint32_t total_bits) {
    DigitSpec s{};
    s.P = (total_bits + RADIX_BITS - 1) / RADIX_BITS;
    for (uint32_t p = 0; p < s.P; ++p) {
      s.shift[p] = (uint8_t)(p * RADIX_BITS);
      s.bits[p] = (uint8_t)std::min<uint32_t>(RADIX_BITS, total_bits - p * RADIX_BITS);
    }
    return s;
  }

  // Rename of round 0 (all suffixes) or of the large groups of a later
  // round; writes the next active list at the device-side offsets `off_in`.
  sa_status rename(uint32_t m, uint32_t round0, uint32_t cb, uint32_t c0, uint32_t W,
                   const uint32_t *base_in, const uint32_t *old_in, uint32_t g_in, int out,
                   const uint32_t *off_in, bool wide = false) {
    RenameArgs ra{};
    ra.sec_buf[0] = wide ? ka : nullptr;
    ra.sec_buf[1] = wide ? kb : nullptr;
    ra.plan = plan;
    ra.m = m;
    ra.round0 = round0;
    ra.cb = cb;
    ra.c0 = c0;
    ra.seg_off = segoff;
    ra.S = S;
    ra.W = W;
    ra.base_in = base_in;
    ra.old_in = old_in;
    ra.g_in = g_in;
    ra.isa = isa;
    ra.upd = upd;
    ra.isa_len = N + S + 1;
    ra.N = (uint32_t)N;
    ra.sa = sa;
    ra.act_out = act[out];
    ra.gstart_out = gstart[out];
    ra.ghead_out = ghead[out];
    ra.gold_out = gold;
    ra.off_in = off_in;
    ra.cnt_out = &ctrl->rc.m_l;
    ra.status = st_ren;
    sa_status s = next_launch(ra.tile_ctr, ra.epoch);
    if (s != SA_OK) return s;
    ra.ctrl = ctrl;
    ra.spin_limit = spin;
    return launch(SA_K_RENAME, 0, 0, [&] { return launch_rename(ra, st); });
  }

  // Large groups and the refine tile map of the list just written.
  sa_status classify(int out, uint32_t apply_bound) {
    ClassifyArgs ca{};
    ca.gstart = gstart[out];
    ca.gname = gname[out];
    ca.ghead = ghead[out];
    ca.gold = gold;
    ca.naming = naming;
    ca.lg = lg;
    ca.loff = loff;
    ca.lbase = lbase;
    ca.lold = lold;
    ca.tfirst = tfirst;
    ca.nominal = nominal;
    ca.small = small;
    ca.cap = REFINE_SHAPE[shape].cap;
    ca.max_groups = L.max_groups;
    ca.max_tiles = L.max_tiles;
    ca.ctrl = ctrl;
    ++pend.classify;
    sa_status s = launch(SA_K_CLASSIFY, 0, PENDING,
                         [&] { return launch_classify(ca, sm_count(), st); });
    if (s != SA_OK) return s;
    // ISA entries of the rename's survivors whose name changed, bucketed by
    // position first when there can be many.
    if (apply_bound == 0) return SA_OK;
    const uint64_t *src = act[out];
    const uint32_t *lo = &ctrl->rc.m_s;
    const uint32_t *count = &ctrl->rc.m_l;
    uint32_t translated = 0;
    if (apply_bound >= bucket_min) {
      // The partition reads the group names while the entries are still in
      // group order and keeps only the changed ones, as (name, i').
      s = bucket(src, lo, &ctrl->rc.m_l, apply_bound, 2, gname[out]);
      if (s != SA_OK) return s;
      src = kb;
      lo = ctrl->zero;
      count = &ctrl->bucket_total;
      translated = 1;
    }
    ++pend.apply;
    return launch(SA_K_APPLY, 0, PENDING, [&] {
      return launch_apply_names(src, lo, count, apply_bound, gname[out], gold, isa, N + S + 1,
                                st, translated);
    });
  }

  // Position bucketing of `count` entries starting at `lo` into keys
  // buffer B (free whenever ISA writes are pending). `src_tag` tells the
  // byte settlement which count applies (0: queued updates, 2: survivors).
  sa_status bucket(const uint64_t *in, const uint32_t *lo, const uint32_t *count,
                   uint32_t max_count, int src_tag, const uint32_t *translate_names = nullptr) {
    BucketArgs ba{};
    if (translate_names) {
      ba.gname = translate_names;
      ba.gold = gold;
      ba.total_out = &ctrl->bucket_total;
    }
    ba.in = in;
    ba.lo = lo;
    ba.count = count;
    ba.max_count = max_count;
    const uint32_t bits = bits_for(N + S);
    ba.shift = bits > 8 ? bits - 8 : 0;
    ba.blocks = std::min<uint32_t>(BUCKET_BLOCKS_MAX, 4 * sm_count());
    ba.counts = bcount;
    ba.out = kb;
    if (src_tag != 4) ++(src_tag ? pend.bucket_surv : pend.bucket_upd);
    sa_status s = launch(SA_K_BUCKET, src_tag, PENDING,
                         [&] { return launch_bucket_count(ba, st); });
    if (s != SA_OK) return s;
    s = launch(SA_K_BUCKET, src_tag, 0, [&] { return launch_bucket_offsets(ba, st); });
    if (s != SA_OK) return s;
    return launch(SA_K_BUCKET, src_tag | 1, PENDING,
                  [&] { return launch_bucket_scatter(ba, st); });
  }

  // ISA[i'] = new for the queued updates (at most `bound` of them).
  sa_status scatter(uint32_t bound) {
    if (bound == 0) return SA_OK;
    const uint64_t *src = upd;
    if (bound >= bucket_min) {
      sa_status s = bucket(upd, nullptr, &ctrl->rc.upd, bound, 0);
      if (s != SA_OK) return s;
      src = kb;
    }
    ++pend.scatter;
    return launch(SA_K_SCATTER, 0, PENDING, [&] {
      return launch_scatter_updates(src, bound, isa, N + S + 1, ctrl, st);
    });
  }

  // Byte counts of the launches whose sizes are known only from this
  // round's control block: scatter and apply read 8 and write 4 bytes per
  // entry; bucketing reads 8 (histogram), then reads and writes 8.
  void settle(const HostCtrl &hc) {
    bytes += pend.scatter * 12ull * hc.upd + pend.apply * 12ull * hc.m_l +
             pend.bucket_upd * 24ull * hc.upd + pend.bucket_surv * 24ull * hc.m_l +
             pend.classify * classify_bytes(hc);
    pend = Pending{};
    for (Rec &r : recs) {
      if (r.bytes != PENDING) continue;
      if (r.cls == SA_K_SCATTER) r.bytes = 12ull * hc.upd;
      if (r.cls == SA_K_APPLY) r.bytes = 12ull * hc.m_l;
      if (r.cls == SA_K_CLASSIFY) r.bytes = classify_bytes(hc);
      if (r.cls == SA_K_BUCKET && (r.pass & 4))
        r.bytes = 0;
      else if (r.cls == SA_K_BUCKET)
        r.bytes = ((r.pass & 1) ? 16ull : 8ull) * ((r.pass & 2) ? hc.m_l : hc.upd);
    }
  }

  // Classification: 4 bytes (start) per group, 12 (head rank, parent's name,
  // name) per group that the rename wrote, 4 per refine tile, 20 (head rank
  // and the four lists) per large group.
  uint64_t classify_bytes(uint32_t items, uint32_t groups, uint32_t renamed, uint32_t large) const {
    return 4ull * groups + 12ull * renamed + 4ull * (items / nominal + 1) + 20ull * large;
  }
  uint64_t classify_bytes(const HostCtrl &hc) const {
    return classify_bytes(hc.m_next(), hc.g_next(), hc.g_l, hc.g_large());
  }

  // Rename (round 0 or large groups) reads 12 bytes per item; writes 4 (SA)
  // and, after round 0, 8 (queued ISA entry) per unique item, 8 per survivor
  // (and 4 of SA in round 0) and 12 per surviving group (start, head rank,
  // parent name).
  static uint64_t rename_bytes(uint32_t m, uint32_t surv, uint32_t groups, bool round0 = false) {
    const uint64_t u = m - surv;
    return 12ull * m + (round0 ? 4 : 12) * u + (round0 ? 12ull : 8ull) * surv + 12ull * groups;
  }

  // Refine: 8 bytes read and a - 1 4-byte gathers per item, 8 bytes of
  // group table per input group, 8 per survivor and per new group, 4 (SA)
  // per unique item, 8 per queued update.
  static uint64_t refine_bytes(uint32_t m, uint32_t G, uint32_t surv, uint32_t groups,
                               uint32_t upd_n, uint32_t a) {
    const uint64_t u = m - surv;
    return (8ull + 4ull * (a - 1)) * m + 8ull * G + 8ull * surv + 8ull * groups + 4 * u +
           8ull * upd_n;
  }

  // Device-driven rounds: only for doubling (a = 2), without the per-launch
  // profile or the per-round name trace; sa_options.device_rounds 1 asks
  // for them, 2 refuses them, 0 leaves the choice to the library.
  bool device_rounds_wanted() const {
    if (mult != 2 || prof || (opt.trace_isa && opt.trace_cap > 1)) return false;
    if (opt.device_rounds == 1) return true;
    if (opt.device_rounds == 2) return false;
    return false;
  }

  // Adds an if-node at the capture point of `outer` (handle h, created on
  // the graph being captured) and starts capturing its body on `inner`.
  static cudaError_t begin_if(cudaStream_t outer, cudaStream_t inner,
                              cudaGraphConditionalHandle h) {
    cudaStreamCaptureStatus cst = cudaStreamCaptureStatusNone;
    cudaGraph_t g = nullptr;
    const cudaGraphNode_t *deps = nullptr;
    size_t nd = 0;
    cudaError_t e = cudaStreamGetCaptureInfo(outer, &cst, nullptr, &g, &deps, nullptr, &nd);
    if (e != cudaSuccess) return e;
    if (cst != cudaStreamCaptureStatusActive) return cudaErrorStreamCaptureInvalidated;
    cudaGraphNodeParams p{};
    p.type = cudaGraphNodeTypeConditional;
    p.conditional.handle = h;
    p.conditional.type = cudaGraphCondTypeIf;
    p.conditional.size = 1;
    cudaGraphNode_t node;
    e = cudaGraphAddNode(&node, g, deps, nullptr, nd, &p);
    if (e != cudaSuccess) return e;
    e = cudaStreamUpdateCaptureDependencies(outer, &node, nullptr, 1,
                                            cudaStreamSetCaptureDependencies);
    if (e != cudaSuccess) return e;
    return cudaStreamBeginCaptureToGraph(inner, p.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                         cudaStreamCaptureModeRelaxed);
  }

  static cudaError_t end_capture(cudaStream_t s) {
    cudaGraph_t g = nullptr;
    return cudaStreamEndCapture(s, &g);
  }

  struct RoundHandles {
    cudaGraphConditionalHandle sort, rename, bucket_upd, bucket_surv;
  };

  // Captures one round (active list and group tables in buffer `cur`) on
  // stream cs, its optional steps in if-nodes captured on cs2. Grids are
  // sized for m1 items (the most any round after round 0 can have) and
  // capped, the kernels looping over their work.
  cudaError_t capture_round(cudaStream_t cs, cudaStream_t cs2, int cur, const RoundHandles &hd,
                            uint32_t m1, uint32_t W) {
    const int nxt = cur ^ 1;
    const uint32_t sms = (uint32_t)sm_count();
    const RoundState *rs = &ctrl->rs;
    RoundBeginArgs rb{};
    rb.ctrl = ctrl;
    rb.hist = hist;
    rb.W = W;
    rb.nominal = nominal;
    rb.bucket_min = bucket_min;
    rb.N = (uint32_t)N;
    rb.if_sort = hd.sort;
    rb.if_rename = hd.rename;
    rb.if_bucket_upd = hd.bucket_upd;
    rb.if_bucket_surv = hd.bucket_surv;
    cudaError_t e = launch_round_begin(rb, cs);
    if (e != cudaSuccess) return e;

    // Large groups: partner names and the global radix sort.
    if ((e = begin_if(cs, cs2, hd.sort)) != cudaSuccess) return e;
    GatherLargeArgs ga{};
    ga.act = act[cur];
    ga.gstart = gstart[cur];
    ga.lg = lg;
    ga.loff = loff;
    ga.mL = m1;
    ga.W = W;
    ga.mult = 2;
    ga.isa = isa;
    ga.isa_len = N + S + 1;
    ga.keys = ka;
    ga.vals = va;
    ga.rs = rs;
    ga.grid_cap = 8 * sms;
    if ((e = launch_gather_large(ga, cs2)) != cudaSuccess) return e;
    const DigitSpec none{};
    if ((e = launch_digit_histogram(ka, m1, none, hist, (int)sms, cs2, rs)) != cudaSuccess) return e;
    if ((e = launch_sort_plan(hist, dbase, none, m1, ka, kb, va, vb, plan, ctrl, cs2, rs)) !=
        cudaSuccess)
      return e;
    for (int p = 0; p < MAX_PASSES; ++p) {
      PassArgs pa{};
      pa.plan = plan;
      pa.p = p;
      pa.digit_base = dbase + p * RADIX;
      pa.m = m1;
      pa.status = st_sort;
      pa.epoch = (uint32_t)p;  // offset from the round's epoch base
      pa.tile_ctr = &ctrl->tile_ctr[p];
      pa.ctrl = ctrl;
      pa.spin_limit = spin;
      pa.items = sort_items;
      pa.rs = rs;
      pa.grid_cap = sms * (sort_items >= 16 ? 3u : (sort_items >= 12 ? 4u : 5u));
      if ((e = launch_onesweep(pa, cs2)) != cudaSuccess) return e;
    }
    if ((e = end_capture(cs2)) != cudaSuccess) return e;

    // Small groups: the tile-local refine.
    RefineArgs rf{};
    rf.act = act[cur];
    rf.gstart = gstart[cur];
    rf.gname = gname[cur];
    rf.ghead = ghead[cur];
    rf.naming = naming;
    rf.tfirst = tfirst;
    rf.m = m1;
    rf.shape = shape;
    rf.small = small;
    rf.tiles = (m1 + nominal - 1) / nominal;
    rf.W = W;
    rf.mult = 2;
    rf.isa = isa;
    rf.isa_len = N + S + 1;
    rf.N = (uint32_t)N;
    rf.sa = sa;
    rf.seg_off = segoff;
    rf.S = S;
    rf.act_out = act[nxt];
    rf.gstart_out = gstart[nxt];
    rf.gname_out = gname[nxt];
    rf.ghead_out = ghead[nxt];
    rf.upd = upd;
    rf.ctrl = ctrl;
    rf.rs = rs;
    {  // two waves of the resident blocks (k_refine's launch bounds)
      const RefineShape sh = REFINE_SHAPE[shape];
      rf.grid_cap = 2 * sms * ((sh.cap / sh.block > 8 ? 512u : 1024u) / sh.block);
    }
    if ((e = launch_refine(rf, cs)) != cudaSuccess) return e;

    // The large groups' rename (after every gather of the round).
    if ((e = begin_if(cs, cs2, hd.rename)) != cudaSuccess) return e;
    RenameArgs ra{};
    ra.plan = plan;
    ra.m = m1;
    ra.W = W;
    ra.seg_off = segoff;
    ra.S = S;
    ra.base_in = lbase;
    ra.old_in = lold;
    ra.g_in = L.max_large;
    ra.isa = isa;
    ra.upd = upd;
    ra.isa_len = N + S + 1;
    ra.N = (uint32_t)N;
    ra.sa = sa;
    ra.act_out = act[nxt];
    ra.gstart_out = gstart[nxt];
    ra.ghead_out = ghead[nxt];
    ra.gold_out = gold;
    ra.off_in = &ctrl->rc.m_s;
    ra.cnt_out = &ctrl->rc.m_l;
    ra.status = st_ren;
    ra.epoch = MAX_PASSES;  // offset from the round's epoch base
    ra.tile_ctr = &ctrl->tile_ctr[MAX_PASSES];
    ra.ctrl = ctrl;
    ra.spin_limit = spin;
    ra.rs = rs;
    ra.grid_cap = 4 * sms;
    if ((e = launch_rename(ra, cs2)) != cudaSuccess) return e;
    if ((e = end_capture(cs2)) != cudaSuccess) return e;

    // The round's queued ISA updates, bucketed by position when many.
    BucketArgs ba{};
    const uint32_t bits = bits_for(N + S);
    ba.shift = bits > 8 ? bits - 8 : 0;
    ba.blocks = std::min<uint32_t>(BUCKET_BLOCKS_MAX, 4 * sms);
    ba.counts = bcount;
    ba.out = kb;
    ba.in = upd;
    ba.count = &ctrl->rc.upd;
    ba.max_count = m1;
    if ((e = begin_if(cs, cs2, hd.bucket_upd)) != cudaSuccess) return e;
    if ((e = launch_bucket_count(ba, cs2)) != cudaSuccess) return e;
    if ((e = launch_bucket_offsets(ba, cs2)) != cudaSuccess) return e;
    if ((e = launch_bucket_scatter(ba, cs2)) != cudaSuccess) return e;
    if ((e = end_capture(cs2)) != cudaSuccess) return e;
    if ((e = launch_scatter_updates(upd, m1, isa, N + S + 1, ctrl, cs, kb, rs, 8 * sms)) !=
        cudaSuccess)
      return e;

    // The new groups, and the ISA entries of the rename's survivors.
    ClassifyArgs ca{};
    ca.gstart = gstart[nxt];
    ca.gname = gname[nxt];
    ca.ghead = ghead[nxt];
    ca.gold = gold;
    ca.naming = naming;
    ca.lg = lg;
    ca.loff = loff;
    ca.lbase = lbase;
    ca.lold = lold;
    ca.tfirst = tfirst;
    ca.nominal = nominal;
    ca.small = small;
    ca.cap = REFINE_SHAPE[shape].cap;
    ca.max_groups = L.max_groups;
    ca.max_tiles = L.max_tiles;
    ca.ctrl = ctrl;
    ca.rs = rs;
    if ((e = launch_classify(ca, (int)sms, cs)) != cudaSuccess) return e;
    ba.in = act[nxt];
    ba.lo = &ctrl->rc.m_s;
    ba.count = &ctrl->rc.m_l;
    ba.gname = gname[nxt];  // translating: (name, i') of the changed names only
    ba.gold = gold;
    ba.total_out = &ctrl->bucket_total;
    if ((e = begin_if(cs, cs2, hd.bucket_surv)) != cudaSuccess) return e;
    if ((e = launch_bucket_count(ba, cs2)) != cudaSuccess) return e;
    if ((e = launch_bucket_offsets(ba, cs2)) != cudaSuccess) return e;
    if ((e = launch_bucket_scatter(ba, cs2)) != cudaSuccess) return e;
    if ((e = end_capture(cs2)) != cudaSuccess) return e;
    return launch_apply_names(act[nxt], &ctrl->rc.m_s, &ctrl->rc.m_l, m1, gname[nxt], gold, isa,
                              N + S + 1, cs, 0, kb, ctrl->zero, &ctrl->bucket_total, rs, 8 * sms);
  }

  // Rounds >= 1 as one graph: while (suffixes active) { round; round }.
  // `round` returns the number of rounds including round 0.
  sa_status run_device_rounds(const HostCtrl &hc0, uint32_t W, uint32_t h1, int cur,
                              uint32_t &round) {
    const uint32_t m1 = hc0.m_next();
    RoundState rs0{};
    rs0.live = 1;
    rs0.round = 0;
    rs0.h_next = h1;
    rs0.epoch = epoch + ROUND_EPOCHS;
    CK(cudaMemcpyAsync(&ctrl->rs, &rs0, sizeof(rs0), cudaMemcpyHostToDevice, st));
    // Kernels that round 0 did not launch (the refine, and the rename where the
    // buckets took its place) set their attributes when first captured, a host
    // call that capture allows.
    cudaStream_t cs = nullptr, cs2 = nullptr;
    cudaGraph_t g = nullptr;
    cudaGraphExec_t exec = nullptr;
    auto cleanup = [&]() {
      if (exec) cudaGraphExecDestroy(exec);
      if (g) cudaGraphDestroy(g);
      if (cs2) cudaStreamDestroy(cs2);
      if (cs) cudaStreamDestroy(cs);
    };
    cudaError_t e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&cs2, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaGraphCreate(&g, 0);
    cudaGraphConditionalHandle loop{};
    cudaGraph_t body = nullptr;
    if (e == cudaSuccess) e = cudaGraphConditionalHandleCreate(&loop, g, 1, cudaGraphCondAssignDefault);
    if (e == cudaSuccess) {
      cudaGraphNodeParams p{};
      p.type = cudaGraphNodeTypeConditional;
      p.conditional.handle = loop;
      p.conditional.type = cudaGraphCondTypeWhile;
      p.conditional.size = 1;
      cudaGraphNode_t node;
      e = cudaGraphAddNode(&node, g, nullptr, nullptr, 0, &p);
      if (e == cudaSuccess) body = p.conditional.phGraph_out[0];
    }
    RoundHandles hd[2];
    for (int k = 0; k < 2 && e == cudaSuccess; ++k) {
      cudaGraphConditionalHandle *hs[4] = {&hd[k].sort, &hd[k].rename, &hd[k].bucket_upd,
                                           &hd[k].bucket_surv};
      for (cudaGraphConditionalHandle *hp : hs)
        if (e == cudaSuccess) e = cudaGraphConditionalHandleCreate(hp, body, 0, 0);
    }
    if (e == cudaSuccess)
      e = cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed);
    if (e == cudaSuccess) {
      cudaError_t ce = capture_round(cs, cs2, cur, hd[0], m1, W);
      if (ce == cudaSuccess) ce = capture_round(cs, cs2, cur ^ 1, hd[1], m1, W);
      if (ce == cudaSuccess) ce = launch_round_end(ctrl, loop, cs);
      cudaStreamCaptureStatus c2 = cudaStreamCaptureStatusNone;
      if (cudaStreamIsCapturing(cs2, &c2) == cudaSuccess && c2 != cudaStreamCaptureStatusNone)
        end_capture(cs2);
      e = end_capture(cs);
      if (ce != cudaSuccess) e = ce;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&exec, g, 0);
    if (e == cudaSuccess) e = cudaGraphLaunch(exec, st);
    if (e != cudaSuccess) {
      cudaGetLastError();
      cleanup();
      return SA_ERR_CUDA;
    }
    launches += 1;  // the graph (its kernels are counted below)
    // One readback of the whole control block (a few KB): error word, the
    // last round's counters, the round state and the per-round records.
    std::vector<uint8_t> raw(sizeof(Ctrl));
    static_assert(sizeof(Ctrl) <= STAGE_BYTES && sizeof(Ctrl) % 4 == 0, "Ctrl fits the stage");
    e = fetch(raw.data(), ctrl, sizeof(Ctrl));
    cleanup();
    if (e != cudaSuccess) return SA_ERR_CUDA;
    const Ctrl &hctrl = *reinterpret_cast<const Ctrl *>(raw.data());
    HostCtrl hc{};
    memcpy(&hc, raw.data(), sizeof(HostCtrl));
    if (hc.error == ERR_TIMEOUT) return SA_ERR_TIMEOUT;
    if (hc.error != ERR_NONE) return SA_ERR_INTERNAL;
    // Statistics and byte counts from the device records.
    const uint32_t last = hctrl.rs.round;
    if (last >= (uint32_t)DEV_MAX_ROUNDS) return SA_ERR_INTERNAL;
    std::vector<RoundRecord> rec(hctrl.rec, hctrl.rec + last + 1);
    if (last >= 1) {  // the last round's outputs are still in the counters
      RoundRecord &r = rec[last];
      r.m_s = hc.m_s;
      r.g_s = hc.g_s;
      r.m_l = hc.m_l;
      r.g_l = hc.g_l;
      r.upd = hc.upd;
      r.passes = hc.passes;
    }
    for (uint32_t r = 1; r <= last; ++r) {
      const RoundRecord &x = rec[r];
      const uint32_t kbits = x.mL ? W + (x.GL > 1 ? bits_for(x.GL - 1) : 0) : 0;
      const uint64_t rbl = x.mL ? rename_bytes(x.mL, x.m_l, x.g_l) : 0;
      const uint64_t rfb = refine_bytes(x.m - x.mL, x.G - x.GL, x.m_s, x.g_s, x.upd, 2);
      const uint32_t next_large = r < last ? rec[r + 1].GL : 0;
      bytes += (x.mL ? (uint64_t)x.passes * 24 * x.mL + 32ull * x.mL : 0) + rbl + rfb +
               classify_bytes(x.m_s + x.m_l, x.g_s + x.g_l, x.g_l, next_large) +
               12ull * x.upd + (x.m >= bucket_min ? 24ull * x.upd : 0) +
               (x.mL ? 12ull * x.m_l + (x.mL >= bucket_min ? 24ull * x.m_l : 0) : 0);
      launches += 5 + (x.mL ? 12 + MAX_PASSES - 1 : 0) + (x.m >= bucket_min ? 3 : 0) +
                  (x.mL && x.mL >= bucket_min ? 3 : 0);
      if (stats && r < SA_MAX_ROUNDS) {
        stats->active[r] = x.m;
        stats->unique[r] = x.m - (x.m_s + x.m_l);
        stats->passes[r] = x.mL ? x.passes : 0;
        stats->key_bits[r] = kbits;
        stats->groups[r] = x.g_s + x.g_l;
      }
    }
    launches += (last + 1) / 2;  // k_round_end, once per body
    round = last + 1;
    return SA_OK;
  }

  // Whether the groups are put in position order after round 0. It pays
  // where the ISA (4 N bytes) is not held by the L2 anyway and enough
  // suffixes stay active to repay the eight launches and the pass over the
  // marks. Measured, position order against rank order: repeated Zipf
  // 2^22 1.82 / 1.74 ms, 2^24 6.53 / 6.69, 2^26 25.6 / 30.8, 2^28 81.7 /
  // 109.3; Markov DNA 2^24 2.29 / 2.21, 2^26 10.40 / 10.49, 2^28 26.3 / 29.9;
  // words 2^26 11.50 / 11.48; with 1.5 % and 3 % active, DNA 2^26 5.38 /
  // 5.30, Zipf bytes 2^26 7.29 / 7.20; below 2^22 about 0.07 ms more.
  bool position_order_wanted(uint32_t m) const {
    if (opt.group_order) return opt.group_order == 1;
    return N >= (1ull << 24) && m >= N / 16;
  }

  // Half a tile as the refine's window and largest group, for the rest of
  // the build, where many of the suffixes active after round 0 are in groups
  // that are above the shape's own limit but fit a tile (REFINE_HALF_SHARE):
  // they are refined in tiles then, at once or after they have split once.
  // Beside groups that no tile can hold, whose rounds sort globally anyway, it
  // must repay the second classification and its readback, 25 us, at 29 ps a
  // suffix and round in a few rounds: prose of 8 M characters with 0.43 M such
  // suffixes took 1.73 ms instead of 1.70.
  // With again, the list is classified again and hc.large re-read.
  sa_status refine_limits(int cur, HostCtrl &hc, bool again) {
    const uint32_t half = REFINE_SHAPE[shape].cap / 2;
    if (hc.mid <= hc.m_next() / REFINE_HALF_SHARE || small == half) return SA_OK;
    if (hc.mid < hc.m_large() && hc.mid < REFINE_HALF_MIN) return SA_OK;
    small = nominal = half;
    if (!again) return SA_OK;
    CK(cudaMemsetAsync(&ctrl->rc.large, 0, sizeof(ctrl->rc.large), st));
    sa_status s = classify(cur, 0);
    if (s != SA_OK) return s;
    HostCtrl h2{};
    s = read_ctrl(h2);
    if (s != SA_OK) return s;
    hc.large = h2.large;
    settle(h2);
    return flush(0, 0);
  }

  // The groups of the active list `cur` (hc: its counts) copied to the
  // other buffer set in order of their smallest member position, then
  // classified again (large groups, refine tile map); hc is re-read.
  sa_status reorder_groups(int cur, HostCtrl &hc) {
    const uint32_t G = hc.g_next(), m = hc.m_next();
    const int nxt = cur ^ 1;
    // Buffers: the records go to the update queue (free now, 8 N bytes >=
    // 16 G), the marks to a key buffer, the scan sums to the other.
    RegroupArgs ra{};
    ra.G = G;
    ra.m = m;
    ra.positions = (uint32_t)std::min<uint64_t>(N + S, 0xFFFFFFFFull);
    ra.act_in = act[cur];
    ra.gstart_in = gstart[cur];
    ra.gname_in = gname[cur];
    ra.ghead_in = ghead[cur];
    ra.lines = reinterpret_cast<uint32_t *>(kb);
    ra.sums = reinterpret_cast<uint32_t *>(ka);
    ra.info = reinterpret_cast<uint4 *>(upd);
    ra.act_out = act[nxt];
    ra.gstart_out = gstart[nxt];
    ra.gname_out = gname[nxt];
    ra.ghead_out = ghead[nxt];
    ra.ctrl = ctrl;
    if (2ull * G > N) return SA_ERR_INTERNAL;
    const uint64_t rank_bytes = 68ull * G + 3 * 32ull * rank_lines(ra.positions);
    sa_status s = launch(SA_K_REORDER, 0, rank_bytes,
                         [&] { return launch_group_rank(ra, sm_count(), st); });
    if (s != SA_OK) return s;
    launches += 4;
    const uint64_t move_bytes = 48ull * G + 16ull * m;
    s = launch(SA_K_REORDER, 1, move_bytes, [&] { return launch_regroup(ra, st); });
    if (s != SA_OK) return s;
    launches += 3;
    bytes += rank_bytes + move_bytes;
    s = classify(nxt, 0);
    if (s != SA_OK) return s;
    HostCtrl h2{};
    s = read_ctrl(h2);
    if (s != SA_OK) return s;
    settle(h2);
    s = flush(0, 0);
    if (s != SA_OK) return s;
    h2.passes = hc.passes;
    h2.pass_mask = hc.pass_mask;
    h2.upd = hc.upd;
    hc = h2;
    return SA_OK;
  }

  // The ISA starts all-ones, so that every end slot reads as the sentinel;
  // once per build, before its first entry (a text that round 0 resolves
  // writes none).
  sa_status clear_isa() {
    if (!isa_cleared) CK(cudaMemsetAsync(isa, 0xFF, (N + S + 1) * 4, st));
    isa_cleared = true;
    return SA_OK;
  }

  // Round 0 after the radix sort of its keys' top `split` digits: the
  // buckets of equal top bits tile by tile, those too large for a tile by
  // the global sort and rename, then the classification. hc: the counts.
  sa_status finish_buckets(int out, uint32_t split, uint32_t bits0, uint32_t cb, uint32_t c0,
                           HostCtrl &hc) {
    const uint32_t m = (uint32_t)N, R = bits0 - split * RADIX_BITS;
    LocalArgs la{};
    la.plan = plan;
    la.m = m;
    la.R = R;
    la.cb = cb;
    la.c0 = c0;
    la.seg_off = segoff;
    la.S = S;
    la.N = m;
    la.naming = naming;
    la.isa_len = N + S + 1;
    la.sa = sa;
    la.act_out = act[out];
    la.gstart_out = gstart[out];
    la.gname_out = gname[out];
    la.ghead_out = ghead[out];
    la.upd = upd;
    la.lg = lg;
    la.loff = loff;
    la.lbase = lbase;
    la.lold = lold;
    la.max_large = L.max_large;
    la.max_groups = L.max_groups;
    la.ctrl = ctrl;
    // The last tile's report saves a copy kernel (about 5 us); a tile's share
    // of it, a fence and an atomic at its end, costs 6 % of long ones.
    if (stage_readbacks && N <= LOCAL_REPORT_MAX) {
      la.host = stage_words() + RADIX;
      la.host_flag = report_flag(1);
    }
    sa_status s = launch(SA_K_RENAME, 0, 0, [&] { return launch_local(la, st); });
    if (s != SA_OK) return s;
    if (la.host) {
      CK(wait_report(la.host_flag));
      memcpy(&hc, la.host, sizeof(hc));
      s = ctrl_status(hc);
    } else {
      s = read_ctrl(hc);
    }
    if (s != SA_OK) return s;
    const uint32_t mL = hc.m_large(), GL = hc.g_large(), passes = hc.passes;
    if (hc.m_s > m || mL > m) return SA_ERR_INTERNAL;
    // 12 bytes read and 4 written per item; 16 per survivor, 12 per group.
    const uint64_t lb = 16ull * m + 16ull * hc.m_s + 12ull * hc.g_s;
    bytes += (uint64_t)passes * 24 * m + lb;
    s = flush(hc.pass_mask, lb);
    if (s != SA_OK) return s;
    if (hc.m_next() == 0 && mL == 0) return SA_OK;
    if (mL > 0) {
      // Every pass was kept, so the sorted keys are in A after an even
      // number of them: the large buckets' items go to the other buffer.
      const bool in_a = split % 2 == 0;
      if (!in_a) std::swap(ka, kb), std::swap(va, vb);
      GatherBigArgs ga{};
      ga.kin = ka;
      ga.vin = va;
      ga.lg = lg;
      ga.loff = loff;
      ga.m = m;
      ga.mL = mL;
      ga.GL = GL;
      ga.R = R;
      ga.keys = kb;
      ga.vals = vb;
      ga.sa = sa;
      ga.ctrl = ctrl;
      s = launch(SA_K_GATHER, 0, 28ull * mL, [&] { return launch_gather_big(ga, st); });
      std::swap(ka, kb), std::swap(va, vb);  // sort from the buffer just written
      if (s == SA_OK) s = sort(mL, spec_for(R + (GL > 1 ? bits_for(GL - 1) : 0)));
      if (in_a) std::swap(ka, kb), std::swap(va, vb);
      if (s != SA_OK) return s;
      s = rename(mL, 2, cb, c0, R, lbase, lold, GL, out, &ctrl->rc.m_s);
      if (s != SA_OK) return s;
      bytes += 28ull * mL;
    }
    s = clear_isa();
    if (s != SA_OK) return s;
    CK(cudaMemsetAsync(&ctrl->rc.large, 0, sizeof(ctrl->rc.large), st));
    s = classify(out, mL);
    if (s != SA_OK) return s;
    s = read_ctrl(hc);
    if (s != SA_OK) return s;
    const uint64_t rb = mL ? rename_bytes(mL, hc.m_l, hc.g_l, true) : 0;
    settle(hc);
    s = flush(hc.pass_mask, rb);
    if (s != SA_OK) return s;
    bytes += (mL ? (uint64_t)hc.passes * 24 * mL : 0) + rb;
    hc.passes = passes + (mL ? hc.passes : 0);
    return SA_OK;
  }

  // ISA entries of the final ranks in the SA: all, or those whose position
  // is in `missing`, into out[0, len). The list goes through the active
  // buffer `buf`.
  sa_status collect(int buf, const uint32_t *missing, uint32_t *out, uint64_t len) {
    CollectArgs ca{};
    ca.sa = sa;
    ca.N = (uint32_t)N;
    ca.seg_off = segoff;
    ca.S = S;
    ca.shift = need_shift(N + S);
    ca.words = L.need_words;
    ca.missing = missing;
    ca.out = act[buf];
    ca.ctrl = ctrl;
    CK(cudaMemsetAsync(&ctrl->need_entries, 0, 4, st));
    sa_status s = launch(SA_K_SCATTER, 2, 4ull * N,
                         [&] { return launch_need_collect(ca, sm_count(), st); });
    if (s != SA_OK) return s;
    bytes += 4ull * N;
    const uint64_t *src = act[buf];
    if (N >= COLLECT_MIN_N && N >= bucket_min) {
      s = bucket(src, nullptr, &ctrl->need_entries, (uint32_t)N, 4);
      if (s != SA_OK) return s;
      src = kb;
    }
    uint32_t *ctr = nullptr, ep = 0;
    s = next_launch(ctr, ep);
    if (s != SA_OK) return s;
    return launch(SA_K_SCATTER, 3, 0, [&] {
      return launch_write_entries(src, &ctrl->need_entries, (uint32_t)N, out, len, ctr,
                                  8 * sm_count(), st);
    });
  }

  // The entries that rounds with partner offsets h, h * mult, .. read (all of
  // them up to NEED_OFFSET_MAX for the first plan, else this round's), of the
  // active list in buffer `from`.
  sa_status fill_needed(int from, uint32_t m, uint64_t h, bool first) {
    NeedArgs na{};
    na.act = act[from];
    na.m = m;
    na.shift = need_shift(N + S);
    for (uint64_t x = h; x <= N && na.offsets + mult <= NEED_OFFSETS; x *= mult) {
      for (uint32_t j = 1; j < mult; ++j)
        if (j * x <= N) na.h[na.offsets++] = (uint32_t)(j * x);
      if (!first || x * mult > NEED_OFFSET_MAX) break;
    }
    na.words = L.need_words;
    na.active = need;
    na.covered = need + L.need_words;
    na.missing = need + 2 * (size_t)L.need_words;
    na.ctrl = ctrl;
    CK(cudaMemsetAsync(&ctrl->need_any, 0, 4, st));
    sa_status s = launch(SA_K_SCATTER, 4, 8ull * m,
                         [&] { return launch_need_plan(na, sm_count(), st); });
    if (s != SA_OK) return s;
    ++launches;
    bytes += 8ull * m;
    return collect(from ^ 1, na.missing, isa, N + S + 1);
  }

  // Digits of the top that the radix sort of round 0 takes before the
  // buckets are sorted tile by tile, or 0 for all digits: the cheapest by
  // the model of the prefixes, in units of one pass over all items. The
  // rename that the tile pass replaces costs RENAME_COST; items
  // in buckets too large for a tile are gathered, sorted by the remaining
  // digits and the bucket ordinal, and renamed.
  // The counts behind the model do not see repeats (copies, words): what the
  // sample finds counts where it is more. Builds by the model alone and with
  // the sample: a Zipf block 4096 and 16384 times in 2^28 characters 202.8, 197.3
  // and 190.4, 186.7 ms, prose of 2^26 13.1 and 11.3, DNA beside Zipf bytes of
  // 2^27 in all 19.6 and 17.5. Batches with half of every one taken to be of two
  // bits, with the sample, unsplit: 48 texts of 10-256 KB, half DNA, half Zipf
  // bytes 0.741, 0.743, 0.733 ms, 64 of Zipf bytes 0.525, 0.485, 0.59, 256 of
  // protein to 1 MB 2.59, 2.17, 3.57.
  // Beyond the sample's characters its last count stands where prefixes that
  // long are repeats (their information exceeds the length's). In a batch only
  // whole characters of it count: a text of few letters has close codes, whose
  // top bits divide nothing.
  uint32_t choose_split(const PrefixModel &model, const KeySample &sample, uint32_t b,
                        uint32_t segbits, uint32_t bits0) const {
    const uint32_t P = (bits0 + RADIX_BITS - 1) / RADIX_BITS;
    double best = P + RENAME_COST;
    uint32_t split = 0;
    // Characters by the logarithm of their text's length.
    uint64_t chars_of[33] = {}, texts_of[33] = {};
    for (uint32_t k = 0; k < S; ++k) {
      const uint32_t len = off[k + 1] - off[k];
      const int l = len ? 31 - __builtin_clz(len) : 32;
      chars_of[l] += len;
      ++texts_of[l];
    }
    double mass[33] = {}, log_len[33] = {};
    for (int l = 0; l < 32; ++l) {
      if (!texts_of[l]) continue;
      mass[l] = (double)chars_of[l] / (double)N;
      log_len[l] = std::log2((double)chars_of[l] / (double)texts_of[l]);
    }
    const uint32_t sampled = b > SAMPLE_MIN_BITS ? sample_blocks(N, S) : 0;
    const bool repeats = SAMPLE_CHARS * model.mean1 >= std::log2((double)N);
    for (uint32_t p = 1; p * RADIX_BITS < bits0; ++p) {
      const uint32_t T = p * RADIX_BITS;
      const double chars = T > segbits ? (double)(T - segbits) / b : 0.0;
      double big = 0.0, cost = p, certain = 1.0;
      for (int l = 0; l < 33; ++l)
        if (mass[l] > 0.0) {
          big += mass[l] * model.large_share(chars, log_len[l], LOCAL_LARGE_LOG2);
          cost += mass[l] * model.local_cost(chars, log_len[l], 8.0 / b);
        }
      if (cost >= best) continue;
      if (sampled && chars >= 1.0 && (chars <= SAMPLE_CHARS || repeats)) {
        const double c = S > 1 ? std::floor(chars) : chars;
        const double found =
            sampled_large_share(sample, std::min(c, (double)SAMPLE_CHARS), sampled, N);
        if (found > big) {
          big = found;
          certain = std::min(1.0, big * N / SAMPLE_CERTAIN);
        }
      }
      const uint32_t R = bits0 - T;
      if (big > 0.0) {  // its share of a pass, each with the fixed part of one
        const double rest = (R + bits_for((uint64_t)(big * N / 4096.0)) + 7) / 8;
        const double share =
            (big * N * PASS_ITEM_US + PASS_FIXED_US * certain) / (N * PASS_ITEM_US + PASS_FIXED_US);
        cost += share * (rest + 3.0 + RENAME_COST);
      }
      if (cost < best) {
        best = cost;
        split = p;
      }
    }
    return split;
  }

  void record(uint32_t r, uint32_t m, const HostCtrl &hc, uint32_t kbits) {
    if (!stats || r >= SA_MAX_ROUNDS) return;
    stats->active[r] = m;
    stats->unique[r] = m - hc.m_next();
    stats->passes[r] = kbits ? hc.passes : 0;
    stats->key_bits[r] = kbits;
    stats->groups[r] = hc.g_next();
  }

  sa_status run() {
    char label[96];
    snprintf(label, sizeof(label), "gbsa:build n=%llu texts=%u", (unsigned long long)N, S);
    NvtxRange build_range(label);
    const uint32_t N32 = (uint32_t)N;
    carve();
    prof = opt.profile != 0 && stats != nullptr;
    naming = opt.paper_names ? NAMES_HEAD : NAMES_RETAIN;
    mult = opt.multiplier ? opt.multiplier : 2;  // checked by the entry points
    CK(cudaMemsetAsync(ws, 0, L.zeroed, st));
    if (S > 1)
      CK(cudaMemcpyAsync(segoff, off.data(), ((size_t)S + 1) * 4, cudaMemcpyHostToDevice, st));

    // ---- A0: alphabet ----
    if (stage_readbacks && stage.get() != cudaSuccess) {
      cudaGetLastError();  // no pinned block to be had: the copy engine instead
      stage_readbacks = false;
    }
    AlphabetArgs aa{};
    aa.text = text;
    aa.n = N;
    aa.hist = bytehist;
    aa.done = &ctrl->done[0];
    aa.code = code;
    aa.seg_off = S == 1 ? segoff : nullptr;
    aa.sample_blocks = sample_blocks(N, S);
    aa.offsets = S > 1 ? segoff : nullptr;
    aa.S = S;
    if (stage_readbacks) {
      aa.host = stage_words();
      aa.host_flag = report_flag(0);
    }
    sa_status s =
        launch(SA_K_BYTE_HIST, 0, N, [&] { return launch_byte_histogram(aa, sm_count(), st); });
    if (s != SA_OK) return s;
    uint32_t hh[RADIX + sizeof(KeySample) / 4];
    if (aa.host) {
      CK(wait_report(aa.host_flag));
      memcpy(hh, aa.host, sizeof(hh));
    } else {
      CK(fetch(hh, bytehist, sizeof(hh)));
    }
    KeySample sample;
    memcpy(&sample, hh + RADIX, sizeof(sample));
    s = flush(0, 0);
    if (s != SA_OK) return s;
    uint32_t sigma = 0;
    for (int c = 0; c < RADIX; ++c) sigma += hh[c] ? 1u : 0u;
    const uint32_t b = std::max<uint32_t>(1, bits_for(sigma - 1));
    const uint32_t segbits = S > 1 ? bits_for(S - 1) : 0;
    // Parameters: the caller's options, else the tuning table's entry for
    // this class (batch or not, bits per character, size), else defaults:
    // 16 keys per radix thread, the 128 x 1024 refine (8 blocks per SM),
    // keys as wide as fit, bucketing from 2^22 pending ISA writes.
    sa_tuned tuned{};
    tuned_params(S > 1, b, N, &tuned);
    bool from_table = false;
    auto pick = [&](uint32_t given, uint32_t table, uint32_t dflt, bool ok_given, bool ok_table) {
      if (given && ok_given) return given;
      if (table && ok_table) {
        from_table = true;
        return table;
      }
      return dflt;
    };
    auto items_ok = [](uint32_t v) { return v == 8 || v == 12 || v == 16; };
    auto shape_ok = [](uint32_t v) { return v >= 1 && v <= (uint32_t)REFINE_SHAPES; };
    sort_items = pick(opt.sort_items, tuned.sort_items, SORT_ITEMS_DEFAULT,
                      items_ok(opt.sort_items), items_ok(tuned.sort_items));
    shape = pick(opt.refine_shape, tuned.refine_shape, 1, shape_ok(opt.refine_shape),
                 shape_ok(tuned.refine_shape)) - 1;
    small = REFINE_SHAPE[shape].small;
    nominal = REFINE_SHAPE[shape].cap - small;
    bucket_min = pick(opt.bucket_min, tuned.bucket_min, BUCKET_MIN, true, true);
    const uint32_t h0 = pick(opt.h0_chars, tuned.h0_chars, 0, true, true);
    uint32_t c0 = (64 - segbits) / b;
    if (h0) c0 = std::min(c0, h0);
    const uint32_t cb = c0 * b;
    bytes += N;
    if (stats) {
      stats->sigma = sigma;
      stats->bits_per_char = b;
      stats->chars_per_key = c0;
      stats->sort_items = sort_items;
      stats->refine_shape = shape + 1;
      stats->bucket_min = bucket_min;
      stats->tuned = from_table ? 1u : 0u;
    }

    // ---- round 0: initial names ----
    snprintf(label, sizeof(label), "gbsa:round 0 m=%u", N32);
    NvtxRange round0_range(label);
    PackArgs pk{};
    pk.text = text;
    pk.N = N32;
    pk.seg_off = segoff;
    pk.S = S;
    pk.code = code;
    pk.b = b;
    pk.c0 = c0;
    pk.cb = cb;
    pk.keys = ka;
    pk.vals = va;
    const uint32_t bits0 = cb + segbits;
    pk.spec = spec_for(bits0);
    pk.hist = hist;
    pk.top_only = (S == 1 && 8 % b == 0 && cb % 8 == 0 && c0 <= 64) ? 1u : 0u;
    // One text with whole-character digits: the first radix pass forms the
    // keys from the text and the pack only counts (no packed copy written
    // and read back).
    const bool keys_in_pass = pk.top_only && opt.initial_keys != 2;
    if (keys_in_pass) {
      pk.keys = nullptr;
      pk.vals = nullptr;
    }
    // How many digits the radix sort takes before the buckets of equal top
    // bits are sorted tile by tile (0: all of them, then the rename).
    PrefixModel model = PrefixModel::characters(hh);
    uint32_t split = 0;
    if (!pk.top_only) {
      split = choose_split(model, sample, b, segbits, bits0);
      if (split) pk.spec = top_spec(bits0, split);
    }
    const uint64_t pack_bytes = keys_in_pass ? (uint64_t)N : 13ull * N;
    s = launch(SA_K_PACK, 0, pack_bytes, [&] { return launch_pack(pk, st); });
    if (s != SA_OK) return s;
    bytes += pack_bytes;
    if (pk.top_only) {
      if (N >= GRAM_MODEL_MIN && b < 8) {
        uint32_t grams[RADIX];
        CK(fetch(grams, hist + (MAX_PASSES - 1) * RADIX, sizeof(grams)));
        model = PrefixModel::grams(grams, b);
      }
      split = choose_split(model, sample, b, segbits, bits0);
      if (split) pk.spec = top_spec(bits0, split);
    }
    inject_pending = opt.inject_stall != 0;
    int cur = 0;  // the active list, group starts and names of this round
    const bool want_trace = opt.trace_isa && opt.trace_cap > 0 && S == 1;
    HostCtrl hc{};
    uint32_t m = N32;
    s = sort(N32, pk.spec, true, 0, keys_in_pass ? &pk : nullptr, split ? 0xFFu : 0u,
             pk.top_only ? &pk : nullptr);
    if (s != SA_OK) return s;
    if (!split) {
      s = clear_isa();
      if (s != SA_OK) return s;
      s = rename(N32, 1, cb, c0, 0, nullptr, nullptr, 0, cur, ctrl->zero);
      if (s != SA_OK) return s;
      s = classify(cur, N32);
      if (s != SA_OK) return s;
      s = read_ctrl(hc);
      if (s != SA_OK) return s;
      const uint64_t rb0 = rename_bytes(m, hc.m_next(), hc.g_next(), true);
      settle(hc);
      s = flush(hc.pass_mask, rb0);
      if (s != SA_OK) return s;
      bytes += (uint64_t)hc.passes * 24 * m + rb0;
    } else {
      s = finish_buckets(cur, split, bits0, cb, c0, hc);
      if (s != SA_OK) return s;
    }
    record(0, m, hc, bits0);
    bytes -= keys_in_pass ? 11ull * m : 0ull;
    // The unique suffixes' ISA entries are needed only by a later round, the
    // ISA output or the trace; a text resolved in round 0 skips them.
    // Without a later round or the trace the ISA output needs no array of its
    // own to be copied from (one text: gapped positions are its own).
    const bool direct = isa_out && hc.m_next() == 0 && !want_trace;
    uint32_t *const fill = direct ? isa_out : isa;
    const uint64_t fill_len = direct ? N : N + S + 1;
    if (hc.m_next() > 0 || isa_out || want_trace) {
      if (!direct) s = clear_isa();
      if (s != SA_OK) return s;
      need_filtered = !isa_out && !opt.trace_isa && !device_rounds_wanted() && N >= NEED_MIN_N &&
                      hc.m_next() <= N / 4;
      if (need_filtered) {
        CK(cudaMemsetAsync(need, 0, 3 * (size_t)L.need_words * 4, st));
        s = fill_needed(cur, hc.m_next(), c0, true);
      } else if (N < COLLECT_MIN_N || bucket_min == 0xFFFFFFFFu) {
        bytes += 8ull * N;
        s = launch(SA_K_SCATTER, 1, 8ull * N, [&] {
          return launch_isa_fill(sa, N32, segoff, S, fill, fill_len, st);
        });
      } else {
        s = collect(cur ^ 1, nullptr, fill, fill_len);
      }
      if (s != SA_OK) return s;
      // Its records settle with round 0's counts, before round 1 reads new ones.
      s = scatter(hc.upd);
      if (s != SA_OK) return s;
      settle(hc);
    }
    if (want_trace) CK(cudaMemcpyAsync(opt.trace_isa, isa, N * 4, cudaMemcpyDeviceToDevice, st));
    const bool reorder = hc.m_next() > 0 && position_order_wanted(hc.m_next());
    s = refine_limits(cur, hc, !reorder);
    if (s != SA_OK) return s;
    if (reorder) {
      // The later rounds read partner names through the ISA: groups in
      // position order make those reads of neighbouring groups neighbours.
      s = reorder_groups(cur, hc);
      if (s != SA_OK) return s;
      cur ^= 1;
    }
    round0_range.end();

    // ---- rounds r >= 1: one doubling step each ----
    const uint32_t W = bits_for(N);  // r2 in [0, N]
    uint64_t h = c0;
    uint32_t round = 1;
    if (hc.m_next() > 0 && device_rounds_wanted()) {
      // The whole loop as one graph launch; rounds, statistics and byte
      // counts come back from the device records.
      s = run_device_rounds(hc, W, (uint32_t)c0, cur, round);
      if (s != SA_OK) return s;
      hc = HostCtrl{};  // no suffix left active
    }
    while (hc.m_next() > 0) {
      if (round >= SA_MAX_ROUNDS || h > N) return SA_ERR_INTERNAL;
      m = hc.m_next();
      snprintf(label, sizeof(label), "gbsa:round %u m=%u", round, m);
      NvtxRange round_range(label);
      const uint32_t G = hc.g_next();
      const uint32_t mL = hc.m_large(), GL = hc.g_large();
      const int nxt = cur ^ 1;
      CK(cudaMemsetAsync(&ctrl->rc, 0, sizeof(RoundCounts), st));
      if (need_filtered && h > NEED_OFFSET_MAX) {  // beyond the first plan
        s = fill_needed(cur, m, h, false);
        if (s != SA_OK) return s;
      }
      // Large groups: keys for the global radix sort (gathered before any
      // name of this round changes).
      uint32_t kbits = 0;
      if (mL > 0) {
        GatherLargeArgs ga{};
        ga.act = act[cur];
        ga.gstart = gstart[cur];
        ga.lg = lg;
        ga.loff = loff;
        ga.mL = mL;
        ga.GL = GL;
        ga.h = (uint32_t)h;
        ga.W = W;
        ga.mult = mult;
        ga.isa = isa;
        ga.isa_len = N + S + 1;
        ga.keys = ka;
        ga.vals = va;
        // a > 2: the queued-update list and the next active list are free
        // until the refine below, and hold the per-item keys until then.
        ga.key1_stash = upd;
        ga.sec_stash = act[nxt];
        const uint64_t gb = mult == 2 ? 24ull * mL : (32ull + 4ull * (mult - 1) + 16ull) * mL;
        s = launch(SA_K_GATHER, 0, gb, [&] { return launch_gather_large(ga, st); });
        if (s != SA_OK) return s;
        bytes += gb;
        kbits = W + (GL > 1 ? bits_for(GL - 1) : 0);
        if (mult > 2) {
          // LSD over the tuple: later partners first, then (group, r2).
          s = sort(mL, spec_for(mult == 4 ? 2 * W : W), false, 1);
          if (s != SA_OK) return s;
          WideArgs wa{};
          wa.plan = plan;
          wa.m = m;
          wa.mL = mL;
          wa.GL = GL;
          wa.W = W;
          wa.act = act[cur];
          wa.gstart = gstart[cur];
          wa.lg = lg;
          wa.loff = loff;
          wa.key1_stash = upd;
          wa.sec_stash = act[nxt];
          wa.ka = ka;
          wa.kb = kb;
          wa.va = va;
          wa.ctrl = ctrl;
          s = launch(SA_K_GATHER, 1, 24ull * mL, [&] { return launch_wide_rekey(wa, st); });
          if (s != SA_OK) return s;
          s = sort(mL, spec_for(kbits));
          if (s != SA_OK) return s;
          s = launch(SA_K_GATHER, 2, 40ull * mL, [&] { return launch_wide_finish(wa, st); });
          if (s != SA_OK) return s;
          bytes += 64ull * mL;
        } else {
          s = sort(mL, spec_for(kbits));
          if (s != SA_OK) return s;
        }
      }
      // Small groups: refined tile by tile; name changes are queued.
      RefineArgs rf{};
      rf.act = act[cur];
      rf.gstart = gstart[cur];
      rf.gname = gname[cur];
      rf.ghead = ghead[cur];
      rf.naming = naming;
      rf.tfirst = tfirst;
      rf.m = m;
      rf.G = G;
      rf.shape = shape;
      rf.small = small;
      rf.tiles = (m + nominal - 1) / nominal;
      rf.h = (uint32_t)h;
      rf.W = W;
      rf.mult = mult;
      rf.isa = isa;
      rf.isa_len = N + S + 1;
      rf.N = N32;
      rf.sa = sa;
      rf.seg_off = segoff;
      rf.S = S;
      rf.act_out = act[nxt];
      rf.gstart_out = gstart[nxt];
      rf.gname_out = gname[nxt];
      rf.ghead_out = ghead[nxt];
      rf.upd = upd;
      rf.ctrl = ctrl;
      s = launch(SA_K_REFINE, 0, 0, [&] { return launch_refine(rf, st); });
      if (s != SA_OK) return s;
      if (mL > 0) {
        s = rename(mL, 0, 0, 0, W, lbase, lold, GL, nxt, &ctrl->rc.m_s, mult > 2);
        if (s != SA_OK) return s;
      }
      s = scatter(m);
      if (s != SA_OK) return s;
      s = classify(nxt, mL);
      if (s != SA_OK) return s;
      if (opt.trace_isa && round < opt.trace_cap && S == 1)
        CK(cudaMemcpyAsync(opt.trace_isa + (size_t)round * N, isa, N * 4,
                           cudaMemcpyDeviceToDevice, st));
      uint32_t p1[2] = {0, 0};  // the first sort's (passes, mask) in a-tuple rounds
      if (mL > 0 && mult > 2) CK(cudaMemcpyAsync(p1, pm1, 8, cudaMemcpyDeviceToHost, st));
      s = read_ctrl(hc);
      if (s != SA_OK) return s;
      hc.passes += p1[0];
      // Settle the byte counts that depend on this round's results.
      const uint64_t rbl = mL ? rename_bytes(mL, hc.m_l, hc.g_l) : 0;
      const uint64_t rfb = refine_bytes(m - mL, G - GL, hc.m_s, hc.g_s, hc.upd, mult);
      for (Rec &r : recs)
        if (r.cls == SA_K_REFINE) r.bytes = rfb;
      settle(hc);
      s = flush(hc.pass_mask, rbl, p1[1]);
      if (s != SA_OK) return s;
      record(round, m, hc, kbits);
      bytes += (mL ? (uint64_t)hc.passes * 24 * mL : 0) + rbl + rfb;
      cur = nxt;
      h *= mult;
      ++round;
    }
    // ---- output ----
    if (isa_out && !direct) {
      s = launch(SA_K_OUTPUT, 0, 8ull * N, [&] {
        return launch_isa_to_local(isa, isa_out, N32, segoff, S, st);
      });
      if (s != SA_OK) return s;
      bytes += 8ull * N;
    }
    // The SA is complete with the last round's readback; the ISA, and the
    // trace of a text resolved in round 0, are written after it.
    if (prof || isa_out || want_trace) {
      CK(cudaStreamSynchronize(st));
      s = flush(0, 0);
      if (s != SA_OK) return s;
    }
    if (stats) {
      stats->rounds = round;
      stats->bytes_model = bytes;
      stats->launches = launches;
    }
    return SA_OK;
  }
};

sa_status check_offsets(const uint64_t *offsets, uint32_t count) {
  if (!offsets || count == 0) return SA_ERR_INVALID_ARG;
  if (offsets[0] != 0) return SA_ERR_INVALID_ARG;
  for (uint32_t k = 0; k < count; ++k)
    if (offsets[k + 1] < offsets[k]) return SA_ERR_INVALID_ARG;
  if (offsets[count] > SA_MAX_N) return SA_ERR_TOO_LARGE;
  return SA_OK;
}

bool bad_options(const sa_options *opt) {
  if (!opt) return false;
  if (opt->multiplier != 0 && (opt->multiplier < 2 || opt->multiplier > 4)) return true;
  if (opt->sort_items != 0 && opt->sort_items != 8 && opt->sort_items != 12 &&
      opt->sort_items != 16)
    return true;
  if (opt->refine_shape > (uint32_t)REFINE_SHAPES) return true;
  return opt->initial_keys > 2;
}

sa_status run_with_workspace(Build &B, void *workspace, size_t ws_bytes) {
  B.L = make_layout(B.N, B.S);
  if (B.opt.spin_limit) B.spin = B.opt.spin_limit;
  PoolBuf own;
  if (workspace) {
    if (ws_bytes < B.L.total || ((uintptr_t)workspace & 255)) return SA_ERR_OOM;
    B.ws = (uint8_t *)workspace;
  } else {
    own.st = B.st;
    if (pool_alloc(&own.p, B.L.total, B.st) != cudaSuccess) {
      own.p = nullptr;
      cudaGetLastError();
      return SA_ERR_OOM;
    }
    B.ws = (uint8_t *)own.p;
  }
  if (B.stats) memset(B.stats, 0, sizeof(sa_stats));
  return B.run();
}

}  // namespace

// The library's private stream-ordered pool, for the other entry points.
cudaError_t library_pool_alloc(void **p, size_t bytes, cudaStream_t st) {
  return pool_alloc(p, bytes, st);
}

int device_sm_count() {
  static std::mutex mu;
  static std::map<int, int> cache;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  std::lock_guard<std::mutex> g(mu);
  auto it = cache.find(dev);
  if (it != cache.end()) return it->second;
  int n = 0;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
    cudaGetLastError();
    return 1;  // not cached: a later call may succeed
  }
  cache[dev] = n;
  return n;
}

namespace {

// Identity of the CUDA context current on this thread (cuCtxGetCurrent and
// cuCtxGetId, reached through the runtime's driver entry points so that
// the library needs no link against libcuda); 0 when it cannot be told.
unsigned long long current_context_id() {
  using GetCurrent = int (*)(void **);
  using GetId = int (*)(void *, unsigned long long *);
  static GetCurrent get_current = nullptr;
  static GetId get_id = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void *f = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      get_current = reinterpret_cast<GetCurrent>(f);
    f = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      get_id = reinterpret_cast<GetId>(f);
    cudaGetLastError();
  });
  if (!get_current || !get_id) return 0;
  void *ctx = nullptr;
  unsigned long long id = 0;
  if (get_current(&ctx) != 0 || !ctx || get_id(ctx, &id) != 0) return 0;
  return id;
}

}  // namespace

cudaError_t ensure_smem_attributes(const void *fn, int smem_bytes, bool max_carveout) {
  static std::mutex mu;
  static std::set<std::pair<const void *, unsigned long long>> done;
  const unsigned long long ctx = current_context_id();
  if (ctx) {
    std::lock_guard<std::mutex> g(mu);
    if (done.count({fn, ctx})) return cudaSuccess;
  }
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
  if (e != cudaSuccess) return e;
  if (max_carveout) {
    e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
  }
  if (ctx) {  // unknown context: set again next time rather than trust a stale entry
    std::lock_guard<std::mutex> g(mu);
    done.insert({fn, ctx});
  }
  return cudaSuccess;
}
}  // namespace gbsa

using namespace gbsa;

GBSA_API size_t sa_workspace_bytes(uint64_t n) { return make_layout(n, 1).total; }

GBSA_API sa_status sa_pool_usage(uint64_t *used, uint64_t *reserved) {
  if (!used || !reserved) return SA_ERR_INVALID_ARG;
  *used = *reserved = 0;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return SA_ERR_CUDA;
  }
  std::lock_guard<std::mutex> g(g_pool_mu);
  auto it = g_pools.find(dev);
  if (it == g_pools.end()) return SA_OK;  // nothing was ever taken from it
  uint64_t u = 0, r = 0;  // the pool attributes are 64-bit values
  if (cudaMemPoolGetAttribute(it->second, cudaMemPoolAttrUsedMemCurrent, &u) != cudaSuccess ||
      cudaMemPoolGetAttribute(it->second, cudaMemPoolAttrReservedMemCurrent, &r) != cudaSuccess) {
    cudaGetLastError();
    return SA_ERR_CUDA;
  }
  *used = u;
  *reserved = r;
  return SA_OK;
}

GBSA_API sa_status sa_pool_trim(uint64_t keep_bytes) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return SA_ERR_CUDA;
  }
  std::lock_guard<std::mutex> g(g_pool_mu);
  auto it = g_pools.find(dev);
  if (it == g_pools.end()) return SA_OK;
  if (cudaMemPoolTrimTo(it->second, (size_t)keep_bytes) != cudaSuccess) {
    cudaGetLastError();
    return SA_ERR_CUDA;
  }
  return SA_OK;
}

GBSA_API size_t sa_batched_workspace_bytes(const uint64_t *offsets, uint32_t count) {
  if (check_offsets(offsets, count) != SA_OK) return 0;
  return make_layout(offsets[count], count).total;
}

GBSA_API sa_status sa_build_ex(const uint8_t *text, uint64_t n, uint32_t *sa_out,
                               uint32_t *isa_out, void *workspace, size_t ws_bytes,
                               const sa_options *opt, sa_stats *stats, gbsa_stream_t stream) {
  return gbsa::build_single(text, n, sa_out, isa_out, workspace, ws_bytes, opt, stats, stream,
                            true);
}

namespace gbsa {
sa_status build_single(const uint8_t *text, uint64_t n, uint32_t *sa_out, uint32_t *isa_out,
                       void *workspace, size_t ws_bytes, const sa_options *opt, sa_stats *stats,
                       gbsa_stream_t stream, bool stage_readbacks) {
  if (n > SA_MAX_N) return SA_ERR_TOO_LARGE;
  if (n > 0 && (!text || !sa_out)) return SA_ERR_INVALID_ARG;
  if (bad_options(opt)) return SA_ERR_INVALID_ARG;
  if (stats) memset(stats, 0, sizeof(sa_stats));
  cudaStream_t st = (cudaStream_t)stream;
  if (n == 0) return SA_OK;
  if (n == 1) {
    if (cudaMemsetAsync(sa_out, 0, 4, st) != cudaSuccess) return SA_ERR_CUDA;
    if (isa_out && cudaMemsetAsync(isa_out, 0, 4, st) != cudaSuccess) return SA_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return SA_ERR_CUDA;
    if (stats) stats->rounds = 1;
    return SA_OK;
  }
  Build B;
  B.stage_readbacks = stage_readbacks;
  B.text = text;
  B.N = n;
  B.S = 1;
  B.off = {0u, (uint32_t)n};
  B.sa = sa_out;
  B.isa_out = isa_out;
  if (opt) B.opt = *opt;
  B.stats = stats;
  B.st = st;
  return run_with_workspace(B, workspace, ws_bytes);
}
}  // namespace gbsa

GBSA_API sa_status sa_build(const uint8_t *text, uint64_t n, uint32_t *sa_out,
                            gbsa_stream_t stream) {
  return sa_build_ex(text, n, sa_out, nullptr, nullptr, 0, nullptr, nullptr, stream);
}

GBSA_API sa_status sa_build_batched_ex(const uint8_t *texts, const uint64_t *offsets,
                                       uint32_t count, uint32_t *sa_out, void *workspace,
                                       size_t ws_bytes, const sa_options *opt,
                                       sa_stats *stats, gbsa_stream_t stream) {
  sa_status s = check_offsets(offsets, count);
  if (s != SA_OK) return s;
  if (count > (1u << 20)) return SA_ERR_TOO_LARGE;
  if (bad_options(opt)) return SA_ERR_INVALID_ARG;
  const uint64_t N = offsets[count];
  if (stats) memset(stats, 0, sizeof(sa_stats));
  if (N == 0) return SA_OK;
  if (!texts || !sa_out) return SA_ERR_INVALID_ARG;
  Build B;
  B.text = texts;
  B.N = N;
  B.S = count;
  B.off.resize((size_t)count + 1);
  for (uint32_t k = 0; k <= count; ++k) B.off[k] = (uint32_t)offsets[k];
  B.sa = sa_out;
  if (opt) {
    B.opt = *opt;
    B.opt.trace_isa = nullptr;
    B.opt.trace_cap = 0;
  }
  B.stats = stats;
  B.st = (cudaStream_t)stream;
  return run_with_workspace(B, workspace, ws_bytes);
}

GBSA_API sa_status sa_build_batched(const uint8_t *texts, const uint64_t *offsets, uint32_t count,
                                    uint32_t *sa_out, gbsa_stream_t stream) {
  return sa_build_batched_ex(texts, offsets, count, sa_out, nullptr, 0, nullptr, nullptr, stream);
}

// Largest request whose host copies run as kernels (sa_build_host).
constexpr uint64_t HOST_KERNEL_COPY_MAX = 4ull << 20;

GBSA_API sa_status sa_build_host(const uint8_t *host_text, uint64_t n, uint32_t *host_sa,
                                 gbsa_stream_t stream) {
  if (n > SA_MAX_N) return SA_ERR_TOO_LARGE;
  if (n > 0 && (!host_text || !host_sa)) return SA_ERR_INVALID_ARG;
  if (n == 0) return SA_OK;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t tb = align256(n), sb = align256(n * 4);
  const size_t wb = sa_workspace_bytes(n);
  PoolBuf buf;
  buf.st = st;
  if (pool_alloc(&buf.p, tb + sb + wb, st) != cudaSuccess) {
    buf.p = nullptr;
    cudaGetLastError();
    return SA_ERR_OOM;
  }
  uint8_t *d_text = (uint8_t *)buf.p;
  uint32_t *d_sa = (uint32_t *)((uint8_t *)buf.p + tb);
  void *d_ws = (uint8_t *)buf.p + tb + sb;
  // Small requests with pinned host buffers copy by kernels, which read and
  // write the buffers through their device mapping: a copy engine runs the
  // copies of all streams in order, so a server's small request would
  // otherwise wait behind the large copies of concurrent builds. Larger or
  // pageable buffers take the copy engine.
  const uint8_t *src_dev = nullptr;
  uint32_t *dst_dev = nullptr;
  if (n <= HOST_KERNEL_COPY_MAX) {
    cudaPointerAttributes at{}, as{};
    if (cudaPointerGetAttributes(&at, host_text) == cudaSuccess &&
        cudaPointerGetAttributes(&as, host_sa) == cudaSuccess && at.type == cudaMemoryTypeHost &&
        as.type == cudaMemoryTypeHost && at.devicePointer && as.devicePointer) {
      src_dev = (const uint8_t *)at.devicePointer;
      dst_dev = (uint32_t *)as.devicePointer;
    }
    cudaGetLastError();  // a pageable pointer is not an error here
  }
  if (src_dev) {
    if (launch_copy_bytes(d_text, src_dev, n, st) != cudaSuccess) return SA_ERR_CUDA;
  } else if (cudaMemcpyAsync(d_text, host_text, n, cudaMemcpyHostToDevice, st) != cudaSuccess) {
    return SA_ERR_CUDA;
  }
  sa_status s = sa_build_ex(d_text, n, d_sa, nullptr, d_ws, wb, nullptr, nullptr, stream);
  if (s != SA_OK) return s;
  if (dst_dev) {
    if (launch_copy_words(dst_dev, d_sa, n, st) != cudaSuccess) return SA_ERR_CUDA;
  } else if (cudaMemcpyAsync(host_sa, d_sa, n * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess) {
    return SA_ERR_CUDA;
  }
  if (cudaStreamSynchronize(st) != cudaSuccess) return SA_ERR_CUDA;
  return SA_OK;
}

GBSA_API sa_status sa_build_batched_host(const uint8_t *const *host_texts, const uint64_t *lengths,
                                         uint32_t *const *host_sas, uint32_t count,
                                         gbsa_stream_t stream) {
  if (count == 0 || !host_texts || !lengths || !host_sas) return SA_ERR_INVALID_ARG;
  if (count > (1u << 20)) return SA_ERR_TOO_LARGE;
  std::vector<uint64_t> off((size_t)count + 1, 0);
  for (uint32_t k = 0; k < count; ++k) {
    if (lengths[k] > SA_MAX_N) return SA_ERR_TOO_LARGE;
    if (lengths[k] > 0 && (!host_texts[k] || !host_sas[k])) return SA_ERR_INVALID_ARG;
    off[k + 1] = off[k] + lengths[k];
    if (off[k + 1] > SA_MAX_N) return SA_ERR_TOO_LARGE;
  }
  const uint64_t N = off[count];
  if (N == 0) return SA_OK;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t tb = align256(N), sb = align256(N * 4);
  const size_t wb = sa_batched_workspace_bytes(off.data(), count);
  PoolBuf buf;
  buf.st = st;
  if (pool_alloc(&buf.p, tb + sb + wb, st) != cudaSuccess) {
    buf.p = nullptr;
    cudaGetLastError();
    return SA_ERR_OOM;
  }
  uint8_t *d_text = (uint8_t *)buf.p;
  uint32_t *d_sa = (uint32_t *)((uint8_t *)buf.p + tb);
  void *d_ws = (uint8_t *)buf.p + tb + sb;
  // As in sa_build_host: a small batch whose buffers are all pinned copies
  // by kernels (one launch per SegCopy::MAX texts each way), so it does not
  // queue behind the copy-engine traffic of other streams; otherwise one
  // copy-engine copy per text and direction.
  std::vector<void *> src_dev, dst_dev;
  bool mapped = N <= HOST_KERNEL_COPY_MAX;
  if (mapped) {
    src_dev.assign(count, nullptr);
    dst_dev.assign(count, nullptr);
    for (uint32_t k = 0; k < count && mapped; ++k) {
      if (lengths[k] == 0) continue;
      cudaPointerAttributes at{}, as{};
      mapped = cudaPointerGetAttributes(&at, host_texts[k]) == cudaSuccess &&
               cudaPointerGetAttributes(&as, host_sas[k]) == cudaSuccess &&
               at.type == cudaMemoryTypeHost && as.type == cudaMemoryTypeHost &&
               at.devicePointer && as.devicePointer;
      src_dev[k] = at.devicePointer;
      dst_dev[k] = as.devicePointer;
    }
    cudaGetLastError();  // a pageable pointer is not an error here
  }
  auto kernel_copies = [&](bool to_flat) -> cudaError_t {
    for (uint32_t k0 = 0; k0 < count; k0 += SegCopy::MAX) {
      SegCopy t{};
      t.count = std::min<uint32_t>(SegCopy::MAX, count - k0);
      for (uint32_t j = 0; j < t.count; ++j) t.ext[j] = to_flat ? src_dev[k0 + j] : dst_dev[k0 + j];
      for (uint32_t j = 0; j <= t.count; ++j) t.off[j] = off[k0 + j];
      const cudaError_t e = launch_copy_segments(to_flat ? (void *)d_text : (void *)d_sa, t,
                                                 to_flat ? 1 : 4, to_flat, st);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  };
  if (mapped) {
    if (kernel_copies(true) != cudaSuccess) return SA_ERR_CUDA;
  } else {
    for (uint32_t k = 0; k < count; ++k)
      if (lengths[k] && cudaMemcpyAsync(d_text + off[k], host_texts[k], lengths[k],
                                        cudaMemcpyHostToDevice, st) != cudaSuccess)
        return SA_ERR_CUDA;
  }
  const sa_status s =
      sa_build_batched_ex(d_text, off.data(), count, d_sa, d_ws, wb, nullptr, nullptr, stream);
  if (s != SA_OK) return s;
  if (mapped) {
    if (kernel_copies(false) != cudaSuccess) return SA_ERR_CUDA;
  } else {
    for (uint32_t k = 0; k < count; ++k)
      if (lengths[k] && cudaMemcpyAsync(host_sas[k], d_sa + off[k], lengths[k] * 4,
                                        cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return SA_ERR_CUDA;
  }
  if (cudaStreamSynchronize(st) != cudaSuccess) return SA_ERR_CUDA;
  return SA_OK;
}

GBSA_API size_t sa_sort_workspace_bytes(uint64_t m) {
  const uint64_t mm = m ? m : 1;
  const uint64_t tiles = (mm + SORT_TILE_MIN - 1) / SORT_TILE_MIN;
  return align256(sizeof(Ctrl)) + align256(sizeof(SortPlan)) + 2 * align256(MAX_PASSES * RADIX * 4) +
         align256(mm * 8) + align256(mm * 4) + align256(tiles * RADIX * 8);
}

GBSA_API sa_status sa_sort_pairs(uint64_t *keys, uint32_t *vals, uint64_t m, uint32_t begin_bit,
                                 uint32_t end_bit, void *workspace, size_t ws_bytes,
                                 gbsa_stream_t stream) {
  if (m > SA_MAX_N) return SA_ERR_TOO_LARGE;
  if (begin_bit >= end_bit || end_bit > 64) return SA_ERR_INVALID_ARG;
  if (m > 0 && (!keys || !vals)) return SA_ERR_INVALID_ARG;
  if (m <= 1) return SA_OK;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t need = sa_sort_workspace_bytes(m);
  PoolBuf own;
  uint8_t *ws = (uint8_t *)workspace;
  if (ws) {
    if (ws_bytes < need || ((uintptr_t)ws & 255)) return SA_ERR_OOM;
  } else {
    own.st = st;
    if (pool_alloc(&own.p, need, st) != cudaSuccess) {
      own.p = nullptr;
      cudaGetLastError();
      return SA_ERR_OOM;
    }
    ws = (uint8_t *)own.p;
  }
  const uint64_t tiles = (m + SORT_TILE_MIN - 1) / SORT_TILE_MIN;
  size_t o = 0;
  auto take = [&](size_t bytes) { uint8_t *r = ws + o; o += align256(bytes); return r; };
  Build B;
  B.st = st;
  B.ctrl = (Ctrl *)take(sizeof(Ctrl));
  B.plan = (SortPlan *)take(sizeof(SortPlan));
  B.hist = (uint32_t *)take(MAX_PASSES * RADIX * 4);
  B.dbase = (uint32_t *)take(MAX_PASSES * RADIX * 4);
  B.kb = (uint64_t *)take(m * 8);
  B.vb = (uint32_t *)take(m * 4);
  B.st_sort = (uint64_t *)take(tiles * RADIX * 8);
  B.ka = keys;
  B.va = vals;
  CK(cudaMemsetAsync(B.ctrl, 0, sizeof(Ctrl), st));
  CK(cudaMemsetAsync(B.st_sort, 0, tiles * RADIX * 8, st));
  DigitSpec spec{};
  const uint32_t span = end_bit - begin_bit;
  spec.P = (span + RADIX_BITS - 1) / RADIX_BITS;
  for (uint32_t p = 0; p < spec.P; ++p) {
    spec.shift[p] = (uint8_t)(begin_bit + p * RADIX_BITS);
    spec.bits[p] = (uint8_t)std::min<uint32_t>(RADIX_BITS, end_bit - spec.shift[p]);
  }
  sa_status s = B.sort((uint32_t)m, spec);
  if (s != SA_OK) return s;
  CK(launch_copy_back(B.plan, keys, vals, (uint32_t)m, sm_count(), st));
  HostCtrl hc{};
  return B.read_ctrl(hc);
}

GBSA_API const char *sa_status_string(sa_status s) {
  switch (s) {
    case SA_OK: return "SA_OK";
    case SA_ERR_INVALID_ARG: return "SA_ERR_INVALID_ARG";
    case SA_ERR_TOO_LARGE: return "SA_ERR_TOO_LARGE";
    case SA_ERR_OOM: return "SA_ERR_OOM";
    case SA_ERR_CUDA: return "SA_ERR_CUDA";
    case SA_ERR_TIMEOUT: return "SA_ERR_TIMEOUT";
    case SA_ERR_INTERNAL: return "SA_ERR_INTERNAL";
  }
  return "SA_ERR_UNKNOWN";
}
