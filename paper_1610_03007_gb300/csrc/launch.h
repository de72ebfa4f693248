// Host-side launchers of the gbsa kernels (one .cu file per step of the
// method). All launches are asynchronous on `stream`.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/gbsa.h"
#include "common.cuh"

namespace gbsa {

// ---- runtime helpers (engine.cu) ----------------------------------------
// SM count of the current device, cached per device; thread-safe.
int device_sm_count();
// Allows `smem_bytes` of dynamic shared memory for kernel `fn` (and, with
// max_carveout, the largest shared-memory carveout), once per kernel and
// CUDA context: function attributes belong to a context, so a process that
// launches on several GPUs, or again after cudaDeviceReset, must set them
// in each. Thread-safe; concurrent first calls may both set them (harmless).
cudaError_t ensure_smem_attributes(const void *fn, int smem_bytes, bool max_carveout);
// sa_build_ex; stage_readbacks false keeps every readback on the copy
// engine through pageable memory (no pinned host allocation, for
// sa_build_noalloc).
sa_status build_single(const uint8_t *text, uint64_t n, uint32_t *sa_out, uint32_t *isa_out,
                       void *workspace, size_t ws_bytes, const sa_options *opt, sa_stats *stats,
                       gbsa_stream_t stream, bool stage_readbacks);
// The tuning table's parameters for a build of this class (tuning.cu); all
// fields 0 when no entry applies.
void tuned_params(bool batched, uint32_t bits, uint64_t n, sa_tuned *out);

// Copies by kernels (k_gather.cu): dst/src may be pinned host memory
// (device-mapped), so the copy does not queue on a copy engine.
cudaError_t launch_copy_words(uint32_t *dst, const uint32_t *src, uint64_t words,
                              cudaStream_t stream);
cudaError_t launch_copy_bytes(uint8_t *dst, const uint8_t *src, uint64_t n, cudaStream_t stream);

// ---- step A0: alphabet (k_alphabet.cu) ----------------------------------
// Of the prefixes drawn: pairs and triples of one block and text that agree in
// 1, 2, .. characters (0 beyond what 64 bits hold beside the text's number).
constexpr uint32_t SAMPLE_KEYS = 512, SAMPLE_CHARS = 8, SAMPLE_BLOCKS_MAX = 64;
struct KeySample {
  unsigned long long triples[SAMPLE_CHARS];
  uint32_t pairs[SAMPLE_CHARS];
};
struct AlphabetArgs {
  const uint8_t *text;
  uint64_t n;
  uint32_t *hist;     // 256 counts (zeroed by the caller), += the text's; then a KeySample
  uint32_t *done;     // blocks finished (zeroed by the caller)
  uint8_t *code;      // out: dense order-preserving code of each byte value
  uint32_t *seg_off;  // out, for one text: {0, n} (NULL otherwise)
  uint32_t *host;     // out: the counts and the sample in pinned host memory, or NULL
  uint32_t sample_blocks;  // blocks that draw SAMPLE_KEYS prefixes each (0: none)
  const uint32_t *offsets;  // S + 1 offsets of a batch (S > 1)
  uint32_t S;
  uint32_t *host_flag;  // set to 1 after them
};
cudaError_t launch_byte_histogram(const AlphabetArgs &a, int num_sms, cudaStream_t stream);

// ---- step A1: initial keys (k_pack.cu) ----------------------------------
struct PackArgs {
  const uint8_t *text;     // concatenated texts
  uint32_t N;              // total characters
  const uint32_t *seg_off; // S+1 ungapped offsets (device)
  uint32_t S;              // number of texts
  const uint8_t *code;     // dense order-preserving code of each byte (device)
  uint32_t b;              // bits per character
  uint32_t c0;             // characters per key
  uint32_t cb;             // c0 * b (segment id sits above these bits)
  uint64_t *keys;          // out: N keys, tail-first order per text
  uint32_t *vals;          // out: N gapped positions
  DigitSpec spec;          // digits of the following radix sort
  uint32_t *hist;          // out: += their histograms (P * 256, zeroed by the caller)
  // 1: one text whose digits hold whole characters (b divides 8, cb a
  // multiple of 8): only the top digit is counted per key and the other
  // histograms are derived from it (launch_sort_plan).
  uint32_t top_only;
};
// keys == NULL (top_only only): only the top digit's histogram (the first
// radix pass then builds the keys from the text, PassArgs.text). With
// top_only the counts go to the last of the MAX_PASSES rows, from which
// launch_sort_plan derives the rows of the digits in spec.
cudaError_t launch_pack(const PackArgs &a, cudaStream_t stream);

// ---- step A2: radix sort (k_sort.cu) ------------------------------------
// hist[P*256] += digit counts of keys[0, m) for the digits in spec.
// rs (device-driven rounds): m and spec come from rs->mL and rs->spec
// instead (m then sizes the grid only).
cudaError_t launch_digit_histogram(const uint64_t *keys, uint32_t m, const DigitSpec &spec,
                                   uint32_t *hist, int num_sms, cudaStream_t stream,
                                   const RoundState *rs = nullptr);
// Exclusive digit offsets, constant-digit skipping and buffer ping-pong.
// keep: bit p keeps pass p even if its digit is constant (the pass that
// reads the text, PassArgs.text; every pass, so that the host knows which
// buffer the result is in).
// grams: the histograms of a text's keys are derived from the last row of
// hist first (PackArgs.top_only).
cudaError_t launch_sort_plan(const uint32_t *hist, uint32_t *digit_base, const DigitSpec &spec,
                             uint32_t m, uint64_t *ka, uint64_t *kb, uint32_t *va,
                             uint32_t *vb, SortPlan *plan, Ctrl *ctrl, cudaStream_t stream,
                             const RoundState *rs = nullptr, uint32_t keep = 0,
                             const PackArgs *grams = nullptr);
// One stable one-sweep pass over digit p of the plan.
struct PassArgs {
  const SortPlan *plan;
  int p;
  uint32_t shift, bits;
  const uint32_t *digit_base;  // 256 entries for this pass
  uint32_t m;
  uint64_t *status;  // >= tiles * 256 words
  uint32_t epoch;
  uint32_t *tile_ctr;
  Ctrl *ctrl;
  uint32_t spin_limit;
  uint32_t inject;
  uint32_t items;    // keys per thread: 8, 12 or 16 (tile = 256 * items)
  // Device-driven rounds: sizes, digit and epoch base from the round state
  // (m then bounds the grid only; epoch is an offset). NULL: the fields above.
  const RoundState *rs;
  uint32_t grid_cap;  // at most this many blocks, each looping over tiles (0: one per tile)
  // Pass 0 of round 0 over one text (text != NULL, p == 0, not persistent):
  // the keys are built from the text in the layout of k_pack.cu (index j <
  // tails: the tail position n-1-j, zero-padded; j >= tails: position j -
  // tails) instead of read from the plan's source buffers.
  const uint8_t *text;
  const uint8_t *code;  // dense code of each byte (256 entries, device)
  uint32_t b, c0, cb, tails;
};
constexpr int SORT_TILE_MIN = 256 * 8;  // smallest tile (sizes the status array)
constexpr uint32_t SORT_ITEMS_DEFAULT = 16;
cudaError_t launch_onesweep(const PassArgs &a, cudaStream_t stream);
// Copies the plan's final buffer back to (ka, va) when it is buffer B.
cudaError_t launch_copy_back(const SortPlan *plan, uint64_t *ka, uint32_t *va, uint32_t m,
                             int num_sms, cudaStream_t stream);

// ---- steps A3+A4: rename, unique test, discard (k_rename.cu) ------------
struct RenameArgs {
  const SortPlan *plan;      // sorted keys / gapped positions
  uint32_t m;
  // 1: initial naming with the end-of-text rules; 2: the same for the
  // buckets k_local left to the global path (keys (bucket << W) | low bits,
  // ranks from base_in).
  uint32_t round0;
  uint32_t cb;               // round 0: segment id = key >> cb (cb < 64)
  uint32_t c0;               // round 0: characters per key
  const uint32_t *seg_off;   // S+1 ungapped offsets
  uint32_t S;
  uint32_t W;                // later rounds: group ordinal g = key >> W
  // a-tuple rounds: {ka, kb}; the later partners of sorted position j are
  // in the buffer that does not hold the keys. {NULL, NULL} otherwise.
  const uint64_t *sec_buf[2];
  const uint32_t *base_in;   // later rounds: head rank - start of group g
  const uint32_t *old_in;    // later rounds: name of group g (round 0: NULL)
  uint32_t g_in;             // later rounds: groups in base_in (bounds guard)
  // Queued ISA entries (head << 32 | i') of new unique suffixes; in round 0
  // (round0 != 0) none: k_isa.cu takes them from the SA.
  uint64_t *upd;
  uint32_t *isa;             // gapped ISA (not written; bounds of gapped positions)
  uint64_t isa_len;          // entries of isa (bounds guard)
  uint32_t N;                // total characters = entries of sa (bounds guard)
  uint32_t *sa;              // SA, written with indices local to each text
                             // (round0 = 1: SA_NONE at the survivors' ranks)
  uint64_t *act_out;         // survivors: (g' << 32) | i'
  uint32_t *gstart_out;      // start of each surviving group in act_out
  uint32_t *ghead_out;       // head rank (SA interval start) of each surviving group
  uint32_t *gold_out;        // name of its parent group (NO_NAME in round 0)
  const uint32_t *off_in;    // device: [survivor offset, group offset] of the output
  uint32_t *cnt_out;         // device: [survivors, groups] written by the last tile
  uint64_t *status;          // >= 2 * tiles words
  uint32_t epoch;
  uint32_t *tile_ctr;
  Ctrl *ctrl;
  uint32_t spin_limit;
  // Device-driven rounds: m = rs->mL, g_in = rs->GL and epoch base
  // rs->epoch (m above then bounds the grid only). NULL: the fields above.
  const RoundState *rs;
  uint32_t grid_cap;         // at most this many blocks, each looping over tiles (0: one per tile)
};
#ifndef GBSA_RN_ITEMS
#define GBSA_RN_ITEMS 8
#endif
constexpr int RENAME_TILE = 256 * GBSA_RN_ITEMS;
cudaError_t launch_rename(const RenameArgs &a, cudaStream_t stream);

// ---- round 0 by buckets of equal top bits (k_local.cu) -------------------
constexpr uint32_t SA_NONE = 0xFFFFFFFFu;  // SA entry of a rank that is not final
constexpr int LOCAL_TILE = 2560;           // window of one tile
struct LocalArgs {
  const SortPlan *plan;     // keys sorted by the bits from R up / gapped positions
  uint32_t m, R;
  uint32_t cb, c0;          // as RenameArgs
  const uint32_t *seg_off;
  uint32_t S, N;
  uint32_t naming;
  uint64_t isa_len;
  uint32_t *sa;             // unique suffixes at their ranks, SA_NONE elsewhere
  uint64_t *act_out;        // survivors of the tiles' buckets, as the refine's
  uint32_t *gstart_out, *gname_out, *ghead_out;
  uint64_t *upd;            // (name << 32) | i' of every survivor
  // Buckets too large for a tile: start, start among their items, start
  // less that, NO_NAME; rc.large counts them (buckets << 32 | items).
  uint32_t *lg, *loff, *lbase, *lold;
  uint32_t max_large, max_groups;
  Ctrl *ctrl;               // rc.m_s / rc.g_s / rc.upd reserve the outputs
  uint32_t *host;           // the last tile copies the head of ctrl here (pinned; or NULL)
  uint32_t *host_flag;      // and sets this to 1
};
cudaError_t launch_local(const LocalArgs &a, cudaStream_t stream);
struct GatherBigArgs {
  const uint64_t *kin;      // the sorted keys and positions k_local read
  const uint32_t *vin;
  const uint32_t *lg, *loff;
  uint32_t m, mL, GL, R;
  uint64_t *keys;           // (bucket << R) | low bits of the key
  uint32_t *vals;
  uint32_t *sa;             // SA_NONE at the buckets' ranks
  Ctrl *ctrl;
};
cudaError_t launch_gather_big(const GatherBigArgs &a, cudaStream_t stream);

// ---- ISA entries of the suffixes final after round 0 (k_isa.cu) ------------
// ISA[i'] = j for every rank j whose SA entry is not SA_NONE.
cudaError_t launch_isa_fill(const uint32_t *sa, uint32_t N, const uint32_t *seg_off, uint32_t S,
                            uint32_t *isa, uint64_t isa_len, cudaStream_t stream);

constexpr uint32_t NEED_WORDS = 1u << 21;        // 2^26 granules
constexpr uint32_t NEED_OFFSETS = 64;
constexpr uint64_t NEED_OFFSET_MAX = 1ull << 17; // rounds the first plan covers
struct NeedArgs {
  const uint64_t *act;  // active entries (their low words are positions)
  uint32_t m;
  uint32_t shift;       // granule of a position: position >> shift
  uint32_t words;       // words of bits in use
  uint32_t offsets;     // partner offsets of the rounds planned for
  uint32_t h[NEED_OFFSETS];
  uint32_t *active, *covered, *missing;  // `words` each
  Ctrl *ctrl;           // need_any is set when a granule is missing
};
cudaError_t launch_need_plan(const NeedArgs &a, int num_sms, cudaStream_t stream);
struct CollectArgs {
  const uint32_t *sa;
  uint32_t N;
  const uint32_t *seg_off;
  uint32_t S;
  uint32_t shift, words;    // as NeedArgs
  const uint32_t *missing;  // NULL: every final rank
  uint64_t *out;            // (rank << 32) | i', ctrl->need_entries of them (N at most)
  Ctrl *ctrl;
};
cudaError_t launch_need_collect(const CollectArgs &a, int num_sms, cudaStream_t stream);

// ---- rounds >= 1: small-group refine and large-group path (k_refine.cu) --
// Groups of up to `small` members are refined inside one tile
// (gather, shared-memory sort, rename, compaction); larger ones go through
// the global radix sort and k_rename.
// Tile shapes of the refine: threads per block, items one tile can hold, and
// the largest small group. Tile t owns the groups whose starts fall in
// [t, t+1) * (cap - small) of the active list, so a tile's groups always fit.
// The first two shapes' wider windows spread a tile's fixed work over more
// items where few groups are above `small`, which cost more in the global
// sort. Refine of the 2^28 repeated Zipf text (groups of about 250) with 256 x
// 2048 tiles and groups of up to 1024, 768, 640, 512: 51.3, 46.4, 44.8, 43.6
// ms; of 2^28 Markov DNA (pairs) with 128 x 1024 and up to 512, 384, 256:
// 3.78, 3.39, 4.00 ms. Where more than one active suffix in REFINE_HALF_SHARE
// is in a group above `small` that a tile can hold, the build takes half a tile
// as window and limit (Build::refine_limits). Builds of 2^27 characters,
// copies of a Zipf block 600, 800, 1000, 1500 times: 87.7, 93.1, 97.4, 101.0 ms
// with groups of up to 512, 40.8, 42.0, 42.8, 96.1 with 1024; of a DNA block
// 400, 500, 600 times 49.8, 72.2, 76.8 with 384, 39.5, 39.3, 69.0 with 512. The
// share at which both take the same time: Zipf 800 copies beside 250 0.08,
// DNA 450 beside 100 0.075. Groups above the tile gain nothing (5000 copies).
struct RefineShape {
  uint32_t block, cap, small;
};
constexpr int REFINE_SHAPES = 4;
constexpr RefineShape REFINE_SHAPE[REFINE_SHAPES] = {
    {128, 1024, 384}, {256, 2048, 512}, {256, 4096, 2048}, {256, 1024, 512}};
constexpr uint32_t REFINE_MIN_NOMINAL = 256;  // least window and least small (buffer sizing)
constexpr uint32_t REFINE_HALF_SHARE = 12;

// Names of groups. A name may be any rank inside the group's SA interval:
// intervals are disjoint and ordered, so such names respect the order of
// the suffixes, and a singleton's only choice is its rank. NAMES_HEAD is the
// paper's rule (Algorithm 5/6: the interval start, r + (subgroup start -
// group start)); NAMES_RETAIN keeps a parent's name in the subgroup whose
// interval contains it and gives every other subgroup the middle of its
// interval, so a majority subgroup keeps its name and fewer ISA entries
// change per round.
enum NamingRule : uint32_t { NAMES_HEAD = 0, NAMES_RETAIN = 1 };
constexpr uint32_t NO_NAME = 0xFFFFFFFFu;

struct ClassifyArgs {
  uint32_t *gstart;         // G entries written by this round; entry G set here
  uint32_t *gname;          // names: final for refine groups, set here for rename groups
  const uint32_t *ghead;    // head rank of every group
  const uint32_t *gold;     // parent names of the rename groups
  uint32_t naming;          // NamingRule
  uint32_t *lg, *loff, *lbase, *lold;  // large groups: index, start in the large
                                       // list, head - start, name
  uint32_t *tfirst;         // first group of each refine tile (tiles + 1 entries)
  uint32_t nominal, small;  // refine tile window; the largest small group
  uint32_t cap;             // items one tile can hold: rc.mid counts those of groups in (small, cap]
  uint32_t max_groups;      // upper bound of G (buffer capacity)
  uint32_t max_tiles;       // upper bound of tiles (buffer capacity - 1)
  Ctrl *ctrl;               // reads rc.m_s + rc.m_l, rc.g_s + rc.g_l; adds to rc.large
  const RoundState *rs;     // device-driven rounds: nothing once the loop ended (else NULL)
};
cudaError_t launch_classify(const ClassifyArgs &a, int num_sms, cudaStream_t stream);

// keys[j] = (k << W) | r2 for the j-th item of the large groups, k = large
// group ordinal; vals[j] = gapped position. With a = 3 or 4 (a-tuples of
// names per round) instead keys[j] = the later partners (r3, or
// (r3 << W) | r4), vals[j] = j, and both keys are also kept by item in the
// stashes for k_wide_rekey / k_wide_finish.
struct GatherLargeArgs {
  const uint64_t *act;
  const uint32_t *gstart;
  const uint32_t *lg, *loff;
  uint32_t mL, GL;
  uint32_t h, W;
  uint32_t mult;            // a: 2, 3 or 4
  const uint32_t *isa;
  uint64_t isa_len;
  uint64_t *keys;
  uint32_t *vals;
  uint64_t *key1_stash;     // a > 2: (k << W) | r2 by item
  uint64_t *sec_stash;      // a > 2: later partners by item
  // Device-driven rounds: mL, GL and h from the round state (mL above then
  // bounds the grid only). NULL: the fields above.
  const RoundState *rs;
  uint32_t grid_cap;        // at most this many blocks (grid-stride; 0: one item per thread)
};
cudaError_t launch_gather_large(const GatherLargeArgs &a, cudaStream_t stream);

// The two steps between and after the sorts of an a-tuple round (a > 2).
// rekey: (ka, va)[x] = (key1_stash[j], j) for j = plan->vfinal[x].
// finish: plan->vfinal[y] = gapped position of item j = plan->vfinal[y];
// the other key buffer (kb if the result is in ka, else ka) gets
// sec_stash[j] at y.
struct WideArgs {
  const SortPlan *plan;
  uint32_t m;               // items in the active list (bounds guard)
  uint32_t mL, GL, W;
  const uint64_t *act;
  const uint32_t *gstart;
  const uint32_t *lg, *loff;
  const uint64_t *key1_stash, *sec_stash;
  uint64_t *ka, *kb;
  uint32_t *va;
  Ctrl *ctrl;
};
cudaError_t launch_wide_rekey(const WideArgs &a, cudaStream_t stream);
cudaError_t launch_wide_finish(const WideArgs &a, cudaStream_t stream);

struct RefineArgs {
  const uint64_t *act;      // current active list (g << 32) | i'
  const uint32_t *gstart;   // G + 1 entries
  const uint32_t *gname;
  const uint32_t *ghead;    // head rank of each group
  uint32_t naming;          // NamingRule
  const uint32_t *tfirst;   // tiles + 1 entries
  uint32_t shape;           // index into REFINE_SHAPE
  uint32_t small;           // largest small group (as classified)
  uint32_t m, G, tiles;
  uint32_t h, W;
  uint32_t mult;            // a: names of i' + h .. i' + (a-1)h are ranked (2, 3, 4)
  const uint32_t *isa;      // read only (updates are deferred)
  uint64_t isa_len;
  uint32_t N;
  uint32_t *sa;             // written with indices local to each text
  const uint32_t *seg_off;  // S + 1 ungapped offsets
  uint32_t S;
  uint64_t *act_out;
  uint32_t *gstart_out, *gname_out, *ghead_out;
  uint64_t *upd;            // (new << 32) | i' for every changed name
  Ctrl *ctrl;               // rc.m_s / rc.g_s / rc.upd reserve the outputs
  // Device-driven rounds: tiles and h from the round state (tiles above
  // then bounds the grid only). NULL: the fields above.
  const RoundState *rs;
  uint32_t grid_cap;        // at most this many blocks, each looping over tiles (0: one per tile)
};
cudaError_t launch_refine(const RefineArgs &a, cudaStream_t stream);

// ISA[i'] = gname[g] for the entries act[*lo, *lo + *count) whose group
// name differs from their parent's (the rename's survivors, or a bucketed
// copy of them); *count <= max_count. Blocks take consecutive chunks in
// launch order.
// translated (host-driven): the entries are (name << 32) | i' of a
// translating bucket pass, all to be written, and *count their number.
// Device-driven rounds (rs): nothing when rs->mL = 0; with rs->bucket_surv
// the entries are the translated bucketed[0, *bucketed_count) instead.
// grid_cap: at most this many blocks (0: one per chunk).
cudaError_t launch_apply_names(const uint64_t *act, const uint32_t *lo, const uint32_t *count,
                               uint32_t max_count, const uint32_t *gname, const uint32_t *gold,
                               uint32_t *isa, uint64_t isa_len, cudaStream_t stream,
                               uint32_t translated = 0, const uint64_t *bucketed = nullptr,
                               const uint32_t *zero = nullptr,
                               const uint32_t *bucketed_count = nullptr,
                               const RoundState *rs = nullptr, uint32_t grid_cap = 0);

// ISA[i'] = new for the min(ctrl->rc.upd, max_upd) queued updates; blocks
// take consecutive chunks in launch order. Device-driven rounds (rs): the
// updates are bucketed[...] when rs->bucket_upd.
cudaError_t launch_scatter_updates(const uint64_t *upd, uint32_t max_upd, uint32_t *isa,
                                   uint64_t isa_len, Ctrl *ctrl, cudaStream_t stream,
                                   const uint64_t *bucketed = nullptr,
                                   const RoundState *rs = nullptr, uint32_t grid_cap = 0);

// ISA[i'] = name for entries[0, min(*count, max_count)) = (name << 32) | i',
// by at most grid_cap blocks.
cudaError_t launch_write_entries(const uint64_t *entries, const uint32_t *count,
                                 uint32_t max_count, uint32_t *isa, uint64_t isa_len,
                                 uint32_t *tile_ctr, uint32_t grid_cap, cudaStream_t stream);

// ---- device-driven rounds (k_rounds.cu) ------------------------------------
// Look-back epochs one device-driven round may use (its launches take the
// offsets 0 .. ROUND_EPOCHS - 1 from the round state's base).
constexpr uint32_t ROUND_EPOCHS = 16;
struct RoundBeginArgs {
  Ctrl *ctrl;               // ctrl->rs, ctrl->rc, ctrl->rec, ctrl->tile_ctr
  uint32_t *hist;           // MAX_PASSES * 256 digit histograms of the large-group sort
  uint32_t W;               // bits of a partner name
  uint32_t nominal;         // refine window (tiles = ceil(m / nominal))
  uint32_t bucket_min;      // discard threshold of the ISA writes
  uint32_t N;               // characters (h never exceeds it)
  // If-nodes of this round: large-group sort, its rename, bucketing of the
  // queued updates, bucketing of the large groups' ISA entries.
  cudaGraphConditionalHandle if_sort, if_rename, if_bucket_upd, if_bucket_surv;
};
cudaError_t launch_round_begin(const RoundBeginArgs &a, cudaStream_t stream);
// Sets `loop` to 1 while suffixes are active and no error was raised.
cudaError_t launch_round_end(const Ctrl *c, cudaGraphConditionalHandle loop, cudaStream_t stream);

// ---- group order after round 0 (k_reorder.cu) -------------------------------
// One line of marks: 7 words of bits and their predecessors' count.
constexpr uint32_t RANK_LINE_BITS = 224;
constexpr uint64_t rank_lines(uint64_t positions) { return positions / RANK_LINE_BITS + 1; }
// Words of `sums` for a build of this many positions and at most N / 2 groups.
constexpr uint64_t rank_sums_words(uint64_t positions, uint64_t groups) {
  return (rank_lines(positions) > groups ? rank_lines(positions) : groups) / 2048 + 1;
}
struct RegroupArgs {
  uint32_t G, m;            // groups and entries of the list
  uint32_t positions;       // gapped positions (N + S)
  const uint64_t *act_in;   // entries in the old order
  const uint32_t *gstart_in, *gname_in, *ghead_in;  // G + 1, G, G entries
  uint32_t *lines;          // rank_lines(positions) * 8 words
  uint32_t *sums;           // rank_sums_words(positions, G) words
  uint4 *info;              // G records (start, size, name, head rank) in the new order
  uint64_t *act_out;        // entries (x << 32) | i' in the new order
  uint32_t *gstart_out, *gname_out, *ghead_out;     // G + 1, G, G entries
  Ctrl *ctrl;               // rc becomes (m, G) of the refine
};
// info[x] = the group with the x-th smallest first position.
cudaError_t launch_group_rank(const RegroupArgs &a, int num_sms, cudaStream_t stream);
// The tables and entries of the new order from info.
cudaError_t launch_regroup(const RegroupArgs &a, cudaStream_t stream);

// ---- position bucketing of ISA writes (k_bucket.cu) ------------------------
constexpr uint32_t BUCKET_BLOCKS_MAX = 1024;
struct BucketArgs {
  const uint64_t *in;     // entries (x << 32) | i'
  const uint32_t *lo;     // device word: first entry (NULL: 0)
  const uint32_t *count;  // device word: number of entries
  const uint32_t *only_if;  // device word: nothing is done when it is 0 (NULL: always)
  uint32_t max_count;     // capacity of `in` past *lo and of `out`
  uint32_t shift;         // bucket of an entry: min(i' >> shift, 255)
  uint32_t blocks;        // partition blocks (<= BUCKET_BLOCKS_MAX)
  uint32_t *counts;       // blocks x 256 words: counts, then run starts
  uint64_t *out;          // entries grouped by bucket
  // Translation (the rename's survivors, entries (g << 32) | i'): when
  // gname is set, an entry whose group's name equals its parent's (gold) is
  // dropped and the others are written as (gname[g] << 32) | i', so that
  // the ISA writes need no group lookups; the number written goes to
  // *total_out. Entries come in group order, so these lookups are nearly
  // sequential here and would be random after the partition.
  const uint32_t *gname, *gold;
  uint32_t *total_out;
};
cudaError_t launch_bucket_count(const BucketArgs &a, cudaStream_t stream);
cudaError_t launch_bucket_offsets(const BucketArgs &a, cudaStream_t stream);
cudaError_t launch_bucket_scatter(const BucketArgs &a, cudaStream_t stream);

// ---- output (k_gather.cu) ------------------------------------------------
// isa_out[p] = isa[p + s] - off_s for text s (single text: a copy).
cudaError_t launch_isa_to_local(const uint32_t *isa, uint32_t *isa_out, uint32_t N,
                                const uint32_t *seg_off, uint32_t S, cudaStream_t stream);

}  // namespace gbsa
