// Step A0 — alphabet of the input: a histogram of the 256 byte values, from
// which the host derives sigma, an order-preserving dense code and the bits
// per character b = ceil(log2 sigma). It generalises the character pairs of
// the initial triples (Section 2.1, Algorithm 1): the initial names are
// built from as many dense codes as fit one 64-bit key.
//
// The block that finishes last turns the counts into the dense codes on the
// device and writes the counts to the host's pinned buffer, so that neither
// an upload of the codes nor a copy kernel of its own stands on a small
// text's critical path.
//
// The counts say nothing of repeats (copies of a block, words), which make
// buckets of equal key bits large however many digits are sorted. So a few more
// blocks each draw 512 positions, sort the prefixes there and count, for 1 to
// SAMPLE_CHARS characters, the pairs and triples that agree in them: the mean
// bucket size and its spread, as they are. They work beside the counting
// blocks, on bytes, which need no codes: +2 us beside 300 000 characters,
// nothing from 2^22 on. (One block with 1024 positions, twice the pairs of two:
// +11 and +7 us; as a step of the last block, on codes, +18.)
//
// Bound: HBM read of n bytes; 16-byte vector loads, per-warp privatised
// shared-memory counters, one global atomic per bin and block.
#include <algorithm>

#include "launch.h"

namespace gbsa {

constexpr int HIST_BLOCK = 512;
constexpr int HIST_COPIES = HIST_BLOCK / 32;  // one private histogram per warp
// Texts of at most this many characters (two bits) are modelled by their grams:
// a block that meets no more stops (5 us of a batch of DNA).
constexpr int SAMPLE_MIN_SIGMA = 4;
static_assert(SAMPLE_KEYS == HIST_BLOCK && SAMPLE_CHARS <= HIST_COPIES,
              "a key to a thread, a count to a warp");

// The 8 characters at pos, first character on top, zeros from `end` on.
__device__ __forceinline__ uint64_t prefix_at(const uint8_t *text, uint64_t n, uint64_t pos,
                                              uint64_t end) {
  const uintptr_t at = (uintptr_t)(text + pos), a0 = at & ~(uintptr_t)7;
  const uint32_t skip = (uint32_t)(at - a0) * 8u;
  uint64_t key = 0;
  if (a0 >= (uintptr_t)text && a0 + 16 <= (uintptr_t)(text + n)) {
    const unsigned long long *w = reinterpret_cast<const unsigned long long *>(a0);
    const uint64_t w0 = __ldg(w), w1 = __ldg(w + 1);
    const uint64_t v = skip ? (w0 >> skip) | (w1 << (64 - skip)) : w0;
    key = ((uint64_t)__byte_perm((uint32_t)v, 0u, 0x0123) << 32) |
          __byte_perm((uint32_t)(v >> 32), 0u, 0x0123);
  } else {  // the text's first and last bytes
    for (uint32_t i = 0; i < 8; ++i) key = (key << 8) | (pos + i < n ? text[pos + i] : 0u);
  }
  return end - pos < 8 ? key & (~0ull << (8 * (8 - (end - pos)))) : key;
}

// One block: a prefix per thread below its text's number (textbits), sorted
// into keys[0, SAMPLE_KEYS); false, and none, when they start with at most
// SAMPLE_MIN_SIGMA characters. `room` words of shared memory follow the keys.
__device__ __forceinline__ bool sample_prefixes(const AlphabetArgs &a, uint64_t *keys,
                                                uint32_t room, uint32_t textbits) {
  const uint32_t tid = threadIdx.x, total = a.sample_blocks * SAMPLE_KEYS;
  const uint32_t *offsets = a.offsets;
  if (a.S > 1 && a.S < room) {  // searched in shared memory
    uint32_t *copy = reinterpret_cast<uint32_t *>(keys + SAMPLE_KEYS);
    for (uint32_t i = tid; i <= a.S; i += HIST_BLOCK) copy[i] = a.offsets[i];
    offsets = copy;
    __syncthreads();
  }
  // Evenly spread, shifted at random: a period of the text must not show.
  const uint32_t i = tid * a.sample_blocks + blockIdx.x;
  uint32_t r = i * 0x9E3779B9u;
  r = (r ^ (r >> 16)) * 0x85EBCA6Bu;
  r ^= r >> 13;
  const uint64_t x = ((uint64_t)i * a.n + (((uint64_t)r * a.n) >> 32)) / total;
  uint64_t end = a.n, text = 0;
  if (a.S > 1) {
    uint32_t lo = 0, hi = a.S - 1;  // the last text with an offset <= x
    while (lo < hi) {
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (offsets[mid] <= x)
        lo = mid;
      else
        hi = mid - 1;
    }
    end = offsets[lo + 1];
    text = (uint64_t)lo << (64 - textbits);
  }
  const uint64_t prefix = prefix_at(a.text, a.n, x, end);
  uint64_t key = text | (prefix >> textbits);
  // The characters that start a prefix: a set of 256 bits.
  __shared__ uint32_t s_seen[RADIX / 32];
  if (tid < RADIX / 32) s_seen[tid] = 0u;
  __syncthreads();
  const uint32_t c = (uint32_t)(prefix >> 56);
  for (uint32_t w = 0; w < RADIX / 32; ++w) {
    const uint32_t in = __reduce_or_sync(0xffffffffu, c / 32 == w ? 1u << (c & 31) : 0u);
    if ((tid & 31) == 0 && in) atomicOr(&s_seen[w], in);
  }
  __syncthreads();
  int seen = 0;
  for (uint32_t w = 0; w < RADIX / 32; ++w) seen += __popc(s_seen[w]);
  if (seen <= SAMPLE_MIN_SIGMA) return false;  // the same for every thread
  // Bitonic: steps inside a warp by shuffles, the others in shared memory.
  for (uint32_t k = 2; k <= SAMPLE_KEYS; k <<= 1) {
    for (uint32_t j = k >> 1; j > 0; j >>= 1) {
      uint64_t q;
      if (j >= 32) {
        __syncthreads();  // the step before is read
        keys[tid] = key;
        __syncthreads();
        q = keys[tid ^ j];
      } else {
        q = __shfl_xor_sync(0xffffffffu, key, j);
      }
      const bool least = ((tid & j) == 0) == ((tid & k) == 0);
      key = (q < key) == least ? q : key;
    }
  }
  __syncthreads();
  keys[tid] = key;
  __syncthreads();
  return true;
}

// One warp: adds the pairs and triples of the sorted keys that agree in their
// top `bits`. A key agrees with every one from its group's head on.
__device__ __forceinline__ void count_agreeing(const uint64_t *keys, uint32_t bits, uint32_t *pairs,
                                               unsigned long long *triples) {
  const uint32_t lane = threadIdx.x & 31, R = 64 - bits;
  uint32_t first = 0, p = 0, t = 0;  // the last head so far; p, t below 2^32 in all
#pragma unroll 4
  for (uint32_t i0 = 0; i0 < SAMPLE_KEYS; i0 += 32) {
    const uint32_t i = i0 + lane;
    const bool head = i == 0 || ((keys[i] ^ keys[i - 1]) >> R) != 0;
    const uint32_t H = __ballot_sync(0xffffffffu, head), m = H & (lanemask_lt() | (1u << lane));
    const uint32_t before = i - (m ? i0 + 31 - __clz(m) : first);
    p += before;
    t += before * (before - 1) / 2;
    if (H) first = i0 + 31 - __clz(H);
  }
  p = __reduce_add_sync(0xffffffffu, p);
  t = __reduce_add_sync(0xffffffffu, t);
  if (lane == 0) {
    atomicAdd(pairs, p);
    atomicAdd(triples, (unsigned long long)t);
  }
}

// Block `block` of `blocks` adds its share of the text to the counts.
__device__ __forceinline__ void count_bytes(const AlphabetArgs &a, uint32_t (*s_hist)[RADIX],
                                            uint32_t block, uint32_t blocks) {
  const uint8_t *__restrict__ text = a.text;
  const uint64_t n = a.n;
  for (int x = threadIdx.x; x < HIST_COPIES * RADIX; x += HIST_BLOCK) (&s_hist[0][0])[x] = 0;
  __syncthreads();
  uint32_t *mine = s_hist[threadIdx.x >> 5];
  // Aligned body with 16-byte loads, then the ragged head and tail bytes.
  const uintptr_t addr = (uintptr_t)text;
  uint64_t head = (16 - (addr & 15)) & 15;
  if (head > n) head = n;
  const uint64_t body = (n - head) / 16;
  const uint4 *vec = (const uint4 *)(text + head);
  const uint64_t stride = (uint64_t)blocks * HIST_BLOCK;
  for (uint64_t v = (uint64_t)block * HIST_BLOCK + threadIdx.x; v < body; v += stride) {
    uint4 q = __ldg(vec + v);
    uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
      for (int s = 0; s < 32; s += 8) atomicAdd(&mine[(w[k] >> s) & 255u], 1u);
    }
  }
  const uint64_t tail0 = head + body * 16;
  const uint64_t gtid = (uint64_t)block * HIST_BLOCK + threadIdx.x;
  if (gtid < head) atomicAdd(&mine[text[gtid]], 1u);
  if (gtid < n - tail0) atomicAdd(&mine[text[tail0 + gtid]], 1u);
  __syncthreads();
  for (int d = threadIdx.x; d < RADIX; d += HIST_BLOCK) {
    uint32_t s = 0;
#pragma unroll
    for (int c = 0; c < HIST_COPIES; ++c) s += s_hist[c][d];
    if (s) atomicAdd(&a.hist[d], s);
  }
}

__global__ void __launch_bounds__(HIST_BLOCK, 4) k_byte_histogram(AlphabetArgs a) {
  __shared__ __align__(16) uint32_t s_hist[HIST_COPIES][RADIX];
  uint32_t *hist = a.hist;
  const uint64_t n = a.n;
  if (blockIdx.x < a.sample_blocks) {
    uint64_t *keys = reinterpret_cast<uint64_t *>(s_hist);
    const uint32_t textbits = a.S > 1 ? 32 - __clz(a.S - 1) : 0;
    const bool taken = sample_prefixes(a, keys, HIST_COPIES * RADIX - 2 * SAMPLE_KEYS, textbits);
    KeySample *out = reinterpret_cast<KeySample *>(hist + RADIX);
    const uint32_t w = threadIdx.x >> 5, bits = textbits + 8 * (w + 1);
    if (taken && w < SAMPLE_CHARS && bits <= 64)
      count_agreeing(keys, bits, &out->pairs[w], &out->triples[w]);
  } else {
    count_bytes(a, s_hist, blockIdx.x - a.sample_blocks, gridDim.x - a.sample_blocks);
  }
  __shared__ uint32_t s_last, s_tmp[HIST_COPIES + 1];
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(a.done, 1u) + 1u == gridDim.x ? 1u : 0u;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const uint32_t d = threadIdx.x;
  const uint32_t c = d < RADIX ? load_volatile_u32(hist + d) : 0u;
  const bool sampled = a.sample_blocks && a.host && d < sizeof(KeySample) / 4;
  const uint32_t w = sampled ? load_volatile_u32(hist + RADIX + d) : 0u;
  uint32_t sigma;
  const uint32_t code = block_exclusive<HIST_BLOCK>(c ? 1u : 0u, OpAdd(), 0u, s_tmp, sigma);
  if (d < RADIX) {
    a.code[d] = (uint8_t)code;
    if (a.host) a.host[d] = c;
  }
  if (sampled) a.host[RADIX + d] = w;
  if (d < 2 && a.seg_off) a.seg_off[d] = d ? (uint32_t)n : 0u;
  if (a.host) report_to_host(a.host_flag);
}

cudaError_t launch_byte_histogram(const AlphabetArgs &a, int num_sms, cudaStream_t stream) {
  if (a.n == 0) return cudaSuccess;
  uint64_t want = (a.n / 16 + HIST_BLOCK - 1) / HIST_BLOCK;
  if (a.sample_blocks > SAMPLE_BLOCKS_MAX) return cudaErrorInvalidValue;
  uint64_t cap = std::max<uint64_t>(1, (uint64_t)num_sms * 4 - a.sample_blocks);  // all resident
  unsigned grid = (unsigned)(want < 1 ? 1 : (want > cap ? cap : want));
  k_byte_histogram<<<grid + a.sample_blocks, HIST_BLOCK, 0, stream>>>(a);
  return cudaGetLastError();
}

}  // namespace gbsa
