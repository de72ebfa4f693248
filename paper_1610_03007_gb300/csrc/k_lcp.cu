// LCP array from the suffix array: a direct consumer of SA named as future
// work at the end of the paper (Section 3). lcp[0] = 0 and, for j >= 1,
// lcp[j] is the longest common prefix of the suffixes SA[j-1] and SA[j]
// (Section 2's suffix order).
//
// Most texts' neighbours in the suffix array agree in a few characters only
// (about log n of the alphabet's size). For those the pairs are compared
// directly: a thread reads 32 aligned bytes at its own suffix, takes its
// neighbour's from the lane before, and has 16 characters settled by one
// round of random reads instead of the six passes below:
//
//   k_lcp_sample: compares up to 2^15 evenly spaced pairs; many long ones, or
//                 one longer than LCP_REST_MAX, send the text to the permuted
//                 form (the kernels of the other form return at once: the
//                 choice is made on the device, in stream order)
//   k_lcp_direct: every pair up to LCP_CAP characters; longer ones listed
//   k_lcp_rest:   a warp per listed pair, 256 characters a step; too many or
//                 too long ones also send the text to the permuted form
//
// Texts of up to LCP_SMALL characters need no other form. Bound: one or two
// random sectors per pair. Measured on 48 M characters of prose (mean LCP 9)
// against the permuted form: 2.30 -> 0.46 ms.
//
// Permuted form of Kasai et al.'s linear-time algorithm (Kasai, Lee,
// Arimura, Arikawa, Park, CPM 2001; permuted LCP of Karkkainen, Manzini and
// Puglisi, CPM 2009): with Phi[SA[j]] = SA[j-1], the permuted array
// PLCP[i] = lcp(i, Phi[i]) satisfies PLCP[i] >= PLCP[i-1] - 1, so a scan in
// text order extends each value from the previous one minus one.
//
//   k_lcp_phi:    Phi[SA[j]] = SA[j-1] (j >= 1); Phi[SA[0]] = n (none).
//                 From 2^20 characters on, the writes are first grouped by
//                 position (k_lcp_entries builds (Phi value, SA[j]) pairs,
//                 the position bucketing of the ISA writes partitions them
//                 into 256 position ranges, k_lcp_apply writes them range
//                 by range), so the Phi being written stays in L2 instead of
//                 each 4-byte write costing a sector read and write.
//   k_lcp_plcp:   the text is cut into chunks of LCP_CHUNK positions, one
//                 thread per chunk scanning it in order; a chunk's first
//                 value is extended from 0, every later one from the
//                 previous minus one. Characters are compared 8 at a time
//                 (two funnel-shifted aligned 32-bit windows per suffix).
//   k_lcp_gather: lcp[j] = PLCP[SA[j]].
// Work: 2n character comparisons plus, per chunk, the first value's LCP.
// Bound: HBM / latency. Algorithmic bytes per position: 8 (Phi: read SA,
// random write) + 10 (PLCP: read Phi, write PLCP, one sequential and one
// random text byte) + 12 (gather: read SA, random read of PLCP, write).
#include <algorithm>

#include "../../include/gbsa.h"
#include "launch.h"

#define GBSA_API extern "C" __attribute__((visibility("default")))

namespace gbsa {

constexpr uint32_t LCP_CHUNK = 256;
constexpr uint32_t LCP_CAP = 64;          // characters a thread compares itself
constexpr uint32_t LCP_REST_MAX = 4096;   // and a warp, in texts above LCP_SMALL
constexpr uint32_t LCP_SMALL = 1u << 16;
constexpr uint32_t LCP_SAMPLES = 1u << 15;
constexpr uint32_t LCP_LISTED = 64;       // at most one pair in this many is listed

// Device words that choose the form (zeroed first).
struct LcpFlags {
  uint32_t permuted;  // k_lcp_rest gave up
  uint32_t samples, longer, too_long;  // k_lcp_sample: pairs, above LCP_CAP, above LCP_REST_MAX
  uint32_t listed;    // pairs k_lcp_direct listed
  uint32_t count;     // entries of the permuted form: n, or 0 when it is not taken
};

// True once the permuted form is chosen; the same for every thread of a
// kernel after the ones that write the flags.
__device__ __forceinline__ bool lcp_permuted(const LcpFlags *f) {
  return f->permuted || f->too_long || f->longer * LCP_LISTED > f->samples;
}

__global__ void __launch_bounds__(256) k_lcp_phi(const uint32_t *__restrict__ sa, uint64_t n,
                                                 uint32_t *__restrict__ phi, const LcpFlags *f) {
  if (!lcp_permuted(f)) return;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride) {
    const uint32_t s = sa[j];
    if (s < n) phi[s] = j ? sa[j - 1] : (uint32_t)n;
  }
}

// Position-bucketed Phi writes: e[j] = (Phi value << 32) | SA[j].
__global__ void __launch_bounds__(256) k_lcp_entries(const uint32_t *__restrict__ sa, uint64_t n,
                                                     uint64_t *__restrict__ e, const LcpFlags *f) {
  if (!lcp_permuted(f)) return;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride)
    e[j] = ((uint64_t)(j ? sa[j - 1] : (uint32_t)n) << 32) | sa[j];
}

__global__ void k_lcp_set_count(LcpFlags *f, uint32_t n) { f->count = lcp_permuted(f) ? n : 0u; }

// Phi[low] = high for the bucketed entries; blocks take consecutive chunks
// of LCP_APPLY entries in launch order, so the positions written stay in a
// narrow window.
constexpr int LCP_APPLY_ITEMS = 8;
constexpr uint32_t LCP_APPLY = 256 * LCP_APPLY_ITEMS;

__global__ void __launch_bounds__(256) k_lcp_apply(const uint64_t *__restrict__ e, uint64_t n,
                                                   uint32_t *__restrict__ phi, const LcpFlags *f) {
  if (!lcp_permuted(f)) return;
  const uint64_t c0 = (uint64_t)blockIdx.x * LCP_APPLY;
  uint64_t u[LCP_APPLY_ITEMS];
#pragma unroll
  for (int k = 0; k < LCP_APPLY_ITEMS; ++k) {
    const uint64_t x = c0 + (uint64_t)k * 256 + threadIdx.x;
    u[k] = x < n ? e[x] : ~0ull;
  }
#pragma unroll
  for (int k = 0; k < LCP_APPLY_ITEMS; ++k) {
    const uint32_t s = (uint32_t)u[k];
    if (u[k] != ~0ull && s < n) phi[s] = (uint32_t)(u[k] >> 32);
  }
}

// Bytes [x, x + 8) of T as two little-endian words; T 4-byte aligned and
// x + 12 <= n (the three aligned words read lie inside the text).
__device__ __forceinline__ void load8(const uint8_t *T, uint64_t x, uint32_t &lo, uint32_t &hi) {
  const uint32_t *w = reinterpret_cast<const uint32_t *>(T + (x & ~3ull));
  const uint32_t sh = (uint32_t)(x & 3u) * 8u;
  const uint32_t w0 = __ldg(w), w1 = __ldg(w + 1), w2 = __ldg(w + 2);
  lo = __funnelshift_r(w0, w1, sh);
  hi = __funnelshift_r(w1, w2, sh);
}

// lcp(i, p) given that the first h characters are known equal.
__device__ __forceinline__ uint64_t lcp_extend(const uint8_t *T, uint64_t n, uint64_t i,
                                               uint64_t p, uint64_t h, bool words) {
  const uint64_t lim = n - (i > p ? i : p);  // the shorter suffix's length
  while (h < lim) {
    if (words && h + 12 <= lim) {
      uint32_t a0, a1, b0, b1;
      load8(T, i + h, a0, a1);
      load8(T, p + h, b0, b1);
      const uint32_t x0 = a0 ^ b0, x1 = a1 ^ b1;
      if (x0) return h + (uint32_t)(__ffs(x0) - 1) / 8u;
      if (x1) return h + 4 + (uint32_t)(__ffs(x1) - 1) / 8u;
      h += 8;
    } else {
      if (T[i + h] != T[p + h]) return h;
      ++h;
    }
  }
  return h;
}

__global__ void __launch_bounds__(256) k_lcp_plcp(const uint8_t *__restrict__ T, uint64_t n,
                                                  const uint32_t *__restrict__ phi,
                                                  uint32_t *__restrict__ plcp, const LcpFlags *f) {
  if (!lcp_permuted(f)) return;
  const bool words = (((uintptr_t)T) & 3u) == 0;
  const uint64_t chunks = (n + LCP_CHUNK - 1) / LCP_CHUNK;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t c = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; c < chunks; c += stride) {
    const uint64_t i0 = c * LCP_CHUNK, i1 = min(n, i0 + LCP_CHUNK);
    uint64_t h = 0;
    for (uint64_t i = i0; i < i1; ++i) {
      const uint32_t p = phi[i];
      if (p >= n) {  // the smallest suffix (or not a suffix array): nothing before it
        h = 0;
        plcp[i] = 0;
        continue;
      }
      h = lcp_extend(T, n, i, p, h, words);
      plcp[i] = (uint32_t)h;
      if (h) --h;
    }
  }
}

__global__ void __launch_bounds__(256) k_lcp_gather(const uint32_t *__restrict__ sa, uint64_t n,
                                                    const uint32_t *__restrict__ plcp,
                                                    uint32_t *__restrict__ lcp, const LcpFlags *f) {
  if (!lcp_permuted(f)) return;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride) {
    const uint32_t s = sa[j];
    lcp[j] = (j == 0 || s >= n) ? 0u : plcp[s];
  }
}

// ---- the direct form --------------------------------------------------------

// Characters [x, x + 16) of T as four little-endian words, zeros past the
// end; T 16-byte aligned, x < n.
__device__ __forceinline__ void load16(const uint8_t *T, uint64_t n, uint64_t x, uint32_t (&w)[4]) {
  const uint64_t a = x & ~15ull;
  uint32_t v[8];
  if (a + 32 <= n) {
    const uint4 p = __ldg(reinterpret_cast<const uint4 *>(T + a));
    const uint4 q = __ldg(reinterpret_cast<const uint4 *>(T + a + 16));
    v[0] = p.x, v[1] = p.y, v[2] = p.z, v[3] = p.w;
    v[4] = q.x, v[5] = q.y, v[6] = q.z, v[7] = q.w;
  } else {  // the last characters of the text
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      uint32_t y = 0;
      for (int c = 3; c >= 0; --c) y = (y << 8) | (a + 4 * i + c < n ? T[a + 4 * i + c] : 0u);
      v[i] = y;
    }
  }
  const uint32_t skip = (uint32_t)(x & 15u) >> 2, sh = (uint32_t)(x & 3u) * 8u;
#pragma unroll
  for (int i = 0; i < 7; ++i) v[i] = (skip & 2u) ? (i + 2 < 8 ? v[i + 2] : 0u) : v[i];
#pragma unroll
  for (int i = 0; i < 5; ++i) v[i] = (skip & 1u) ? v[i + 1] : v[i];
#pragma unroll
  for (int i = 0; i < 4; ++i) w[i] = __funnelshift_r(v[i], v[i + 1], sh);
}

__device__ __forceinline__ uint32_t first_difference(const uint32_t (&a)[4], const uint32_t (&b)[4]) {
  uint32_t at = 16;
#pragma unroll
  for (int i = 3; i >= 0; --i) {
    const uint32_t x = a[i] ^ b[i];
    if (x) at = 4 * i + (uint32_t)(__ffs(x) - 1) / 8u;
  }
  return at;
}

// lcp(i, p) by a warp (every lane gets it), the first h characters known
// equal; stops at `most` or a little later.
__device__ __forceinline__ uint64_t lcp_warp(const uint8_t *T, uint64_t n, uint64_t i, uint64_t p,
                                             uint64_t h, uint64_t most) {
  const int lane = threadIdx.x & 31;
  const uint64_t lim = n - (i > p ? i : p);
  while (h < lim && h < most) {
    const uint64_t at = h + 8 * lane;
    uint32_t equal = 8;  // equal characters of this lane's eight
    if (at + 12 <= lim) {
      uint32_t a0, a1, b0, b1;
      load8(T, i + at, a0, a1);
      load8(T, p + at, b0, b1);
      if (a0 != b0)
        equal = (uint32_t)(__ffs(a0 ^ b0) - 1) / 8u;
      else if (a1 != b1)
        equal = 4 + (uint32_t)(__ffs(a1 ^ b1) - 1) / 8u;
    } else {
      equal = 0;
      while (equal < 8 && at + equal < lim && T[i + at + equal] == T[p + at + equal]) ++equal;
    }
    const uint32_t stop = __ballot_sync(0xffffffffu, equal < 8);
    if (stop) {
      const int first = __ffs(stop) - 1;
      return h + 8 * first + __shfl_sync(0xffffffffu, equal, first);
    }
    h += 256;
  }
  return h < lim ? h : lim;
}

__global__ void __launch_bounds__(256) k_lcp_sample(const uint8_t *__restrict__ T, uint64_t n,
                                                    const uint32_t *__restrict__ sa, LcpFlags *f) {
  const uint32_t k = blockIdx.x * 8 + (threadIdx.x >> 5);  // this warp's sample
  const uint64_t j = 1 + (uint64_t)k * (n - 1) / LCP_SAMPLES;
  const uint64_t i = sa[j], p = sa[j - 1];
  if (i >= n || p >= n) return;  // not a suffix array
  const uint64_t h = lcp_warp(T, n, i, p, 0, LCP_REST_MAX + 1);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&f->samples, 1u);
    if (h > LCP_CAP) atomicAdd(&f->longer, 1u);
    if (h > LCP_REST_MAX) atomicAdd(&f->too_long, 1u);
  }
}

// LCP_ROWS rows of 32 consecutive pairs per warp and iteration: the suffix
// before a row's first is the row before's last.
constexpr int LCP_ROWS = 4;
__global__ void __launch_bounds__(256) k_lcp_direct(const uint8_t *__restrict__ T, uint64_t n,
                                                    const uint32_t *__restrict__ sa,
                                                    uint32_t *__restrict__ lcp,
                                                    uint32_t *__restrict__ list, uint32_t cap,
                                                    LcpFlags *f) {
  if (lcp_permuted(f)) return;
  const int lane = threadIdx.x & 31;
  const uint64_t warps = (uint64_t)gridDim.x * 8;
  for (uint64_t j0 = ((uint64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * (32 * LCP_ROWS); j0 < n;
       j0 += warps * (32 * LCP_ROWS)) {
    uint32_t s[LCP_ROWS], before;
#pragma unroll
    for (int r = 0; r < LCP_ROWS; ++r) {
      const uint64_t j = j0 + 32 * r + lane;
      s[r] = j < n ? sa[j] : 0xFFFFFFFFu;
    }
    before = j0 > 0 ? sa[j0 - 1] : 0xFFFFFFFFu;
    uint32_t w[LCP_ROWS][4], pw[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int r = 0; r < LCP_ROWS; ++r) {
      if (s[r] < n)
        load16(T, n, s[r], w[r]);
      else
        w[r][0] = w[r][1] = w[r][2] = w[r][3] = 0u;
    }
    if (lane == 0 && before < n) load16(T, n, before, pw);
#pragma unroll
    for (int r = 0; r < LCP_ROWS; ++r) {
      const uint64_t j = j0 + 32 * r + lane;
      uint32_t p = __shfl_up_sync(0xffffffffu, s[r], 1), b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) b[i] = __shfl_up_sync(0xffffffffu, w[r][i], 1);
      if (lane == 0) {
        p = before;
#pragma unroll
        for (int i = 0; i < 4; ++i) b[i] = pw[i];
      }
      before = __shfl_sync(0xffffffffu, s[r], 31);  // the next row's
#pragma unroll
      for (int i = 0; i < 4; ++i) pw[i] = __shfl_sync(0xffffffffu, w[r][i], 31);
      uint64_t h = 0;
      bool more = false;
      if (j > 0 && s[r] < n && p < n) {
        const uint64_t lim = n - (s[r] > p ? s[r] : p);
        h = first_difference(w[r], b);
        more = h == 16;
        while (more && h + 12 <= lim && h < LCP_CAP) {
          uint32_t a0, a1, b0, b1;
          load8(T, s[r] + h, a0, a1);
          load8(T, p + h, b0, b1);
          const uint32_t x0 = a0 ^ b0, x1 = a1 ^ b1;
          more = !(x0 | x1);
          h += x0 ? (uint32_t)(__ffs(x0) - 1) / 8u : (x1 ? 4 + (uint32_t)(__ffs(x1) - 1) / 8u : 8u);
        }
        while (more && h < lim && h < LCP_CAP) {  // the last characters of the text
          more = T[s[r] + h] == T[p + h];
          h += more ? 1u : 0u;
        }
        if (h >= lim) {
          h = lim;
          more = false;
        }
      }
      if (j < n) lcp[j] = (uint32_t)h;
      const uint32_t L = __ballot_sync(0xffffffffu, more);
      if (L) {  // the pairs that agree in LCP_CAP characters or more
        uint32_t base = 0;
        if (lane == 0) base = atomicAdd(&f->listed, (uint32_t)__popc(L));
        base = __shfl_sync(0xffffffffu, base, 0) + __popc(L & lanemask_lt());
        if (more && base < cap) list[base] = (uint32_t)j;
      }
    }
  }
}

__global__ void __launch_bounds__(256) k_lcp_rest(const uint8_t *__restrict__ T, uint64_t n,
                                                  const uint32_t *__restrict__ sa,
                                                  uint32_t *__restrict__ lcp,
                                                  const uint32_t *__restrict__ list, uint32_t cap,
                                                  uint64_t most, LcpFlags *f) {
  if (f->too_long || f->longer * LCP_LISTED > f->samples) return;  // the sample's choice
  const uint32_t listed = f->listed;
  if (listed > cap) {
    if (threadIdx.x == 0 && blockIdx.x == 0) f->permuted = 1u;
    return;
  }
  for (uint32_t k = blockIdx.x * 8 + (threadIdx.x >> 5); k < listed; k += gridDim.x * 8) {
    const uint32_t j = list[k];
    const uint64_t h = lcp_warp(T, n, sa[j], sa[j - 1], LCP_CAP, most);
    if ((threadIdx.x & 31) == 0) {
      lcp[j] = (uint32_t)h;
      if (h >= most && h < n) f->permuted = 1u;
    }
  }
}

}  // namespace gbsa

namespace {

int lcp_sm_count() { return gbsa::device_sm_count(); }

unsigned grid_for(uint64_t units, int per_sm) {
  const uint64_t want = (units + 255) / 256, cap = (uint64_t)lcp_sm_count() * per_sm;
  return (unsigned)(want < cap ? (want ? want : 1) : cap);
}

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

constexpr uint64_t LCP_BUCKET_MIN = 1ull << 20;  // bucket the Phi writes from this size on

// Phi (4n; the direct form's list) | entries (8n; PLCP reuses its first half)
// | bucketed entries (8n) | bucket counts | the flags.
struct LcpLayout {
  size_t phi, ent, ent2, counts, count, total;
};

LcpLayout lcp_layout(uint64_t n) {
  LcpLayout L{};
  size_t o = 0;
  auto take = [&](size_t b) {
    const size_t r = o;
    o += align256(b);
    return r;
  };
  L.phi = take((size_t)n * 4);
  L.ent = take((size_t)n * 8);
  L.ent2 = take((size_t)n * 8);
  L.counts = take((size_t)gbsa::BUCKET_BLOCKS_MAX * 256 * 4);
  L.count = take(sizeof(gbsa::LcpFlags));
  L.total = o;
  return L;
}

cudaError_t launch_lcp(const uint8_t *text, uint64_t n, const uint32_t *sa, uint32_t *lcp_out,
                       uint8_t *base, const LcpLayout &L, gbsa::LcpFlags *f, cudaStream_t st) {
  uint32_t *phi = reinterpret_cast<uint32_t *>(base + L.phi);
  uint32_t *plcp = reinterpret_cast<uint32_t *>(base + L.ent);
  const uint64_t chunks = (n + gbsa::LCP_CHUNK - 1) / gbsa::LCP_CHUNK;
  cudaError_t e = cudaSuccess;
  // The direct form reads the text in aligned 16-byte words.
  const bool direct = ((uintptr_t)text & 15u) == 0, small = n <= gbsa::LCP_SMALL;
  if (direct) {
    uint32_t *list = phi;
    const uint32_t cap = (uint32_t)(small ? n : n / gbsa::LCP_LISTED);
    const uint64_t rows = (n + gbsa::LCP_ROWS - 1) / gbsa::LCP_ROWS;
    if (!small) gbsa::k_lcp_sample<<<gbsa::LCP_SAMPLES / 8, 256, 0, st>>>(text, n, sa, f);
    gbsa::k_lcp_direct<<<grid_for(rows, 8), 256, 0, st>>>(text, n, sa, lcp_out, list, cap, f);
    gbsa::k_lcp_rest<<<grid_for((uint64_t)cap * 32, 8), 256, 0, st>>>(
        text, n, sa, lcp_out, list, cap, small ? n : (uint64_t)gbsa::LCP_REST_MAX, f);
    if (small) return cudaGetLastError();
  } else {
    e = cudaMemsetAsync(&f->permuted, 1, 1, st);  // non-zero: the permuted form
    if (e != cudaSuccess) return e;
  }
  if (n >= LCP_BUCKET_MIN) {
    uint64_t *ent = reinterpret_cast<uint64_t *>(base + L.ent);
    gbsa::k_lcp_entries<<<grid_for(n, 8), 256, 0, st>>>(sa, n, ent, f);
    gbsa::k_lcp_set_count<<<1, 1, 0, st>>>(f, (uint32_t)n);
    gbsa::BucketArgs ba{};
    ba.in = ent;
    ba.lo = nullptr;
    ba.count = &f->count;
    ba.only_if = &f->count;
    ba.max_count = (uint32_t)n;
    uint32_t bits = 0;
    while (bits < 64 && (n >> bits)) ++bits;
    ba.shift = bits > 8 ? bits - 8 : 0;
    ba.blocks = std::min<uint32_t>(gbsa::BUCKET_BLOCKS_MAX, 4u * (uint32_t)lcp_sm_count());
    ba.counts = reinterpret_cast<uint32_t *>(base + L.counts);
    ba.out = reinterpret_cast<uint64_t *>(base + L.ent2);
    if ((e = gbsa::launch_bucket_count(ba, st)) == cudaSuccess &&
        (e = gbsa::launch_bucket_offsets(ba, st)) == cudaSuccess &&
        (e = gbsa::launch_bucket_scatter(ba, st)) == cudaSuccess) {
      gbsa::k_lcp_apply<<<(unsigned)((n + gbsa::LCP_APPLY - 1) / gbsa::LCP_APPLY), 256, 0, st>>>(
          ba.out, n, phi, f);
    }
  } else {
    gbsa::k_lcp_phi<<<grid_for(n, 8), 256, 0, st>>>(sa, n, phi, f);
  }
  gbsa::k_lcp_plcp<<<grid_for(chunks, 8), 256, 0, st>>>(text, n, phi, plcp, f);
  gbsa::k_lcp_gather<<<grid_for(n, 8), 256, 0, st>>>(sa, n, plcp, lcp_out, f);
  return e == cudaSuccess ? cudaGetLastError() : e;
}

}  // namespace

GBSA_API size_t sa_lcp_workspace_bytes(uint64_t n) { return lcp_layout(n).total; }

GBSA_API sa_status sa_lcp(const uint8_t *text, uint64_t n, const uint32_t *sa, uint32_t *lcp_out,
                          void *workspace, size_t ws_bytes, gbsa_stream_t stream) {
  if (n > SA_MAX_N) return SA_ERR_TOO_LARGE;
  if (n > 0 && (!text || !sa || !lcp_out)) return SA_ERR_INVALID_ARG;
  if (n == 0) return SA_OK;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t need = sa_lcp_workspace_bytes(n);
  void *ws = workspace;
  if (ws) {
    if (ws_bytes < need || ((uintptr_t)ws & 255)) return SA_ERR_INVALID_ARG;
  } else if (cudaMallocAsync(&ws, need, st) != cudaSuccess) {
    return SA_ERR_OOM;
  }
  const LcpLayout L = lcp_layout(n);
  uint8_t *base = static_cast<uint8_t *>(ws);
  gbsa::LcpFlags *f = reinterpret_cast<gbsa::LcpFlags *>(base + L.count);
  cudaError_t e = cudaMemsetAsync(f, 0, sizeof(*f), st);
  if (e == cudaSuccess) e = launch_lcp(text, n, sa, lcp_out, base, L, f, st);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (!workspace) {
    const cudaError_t f = cudaFreeAsync(ws, st);
    if (e == cudaSuccess) e = f;
  }
  return e == cudaSuccess ? SA_OK : SA_ERR_CUDA;
}
