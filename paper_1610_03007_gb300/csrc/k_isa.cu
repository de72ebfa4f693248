// ISA entries of the suffixes that are unique after round 0 (Section 2.1,
// Algorithm 5 in inverse-suffix-array form: a discarded suffix keeps its
// rank, which later rounds read as a partner name).
//
// Their ranks stand in the SA (SA_NONE at every other rank), so they need no
// queue: one pass over the SA in rank order writes ISA[SA[j]] = j. But few of
// them are ever read. A round reads ISA[i + h] for its active suffixes i
// alone, the active sets only shrink, and active suffixes lie in the repeats
// of the text; so a position is needed only if it lies some round's h after
// an active one. k_need_* keep that set as bits, one per granule of 2^shift
// positions (at most 2^26 bits, 8 MB that stay in L2 under random reads; up
// to 2^26 characters the set is exact):
//
//   k_need_mark: the granules of the active suffixes
//   k_need_plan: their translates by the offsets of the coming rounds, less
//                the granules already covered
//   k_need_collect: reads the SA and keeps the (rank, position) entries in a
//                needed granule, which are then written (bucketed by position
//                first when there are many, k_bucket.cu)
//
// Granules only add entries (a written entry is always right), so the filter
// needs no exactness. One plan covers the rounds up to NEED_OFFSET_MAX; later
// ones, which only texts with longer repeats reach, plan again per round and
// collect nothing when all is covered.
//
// Bound: random reads of the bits from L2, one sector per rank; 4 bytes of
// SA read per rank and 8 per active suffix.
#include "launch.h"

namespace gbsa {

namespace {

constexpr int IF_ITEMS = 8;
constexpr int IF_CHUNK = 256 * IF_ITEMS;

// The last text in [lo, hi] with an offset <= j.
__device__ __forceinline__ uint32_t text_of(const uint32_t *seg_off, uint32_t lo, uint32_t hi,
                                            uint32_t j) {
  while (lo < hi) {
    const uint32_t mid = (lo + hi + 1) >> 1;
    if (__ldg(seg_off + mid) <= j)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

}  // namespace

// Every final rank, directly. Blocks take consecutive chunks of ranks; the
// ranks of a text are consecutive, so the chunk's texts are found once.
__global__ void __launch_bounds__(256) k_isa_fill(const uint32_t *__restrict__ sa, uint32_t N,
                                                 const uint32_t *__restrict__ seg_off, uint32_t S,
                                                 uint32_t *isa, uint64_t isa_len) {
  __shared__ uint32_t s_seg[2];
  const uint32_t j0 = blockIdx.x * (uint32_t)IF_CHUNK;
  if (S > 1) {
    if (threadIdx.x < 2)
      s_seg[threadIdx.x] =
          segment_of(seg_off, S, threadIdx.x ? min(j0 + IF_CHUNK - 1u, N - 1u) : j0);
    __syncthreads();
  }
  uint32_t v[IF_ITEMS];
#pragma unroll
  for (int k = 0; k < IF_ITEMS; ++k) {
    const uint32_t j = j0 + k * 256 + threadIdx.x;
    v[k] = j < N ? sa[j] : SA_NONE;
  }
#pragma unroll
  for (int k = 0; k < IF_ITEMS; ++k) {
    if (v[k] == SA_NONE) continue;
    const uint32_t j = j0 + k * 256 + threadIdx.x;
    uint64_t ip = v[k];
    if (S > 1) {
      const uint32_t t = text_of(seg_off, s_seg[0], s_seg[1], j);
      ip += __ldg(seg_off + t) + t;
    }
    if (ip < isa_len) isa[ip] = j;
  }
}

cudaError_t launch_isa_fill(const uint32_t *sa, uint32_t N, const uint32_t *seg_off, uint32_t S,
                            uint32_t *isa, uint64_t isa_len, cudaStream_t stream) {
  if (N == 0) return cudaSuccess;
  k_isa_fill<<<(unsigned)(((uint64_t)N + IF_CHUNK - 1) / IF_CHUNK), 256, 0, stream>>>(
      sa, N, seg_off, S, isa, isa_len);
  return cudaGetLastError();
}

// Granules of the active suffixes. Most of a repeat's suffixes find their
// granule marked already, so the bit is read first.
constexpr int NM_UNROLL = 8;
__global__ void __launch_bounds__(256) k_need_mark(NeedArgs a) {
  const uint64_t stride = (uint64_t)gridDim.x * 256;
  for (uint64_t x0 = (uint64_t)blockIdx.x * 256 + threadIdx.x; x0 < a.m; x0 += NM_UNROLL * stride) {
    uint32_t g[NM_UNROLL], old[NM_UNROLL];
#pragma unroll
    for (int u = 0; u < NM_UNROLL; ++u) {
      const uint64_t x = x0 + u * stride;
      g[u] = x < a.m ? (uint32_t)a.act[x] >> a.shift : 0xFFFFFFFFu;
    }
#pragma unroll
    for (int u = 0; u < NM_UNROLL; ++u)
      old[u] = (g[u] >> 5) < a.words ? load_volatile_u32(a.active + (g[u] >> 5)) : 0xFFFFFFFFu;
#pragma unroll
    for (int u = 0; u < NM_UNROLL; ++u)
      if (!((old[u] >> (g[u] & 31)) & 1u)) atomicOr(&a.active[g[u] >> 5], 1u << (g[u] & 31));
  }
}

// missing = the needed granules not covered yet; they are from now on.
__global__ void __launch_bounds__(256) k_need_plan(NeedArgs a) {
  const uint32_t w = blockIdx.x * 256 + threadIdx.x;
  if (w >= a.words) return;
  uint32_t need = 0;
  for (uint32_t i = 0; i < a.offsets; ++i) {
    // A position p of granule q moves to granule q + (h >> shift) or the next.
    const uint32_t h = a.h[i], q = h >> a.shift;
    for (uint32_t extra = 0; extra < ((h & ((1u << a.shift) - 1u)) ? 2u : 1u); ++extra) {
      const uint32_t by = q + extra, bw = by >> 5, bb = by & 31;
      if (w < bw) continue;
      const uint32_t lo = a.active[w - bw];
      const uint32_t before = w > bw ? a.active[w - bw - 1] : 0u;
      need |= bb ? (lo << bb) | (before >> (32 - bb)) : lo;
    }
  }
  const uint32_t miss = need & ~a.covered[w];
  a.covered[w] |= miss;
  a.missing[w] = miss;
  if (miss) a.ctrl->need_any = 1u;
}

// Entries (rank << 32) | i' of the final ranks whose position lies in a
// missing granule (bits NULL: every final rank), in any order.
constexpr int NC_BLOCK = 256;
constexpr int NC_ITEMS = 16;
constexpr int NC_CHUNK = NC_BLOCK * NC_ITEMS;
__global__ void __launch_bounds__(NC_BLOCK) k_need_collect(CollectArgs a) {
  __shared__ uint32_t s_cnt[NC_BLOCK / 32], s_seg[2], s_base;
  if (a.missing && !a.ctrl->need_any) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (uint64_t c0 = (uint64_t)blockIdx.x * NC_CHUNK; c0 < a.N;
       c0 += (uint64_t)gridDim.x * NC_CHUNK) {
    const uint32_t j0 = (uint32_t)c0;
    __syncthreads();  // the previous chunk's shared words are read
    if (a.S > 1 && threadIdx.x < 2)
      s_seg[threadIdx.x] =
          segment_of(a.seg_off, a.S, threadIdx.x ? min(j0 + NC_CHUNK - 1u, a.N - 1u) : j0);
    uint32_t v[NC_ITEMS];
#pragma unroll
    for (int k = 0; k < NC_ITEMS; ++k) {
      const uint64_t j = c0 + k * NC_BLOCK + threadIdx.x;
      v[k] = j < a.N ? a.sa[j] : SA_NONE;
    }
    if (a.S > 1) __syncthreads();
    if (a.S > 1) {
#pragma unroll
      for (int k = 0; k < NC_ITEMS; ++k) {
        if (v[k] == SA_NONE) continue;
        const uint32_t t = text_of(a.seg_off, s_seg[0], s_seg[1], j0 + k * NC_BLOCK + threadIdx.x);
        v[k] += __ldg(a.seg_off + t) + t;
      }
    }
    uint32_t bits[NC_ITEMS];
#pragma unroll
    for (int k = 0; k < NC_ITEMS; ++k) {
      const uint32_t g = v[k] >> a.shift;
      bits[k] = a.missing && v[k] != SA_NONE && (g >> 5) < a.words ? __ldg(a.missing + (g >> 5)) : 0u;
    }
    uint32_t keep = 0, mine = 0;
#pragma unroll
    for (int k = 0; k < NC_ITEMS; ++k) {
      const bool in = v[k] != SA_NONE && (!a.missing || ((bits[k] >> ((v[k] >> a.shift) & 31)) & 1u));
      const uint32_t B = __ballot_sync(0xffffffffu, in);
      if (in) keep |= 1u << k;
      mine += __popc(B);
    }
    if (lane == 0) s_cnt[warp] = mine;
    __syncthreads();
    if (warp == 0) {
      const uint32_t c = lane < NC_BLOCK / 32 ? s_cnt[lane] : 0u;
      const uint32_t incl = warp_inclusive(c, OpAdd());
      if (lane < NC_BLOCK / 32) s_cnt[lane] = incl - c;
      if (lane == 31) s_base = incl ? atomicAdd(&a.ctrl->need_entries, incl) : 0u;
    }
    __syncthreads();
    uint32_t at = s_base + s_cnt[warp];
#pragma unroll
    for (int k = 0; k < NC_ITEMS; ++k) {
      const bool in = (keep >> k) & 1u;
      const uint32_t B = __ballot_sync(0xffffffffu, in);
      const uint32_t x = at + __popc(B & lanemask_lt());
      if (in && x < a.N)
        a.out[x] = ((uint64_t)(j0 + k * NC_BLOCK + threadIdx.x) << 32) | v[k];
      at += __popc(B);
    }
  }
}

cudaError_t launch_need_plan(const NeedArgs &a, int num_sms, cudaStream_t stream) {
  cudaError_t e = cudaMemsetAsync(a.active, 0, (size_t)a.words * 4, stream);
  if (e != cudaSuccess) return e;
  const uint64_t per = 256 * NM_UNROLL, want = ((uint64_t)a.m + per - 1) / per;
  const uint64_t cap = (uint64_t)num_sms * 8;
  k_need_mark<<<(unsigned)(want < 1 ? 1 : (want < cap ? want : cap)), 256, 0, stream>>>(a);
  k_need_plan<<<(a.words + 255) / 256, 256, 0, stream>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_need_collect(const CollectArgs &a, int num_sms, cudaStream_t stream) {
  if (a.N == 0) return cudaSuccess;
  const uint64_t want = ((uint64_t)a.N + NC_CHUNK - 1) / NC_CHUNK, cap = (uint64_t)num_sms * 8;
  k_need_collect<<<(unsigned)(want < cap ? want : cap), NC_BLOCK, 0, stream>>>(a);
  return cudaGetLastError();
}

}  // namespace gbsa
