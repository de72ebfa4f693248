// Group order for the rounds after round 0 (Section 2.1, Algorithm 5: the
// order of the groups in the active list is free, since names are
// absolute ranks and a round only needs each group contiguous).
//
// Round 0 leaves the groups in rank order, in which neighbouring groups
// are unrelated text positions: every partner-name read ISA[i' + h] of a
// later round is then a random 4-byte access (a DRAM sector or two per
// read on a text far larger than L2). Repeats make groups of positions
// that move together: the suffixes of a copied segment and of its source
// form pairs (p, p + d), (p + 1, p + 1 + d), ..., and the copies of a
// repeated text groups {p, p + B, p + 2B, ...}, {p + 1, ...}. With the
// groups ordered by their first member's position, neighbouring groups --
// handled by neighbouring threads and by tiles in flight at the same time
// -- read neighbouring ISA entries, so the reads share cache lines and L2
// sectors. The rounds keep the order approximately (each tile writes its
// subgroups in place of its groups, and tiles start in order), so the
// groups are reordered once, after round 0.
//
// The first positions are distinct integers below N + S, so the order needs
// no sort: a bit per position marks them, and a group's new index is the
// number of marks below its own.
//
//   k_group_mark:  sets the bit of each group's first member
//   k_rank_sums / k_scan_top / k_rank_apply: the marks before every line
//                  (224 bits and their count share one 32-byte sector, so a
//                  rank is one sector read)
//   k_group_place: each group's record (start, size, name, head rank) to
//                  its new index (one random sector read, one 16-byte write)
//   k_info_sums / k_scan_top / k_info_apply: starts in the new order, names
//                  and head ranks
//   k_regroup:     the entries (g' << 32) | i' of the new list, tile by tile
//                  over its items, so a group's size does not matter
//
// then the classification runs again on the new tables.
//
// Bound: the random accesses of the marks and records, 16 bytes written and
// two sectors touched per group, and 16 bytes streamed per entry. Measured
// against a radix sort of (first position, group) with a gather of the
// records, and one thread per group copying its entries: the 256 copies of a
// 2^20-byte Zipf block 3.7 -> 0.88 ms (1 M groups of about 250), prose of
// 8 M characters 12.2 -> 0.07 ms (0.5 M groups of up to tens of thousands),
// 2^30 Markov DNA 6.8 -> 6.9 ms (72 M pairs: bound by the random records).
#include "dcx.cuh"

namespace gbsa {

namespace {

constexpr uint32_t RK_BITS = RANK_LINE_BITS;  // marks per line: 7 words; word 7 is the count
constexpr int RG_UNROLL = 4;  // groups per thread and iteration, loads before uses
constexpr int RK_TILE = 2048;  // lines, or groups, per scan tile

// After round 0 a group's members are in increasing position order, so the
// smallest is the first: one read per group. (Were it not, the order would
// only be approximate, and every order of the groups is valid.)
__global__ void __launch_bounds__(256) k_group_mark(const uint64_t *__restrict__ act,
                                                   const uint32_t *__restrict__ gstart,
                                                   uint32_t G, uint32_t *__restrict__ lines,
                                                   uint32_t positions, Ctrl *ctrl) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t g0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; g0 < G;
       g0 += RG_UNROLL * stride) {
    uint32_t s[RG_UNROLL], p[RG_UNROLL];
#pragma unroll
    for (int u = 0; u < RG_UNROLL; ++u) s[u] = g0 + u * stride < G ? gstart[g0 + u * stride] : 0u;
#pragma unroll
    for (int u = 0; u < RG_UNROLL; ++u) p[u] = (uint32_t)act[s[u]];
#pragma unroll
    for (int u = 0; u < RG_UNROLL; ++u) {
      if (g0 + u * stride >= G) break;
      if (p[u] >= positions) {  // never taken unless a logic error
        raise_error(ctrl, ERR_INTERNAL, 17);
        return;
      }
      const uint32_t line = p[u] / RK_BITS, bit = p[u] - line * RK_BITS;
      atomicOr(&lines[(uint64_t)line * 8 + (bit >> 5)], 1u << (bit & 31));
    }
  }
}

__device__ __forceinline__ uint32_t line_count(const uint4 &a, const uint4 &b) {
  return __popc(a.x) + __popc(a.y) + __popc(a.z) + __popc(a.w) + __popc(b.x) + __popc(b.y) +
         __popc(b.z);
}

__global__ void __launch_bounds__(256) k_rank_sums(const uint4 *__restrict__ lines, uint32_t L,
                                                  uint32_t *__restrict__ sums) {
  __shared__ uint32_t tmp[8];
  const uint64_t base = (uint64_t)blockIdx.x * RK_TILE + threadIdx.x;
  uint32_t v = 0;
#pragma unroll
  for (int k = 0; k < RK_TILE / 256; ++k) {
    const uint64_t x = base + k * 256;
    if (x < L) v += line_count(lines[2 * x], lines[2 * x + 1]);
  }
  uint32_t total;
  block_incl_sum(v, tmp, total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(256) k_rank_apply(uint4 *__restrict__ lines, uint32_t L,
                                                   const uint32_t *__restrict__ sums) {
  __shared__ uint32_t tmp[8];
  uint32_t before = sums[blockIdx.x];
  for (int k = 0; k < RK_TILE / 256; ++k) {  // 256 consecutive lines at a time
    const uint64_t x = (uint64_t)blockIdx.x * RK_TILE + k * 256 + threadIdx.x;
    const uint32_t c = x < L ? line_count(lines[2 * x], lines[2 * x + 1]) : 0u;
    uint32_t total;
    const uint32_t incl = block_incl_sum(c, tmp, total);
    if (x < L) reinterpret_cast<uint32_t *>(lines)[8 * x + 7] = before + incl - c;
    before += total;
  }
}

__global__ void __launch_bounds__(256) k_group_place(const uint64_t *__restrict__ act,
                                                    const uint32_t *__restrict__ gstart,
                                                    const uint32_t *__restrict__ gname,
                                                    const uint32_t *__restrict__ ghead, uint32_t G,
                                                    const uint4 *__restrict__ lines,
                                                    uint4 *__restrict__ info, Ctrl *ctrl) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t g0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; g0 < G;
       g0 += RG_UNROLL * stride) {
    uint32_t s[RG_UNROLL], e[RG_UNROLL], p[RG_UNROLL];
#pragma unroll
    for (int u = 0; u < RG_UNROLL; ++u) {
      const uint64_t g = g0 + u * stride;
      s[u] = g < G ? gstart[g] : 0u;
      e[u] = g < G ? gstart[g + 1] : 0u;
    }
#pragma unroll
    for (int u = 0; u < RG_UNROLL; ++u) p[u] = (uint32_t)act[s[u]];
    uint4 a[RG_UNROLL], b[RG_UNROLL];
#pragma unroll
    for (int u = 0; u < RG_UNROLL; ++u) {
      const uint64_t line = p[u] / RK_BITS;
      a[u] = lines[2 * line];
      b[u] = lines[2 * line + 1];
    }
#pragma unroll
    for (int u = 0; u < RG_UNROLL; ++u) {
      const uint64_t g = g0 + u * stride;
      if (g >= G) break;
      const uint32_t bit = p[u] % RK_BITS;
      const uint32_t w[7] = {a[u].x, a[u].y, a[u].z, a[u].w, b[u].x, b[u].y, b[u].z};
      uint32_t x = b[u].w;
#pragma unroll
      for (int i = 0; i < 7; ++i) {
        const uint32_t lo = 32 * i;
        const uint32_t m = bit >= lo + 32 ? 0xFFFFFFFFu : (bit <= lo ? 0u : (1u << (bit - lo)) - 1u);
        x += __popc(w[i] & m);
      }
      if (x >= G) {  // never taken unless a logic error
        raise_error(ctrl, ERR_INTERNAL, 18);
        return;
      }
      info[x] = make_uint4(s[u], e[u] - s[u], gname[g], ghead[g]);
    }
  }
}

__global__ void __launch_bounds__(256) k_info_sums(const uint4 *__restrict__ info, uint32_t G,
                                                  uint32_t *__restrict__ sums) {
  __shared__ uint32_t tmp[8];
  const uint64_t base = (uint64_t)blockIdx.x * RK_TILE + threadIdx.x;
  uint32_t v = 0;
#pragma unroll
  for (int k = 0; k < RK_TILE / 256; ++k)
    if (base + k * 256 < G) v += info[base + k * 256].y;
  uint32_t total;
  block_incl_sum(v, tmp, total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(256) k_info_apply(RegroupArgs a) {
  __shared__ uint32_t tmp[8];
  uint32_t before = a.sums[blockIdx.x];
  for (int k = 0; k < RK_TILE / 256; ++k) {
    const uint64_t x = (uint64_t)blockIdx.x * RK_TILE + k * 256 + threadIdx.x;
    const uint4 r = x < a.G ? a.info[x] : make_uint4(0u, 0u, 0u, 0u);
    uint32_t total;
    const uint32_t incl = block_incl_sum(r.y, tmp, total);
    if (x < a.G) {
      a.gstart_out[x] = before + incl - r.y;
      a.gname_out[x] = r.z;
      a.ghead_out[x] = r.w;
      if (x + 1 == a.G) a.gstart_out[a.G] = a.m;
    }
    before += total;
  }
}

// Items per block of the regroup: each holds at most 1024 group starts
// (groups have two members or more) besides the group it opens in.
constexpr int RG_TILE = 2048;

__global__ void __launch_bounds__(256) k_regroup(RegroupArgs a) {
  __shared__ uint32_t s_shift[RG_TILE / 2 + 1];  // source minus new index of a group's items
  __shared__ __align__(8) uint8_t s_head[RG_TILE];
  __shared__ uint32_t s_seg[RG_TILE / 32];
  __shared__ uint32_t s_x0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t base = blockIdx.x * (uint32_t)RG_TILE;
  const uint32_t count = min((uint32_t)RG_TILE, a.m - base);
  if (blockIdx.x == 0 && tid == 0) {  // every group is now a refine group with its final name
    RoundCounts rc{};
    rc.m_s = a.m;
    rc.g_s = a.G;
    a.ctrl->rc = rc;
  }
  reinterpret_cast<uint2 *>(s_head)[tid] = make_uint2(0u, 0u);
  if (warp == 0) {  // the last group starting at or before base, 32 probes at a time
    uint32_t lo = 0, n = a.G;  // gstart[lo] <= base; candidates [lo, lo + n)
    while (n > 1) {
      const uint32_t step = (n + 31) / 32;
      const uint64_t x = (uint64_t)lo + (uint64_t)lane * step;
      const bool le = (uint64_t)lane * step < n && a.gstart_out[x] <= base;
      const uint32_t k = 31 - __clz(__ballot_sync(0xffffffffu, le));  // lane 0 always holds
      lo += k * step;
      n = min(step, n - k * step);
    }
    if (lane == 0) s_x0 = lo;
  }
  __syncthreads();
  const uint32_t x0 = s_x0;
  for (uint32_t k = tid; k <= (uint32_t)RG_TILE / 2 && x0 + k < a.G; k += 256) {
    const uint32_t s = a.gstart_out[x0 + k];
    if (s >= base + count) break;
    s_shift[k] = a.info[x0 + k].x - s;
    if (k) s_head[s - base] = 1;
  }
  __syncthreads();
  uint32_t heads[RG_TILE / 256];
#pragma unroll
  for (int k = 0; k < RG_TILE / 256; ++k) {
    heads[k] = __ballot_sync(0xffffffffu, s_head[k * 256 + tid] != 0);
    if (lane == 0) s_seg[k * 8 + warp] = __popc(heads[k]);
  }
  __syncthreads();
  if (warp == 0) {  // exclusive sums over the 64 segments, in item order
    const uint32_t c0 = s_seg[2 * lane], c1 = s_seg[2 * lane + 1];
    const uint32_t ex = warp_inclusive(c0 + c1, OpAdd()) - c0 - c1;
    s_seg[2 * lane] = ex;
    s_seg[2 * lane + 1] = ex + c0;
  }
  __syncthreads();
  uint32_t x[RG_TILE / 256], src[RG_TILE / 256];
  uint32_t ip[RG_TILE / 256];
#pragma unroll
  for (int k = 0; k < RG_TILE / 256; ++k) {
    const uint32_t e = k * 256 + tid;
    x[k] = s_seg[k * 8 + warp] + __popc(heads[k] & (lanemask_lt() | (1u << lane)));
    src[k] = e < count ? s_shift[x[k]] + base + e : 0u;
    if (src[k] >= a.m) {  // never taken unless a logic error
      raise_error(a.ctrl, ERR_INTERNAL, 19);
      src[k] = 0;
    }
  }
#pragma unroll
  for (int k = 0; k < RG_TILE / 256; ++k) ip[k] = (uint32_t)a.act_in[src[k]];
#pragma unroll
  for (int k = 0; k < RG_TILE / 256; ++k) {
    const uint32_t e = k * 256 + tid;
    if (e < count) a.act_out[base + e] = ((uint64_t)(x0 + x[k]) << 32) | ip[k];
  }
}

}  // namespace

cudaError_t launch_group_rank(const RegroupArgs &a, int num_sms, cudaStream_t stream) {
  if (a.G == 0) return cudaSuccess;
  const uint32_t L = (uint32_t)rank_lines(a.positions);
  const uint64_t want = ((uint64_t)a.G + 255) / 256, cap = (uint64_t)num_sms * 16;
  const unsigned grid = (unsigned)(want < cap ? want : cap);
  const unsigned lt = (L + RK_TILE - 1) / RK_TILE;
  cudaError_t e = cudaMemsetAsync(a.lines, 0, (size_t)L * 32, stream);
  if (e != cudaSuccess) return e;
  k_group_mark<<<grid, 256, 0, stream>>>(a.act_in, a.gstart_in, a.G, a.lines, a.positions, a.ctrl);
  uint4 *lines = reinterpret_cast<uint4 *>(a.lines);
  k_rank_sums<<<lt, 256, 0, stream>>>(lines, L, a.sums);
  k_scan_top<<<1, DC_BLOCK, 0, stream>>>(a.sums, lt);
  k_rank_apply<<<lt, 256, 0, stream>>>(lines, L, a.sums);
  k_group_place<<<grid, 256, 0, stream>>>(a.act_in, a.gstart_in, a.gname_in, a.ghead_in, a.G,
                                          lines, a.info, a.ctrl);
  return cudaGetLastError();
}

cudaError_t launch_regroup(const RegroupArgs &a, cudaStream_t stream) {
  if (a.G == 0) return cudaSuccess;
  const unsigned gt = (a.G + RK_TILE - 1) / RK_TILE;
  k_info_sums<<<gt, 256, 0, stream>>>(a.info, a.G, a.sums);
  k_scan_top<<<1, DC_BLOCK, 0, stream>>>(a.sums, gt);
  k_info_apply<<<gt, 256, 0, stream>>>(a);
  k_regroup<<<(a.m + RG_TILE - 1) / RG_TILE, 256, 0, stream>>>(a);
  return cudaGetLastError();
}

}  // namespace gbsa
