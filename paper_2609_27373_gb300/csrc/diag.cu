// Routing diagnostics: the block attention mass of a step retained by a
// support, and the overlap of two supports (rolling-set Jaccard).
#include <cooperative_groups.h>
#include <limits.h>

#include <algorithm>

#include "internal.cuh"

namespace wise {
namespace {

// The row of query head bh and query block q of a support list.  Rows are
// divided in 32 bits (those of a launch, n_blocks masses each and n_blocks to a
// head, do not reach 2^32 in any memory); 64-bit division was half of the time
// of a row of eight entries.
struct MassRow {
  int q;
  long long support;  // row of the support lists: heads lie in whole groups, so bh / group counts (b, kv head)
};
__device__ __forceinline__ MassRow mass_row(const SupportMassParams& p, uint32_t row) {
  const uint32_t bh = row / (uint32_t)p.n_blocks;
  return {(int)(row - bh * (uint32_t)p.n_blocks), (long long)(bh / (uint32_t)p.group) * p.n_blocks + row - bh * (uint32_t)p.n_blocks};
}

// Eight lanes per query-head row (b, h, q): the row's masses r_qb summed over
// the key blocks of its kv-group's support list, in list order.  Entries that
// are negative, beyond the query block, or not strictly above the previous
// accepted entry are skipped (the attention kernels' rule) and reported.
// Latency-bound: one lane per row took two dependent loads per entry; here
// eight entries, and then their masses, are loaded at once, a prefix maximum
// over the eight decides which entries count, and the sum still adds them one
// after the other (4K, 32 heads, 8 entries: 3.5 us, here 1.9).
__global__ void __launch_bounds__(256) support_mass_kernel(const SupportMassParams p) {
  constexpr int kLanes = 8;
  const long long row = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / kLanes;
  if (row >= p.rows) return;  // for all lanes of a row
  const int lane = threadIdx.x % kLanes;
  const unsigned mask = 0xFFu << (threadIdx.x & 31 & ~(kLanes - 1));
  const auto [q, srow] = mass_row(p, (uint32_t)row);
  const int32_t* list = p.idx + srow * p.cap;
  const float* m = p.blockmass + row * p.n_blocks;
  int n = __ldg(p.counts + srow);
  int v = lane < p.cap ? __ldg(list + lane) : -1;
  int bad = 0;
  if (n < 0 || n > p.cap) {
    bad = 1;
    n = n < 0 ? 0 : p.cap;
  }
  float acc = 0.0f;
  int carry = -1;  // largest in-range entry so far
  for (int x = 0; x < n; x += kLanes) {
    const int next = x + kLanes + lane < n ? __ldg(list + x + kLanes + lane) : -1;
    const bool live = x + lane < n;
    const bool in_range = live && v >= 0 && v <= q;
    int best = in_range ? v : -1;
#pragma unroll
    for (int o = 1; o < kLanes; o <<= 1) {
      const int other = __shfl_up_sync(mask, best, o, kLanes);
      if (lane >= o) best = max(best, other);
    }
    int before = __shfl_up_sync(mask, best, 1, kLanes);
    before = max(lane == 0 ? -1 : before, carry);
    const bool take = in_range && v > before;
    if (live && !take) bad = 1;
    carry = max(carry, __shfl_sync(mask, best, kLanes - 1, kLanes));
    const float mass = take ? __ldg(m + v) : 0.0f;
#pragma unroll
    for (int i = 0; i < kLanes; ++i) acc += __shfl_sync(mask, mass, i, kLanes);
    v = next;
  }
  if (lane == 0) p.retained[row] = acc;
  if (bad) atomicOr(p.status, kStatusBadSupport);
}

// One lane per row, for many rows: bound by their loads then, not by one row's
// chain of them.
__global__ void __launch_bounds__(256) support_mass_rows_kernel(const SupportMassParams p) {
  const uint32_t row = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= p.rows) return;
  const auto [q, srow] = mass_row(p, row);
  int n = __ldg(p.counts + srow);
  int bad = 0;
  if (n < 0 || n > p.cap) {
    bad = 1;
    n = n < 0 ? 0 : p.cap;
  }
  const int32_t* list = p.idx + srow * p.cap;
  const float* m = p.blockmass + (long long)row * p.n_blocks;
  float acc = 0.0f;
  int prev = -1;
  for (int i = 0; i < n; ++i) {
    const int v = __ldg(list + i);
    if (v >= 0 && v <= q && v > prev) {
      acc += __ldg(m + v);
      prev = v;
    } else {
      bad = 1;
    }
  }
  p.retained[row] = acc;
  if (bad) atomicOr(p.status, kStatusBadSupport);
}

// Next entry of a support list that the attention kernels use (in [0, q] and
// strictly above the last accepted one), or INT_MAX when the list is done.
__device__ __forceinline__ int next_valid(const int32_t* list, int n, int q, int& i, int& prev, int& bad) {
  while (i < n) {
    const int v = __ldg(list + i);
    ++i;
    if (v >= 0 && v <= q && v > prev) {
      prev = v;
      return v;
    }
    bad = 1;
  }
  return INT_MAX;
}

__device__ __forceinline__ int clamp_list(int n, int cap, int& bad) {
  if (n < 0 || n > cap) {
    bad = 1;
    return n < 0 ? 0 : cap;
  }
  return n;
}

// Lists over more than 1024 blocks, and many short ones.  One CTA per batch
// element; each thread merges the two (ascending) lists of its rows (b, kv head,
// q) and counts the blocks in both and in either.  The counts are integers, so
// the result does not depend on the reduction order.
__global__ void __launch_bounds__(256) support_overlap_merge_kernel(const SupportOverlapParams p) {
  const int b = blockIdx.x;
  unsigned long long inter = 0, uni = 0;
  int bad = 0;
  for (int r = threadIdx.x; r < p.rows; r += blockDim.x) {
    const long long row = (long long)b * p.rows + r;
    const int q = r % p.n_blocks;
    const int na = clamp_list(__ldg(p.counts_a + row), p.cap_a, bad);
    const int nb = clamp_list(__ldg(p.counts_b + row), p.cap_b, bad);
    const int32_t* la = p.idx_a + row * p.cap_a;
    const int32_t* lb = p.idx_b + row * p.cap_b;
    int ia = 0, ib = 0, pa = -1, pb = -1;
    int va = next_valid(la, na, q, ia, pa, bad), vb = next_valid(lb, nb, q, ib, pb, bad);
    while (va != INT_MAX || vb != INT_MAX) {
      ++uni;
      if (va == vb) {
        ++inter;
        va = next_valid(la, na, q, ia, pa, bad);
        vb = next_valid(lb, nb, q, ib, pb, bad);
      } else if (va < vb) {
        va = next_valid(la, na, q, ia, pa, bad);
      } else {
        vb = next_valid(lb, nb, q, ib, pb, bad);
      }
    }
  }
  __shared__ unsigned long long part[2][8];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    inter += __shfl_xor_sync(0xffffffffu, inter, off);
    uni += __shfl_xor_sync(0xffffffffu, uni, off);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    part[0][warp] = inter;
    part[1][warp] = uni;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long ti = 0, tu = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      ti += part[0][w];
      tu += part[1][w];
    }
    p.inter_union[2 * b] = ti;
    p.inter_union[2 * b + 1] = tu;
  }
  if (bad) atomicOr(p.status, kStatusBadSupport);
}

// Up to 1024 blocks.  One to kOvCtas CTAs per batch element, a cluster of
// them, and kLanes lanes per row at a time: kLanes entries of a list are loaded
// at once, judged (TileIter's rule), and set bits in the row's two bitmaps of
// kLanes words.  The CTAs' counts meet in the first CTA through distributed
// shared memory.
// Bound by latency with few rows, by instruction issue with many, and by the
// launch of CTAs with many elements; hence no more warps than about half of the
// chip holds, 8 lanes a row (32 over 256 blocks, or with under 1024 rows, which
// are single then: 64 rows 3.6 us at both), and clusters of small CTAs only for few
// elements.  Lists of up to 24 entries against 8 (us, merging / a cluster of 8 full
// CTAs and 32 lanes for every element / here): 1 element of 1024 rows 34 / 7.8 / 5.0,
// of 2048 (256 blocks) 98 / 11.9 / 7.2, 4 of 8192 391 / 36 / 17, 64 of 256 10.3 / 20.4 / 4.9,
// 64 of 8 3.6 / 13.0 / 2.3, 4096 of 16 19.4 / 804 / 8.6.
constexpr int kOvCtas = 8;
constexpr int kOvThreads = 1024;
constexpr int kOvBlocks = 1024;
constexpr int kOvWarps = 4864;         // of a launch, as far as rows and kOvMinWarps go
constexpr int kOvMinWarps = 4;         // of an element
constexpr int kOvFewElements = 19;     // with up to 8 CTAs each they fit the chip at once
constexpr long long kOvNarrowRows = 1024;

// n, list, q and bits are the row's, lane its lane, mask its lanes.
template <int kLanes>
__device__ __forceinline__ void set_list_bits(const int32_t* list, int n, int first, int q, int lane, unsigned mask,
                                              uint32_t* bits, int& bad) {
  int carry = -1, v = first;
  for (int x = 0; x < n; x += kLanes) {
    const int next = x + kLanes + lane < n ? __ldg(list + x + kLanes + lane) : -1;
    const bool live = x + lane < n;
    const bool in_range = live && v >= 0 && v <= q;
    int best = in_range ? v : -1;
    // Each above its neighbour, as in a list that is as it should be, or a
    // prefix maximum, which costs 8 lanes no more.
    bool take = false;
    unsigned lanes = 0;
    if constexpr (kLanes == 32) {
      int before = __shfl_up_sync(mask, best, 1);
      if (lane == 0) before = carry;
      take = in_range && best > before;
      lanes = __ballot_sync(mask, live);
    }
    if (kLanes == 32 && __ballot_sync(mask, take) == lanes) {
      carry = __shfl_sync(mask, best, 31 - __clz(lanes));
    } else {
#pragma unroll
      for (int o = 1; o < kLanes; o <<= 1) {
        const int other = __shfl_up_sync(mask, best, o, kLanes);
        if (lane >= o) best = max(best, other);
      }
      int before = __shfl_up_sync(mask, best, 1, kLanes);
      before = max(lane == 0 ? -1 : before, carry);
      take = in_range && v > before;
      if (live && !take) bad = 1;
      carry = max(carry, __shfl_sync(mask, best, kLanes - 1, kLanes));
    }
    if (take) atomicOr(bits + (v >> 5), 1u << (v & 31));
    v = next;
  }
}

template <int kLanes>
__global__ void __launch_bounds__(kOvThreads) support_overlap_kernel(const SupportOverlapParams p) {
  namespace cg = cooperative_groups;
  constexpr int kRows = 32 / kLanes;  // of a warp at a time
  __shared__ uint32_t bits[kOvThreads / 32][2][32];
  __shared__ unsigned long long warp_part[2][kOvThreads / 32], part[2];
  cg::cluster_group cluster = cg::this_cluster();
  const int ctas = cluster.num_blocks(), warps = blockDim.x >> 5;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x % kLanes, sub = (threadIdx.x & 31) / kLanes;
  const unsigned mask = (kLanes == 32 ? 0xffffffffu : (1u << (kLanes & 31)) - 1u) << (sub * kLanes);
  const int b = blockIdx.x / ctas, cta = blockIdx.x % ctas;
  uint32_t* bits_a = bits[warp][0] + sub * kLanes;
  uint32_t* bits_b = bits[warp][1] + sub * kLanes;
  unsigned long long inter = 0, uni = 0;
  int bad = 0;
  for (int r = (cta * warps + warp) * kRows + sub; r < p.rows; r += ctas * warps * kRows) {
    const long long row = (long long)b * p.rows + r;
    const int q = r % p.n_blocks;
    const int32_t* la = p.idx_a + row * p.cap_a;
    const int32_t* lb = p.idx_b + row * p.cap_b;
    const int ca = __ldg(p.counts_a + row), cb = __ldg(p.counts_b + row);
    const int fa = lane < p.cap_a ? __ldg(la + lane) : -1, fb = lane < p.cap_b ? __ldg(lb + lane) : -1;
    bits_a[lane] = 0u;
    bits_b[lane] = 0u;
    __syncwarp(mask);
    set_list_bits<kLanes>(la, clamp_list(ca, p.cap_a, bad), fa, q, lane, mask, bits_a, bad);
    set_list_bits<kLanes>(lb, clamp_list(cb, p.cap_b, bad), fb, q, lane, mask, bits_b, bad);
    __syncwarp(mask);
    const uint32_t wa = bits_a[lane], wb = bits_b[lane];
    inter += __popc(wa & wb);
    uni += __popc(wa | wb);
    __syncwarp(mask);
  }
  __syncwarp();
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    inter += __shfl_xor_sync(0xffffffffu, inter, off);
    uni += __shfl_xor_sync(0xffffffffu, uni, off);
  }
  if ((threadIdx.x & 31) == 0) {
    warp_part[0][warp] = inter;
    warp_part[1][warp] = uni;
  }
  if (bad) atomicOr(p.status, kStatusBadSupport);
  __syncthreads();
  unsigned long long total = 0;
  if (threadIdx.x < 2)
    for (int i = 0; i < warps; ++i) total += warp_part[threadIdx.x][i];
  if (ctas > 1) {
    if (threadIdx.x < 2) part[threadIdx.x] = total;
    cluster.sync();  // every CTA's counts are in its `part`
    if (cta == 0 && threadIdx.x < 2)
      for (int i = 1; i < ctas; ++i) total += *cluster.map_shared_rank(&part[threadIdx.x], i);
    cluster.sync();  // they have been read before a CTA ends
  }
  if (cta == 0 && threadIdx.x < 2) p.inter_union[2 * b + threadIdx.x] = total;
}

template <int kLanes>
cudaError_t launch_overlap_lanes(const SupportOverlapParams& p, cudaStream_t stream) {
  constexpr int kRows = 32 / kLanes;
  const int all = (p.rows + kRows - 1) / kRows;
  const int warps = std::max(1, std::min(all, std::max(kOvMinWarps, kOvWarps / p.batch)));
  int ctas = 1;
  const int per_cta = p.batch <= kOvFewElements ? 8 : kOvThreads / 32;
  while (ctas < kOvCtas && ctas * per_cta < warps) ctas *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)p.batch * ctas);
  cfg.blockDim = dim3(32 * std::min(kOvThreads / 32, (warps + ctas - 1) / ctas));
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ctas;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = ctas > 1 ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, support_overlap_kernel<kLanes>, p);
  return e == cudaSuccess ? cudaGetLastError() : e;
}

}  // namespace

cudaError_t launch_support_overlap(const SupportOverlapParams& p, cudaStream_t stream) {
  const long long rows = (long long)p.batch * p.rows;
  // Many rows of short lists, as many in an element as its CTA has threads for:
  // a merge is done before the bitmaps are (256 elements of 128 rows, rows of 16 and 8:
  // lists of 6 and 2 3.2 us, of 16 and 8 6.2, bitmaps 6.6 and 7.5).
  const bool short_rows = p.rows >= 32 && p.rows <= 256 && rows >= 4096 && (long long)p.cap_a + p.cap_b <= 24;
  if (p.n_blocks > kOvBlocks || short_rows) {
    support_overlap_merge_kernel<<<p.batch, 256, 0, stream>>>(p);
    return cudaGetLastError();
  }
  if (p.n_blocks <= 256 && rows >= kOvNarrowRows) return launch_overlap_lanes<8>(p, stream);
  return launch_overlap_lanes<32>(p, stream);
}

cudaError_t launch_support_mass(const SupportMassParams& p, cudaStream_t stream) {
  // Many rows, of lists of up to 16 entries: one lane
  // each (131072 rows of 12, lists of 2 / 8: 8.7 / 8.6 us with eight lanes and 64-bit
  // division, 6.9 / 6.9 without, 3.3 / 5.0 with one; rows of 64, lists of 32: 13 with
  // one, 7.6 with eight).
  if (p.rows > 32768 && p.cap <= 16) {
    support_mass_rows_kernel<<<(unsigned)((p.rows + 255) / 256), 256, 0, stream>>>(p);
    return cudaGetLastError();
  }
  const long long blocks = (p.rows * 8 + 255) / 256;
  support_mass_kernel<<<(unsigned)blocks, 256, 0, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace wise
