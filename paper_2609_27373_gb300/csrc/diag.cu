// Routing diagnostics: the block attention mass of a step retained by a
// support, and the overlap of two supports (rolling-set Jaccard).
#include <cooperative_groups.h>
#include <limits.h>

#include "internal.cuh"

namespace wise {
namespace {

// Eight lanes per query-head row (b, h, q): the row's masses r_qb summed over
// the key blocks of its kv-group's support list, in list order.  Entries that
// are negative, beyond the query block, or not strictly above the previous
// accepted entry are skipped (the attention kernels' rule) and reported.
// Latency-bound: one lane per row took two dependent loads per entry; here
// eight entries, and then their masses, are loaded at once, a prefix maximum
// over the eight decides which entries count, and the sum still adds them one
// after the other (4K, 32 heads, 8 entries: 3.3 us, here 1.9).
__global__ void __launch_bounds__(256) support_mass_kernel(const SupportMassParams p) {
  constexpr int kLanes = 8;
  const long long row = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / kLanes;
  if (row >= p.rows) return;  // for all lanes of a row
  const int lane = threadIdx.x % kLanes;
  const unsigned mask = 0xFFu << (threadIdx.x & 31 & ~(kLanes - 1));
  const int q = (int)(row % p.n_blocks);
  const long long bh = row / p.n_blocks;
  const int h = (int)(bh % p.n_heads);
  const int b = (int)(bh / p.n_heads);
  const long long srow = ((long long)b * p.n_kv_heads + h / p.group) * p.n_blocks + q;
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

// Lists over more than 1024 blocks.  One CTA per batch element; each thread
// merges the two (ascending) lists of its rows (b, kv head, q) and counts the
// blocks in both and in either.  The counts are integers, so the result does
// not depend on the reduction order.
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

// Up to 1024 blocks.  A cluster of kOvCtas CTAs per batch element, one warp per
// row at a time: 32 entries of a list are loaded at once, a prefix maximum
// decides which the attention kernels would use (TileIter's rule), and those
// set bits in the warp's two bitmaps.  The CTAs' counts meet in the first CTA
// through distributed shared memory.  (One CTA per element with a merge per
// thread was bound by its chain of dependent loads: 4K, 32 heads, lists of up
// to 32 against 8: 36 us, here 7.6.)
constexpr int kOvCtas = 8;
constexpr int kOvThreads = 1024;
constexpr int kOvBlocks = 1024;

__device__ __forceinline__ void set_list_bits(const int32_t* list, int n, int first, int q, int lane, uint32_t* bits,
                                              int& bad) {
  int carry = -1, v = first;
  for (int x = 0; x < n; x += 32) {
    const int next = x + 32 + lane < n ? __ldg(list + x + 32 + lane) : -1;
    const bool live = x + lane < n;
    const bool in_range = live && v >= 0 && v <= q;
    int best = in_range ? v : -1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int other = __shfl_up_sync(0xffffffffu, best, o);
      if (lane >= o) best = max(best, other);
    }
    int before = __shfl_up_sync(0xffffffffu, best, 1);
    before = max(lane == 0 ? -1 : before, carry);
    const bool take = in_range && v > before;
    if (live && !take) bad = 1;
    carry = max(carry, __shfl_sync(0xffffffffu, best, 31));
    if (take) atomicOr(bits + (v >> 5), 1u << (v & 31));
    v = next;
  }
}

__global__ void __cluster_dims__(kOvCtas, 1, 1) __launch_bounds__(kOvThreads)
    support_overlap_kernel(const SupportOverlapParams p) {
  namespace cg = cooperative_groups;
  __shared__ uint32_t bits[kOvThreads / 32][2][kOvBlocks / 32];
  __shared__ unsigned long long part[2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.x / kOvCtas, cta = blockIdx.x % kOvCtas;
  if (threadIdx.x < 2) part[threadIdx.x] = 0;
  __syncthreads();
  unsigned long long inter = 0, uni = 0;
  int bad = 0;
  for (int r = cta * (kOvThreads / 32) + warp; r < p.rows; r += kOvCtas * (kOvThreads / 32)) {
    const long long row = (long long)b * p.rows + r;
    const int q = r % p.n_blocks;
    const int32_t* la = p.idx_a + row * p.cap_a;
    const int32_t* lb = p.idx_b + row * p.cap_b;
    const int ca = __ldg(p.counts_a + row), cb = __ldg(p.counts_b + row);
    const int fa = lane < p.cap_a ? __ldg(la + lane) : -1, fb = lane < p.cap_b ? __ldg(lb + lane) : -1;
    bits[warp][0][lane] = 0u;
    bits[warp][1][lane] = 0u;
    __syncwarp();
    set_list_bits(la, clamp_list(ca, p.cap_a, bad), fa, q, lane, bits[warp][0], bad);
    set_list_bits(lb, clamp_list(cb, p.cap_b, bad), fb, q, lane, bits[warp][1], bad);
    __syncwarp();
    const uint32_t wa = bits[warp][0][lane], wb = bits[warp][1][lane];
    inter += __popc(wa & wb);
    uni += __popc(wa | wb);
    __syncwarp();
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    inter += __shfl_xor_sync(0xffffffffu, inter, off);
    uni += __shfl_xor_sync(0xffffffffu, uni, off);
  }
  if (lane == 0) {
    atomicAdd(&part[0], inter);
    atomicAdd(&part[1], uni);
  }
  if (bad) atomicOr(p.status, kStatusBadSupport);
  cg::cluster_group cluster = cg::this_cluster();
  cluster.sync();  // every CTA's counts are in its `part`
  if (cta == 0 && threadIdx.x < 2) {
    unsigned long long total = 0;
    for (int i = 0; i < kOvCtas; ++i) total += *cluster.map_shared_rank(&part[threadIdx.x], i);
    p.inter_union[2 * b + threadIdx.x] = total;
  }
  cluster.sync();  // they have been read before a CTA ends
}

}  // namespace

cudaError_t launch_support_overlap(const SupportOverlapParams& p, cudaStream_t stream) {
  if (p.n_blocks <= kOvBlocks) {
    support_overlap_kernel<<<(unsigned)p.batch * kOvCtas, kOvThreads, 0, stream>>>(p);
  } else {
    support_overlap_merge_kernel<<<p.batch, 256, 0, stream>>>(p);
  }
  return cudaGetLastError();
}

cudaError_t launch_support_mass(const SupportMassParams& p, cudaStream_t stream) {
  const long long blocks = (p.rows * 8 + 255) / 256;
  support_mass_kernel<<<(unsigned)blocks, 256, 0, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace wise
