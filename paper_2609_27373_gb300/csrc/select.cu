// Support selection (Eq. 6, single-pass form over accumulated block mass) and
// the working sets of the paper's own form.
//
// One warp per (batch, kv-head, query block) row.  Lane l owns key blocks
// l, l + 32, ... (KPL of them).  Masses of the kv-head group's query heads are
// pooled in exact 64-bit fixed point, the forced sink/local blocks are marked,
// and the remaining admissible blocks are taken in rank order (pooled mass
// descending, block index ascending) until the rule is met: top-k reached, or
// the kept mass covering eta of the row's admissible mass
// (cum * 65536 >= eta16 * total, compared in 128 bits), never beyond `cap`.
// The chosen set is written in ascending order with ballots and prefix
// popcounts, padded with -1.
//
// Bound: latency and instruction issue (the masses of a 32K launch are 4 MB).
// The fixed-point conversion is integer arithmetic, not double precision, whose
// rate on this chip is 1/64 of single precision's, and reductions use the warp
// reduction instructions.  Ranking (take_ranked) depends on the row: up to 32
// blocks are compared all with all; otherwise picks are taken one by one, and
// where four do not suffice and many may follow, a search over the mass of the
// last pick narrows the rest down to a few.  Measured back to back in a graph
// (us, with double precision, one-by-one picks and shuffles / here): 32K, 4 heads
// per kv head, top 12 22.6 / 12.8; 32 heads of 128 blocks, masses a softmax of
// normals, coverage up to 32 blocks: std 1 33.6 / 10.7, std 12 (one block holds most
// of a row) 8.9 / 6.0; working sets of two steps: std 1 160 / 21, std 12 13.0 / 8.5;
// of 256 blocks 575 / 53, 31 / 20; 4 heads of 1024 blocks 2560 / 131, 91 / 52.
// With the search from the first pick on, down to the last bit, concentrated
// rows were bound by it: the cases at std 12 took 19.6, 32.7, 84 and 151.
#include <limits.h>

#include <algorithm>

#include "internal.cuh"

namespace wise {

// floor(min(x, 4096) * 2^32); negative, zero and NaN masses count as zero.
__device__ __forceinline__ uint64_t mass_units(float x) {
  if (!(x > 0.0f)) return 0ull;
  const uint32_t bits = __float_as_uint(fminf(x, 4096.0f));
  const int shift = (int)(bits >> 23) - 118;  // x = m * 2^(e - 150)
  const uint64_t m = (bits & 0x7FFFFFu) | 0x800000u;
  // Below 2^-32 (denormals among them) the result is 0: m < 2^24.
  return shift >= 0 ? m << shift : shift > -24 ? m >> -shift : 0ull;
}

// Sum over the warp of values below 2^59 (the total below 2^64): 26-bit limbs,
// whose sums of 32 fit a 32-bit reduction.
__device__ __forceinline__ uint64_t warp_sum_u64(uint64_t v) {
  constexpr uint32_t kLimb = (1u << 26) - 1u;
  const uint32_t s0 = __reduce_add_sync(0xffffffffu, (uint32_t)v & kLimb);
  const uint32_t s1 = __reduce_add_sync(0xffffffffu, (uint32_t)(v >> 26) & kLimb);
  const uint32_t s2 = __reduce_add_sync(0xffffffffu, (uint32_t)(v >> 52));
  return (uint64_t)s0 + ((uint64_t)s1 << 26) + ((uint64_t)s2 << 52);
}

__device__ __forceinline__ uint64_t warp_max_u64(uint64_t v) {
  const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32));
  const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32) == hi ? (uint32_t)v : 0u);
  return ((uint64_t)hi << 32) | lo;
}

// cum * 65536 < eta16 * total, exactly.
__device__ __forceinline__ bool below_threshold(uint64_t cum, uint64_t eta16, uint64_t total) {
  const uint64_t lhs_hi = cum >> 48, lhs_lo = cum << 16;
  const uint64_t rhs_hi = __umul64hi(eta16, total), rhs_lo = eta16 * total;
  return lhs_hi < rhs_hi || (lhs_hi == rhs_hi && lhs_lo < rhs_lo);
}

// Rows that may take up to kFewPicks blocks take them one by one.  In the others
// the search follows kFirstPicks picks (2 and 0 were slower on concentrated rows,
// 128 blocks, std 12: 8.5 / 9.9 / 12.8 us) and ends when kLeft blocks are undecided
// (2 and 8 within 3 %).  A launch in which no row may take more has an instance
// without the search: its registers cost top 8 of 256 blocks 13.7 -> 14.2 us.
constexpr int kFewPicks = 16;
constexpr int kFirstPicks = 4;
constexpr int kLeft = 4;

// Adds candidates in rank order to `chosen` until done(kept mass, number
// added), which stays true once it is true; `cum` is the mass kept before, and
// `most` an upper bound on the number added.  Bit i of cand / chosen is block
// lane + 32 i.
template <int KPL, bool kFew, class Done>
__device__ __forceinline__ void take_ranked(const uint64_t (&U)[KPL], uint32_t cand, uint32_t& chosen, uint64_t cum,
                                            int most, int lane, Done done) {
  if (done(cum, 0)) return;
  if constexpr (KPL == 1) {
    // Lane l's block is taken unless the blocks ranked before it (mass and
    // number summed over all of them) already suffice.
    uint64_t before = 0;
    int rank = 0;
    const uint32_t all = __ballot_sync(0xffffffffu, cand != 0u);
    const uint64_t mine = U[0];
#pragma unroll 8
    for (int o = 0; o < 32; ++o) {
      const uint64_t u = __shfl_sync(0xffffffffu, mine, o);
      const bool ahead = ((all >> o) & 1u) && (u > mine || (u == mine && o < lane));
      before += ahead ? u : 0ull;
      rank += ahead;
    }
    if (cand && !done(cum + before, rank)) chosen |= 1u;
  } else {
    // One at a time: the largest mass, then the lowest block.
    int added = 0;
    for (int first = !kFew && most > kFewPicks ? kFirstPicks : INT_MAX;; --first) {
      if (!kFew && first == 0) {
        // Masses lo and hi such that the blocks of mass >= lo suffice and those of
        // mass >= hi do not, closed in bit by bit until few blocks lie between.
        uint64_t top = 0, part = 0;
#pragma unroll
        for (int i = 0; i < KPL; ++i) {
          if ((cand >> i) & 1u) {
            top = max(top, U[i]);
            part += U[i];
          }
        }
        int n_lo = __reduce_add_sync(0xffffffffu, __popc(cand)), n_hi = 0;  // blocks of mass >= lo, >= hi
        if (!done(cum + warp_sum_u64(part), added + n_lo)) {
          chosen |= cand;  // all of them do not suffice
          return;
        }
        top = warp_max_u64(top);
        uint64_t lo = 0, hi = ~0ull, s_hi = 0;
        for (int bit = 63 - __clzll((long long)(top | 1ull)); bit >= 0 && n_lo - n_hi > kLeft; --bit) {
          const uint64_t t = lo | (1ull << bit);
          uint64_t s = 0;
          int n = 0;
#pragma unroll
          for (int i = 0; i < KPL; ++i) {
            const bool in = ((cand >> i) & 1u) && U[i] >= t;
            s += in ? U[i] : 0ull;
            n += in;
          }
          s = warp_sum_u64(s);
          n = __reduce_add_sync(0xffffffffu, n);
          if (done(cum + s, added + n)) {
            lo = t;
            n_lo = n;
          } else {
            hi = t;
            n_hi = n;
            s_hi = s;
          }
        }
        // The blocks of mass >= hi, and of those between one by one below.
        uint32_t above = 0, between = 0;
#pragma unroll
        for (int i = 0; i < KPL; ++i) {
          if (!((cand >> i) & 1u)) continue;
          if (U[i] >= hi) {
            above |= 1u << i;
          } else if (U[i] >= lo) {
            between |= 1u << i;
          }
        }
        chosen |= above;
        cum += s_hi;
        added += n_hi;
        cand = between;
        const int n_eq = n_lo - n_hi;
        if (n_eq > kLeft) {
          // No bit is left: all of them have mass lo.  The fewest that suffice,
          // the lowest blocks first.
          int take = 0;
          for (int step = 1 << (31 - __clz(n_eq)); step > 0; step >>= 1)
            if (take + step <= n_eq && !done(cum + (uint64_t)(take + step) * lo, added + take + step)) take += step;
          ++take;
#pragma unroll
          for (int i = 0; i < KPL; ++i) {
            const uint32_t ball = __ballot_sync(0xffffffffu, (between >> i) & 1u);
            if (((between >> i) & 1u) && __popc(ball & ((1u << lane) - 1u)) < take) chosen |= 1u << i;
            take -= __popc(ball);
          }
          return;
        }
      }
      uint64_t best_u = 0;
      int best_kb = INT_MAX;
#pragma unroll
      for (int i = 0; i < KPL; ++i) {
        if (((cand >> i) & 1u) && (best_kb == INT_MAX || U[i] > best_u)) {
          best_u = U[i];
          best_kb = lane + 32 * i;
        }
      }
      const uint64_t u = warp_max_u64(best_u);
      const int kb = (int)__reduce_min_sync(0xffffffffu, best_u == u ? (uint32_t)best_kb : (uint32_t)INT_MAX);
      if (kb == INT_MAX) return;  // no candidate left
      if ((kb & 31) == lane) {
        cand &= ~(1u << (kb >> 5));
        chosen |= 1u << (kb >> 5);
      }
      cum += u;
      ++added;
      if (done(cum, added)) return;
    }
  }
}

// Pooled masses of this lane's blocks in one row set of masses
// [batch][n_heads][nb][nb].
template <int KPL>
__device__ __forceinline__ void pool_masses(const float* masses, int n_heads, int group, int nb, int b, int g, int q,
                                            int lane, uint64_t (&U)[KPL]) {
  const float* row = masses + (((size_t)b * n_heads + (size_t)g * group) * nb + q) * nb;
  const size_t head = (size_t)nb * nb;
#pragma unroll
  for (int i = 0; i < KPL; ++i) U[i] = 0;
#pragma unroll 4
  for (int h = 0; h < group; ++h) {
#pragma unroll
    for (int i = 0; i < KPL; ++i) {
      const int kb = lane + 32 * i;
      if (kb <= q) U[i] += mass_units(__ldg(row + h * head + kb));
    }
  }
}

// Writes the chosen blocks of a row in ascending order, -1 padded, and their
// number.
template <int KPL>
__device__ __forceinline__ void write_row(uint32_t chosen, int32_t* out, int cap, int32_t* count, int lane) {
  int n = 0;
#pragma unroll
  for (int i = 0; i < KPL; ++i) {
    const uint32_t ball = __ballot_sync(0xffffffffu, (chosen >> i) & 1u);
    if ((chosen >> i) & 1u) out[n + __popc(ball & ((1u << lane) - 1u))] = lane + 32 * i;
    n += __popc(ball);
  }
  for (int pos = n + lane; pos < cap; pos += 32) out[pos] = -1;
  if (lane == 0) *count = n;
}

template <int KPL, bool kFew>
__global__ void __launch_bounds__(256) select_kernel(const SelectParams p) {
  const long row = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const long n_rows = (long)p.batch * p.n_kv_heads * p.n_blocks;
  if (row >= n_rows) return;
  const int lane = threadIdx.x & 31;
  const int nb = p.n_blocks;
  const int q = (int)(row % nb);
  const int g = (int)((row / nb) % p.n_kv_heads);
  const int b = (int)(row / ((long)nb * p.n_kv_heads));

  uint64_t U[KPL];
  pool_masses(p.blockmass, p.n_heads, p.group, nb, b, g, q, lane, U);
  uint32_t cand = 0, chosen = 0;  // bit i <-> block lane + 32 i
  uint64_t total_part = 0, cum_part = 0;
#pragma unroll
  for (int i = 0; i < KPL; ++i) {
    const int kb = lane + 32 * i;
    if (kb <= q) {
      total_part += U[i];
      const bool forced = kb < p.n_sink || kb > q - p.n_local;
      if (forced) {
        chosen |= 1u << i;
        cum_part += U[i];
      } else {
        cand |= 1u << i;
      }
    }
  }
  const uint64_t total = warp_sum_u64(total_part);
  const uint64_t cum = warp_sum_u64(cum_part);
  const int n_forced = __reduce_add_sync(0xffffffffu, __popc(chosen));
  const int budget = (p.mode == 0) ? min(p.topk, p.cap - n_forced) : p.cap - n_forced;
  const bool coverage = p.mode != 0;
  take_ranked<KPL, kFew>(U, cand, chosen, cum, budget, lane, [&](uint64_t c, int n) {
    return n >= budget || (coverage && !below_threshold(c, p.eta16, total));
  });
  write_row<KPL>(chosen, p.idx + row * p.cap, p.cap, p.counts + row, lane);
}

template <int KPL>
static cudaError_t launch_select_kpl(const SelectParams& p, cudaStream_t stream) {
  const long rows = (long)p.batch * p.n_kv_heads * p.n_blocks;
  const int warps = 8;
  const long grid = (rows + warps - 1) / warps;
  const int most = p.mode == 0 ? std::min(p.topk, p.cap) : p.cap;
  if (KPL > 1 && most <= kFewPicks)
    select_kernel<KPL, true><<<(unsigned)grid, warps * 32, 0, stream>>>(p);
  else
    select_kernel<KPL, false><<<(unsigned)grid, warps * 32, 0, stream>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_select(const SelectParams& p, cudaStream_t stream) {
  if (p.n_blocks <= 32) return launch_select_kpl<1>(p, stream);
  if (p.n_blocks <= 64) return launch_select_kpl<2>(p, stream);
  if (p.n_blocks <= 128) return launch_select_kpl<4>(p, stream);
  if (p.n_blocks <= 256) return launch_select_kpl<8>(p, stream);
  if (p.n_blocks <= 512) return launch_select_kpl<16>(p, stream);
  return launch_select_kpl<32>(p, stream);
}

// ----------------------------------------------------------- working sets
// wise_select_working_set: the paper's own working set and its controls,
// one warp per (batch, kv-head, query block) row, same fixed-point masses,
// ranking and exact threshold comparison as select_kernel, no cap (the host
// requires cap >= nKB).  Modes: 0 union of per-step eta coverage sets (Eq. 6
// with the window union), 1 static (the first step's eta coverage set),
// 2 mass matched, 3 size matched (first step's ranking against a reference
// working set).  Forced sink/local blocks belong to every set.

// Two CTAs per SM at 32 blocks a lane (1024 blocks, std 12: 67 -> 52 us).
template <int KPL>
__global__ void __launch_bounds__(256, KPL >= 32 ? 2 : 0) working_set_kernel(const WorkingSetParams p) {
  const long row = (long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const long n_rows = (long)p.batch * p.n_kv_heads * p.n_blocks;
  if (row >= n_rows) return;
  const int lane = threadIdx.x & 31;
  const int nb = p.n_blocks;
  const int q = (int)(row % nb);
  const int g = (int)((row / nb) % p.n_kv_heads);
  const int b = (int)(row / ((long)nb * p.n_kv_heads));

  uint32_t admissible = 0, forced = 0;
#pragma unroll
  for (int i = 0; i < KPL; ++i) {
    const int kb = lane + 32 * i;
    if (kb <= q) {
      admissible |= 1u << i;
      if (kb < p.n_sink || kb > q - p.n_local) forced |= 1u << i;
    }
  }
  uint64_t U[KPL];
  const size_t step_size = (size_t)p.batch * p.n_heads * nb * nb;
  uint32_t result = forced;
  if (p.mode <= 1) {
    // Union over the steps of each step's eta coverage set (one step: static).
    for (int st = 0; st < p.n_steps; ++st) {
      pool_masses(p.masses + (size_t)st * step_size, p.n_heads, p.group, nb, b, g, q, lane, U);
      uint64_t total_part = 0, cum_part = 0;
#pragma unroll
      for (int i = 0; i < KPL; ++i) {
        if ((admissible >> i) & 1u) total_part += U[i];
        if ((forced >> i) & 1u) cum_part += U[i];
      }
      const uint64_t total = warp_sum_u64(total_part);
      uint32_t chosen = forced;
      take_ranked<KPL, false>(U, admissible & ~forced, chosen, warp_sum_u64(cum_part), nb, lane,
                  [&](uint64_t c, int) { return !below_threshold(c, p.eta16, total); });
      result |= chosen;
    }
  } else {
    // The reference working set of this row: its size and its first-step mass.
    pool_masses(p.masses, p.n_heads, p.group, nb, b, g, q, lane, U);
    const int32_t* ref = p.ref_idx + row * p.ref_cap;
    int n_ref = __ldg(p.ref_counts + row);
    int bad = 0;
    if (n_ref < 0 || n_ref > p.ref_cap) {
      bad = 1;
      n_ref = n_ref < 0 ? 0 : p.ref_cap;
    }
    uint32_t in_ref = 0;
    int prev = -1, k_ref = 0;
    for (int e = 0; e < n_ref; ++e) {
      const int v = __ldg(ref + e);  // the same value for every lane
      if (v >= 0 && v <= q && v > prev) {
        prev = v;
        ++k_ref;
        if ((v & 31) == lane) in_ref |= 1u << (v >> 5);
      } else {
        bad = 1;
      }
    }
    if (bad && lane == 0) atomicOr(p.status, kStatusBadSupport);
    uint64_t ref_part = 0, cum_part = 0;
    int n_forced_part = 0;
#pragma unroll
    for (int i = 0; i < KPL; ++i) {
      if ((in_ref >> i) & 1u) ref_part += U[i];
      if ((forced >> i) & 1u) {
        cum_part += U[i];
        ++n_forced_part;
      }
    }
    const uint64_t target = warp_sum_u64(ref_part);
    const uint64_t cum = warp_sum_u64(cum_part);
    const int k_more = k_ref - __reduce_add_sync(0xffffffffu, n_forced_part);
    uint32_t chosen = forced;
    if (p.mode == 2)
      take_ranked<KPL, false>(U, admissible & ~forced, chosen, cum, nb, lane, [&](uint64_t c, int) { return c >= target; });
    else
      take_ranked<KPL, false>(U, admissible & ~forced, chosen, cum, k_more, lane, [&](uint64_t, int n) { return n >= k_more; });
    result = chosen;
  }
  write_row<KPL>(result, p.idx + row * p.cap, p.cap, p.counts + row, lane);
}

template <int KPL>
static cudaError_t launch_ws_kpl(const WorkingSetParams& p, cudaStream_t stream) {
  const long rows = (long)p.batch * p.n_kv_heads * p.n_blocks;
  const int warps = 8;
  const long grid = (rows + warps - 1) / warps;
  working_set_kernel<KPL><<<(unsigned)grid, warps * 32, 0, stream>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_working_set(const WorkingSetParams& p, cudaStream_t stream) {
  if (p.n_blocks <= 32) return launch_ws_kpl<1>(p, stream);
  if (p.n_blocks <= 64) return launch_ws_kpl<2>(p, stream);
  if (p.n_blocks <= 128) return launch_ws_kpl<4>(p, stream);
  if (p.n_blocks <= 256) return launch_ws_kpl<8>(p, stream);
  if (p.n_blocks <= 512) return launch_ws_kpl<16>(p, stream);
  return launch_ws_kpl<32>(p, stream);
}

}  // namespace wise
