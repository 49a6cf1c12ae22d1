// Causal flash attention with two query tiles in flight per CTA: the kernel
// for launches with several units per SM (attn_kernel.cuh, which puts both
// softmax warpgroups on one query tile, is the one for few units).  Same three
// variants (kDense, kDenseMass, kSparse), same arithmetic per row and tile.
//
// A stream is one 128-row query tile of one (batch, head) at a time, with its
// own softmax warpgroup (thread t owns row t = TMEM lane t), S buffer and O
// accumulator.  The tile chain of one stream (S product -> softmax -> P V) is
// latency-bound; the other stream's products fill the tensor pipe meanwhile,
// and one stream's epilogue, Q load and first tile overlap the other's tiles.
//
// Pairing (AttnParams::pair):
//   kPairNone   the streams take units of their own (each with its own support
//               list); the producer gives the next unit to the stream with
//               fewer tiles so far.
//   kPairHeads  stream s takes head 2 v + s of the same kv-head group, same
//               query tile: the same key tiles, so each K and V tile is loaded
//               once for both.
//   kPairTiles  (dense variants) stream s takes query tile 2 v + s of the same
//               head, less AttnParams::lone_first: K and V tiles shared up to the
//               diagonal.  Of an odd number of tiles the last, or the first, has
//               no partner and leaves one stream without work.
//
// Tensor memory (512 columns): S of stream s at 128 s, with P (bf16 pairs)
// written over its first 64 columns, and O of stream s at 256 + 128 s.
// S(j+1) of a stream overwrites P(j), so it is issued right behind P V(j) by
// the same thread, with no barrier between them.  This relies on the tensor
// pipe running one thread's tcgen05.mma of one CTA group in the order of issue.
// The ISA states that for products of the same shape and accumulator; these two
// have different accumulators (and, at head dims 64 and 96, shapes), so here it
// is the hardware's behaviour that is relied on, not a documented guarantee.
// An S product that ran ahead would change P under P V: outputs that differ
// between runs (the repeated launches of test_determinism_gpu.py) or from the
// oracle (test_duo_gpu.py).  It also follows that S(j+1) complete means P V(j)
// complete (a commit tracks all earlier products of its thread, which is
// documented): the softmax may rescale O without a further wait, and the
// epilogue's read of O precedes the next unit's first P V because the same
// warpgroup writes that P.
//
// Shared memory at head dim 128: a Q tile per stream (2 x 32 KB) and five
// more tiles.  Paired, they are one ring of K and V tiles.  Unpaired, each
// stream has one V tile and one and a half K tiles (three 64-column boxes; at
// head dim 96 two V tiles and five 32-column boxes): with rings of their own a
// stream that stands still does not hold up the other's loads.  That leaves 3 KB for everything else (hence the packed tile
// masks and the small schedule rings).
//
// Warp roles (512 threads; warps 14 and 15 only complete the warpgroup):
//   warps 0-3, 4-7  softmax of stream 0 and 1, epilogues included
//   warps 8, 11     producers: tile schedule, K and V loads (warp 8 for both
//                   streams of a paired launch)
//   warps 9, 10     products and Q loads of stream 0 and 1
//   warp 12         stager: the units and, sparse, their tile masks
//   warp 13         watchdog
//
// What bounds it (a timeline of one CTA, head dim 128): a stream's tile chain,
// 2830 clk for a tile of each stream against 2048 clk of tensor work: S product
// 740 to its softmax's first load, load and row maximum 440, exponentials and P
// 730 (550 of it the ex2 rate, 4.3 clk per warp instruction), 200 until the
// issuing warp sees P, P V and S(j+1) behind one another.  attn_kernel takes
// 1930 clk a tile.  A unit boundary costs a sparse stream 4400 clk more (16K, 11
// tiles a unit): the diagonal's mask 600-1000, O's last product and the
// epilogue 3100, the rest of the wait for the next unit's Q and first S.  These
// do not add up to an unpaired launch: 16K, 142 tiles and 13.5 units a stream in
// 302 us, leaves 3660 clk a tile besides the boundaries (paired 32K 3130); the
// likely part is the wait for V and K, whose buffers are one and a half tiles.
// Measured against attn_kernel (us, before / here): dense 120 / 102, dense + mass
// 130 / 111, sparse block 128 64 / 57, block 32 150 / 110; 16K sparse 352 / 286; 32K,
// four heads to a kv head 855 / 690 (paired); 4 x 4K, head dim 96 405 / 298.
//
// Every wait is bounded (the watchdog); a stream that stands still for the
// launch's limit sets the status word and an abort flag, and every role unwinds.
#pragma once

#include <type_traits>

#include "attn_common.cuh"

namespace wise {

constexpr int kDuoSlots = 8;        // schedule entries per stream
constexpr int kDuoStageTiles = 256; // sparse: key tiles a unit may span (longer launches use attn_kernel)
constexpr int kDuoMassCols = 32;    // key blocks per pass of the mass epilogue
constexpr int kEntSolo = 64;        // the tile is used by this stream only (paired launches)

// Units staged by warp 12.
template <int S, bool kMask>
struct DuoStage {
  // Units staged ahead.  At least two: a producer that takes the unit of a
  // slot then knows the slot's earlier phase complete (the unit two before has
  // been taken); with one, the second producer may wait for a phase while the
  // one before it is still open, and a parity wait would return at once.
  static constexpr int kSlots = 2;
  // Sparse: S * S bits per key tile, packed.
  static constexpr int kWords = kMask ? kDuoStageTiles * S * S / 32 : 1;
  uint64_t full[kSlots], empty[kSlots];
  int4 unit[kSlots];  // {tiles (-1: no more units), b * n_heads + h, b * n_kv_heads + kv head, query tile}, of stream 0
  uint32_t mask[kSlots][kWords];
  uint32_t taken[2][kWords];  // masks of the unit each producer works on
  int next;                   // units taken by the producers
};

struct DuoMassSums {
  float sum[2][2][4][kDuoMassCols];  // [stream][buffer][warp][key block]
};
struct DuoNoMass {};

template <int D, bool kPaired>
struct DuoCfg {
  // 128-row boxes of 64 columns (128-byte swizzle).  Unpaired at head dim 96,
  // of 32 columns (64-byte swizzle): a tile then takes 24 KB instead of 32
  // (half of the second 64-column box is not used), and a stream has room for a
  // second V tile (4 x 4K, 55 heads: 316 -> 305 us; block 32, 2 x 4K, 32 heads:
  // 204 -> 200).  Paired launches gained nothing from 7 ring entries instead of
  // 5, and dense + mass lost 1 %.
  static constexpr int kCols = duo_box_cols(D, kPaired);
  static constexpr int kBoxes = (D + kCols - 1) / kCols;
  static constexpr int kBox = 128 * kCols * 2;      // bytes
  static constexpr int kTile = kBoxes * kBox;       // bytes of a 128-row Q, K or V tile
  static constexpr int kBudget = 227 * 1024;
  static constexpr int kStateBytes = (D > 64 ? 3 : 4) * 1024;
  // Paired: ring of K and V tiles.
  static constexpr int kFit = (kBudget - kStateBytes - 2 * kTile) / kTile;
  static constexpr int kRing = kFit > 8 ? 8 : kFit;
  // Unpaired, per stream: K boxes (used as a ring) and one or two V tiles.
  static constexpr int kVTiles = kCols == 32 ? 2 : 1;
  static constexpr int kKBoxes = 2 * kBoxes - (D == 64 ? 0 : 1);
  static constexpr int kStream = kKBoxes * kBox + kVTiles * kTile;
  static constexpr int kKVBytes = kPaired ? kRing * kTile : 2 * kStream;
  // The dynamic shared memory of a kernel without static shared memory starts
  // 1024-byte aligned (checked by the kernel's set-up).  At least 116 KB, so
  // that one CTA runs per SM (it owns all 512 TMEM columns).
  static constexpr int kUsed = 2 * kTile + kKVBytes + kStateBytes;
  static constexpr int kSmem = kUsed > 116 * 1024 ? kUsed : 116 * 1024;
  static constexpr uint32_t kTmemS = 0, kTmemO = 256;
  static constexpr int kThreads = 512;
  static constexpr int kRegsSoftmax = 200, kRegsOther = 56;  // 256 x 200 + 256 x 56 = 512 x 128
  static constexpr int kProducerWarp = 8, kMmaWarp = 9, kProducerWarp1 = 11, kStageWarp = 12, kWatchWarp = 13;
  static_assert(kRing >= 4 && kSmem <= kBudget, "shared memory budget");
};

template <int R, int BLK, int MODE>
struct DuoShared {
  static constexpr int S = kTileN / BLK;
  using Stage = DuoStage<S, MODE == kSparse>;
  uint64_t full[R], empty[R];                // paired: K/V ring
  uint64_t k_full[2][2], v_full[2][2], v_free[2];  // unpaired: K(j), V(j) landed, by j & 1; P V(j) complete
  uint64_t sched_full[2][kDuoSlots], sched_empty[2][kDuoSlots];  // schedule entry written / read by all
  uint64_t q_full[2];
  uint64_t s_full[2];     // S(j) complete, and with it P V(j-1)
  uint64_t p_full[2];     // P(j) written
  uint64_t o_full[2];     // the unit's last P V complete
  uint64_t epi[2];        // the 4 warps of a stream wrote their mass sums of a pass
  uint64_t done[2];
  // {key tile | mask << 16, b * n_heads + h, flags | paired: tile counter << 8, tile of the unit | query tile << 16}
  int4 sched[2][kDuoSlots];
  Stage stage;
  typename std::conditional<MODE == kDenseMass, DuoMassSums, DuoNoMass>::type mass;
  uint32_t tmem_base;
  int abort;
  int beat[2];  // per stream, by its softmax: twice the entries taken, less one while it works on the last of them
};

// Unit u -> (batch, virtual head, virtual query tile): see decode_unit; a
// virtual head is a pair of heads with kPairHeads, a virtual query tile a pair
// of query tiles with kPairTiles.
__device__ __forceinline__ void decode_duo(const AttnParams& p, int u, int& b, int& vh, int& vq) {
  const int bh_count = p.batch * p.v_heads;
  int bh;
  if (p.v_group_heads > 0) {
    const int per_group = p.v_group_heads * p.v_qtiles;
    const int g = u / per_group, v = u - g * per_group;
    const int gh = min(p.v_group_heads, bh_count - g * p.v_group_heads);
    vq = p.v_qtiles - 1 - v / gh;
    bh = g * p.v_group_heads + v % gh;
  } else {
    vq = p.v_qtiles - 1 - u / bh_count;
    bh = u % bh_count;
  }
  b = bh / p.v_heads;
  vh = bh % p.v_heads;
}

// The CTA's units in order: round k of the snake; false when round k holds no
// unit for this CTA.
__device__ __forceinline__ bool duo_unit(const AttnParams& p, int k, int& u) {
  const int G = gridDim.x, c = blockIdx.x;
  u = k * G + ((k & 1) ? G - 1 - c : c);
  return u < p.v_units;
}

// Waits end when the phase completes or the abort flag is set; the watchdog
// (warp 13) sets the flag when a stream stands still for the launch's limit.
// Code size matters in this kernel: its roles together run more instructions
// than the SM's instruction cache holds, and with a timed loop at every wait
// and everything unrolled (99 KB) a fifth of the fetches missed and the warps
// stalled 1.6 cycles per instruction for instructions; hence also the rolled
// loops on whatever is not the tile loop.
__device__ __forceinline__ bool duo_wait(uint64_t* bar, uint32_t parity, const volatile int* abort) {
  const uint32_t at = smem_u32(bar);
#pragma unroll 1
  while (!mbar_try_wait_at(at, parity))
    if (*abort) return false;
  return true;
}

// By all lanes of a warp together; the outcome is the same for all of them.
__device__ __forceinline__ bool duo_warp_wait(uint64_t* bar, uint32_t parity, const volatile int* abort) {
  return __all_sync(0xffffffffu, duo_wait(bar, parity, abort));
}

// On the way out: a wait for work in flight, with its own limit.
__device__ __forceinline__ void duo_drain(uint64_t* bar, uint32_t parity) {
  const uint64_t t0 = global_timer_ns();
#pragma unroll 1
  while (!mbar_try_wait(bar, parity))
    if (global_timer_ns() - t0 > kWaitLimitNs) return;
}

// Warp 13, one lane.  A stream's clock runs from the moment its softmax takes a
// schedule entry until it is ready for the next one (a key tile, the unit's
// epilogue with its last).  A stream that waits for an entry has nothing to do
// as long as the other one moves: a paired unit may hold tiles for one stream
// only, and a stream may run out of units early.  Both standing still, working
// or not, is a wait of the producers or the stager that does not end.
template <class Sh>
__device__ void duo_watchdog(const AttnParams& p, Sh& sb) {
  volatile int* beat = sb.beat;
  int last0 = 0, last1 = 0;
  uint64_t t0 = global_timer_ns(), t1 = t0;
#pragma unroll 1
  for (uint32_t it = 0;; ++it) {
    const bool d0 = mbar_test_wait(&sb.done[0], 0);
    if (d0 && mbar_try_wait(&sb.done[1], 0)) return;
    if (!d0 && mbar_try_wait(&sb.done[0], 0)) continue;
    const int b0 = beat[0], b1 = beat[1];
    const bool d1 = mbar_test_wait(&sb.done[1], 0);
    const uint64_t now = global_timer_ns();
    if (b0 != last0) t0 = now;
    if (b1 != last1) t1 = now;
    last0 = b0;
    last1 = b1;
    // Unsigned, like mbar_wait: the limit may be any 64-bit number.
    const uint64_t both = max(t0, t1);
    if ((!d0 && now - ((b0 & 1) ? t0 : both) > p.wait_ns) || (!d1 && now - ((b1 & 1) ? t1 : both) > p.wait_ns)) {
      raise_status(p, &sb.abort, kStatusTimeout);
      return;
    }
    if (it >= 16) __nanosleep(200);
  }
}

// ------------------------------------------------------------------- stager
// Warp 12: the CTA's units in order and, sparse, the masks of their key tiles
// from their S support lists.  An entry of list q is accepted if it lies in
// [0, q0 + q] and exceeds every in-range entry before it (TileIter's rule).  32
// entries are judged at a time, the next 32 being loaded meanwhile: each above
// its neighbour, as in a list that is as it should be, or by a warp prefix max.
// Units of few tiles are bound by this warp.  Lists of three entries at block 32
// (us, every row walked to its end with a prefix max for all / here): 16K,
// 32 heads, rows of 32 171 / 173, rows of 512 954 / 174; 32K, 8 heads, rows of
// 1024 971 / 97.  After the last unit come two end markers, one for each producer.
template <int D, int BLK, int MODE, class Sh>
__device__ void duo_stager(const AttnParams& p, Sh& sb) {
  constexpr int S = kTileN / BLK;
  constexpr int kSlots = Sh::Stage::kSlots;
  auto& st = sb.stage;
  const int lane = threadIdx.x & 31;
  volatile int* abort = &sb.abort;
  int bad = 0, ends = 0;
  bool ok = true;
  for (int k = 0, n_st = 0; ends < 2; ++k) {
    int u, b = 0, vh = 0, vq = 0;
    const bool more = k * (int)gridDim.x < p.v_units;
    if (more) {
      if (!duo_unit(p, k, u)) continue;
      decode_duo(p, u, b, vh, vq);
    } else {
      ++ends;
    }
    const int slot = n_st % kSlots;
    if (n_st >= kSlots && !duo_warp_wait(&st.empty[slot], ((n_st / kSlots) - 1) & 1, abort)) {
      ok = false;
      break;
    }
    const int h = p.pair == kPairHeads ? 2 * vh : vh;
    const int z = b * p.n_kv_heads + h / p.group;
    const int qt = p.pair == kPairTiles ? 2 * vq - p.lone_first : vq;  // of stream 0 (-1: stream 1 alone)
    int n = -1;
    if (more) {
      if constexpr (MODE != kSparse) {
        n = (p.pair == kPairTiles ? min(qt + 1, p.n_qtiles - 1) : qt) + 1;
      } else {
        const int q0 = vq * S;
        const int n_lists = min(S, p.n_blocks - q0);
        const int n_words = ((vq + 1) * S * S + 31) / 32;
        for (int i = lane; i < n_words; i += 32) st.mask[slot][i] = 0u;
        __syncwarp();
        const size_t row0 = (size_t)z * p.n_blocks + q0;
        const int32_t* list = p.idx + row0 * p.cap;
        const int32_t* counts = p.counts + row0;
        int q = 0, x = 0, carry = -1;  // list, first entry
        int cnt = __ldg(counts);
        int v = lane < p.cap ? __ldg(list + lane) : -1;
#pragma unroll 1
        while (q < n_lists) {
          // A list is read as far as its count goes.  In rows of up to 32 the next
          // load need not wait for the count: the next list follows in any case.
          bool more_of = false;
          if (p.cap > 32) more_of = x + 32 < clamp_count(cnt, p.cap, bad);
          const int nx = more_of ? x + 32 : 0, nq = more_of ? q : q + 1;
          int n_cnt = 0, n_v = -1;
          if (nq < n_lists) {
            n_cnt = __ldg(counts + nq);
            if (nx + lane < p.cap) n_v = __ldg(list + (size_t)nq * p.cap + nx + lane);
          }
          if (x == 0) carry = -1;
          const bool live = x + lane < clamp_count(cnt, p.cap, bad);
          const bool in_range = live && v >= 0 && v <= q0 + q;
          int m = in_range ? v : -1;
          int before = __shfl_up_sync(0xffffffffu, m, 1);
          if (lane == 0) before = carry;
          const unsigned lanes = __ballot_sync(0xffffffffu, live);
          bool acc = in_range && m > before;
          if (__ballot_sync(0xffffffffu, acc) != lanes) {
            // Something not ascending or out of range: a prefix maximum decides.
#pragma unroll 1
            for (int o = 1; o < 32; o <<= 1) {
              const int other = __shfl_up_sync(0xffffffffu, m, o);
              if (lane >= o) m = max(m, other);
            }
            before = __shfl_up_sync(0xffffffffu, m, 1);
            before = max(lane == 0 ? -1 : before, carry);
            acc = in_range && v > before;
            bad = 1;
            carry = max(carry, __shfl_sync(0xffffffffu, m, 31));
          } else if (lanes) {
            carry = __shfl_sync(0xffffffffu, m, 31 - __clz(lanes));
          }
          if (acc) {
            const int bit = (v / S) * (S * S) + q * S + v % S;
            atomicOr(&st.mask[slot][bit >> 5], 1u << (bit & 31));
          }
          q = nq;
          x = nx;
          cnt = n_cnt;
          v = n_v;
        }
        __syncwarp();
        n = 0;
        for (int i = lane; i < n_words; i += 32) {
          uint32_t m = st.mask[slot][i];
          if (S == 2) m = (m | m >> 1 | m >> 2 | m >> 3) & 0x11111111u;
          if (S == 4) m = ((m & 0xFFFFu) ? 1u : 0u) | ((m >> 16) ? 2u : 0u);
          n += __popc(m);
        }
        n = __reduce_add_sync(0xffffffffu, n);
      }
    }
    if (lane == 0) {
      st.unit[slot] = make_int4(n, b * p.n_heads + h, z, qt);
      mbar_arrive(&st.full[slot]);
    }
    ++n_st;
  }
  if (MODE == kSparse && __any_sync(0xffffffffu, bad) && lane == 0) {
    griddep_wait();  // the status word is written after the previous kernel of the stream
    atomicOr(p.status, kStatusBadSupport);
  }
  if (!ok && lane == 0) raise_status(p, &sb.abort, kStatusTimeout);
}

// ----------------------------------------------------------------- producers
// Takes the next staged unit, all lanes together; its masks move to the
// producer's own copy, so that the slot is free at once.
template <int MODE, class Sh>
__device__ __forceinline__ bool duo_take_unit(const AttnParams& p, int own, int4& unit, Sh& sb) {
  constexpr int kSlots = Sh::Stage::kSlots;
  auto& st = sb.stage;
  const int lane = threadIdx.x & 31;
  int n = 0;
  if (lane == 0) n = atomicAdd(&st.next, 1);
  n = __shfl_sync(0xffffffffu, n, 0);
  const int slot = n % kSlots;
  if (!duo_warp_wait(&st.full[slot], (n / kSlots) & 1, &sb.abort)) return false;
  unit = st.unit[slot];
  if constexpr (MODE == kSparse) {
#pragma unroll 1
    for (int i = lane; i < Sh::Stage::kWords; i += 32) st.taken[own][i] = st.mask[slot][i];
  }
  __syncwarp();
  if (lane == 0) mbar_arrive(&st.empty[slot]);
  return true;
}

// The key tiles of a unit in ascending order: the dense prefix, or the set
// bits of the masks.
template <int BLK, int MODE>
struct DuoWalk {
  static constexpr int S = kTileN / BLK;
  int kt = 0, word = -1;
  uint32_t cur = 0;
  // key tile | mask << 16
  __device__ __forceinline__ uint32_t next(const uint32_t* mask) {
    if constexpr (MODE != kSparse) {
      return (uint32_t)kt++ | ((S == 1 ? 1u : S == 2 ? 0xFu : 0xFFFFu) << 16);
    } else {
      constexpr int kBits = S * S, kPer = 32 / kBits;
      constexpr uint32_t kOne = kBits == 1 ? 1u : (1u << kBits) - 1u;
      while (cur == 0) cur = mask[++word];
      const int b = (__ffs(cur) - 1) / kBits;
      const uint32_t m = (cur >> (b * kBits)) & kOne;
      cur &= ~(kOne << (b * kBits));
      return (uint32_t)(word * kPer + b) | (m << 16);
    }
  }
};

template <class Sh>
__device__ __forceinline__ bool duo_emit(const AttnParams& p, int s, int& pos, int4 ent, Sh& sb) {
  const int slot = pos % kDuoSlots;
  if (pos >= kDuoSlots && !duo_wait(&sb.sched_empty[s][slot], ((pos / kDuoSlots) - 1) & 1, &sb.abort))
    return false;
  sb.sched[s][slot] = ent;
  mbar_arrive(&sb.sched_full[s][slot]);
  ++pos;
  return true;
}

// Unpaired: stream s's producer (lane 0 does the loads).  The boxes of K(j)
// follow those of K(j-1) in a ring of one box less than two tiles (two tiles at
// head dim 64): all but the last are free once S(j-2) has completed, which
// V(j-1)'s wait or the one for the last box of K(j-1) has seen, the last one
// once S(j-1) has.  With one V tile, V(j) may be loaded once P V(j-1) is
// complete; with two, once P V(j-2) is, and S(j-1) complete means that.
template <int D, int BLK, int MODE, class Sh>
__device__ void duo_producer(const CUtensorMap* mapK, const CUtensorMap* mapV, const AttnParams& p, int s,
                             uint8_t* kv, Sh& sb) {
  using C = DuoCfg<D, false>;
  const int lane = threadIdx.x & 31;
  volatile int* abort = &sb.abort;
  uint8_t* k_boxes = kv + s * C::kStream;
  uint8_t* v_tiles = k_boxes + C::kKBoxes * C::kBox;
  int pos = 0, j = 0, box = 0, nk = 0, nv = 0;  // tiles, next K box, K and V tiles loaded
  bool ok = true, waited = false;
  for (;;) {
    int4 unit;
    if (!duo_take_unit<MODE>(p, s, unit, sb)) {
      ok = false;
      break;
    }
    if (unit.x > 0 && !waited) {
      griddep_wait();  // the first copy: the previous kernel of the stream has completed
      waited = true;
    }
    if (lane == 0) {
      if (unit.x <= 0) {
        ok = duo_emit(p, s, pos, make_int4(0, unit.y, unit.x < 0 ? kEntEnd : kEntEmpty, unit.w << 16), sb);
      }
      DuoWalk<BLK, MODE> walk;
#pragma unroll 1
      for (int t = 0; t < unit.x; ++t, ++j) {
        const uint32_t key = walk.next(sb.stage.taken[s]);
        const int y = (int)(key & 0xFFFFu) * kTileN;
        const int fl = (t == 0 ? kEntFirst : 0) | (t + 1 == unit.x ? kEntLast : 0);
        if (!duo_emit(p, s, pos, make_int4((int)key, unit.y, fl, t | (unit.w << 16)), sb)) {
          ok = false;
          break;
        }
        uint64_t* k_full = &sb.k_full[s][j & 1];
        mbar_arrive_expect_tx(k_full, C::kTile);
        bool free = true;
#pragma unroll
        for (int i = 0; i < C::kBoxes; ++i) {
          // Issued after a wait that gave up as well: the barrier expects the
          // whole tile, and nothing is read from it any more.
          if (D > 64 && i + 1 == C::kBoxes) free = j < 1 || duo_wait(&sb.s_full[s], (j - 1) & 1, abort);
          tma_load_3d(k_boxes + box * C::kBox, mapK, k_full, C::kCols * i, y, unit.z);
          box = box + 1 == C::kKBoxes ? 0 : box + 1;
        }
        ++nk;
        if (C::kVTiles == 1 && free) free = j < 1 || duo_wait(&sb.v_free[s], (j - 1) & 1, abort);
        if (!free) {
          ok = false;
          break;
        }
        const int v_buf = C::kVTiles == 1 ? 0 : j & 1;
        mbar_arrive_expect_tx(&sb.v_full[s][v_buf], C::kTile);
#pragma unroll
        for (int i = 0; i < C::kBoxes; ++i)
          tma_load_3d(v_tiles + v_buf * C::kTile + i * C::kBox, mapV, &sb.v_full[s][v_buf], C::kCols * i, y, unit.z);
        ++nv;
      }
    }
    ok = __all_sync(0xffffffffu, ok);
    if (!ok || unit.x < 0) break;
  }
  if (!ok && lane == 0) {
    raise_status(p, &sb.abort, kStatusTimeout);
    // Copies already issued land before shared memory is released.
    for (int i = max(0, nk - 2); i < nk; ++i) duo_drain(&sb.k_full[s][i & 1], (i >> 1) & 1);
    for (int i = max(0, nv - C::kVTiles); i < nv; ++i)
      duo_drain(&sb.v_full[s][i % C::kVTiles], (i / C::kVTiles) & 1);
  }
}

// Paired: one producer for both streams.  The n-th tile's K is load 2 n and
// its V load 2 n + 1 of the ring.  Its entries are published when both ring
// slots have been given back, so that whoever reads an entry is at most one
// phase away from either slot's barrier.
template <int D, int BLK, int MODE, class Sh>
__device__ void duo_producer_paired(const CUtensorMap* mapK, const CUtensorMap* mapV, const AttnParams& p,
                                    uint8_t* ring, Sh& sb) {
  using C = DuoCfg<D, true>;
  constexpr int R = C::kRing;
  const int lane = threadIdx.x & 31;
  const bool heads = p.pair == kPairHeads;
  volatile int* abort = &sb.abort;
  int pos0 = 0, pos1 = 0, n = 0, slot = 0;
  uint32_t par = 1;  // parity of the slot's release before this use (waits on a fresh barrier pass)
  bool ok = true, waited = false;
  auto step = [&]() {
    if (++slot == R) {
      slot = 0;
      par ^= 1u;
    }
  };
  auto load = [&](const CUtensorMap* map, int y, int z) {
    mbar_arrive_expect_tx(&sb.full[slot], C::kTile);
#pragma unroll
    for (int i = 0; i < C::kBoxes; ++i)
      tma_load_3d(ring + slot * C::kTile + i * C::kBox, map, &sb.full[slot], C::kCols * i, y, z);
    step();
  };
  int loads = 0;
  for (;;) {
    int4 unit;
    if (!duo_take_unit<MODE>(p, 0, unit, sb)) {
      ok = false;
      break;
    }
    if (unit.x > 0 && !waited) {
      griddep_wait();
      waited = true;
    }
    if (lane == 0) {
      const int bh1 = unit.y + (heads ? 1 : 0), qt1 = heads ? unit.w : unit.w + 1;
      const bool two = qt1 < p.n_qtiles;  // not the last of an odd number of query tiles
      if (unit.x <= 0) {  // no tile (sparse, head pairs), or the end
        const int fl = unit.x < 0 ? kEntEnd : kEntEmpty;
        ok = duo_emit(p, 0, pos0, make_int4(0, unit.y, fl, qt1 << 16), sb) &&
             duo_emit(p, 1, pos1, make_int4(0, bh1, fl, qt1 << 16), sb);
      }
      DuoWalk<BLK, MODE> walk;
#pragma unroll 1
      for (int t = 0; t < unit.x; ++t, ++n) {
        const uint32_t key = walk.next(sb.stage.taken[0]);
        const int kt = (int)(key & 0xFFFFu);
        // kPairTiles: stream 0 ends one tile before stream 1, or has none.
        const bool use0 = heads || kt <= unit.w;
        const int last = t + 1 == unit.x ? kEntLast : 0;
        const int fl = (n << 8) | (t == 0 ? kEntFirst : 0) | (use0 && two ? 0 : kEntSolo);
        if (!duo_wait(&sb.empty[slot], par, abort)) {
          ok = false;
          break;
        }
        load(mapK, kt * kTileN, unit.z);
        ++loads;
        if (!duo_wait(&sb.empty[slot], par, abort) ||
            (use0 && !duo_emit(p, 0, pos0,
                               make_int4((int)key, unit.y, fl | (!heads && kt == unit.w ? kEntLast : last),
                                         t | (unit.w << 16)), sb)) ||
            (two && !duo_emit(p, 1, pos1, make_int4((int)key, bh1, fl | last, t | (qt1 << 16)), sb))) {
          ok = false;
          break;
        }
        load(mapV, kt * kTileN, unit.z);
        ++loads;
      }
    }
    ok = __all_sync(0xffffffffu, ok);
    if (!ok || unit.x < 0) break;
  }
  if (!ok && lane == 0) {
    raise_status(p, &sb.abort, kStatusTimeout);
    for (int i = max(0, loads - R); i < loads; ++i) duo_drain(&sb.full[i % R], (i / R) & 1);
  }
}

// ------------------------------------------------------------------ products
// Warps 9 and 10, one per stream, all lanes together; one elected lane issues.
// Everything a product needs besides P is looked up before the wait for P, so
// that P V(j) and S(j+1) follow at once; the rest of the bookkeeping runs under
// the softmax.  (One warp serving both streams spent 2200 clk per tile, more
// than the 1024 clk of the products: a warp beside two busy softmax warps
// issues an instruction every 5 to 10 clk.)  The stream's Q is loaded here as
// well: the last P of a unit being written means that its last S has read Q.
template <int D, bool kPaired, class Sh>
__device__ void duo_mma(const CUtensorMap* mapQ, const AttnParams& p, int s, uint32_t tmem, uint8_t* q_tiles,
                        uint8_t* kv, Sh& sb) {
  using C = DuoCfg<D, kPaired>;
  constexpr int R = C::kRing;
  constexpr int kRow = C::kCols * 2;   // bytes of a box row, and its swizzle
  constexpr int kSteps = C::kCols / 16;  // products (of 16 columns) per box
  constexpr uint32_t idesc_s = idesc_bf16_f32(128, kTileN, false, false);
  constexpr uint32_t idesc_o = idesc_bf16_f32(128, D, false, true);
  volatile int* abort = &sb.abort;
  const bool leader = elect_one();
  // Shared-memory descriptors: constant high halves, low halves that hold the
  // address.
  auto low = [](const uint8_t* at, uint32_t lbo) {
    return __shfl_sync(0xffffffffu, (uint32_t)smem_desc<kRow>(smem_u32(at), lbo, 8 * kRow), 0);
  };
  constexpr uint32_t hi = (uint32_t)(smem_desc<kRow>(0, 0, 8 * kRow) >> 32);
  uint8_t* q_tile = q_tiles + s * C::kTile;
  const uint32_t q_lo = low(q_tile, 16);
  const uint32_t s_tm = tmem + C::kTmemS + s * 128, o_tm = tmem + C::kTmemO + s * 128;
  const uint8_t* k_boxes = kv + s * C::kStream;  // unpaired

  int pos = 0;  // entries taken
  int j = 0;    // tiles whose P V has been issued
  int nq = 0;   // units begun
  int fl = 0;   // flags of the tile whose P V is due
  int box = 0;  // unpaired: first K box of the next tile
  bool due = false, ok = true;
#pragma unroll 1
  for (;;) {
    // V of the tile whose P V is due.
    int v_slot = 0;
    uint32_t v_lo = 0;
    if (due) {
      const int v_buf = C::kVTiles == 1 ? 0 : j & 1;
      uint64_t* v_bar = &sb.v_full[s][v_buf];
      uint32_t v_par = (C::kVTiles == 1 ? j : j >> 1) & 1;
      const uint8_t* v_at = k_boxes + C::kKBoxes * C::kBox + v_buf * C::kTile;
      if constexpr (kPaired) {
        const int l = 2 * (fl >> 8) + 1;
        v_slot = l % R;
        v_bar = &sb.full[v_slot];
        v_par = (l / R) & 1;
        v_at = kv + v_slot * C::kTile;
      }
      v_lo = low(v_at, C::kBox);
      if (!duo_warp_wait(v_bar, v_par, abort)) {
        ok = false;
        break;
      }
    }
    // The next entry, if it is there (the producer publishes it right after
    // the copy of that V is started; looked for before the wait above it was
    // missed at every other tile, and S(j+1) then came 700 clk later).
    const int slot = pos % kDuoSlots;
    const uint32_t slot_par = (pos / kDuoSlots) & 1;
    bool got = __all_sync(0xffffffffu, mbar_test_wait(&sb.sched_full[s][slot], slot_par));
    int4 ent = make_int4(0, 0, 0, 0);
    int k_slot = 0;
    uint64_t* k_bar = nullptr;
    uint32_t k_par = 0, k_lo[C::kBoxes] = {};  // K: barrier, descriptors of its boxes
    auto look = [&](int jn) {            // jn: the tile of the entry
      ent = sb.sched[s][slot];
      if constexpr (kPaired) {
        const int l = 2 * (ent.z >> 8);
        k_slot = l % R;
        k_bar = &sb.full[k_slot];
        k_par = (l / R) & 1;
        const uint32_t k0 = low(kv + k_slot * C::kTile, 16);
#pragma unroll
        for (int i = 0; i < C::kBoxes; ++i) k_lo[i] = k0 + i * (C::kBox >> 4);
      } else {
        k_bar = &sb.k_full[s][jn & 1];
        k_par = (jn >> 1) & 1;
        const uint32_t k0 = low(k_boxes, 16);
#pragma unroll
        for (int i = 0; i < C::kBoxes; ++i)
          k_lo[i] = k0 + (box + i - (box + i >= C::kKBoxes ? C::kKBoxes : 0)) * (C::kBox >> 4);
      }
    };
    if (got) look(j + (due ? 1 : 0));
    // S(j+1) may follow P V(j) at once if its K is there by then.
    const bool next = got && !(ent.z & (kEntEnd | kEntEmpty | kEntFirst));
    bool chain = false;
    auto issue_s = [&]() {
#pragma unroll
      for (int kk = 0; kk < D / 16; ++kk) {
        const int i = kk / kSteps;
        const uint32_t off = ((kk % kSteps) * 32) >> 4;
        umma_ss_split(s_tm, q_lo + i * (C::kBox >> 4) + off, hi, k_lo[i] + off, hi, idesc_s, kk > 0 ? 1u : 0u);
      }
      umma_commit(&sb.s_full[s]);
      if constexpr (kPaired) {
        umma_commit(&sb.empty[k_slot]);
        if (ent.z & kEntSolo) umma_commit(&sb.empty[k_slot]);
      }
    };
    if (due) {
      const uint32_t acc = (fl & kEntFirst) ? 0u : 1u;
      if (!duo_warp_wait(&sb.p_full[s], j & 1, abort)) {
        ok = false;
        break;
      }
      if (leader) {
        tc_fence_after_sync();
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
          umma_ts_split(o_tm, s_tm + kk * 8, v_lo + ((kk * 16 * kRow) >> 4), hi, idesc_o, kk > 0 ? 1u : acc);
        if (kPaired || C::kVTiles == 1) umma_commit(kPaired ? &sb.empty[v_slot] : &sb.v_free[s]);
        if (fl & kEntLast) umma_commit(&sb.o_full[s]);
        chain = next && mbar_test_wait(k_bar, k_par);
        if (chain) issue_s();
        if (kPaired && (fl & kEntSolo)) umma_commit(&sb.empty[v_slot]);
        mbar_arrive(&sb.sched_empty[s][(pos - 1) % kDuoSlots]);
      }
      chain = __any_sync(0xffffffffu, chain);
      due = false;
      ++j;
    }
    if (!got) {
      if (!duo_warp_wait(&sb.sched_full[s][slot], slot_par, abort)) {
        ok = false;
        break;
      }
      look(j);
    }
    ++pos;
    if (!chain) {
      if (ent.z & kEntEnd) break;
      if (ent.z & kEntEmpty) {
        if (leader) mbar_arrive(&sb.sched_empty[s][slot]);
        __syncwarp();
        continue;
      }
      if (ent.z & kEntFirst) {
        if (leader) {
          mbar_arrive_expect_tx(&sb.q_full[s], C::kTile);
#pragma unroll 1
          for (int i = 0; i < C::kBoxes; ++i)
            tma_load_3d(q_tile + i * C::kBox, mapQ, &sb.q_full[s], C::kCols * i, (ent.w >> 16) * 128, ent.y);
        }
        __syncwarp();
        ++nq;
        if (!duo_warp_wait(&sb.q_full[s], (nq - 1) & 1, abort)) {
          ok = false;
          break;
        }
      }
      if (!duo_warp_wait(k_bar, k_par, abort)) {
        ok = false;
        break;
      }
      if (leader) {
        tc_fence_after_sync();
        issue_s();
      }
      __syncwarp();
    }
    fl = ent.z;
    due = true;
    if constexpr (!kPaired) {
      box += C::kBoxes;
      if (box >= C::kKBoxes) box -= C::kKBoxes;
    }
  }
  if (!ok && (threadIdx.x & 31) == 0) raise_status(p, &sb.abort, kStatusTimeout);
  __syncwarp();
  // Every product issued completes before TMEM is released, every copy before
  // shared memory is.
  if (leader) umma_commit(&sb.done[s]);
  __syncwarp();
  duo_drain(&sb.done[s], 0);
  if (!ok && nq > 0) duo_drain(&sb.q_full[s], (nq - 1) & 1);
}

// ------------------------------------------------------------------- softmax
// p = 2^(s * scale - shift) of N columns, the sum added to acc; the packed
// bf16 pairs go to out.
template <int N>
__device__ __forceinline__ void exp2_pack(const float* s, float scale, float shift, float2 (&acc)[4], uint32_t* out) {
  const float2 sc = make_float2(scale, scale), sh = make_float2(-shift, -shift);
#pragma unroll
  for (int c = 0; c < N; c += 2) {
    const float2 x = __ffma2_rn(make_float2(s[c], s[c + 1]), sc, sh);
    const float2 y = make_float2(ex2_approx(x.x), ex2_approx(x.y));
    acc[(c / 2) & 3] = __fadd2_rn(acc[(c / 2) & 3], y);
    out[c / 2] = pack_bf16x2(y.x, y.y);
  }
}

__device__ __forceinline__ float sum4(const float2 (&a)[4]) {
  const float2 b = __fadd2_rn(__fadd2_rn(a[0], a[1]), __fadd2_rn(a[2], a[3]));
  return b.x + b.y;
}

// The masks of an S tile, 32 keys (a chunk) at a time: the 32 rows of a warp
// lie in one query block and start at a multiple of 32, so that a chunk is
// kept, dropped (its bit in `off`), or crossed by the diagonal (chunk `diag`)
// for the whole warp.
__device__ __forceinline__ uint32_t masked_key(uint32_t v, int i, int lane) { return i > lane ? 0xFF800000u : v; }

// Block 128, and the dense variants: only a unit's last tile has masked keys.
// They are set to -inf in tensor memory by a small loop that costs this tile about 700 clk: as
// straight-line code on the registers it was fetched from beyond the
// instruction cache once a unit, 2000 to 4000 clk.
__device__ __forceinline__ void mask_in_tmem(uint32_t s_col, int diag, int lane) {
  uint32_t v[32];
  if (diag >= 0) {
    tmem_ld_32x32b_x32(s_col + 32 * diag, v);
    tmem_ld_wait(v);
#pragma unroll
    for (int i = 1; i < 32; ++i) v[i] = masked_key(v[i], i, lane);
    tmem_st_32x32b_x32(s_col + 32 * diag, v);
  }
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = 0xFF800000u;
#pragma unroll 1
  for (int c = max(diag + 1, 0); c < kTileN / 32; ++c) tmem_st_32x32b_x32(s_col + 32 * c, v);
  tmem_st_wait();
}

// Sparse with blocks of 32 and 64, where most tiles have masked keys: the row's maximum
// over the chunks that are kept, masking the one the diagonal crosses.  Dropped
// chunks are not touched (their exponentials are skipped as well); set to -inf
// like the others' masked keys they cost 700 clk a tile.
__device__ __forceinline__ float masked_row_max(float (&s)[kTileN], uint32_t off, int diag, int lane) {
  float m[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
  for (int c = 0; c < kTileN / 32; ++c) {
    if ((off >> c) & 1u) continue;
    if (c == diag) {
#pragma unroll
      for (int i = 1; i < 32; ++i) s[32 * c + i] = i > lane ? -INFINITY : s[32 * c + i];
    }
#pragma unroll
    for (int i = 0; i < 32; i += 2) m[(i / 2) & 3] = fmax3(m[(i / 2) & 3], s[32 * c + i], s[32 * c + i + 1]);
  }
  return fmaxf(fmax3(m[0], m[1], m[2]), m[3]);
}

// Words w[4 k + q] of a row lie in lane q of a quad (k = 0 .. 4 M - 1 in its
// registers); afterwards lane q holds the M * 4 consecutive words from
// 4 M q.  Two exchanges, across lane bit 1 and bit 0.
template <int M>
__device__ __forceinline__ void quad_rows(const uint32_t (&w)[4 * M], int lane, uint32_t (&out)[4 * M]) {
  const bool hi = (lane & 2) != 0, lo = (lane & 1) != 0;
  uint32_t a[2 * M], b[2 * M];  // words of lanes 0, 1 / 2, 3 of the quad
#pragma unroll
  for (int i = 0; i < 2 * M; ++i) {
    const uint32_t keep = hi ? w[2 * M + i] : w[i];
    const uint32_t recv = __shfl_xor_sync(0xffffffffu, hi ? w[i] : w[2 * M + i], 2);
    a[i] = hi ? recv : keep;
    b[i] = hi ? keep : recv;
  }
#pragma unroll
  for (int i = 0; i < M; ++i) {
    const uint32_t ka = lo ? a[M + i] : a[i], kb = lo ? b[M + i] : b[i];
    const uint32_t ra = __shfl_xor_sync(0xffffffffu, lo ? a[i] : a[M + i], 1);
    const uint32_t rb = __shfl_xor_sync(0xffffffffu, lo ? b[i] : b[M + i], 1);
    out[4 * i + 0] = lo ? ra : ka;
    out[4 * i + 1] = lo ? ka : ra;
    out[4 * i + 2] = lo ? rb : kb;
    out[4 * i + 3] = lo ? kb : rb;
  }
}

// 16 columns of O.
__device__ __forceinline__ void store_16(__nv_bfloat16* dst, const uint32_t (&q)[8], bool wide) {
  if (wide) {
    st_global_v8(dst, q);
  } else {
    *reinterpret_cast<uint4*>(dst) = make_uint4(q[0], q[1], q[2], q[3]);
    *reinterpret_cast<uint4*>(dst + 8) = make_uint4(q[4], q[5], q[6], q[7]);
  }
}

// Writes the first `cols` of 64 columns of 8 rows from a fragment
// (`acc[4 k + at]` and the next: columns 8 k + 2 (lane % 4) of row lane / 4),
// scaled by the row's f: each lane ends with 16 consecutive columns, so that a
// warp's store covers whole 128-byte row segments of 8 rows.  (Each thread
// storing the row it owns took 2300 clk a unit with 16-byte stores: 32 lines
// per store.)
__device__ __forceinline__ void store_fragment(__nv_bfloat16* dst, const uint32_t (&acc)[32], int at, float f, int lane,
                                               int cols, bool in, bool wide) {
  uint32_t w[8], q[8];
  const float2 f2 = make_float2(f, f);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const float2 x =
        __fmul2_rn(make_float2(__uint_as_float(acc[4 * k + at]), __uint_as_float(acc[4 * k + at + 1])), f2);
    w[k] = pack_bf16x2(x.x, x.y);
  }
  quad_rows<2>(w, lane, q);
  const int c = 16 * (lane & 3);
  if (in && c < cols) store_16(dst + c, q, wide);
}

template <int D, int BLK, int MODE, class Sh>
__device__ void duo_softmax(const AttnParams& p, int w, uint32_t tmem, Sh& sb) {
  using C = DuoCfg<D, true>;
  constexpr float kRescaleThreshold = 8.0f;  // log2 units: P stays <= 256
  constexpr int S = kTileN / BLK;
  constexpr uint32_t kAllPairs = S == 1 ? 1u : S == 2 ? 0xFu : 0xFFFFu;
  volatile int* abort = &sb.abort;
  const int r = threadIdx.x & 127;
  const int wq = r >> 5, lane = r & 31;
  const uint32_t lane_tmem = tmem + ((uint32_t)(wq * 32) << 16);
  const uint32_t s_col = lane_tmem + C::kTmemS + w * 128, o_col = lane_tmem + C::kTmemO + w * 128;
  const int qsub = r / BLK;
  // kDenseMass: log2 partial masses of the row, [stream][key tile][S][128 rows].
  float* lc = p.scratch + (size_t)blockIdx.x * scratch_floats_per_cta(p.n_qtiles, S, p.n_blocks) +
              (size_t)w * p.n_qtiles * S * 128 + r;
  int pos = 0, j = 0, nu = 0, n_pass = 0;
  float l = 0.0f, m = -INFINITY;
  bool ok = true;

  for (;;) {
    const int slot = pos % kDuoSlots;
    if (r == 0) sb.beat[w] = 2 * pos;
    if (!duo_warp_wait(&sb.sched_full[w][slot], (pos / kDuoSlots) & 1, abort)) {
      ok = false;
      break;
    }
    const int4 ent = sb.sched[w][slot];
    __syncwarp();
    if (lane == 0) mbar_arrive(&sb.sched_empty[w][slot]);
    ++pos;
    if (r == 0) sb.beat[w] = 2 * pos - 1;
    if (ent.z & kEntEnd) break;
    const int qt = ent.w >> 16, t = ent.w & 0xFFFF;
    const int row = qt * 128 + r;
    if (ent.z & kEntEmpty) {
      if (row < p.seqlen) {
        uint4* dst = reinterpret_cast<uint4*>(p.O + ((size_t)ent.y * p.seqlen + row) * D);
#pragma unroll 1
        for (int c = 0; c < D / 8; ++c) dst[c] = make_uint4(0u, 0u, 0u, 0u);
      }
      continue;
    }
    const bool first = (ent.z & kEntFirst) != 0;
    if (first) {
      l = 0.0f;
      m = -INFINITY;
    }

    // ---- one tile
    if (!duo_warp_wait(&sb.s_full[w], j & 1, abort)) {
      ok = false;
      break;
    }
    tc_fence_after_sync();
    const int kt = ent.x & 0xFFFF;
    uint32_t off = 0;
    int diag = 4;
    if (((uint32_t)ent.x >> 16) != kAllPairs || kt >= qt) {
      diag = (row - lane - kt * kTileN) >> 5;
      if constexpr (S == 1 || MODE != kSparse) {
        mask_in_tmem(s_col, diag, lane);
      } else {
        const uint32_t sub = (uint32_t)ent.x >> (16 + qsub * S);
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (c > diag || !((sub >> (32 * c / BLK)) & 1u)) off |= 1u << c;
      }
    }
    float s[kTileN];
    tmem_load_row<kTileN>(s_col, s);
    constexpr bool kChunks = MODE == kSparse && S > 1;  // chunks of 32 keys one by one
    const float m_tile = (kChunks ? masked_row_max(s, off, diag, lane) : row_max(s)) * p.scale_log2;
    const float m_new = (m_tile > m + kRescaleThreshold) ? m_tile : m;
    const float shift = m_new == -INFINITY ? 0.0f : m_new;
    if (m_new != m) {
      const float f = ex2_approx(m - m_new);  // 0 while m is -inf
      l *= f;
    }
    // O (P V(j-1) has completed with S(j)) is rescaled only when the max
    // moved; the warp does it together, lanes whose max did not move by 1.
    const bool rescale = !first && m_new != m && m != -INFINITY;
    if (__any_sync(0xffffffffu, rescale)) {
      const float f = rescale ? ex2_approx(m - m_new) : 1.0f;
#pragma unroll 1
      for (int c = 0; c < D / 16; ++c) {
        uint32_t v[16];
        tmem_ld_32x32b_x16(o_col + 16 * c, v);
        tmem_ld_wait(v);
#pragma unroll
        for (int e = 0; e < 16; ++e) v[e] = __float_as_uint(__uint_as_float(v[e]) * f);
        tmem_st_32x32b_x16(o_col + 16 * c, v);
      }
    }
    m = m_new;
    float2 acc[4];
    float tile_sum = 0.0f;
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[e] = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      // P of 32 keys, over S, which this warp has read.  Chunks without a key
      // are skipped where there are many (blocks of 32 and 64).
      uint32_t pw[16];
      if (kChunks && ((off >> c) & 1u)) {
#pragma unroll
        for (int e = 0; e < 16; ++e) pw[e] = 0u;
      } else {
        exp2_pack<32>(s + 32 * c, p.scale_log2, shift, acc, pw);
      }
      tmem_st_32x32b_x16(s_col + 16 * c, pw);
      if constexpr (MODE == kDenseMass && S > 1) {
        if ((32 * (c + 1)) % BLK == 0) {
          const float g = sum4(acc);
          lc[((size_t)t * S + 32 * c / BLK) * 128] = g > 0.0f ? m + lg2_approx(g) : -INFINITY;
          tile_sum += g;
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[e] = make_float2(0.0f, 0.0f);
        }
      }
    }
    tmem_st_wait();
    tc_fence_before_sync();
    __syncwarp();
    if (lane == 0) mbar_arrive(&sb.p_full[w]);
    if constexpr (!(MODE == kDenseMass && S > 1)) {
      tile_sum = sum4(acc);
      if constexpr (MODE == kDenseMass) lc[(size_t)t * 128] = tile_sum > 0.0f ? m + lg2_approx(tile_sum) : -INFINITY;
    }
    l += tile_sum;
    ++j;
    if (!(ent.z & kEntLast)) continue;

    // ---- epilogue of the unit
    if constexpr (MODE == kDenseMass) {
      // Block mass (Eq. 5), under the unit's last P V: per row 2^(lc - lse),
      // 32 key blocks per pass, their warp column sums one per lane, then the
      // sum over the warps of each query block.
      constexpr int kWarpsPerBlock = BLK / 32;
      const float lse = m + lg2_approx(l);
      const int n_kb = min((t + 1) * S, p.n_blocks);
      const int end = p.step == 0 ? p.n_blocks : n_kb;  // the first step zeroes the future blocks
      const int qblock = qt * S + wq;                   // query block this warp writes (warps 0 .. S-1)
      const bool writer = wq < S && qblock < p.n_blocks;
      float* out = p.blockmass + ((size_t)ent.y * p.n_blocks + qblock) * p.n_blocks;
      for (int kb0 = 0; kb0 < end; kb0 += kDuoMassCols) {
        const int kb = kb0 + lane;
        float sum = 0.0f;
        if (kb0 < n_kb) {
          const float before = (writer && p.step > 0 && kb < n_kb) ? out[kb] : 0.0f;
          float v[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] = (kb0 + i < n_kb) ? lc[(size_t)(kb0 + i) * 128] : -INFINITY;
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] = (row < p.seqlen) ? ex2_approx(v[i] - lse) : 0.0f;
          sum = warp_column_sums(v, lane);
          if constexpr (kWarpsPerBlock > 1) {
            auto& ws = sb.mass.sum[w][n_pass & 1];
            ws[wq][lane] = sum;
            __syncwarp();
            if (lane == 0) mbar_arrive(&sb.epi[w]);
            if (!duo_warp_wait(&sb.epi[w], n_pass & 1, abort)) {
              ok = false;
              break;
            }
            ++n_pass;
            sum = 0.0f;
            if (writer) {
#pragma unroll
              for (int q = 0; q < kWarpsPerBlock; ++q) sum += ws[wq * kWarpsPerBlock + q][lane];
            }
          }
          sum = before + sum * (1.0f / (float)BLK);
        }
        if (writer && kb < end) out[kb] = kb < n_kb ? sum : 0.0f;
      }
      if (!ok) break;
    }
    if (!duo_warp_wait(&sb.o_full[w], nu & 1, abort)) {
      ok = false;
      break;
    }
    ++nu;
    tc_fence_after_sync();
    const float inv_l = l > 0.0f ? 1.0f / l : 0.0f;
    const bool wide = p.o_align32 != 0;
    if constexpr (D % 64 == 0 || MODE == kDense) {
      // Rolled, 16 rows x 64 columns at a time (this code runs once a unit, its
      // first pass from beyond the instruction cache): rows lane / 4 and
      // lane / 4 + 8 of them in each lane.  At head dim 96 the second 64 have
      // 32 columns: the TMEM columns after them are read but not stored.
#pragma unroll 1
      for (int i = 0; i < 2 * ((D + 63) / 64); ++i) {
        const int h = i & 1, c0 = (i >> 1) * 64;
        const int ra = 16 * h + (lane >> 2), rb = ra + 8;
        const float fa = __shfl_sync(0xffffffffu, inv_l, ra), fb = __shfl_sync(0xffffffffu, inv_l, rb);
        const int row0 = qt * 128 + wq * 32;
        __nv_bfloat16* da = p.O + ((size_t)ent.y * p.seqlen + row0 + ra) * D + c0;
        uint32_t v[32];
        tmem_ld_16x256b_x8(o_col + ((uint32_t)(16 * h) << 16) + c0, v);
        tmem_ld_wait(v);
        const int q_cols = D % 64 == 0 ? 64 : min(D - c0, 64);
        store_fragment(da, v, 0, fa, lane, q_cols, row0 + ra < p.seqlen, wide);
        store_fragment(da + 8 * D, v, 2, fb, lane, q_cols, row0 + rb < p.seqlen, wide);
      }
    } else {
      // Head dim 96: each thread its own row (half of the second fragment's
      // lanes would have nothing to store).  4 x 4K, 55 heads: 308 us with
      // fragments, 299 with rows (rolled 297, but 8K at block 64 108 -> 113);
      // block 32, 2 x 4K, 32 heads: 201 -> 198; dense + mass 4K, 24 heads: 77.1
      // -> 75.6.  Dense gains 2 % with query tiles paired and loses 1 % with
      // heads paired, and keeps the fragments, as does head dim 128 (16K: 285 us
      // with fragments, 294 with rows).
#pragma unroll
      for (int c0 = 0; c0 < D; c0 += 32) {
        uint32_t v[32];
        tmem_ld_32x32b_x32(o_col + c0, v);
        tmem_ld_wait(v);
        if (row < p.seqlen) {
          __nv_bfloat16* dst = p.O + ((size_t)ent.y * p.seqlen + row) * D + c0;
          const float2 f2 = make_float2(inv_l, inv_l);
#pragma unroll
          for (int c = 0; c < 32; c += 16) {
            uint32_t q[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const float2 x = __fmul2_rn(
                  make_float2(__uint_as_float(v[c + 2 * k]), __uint_as_float(v[c + 2 * k + 1])), f2);
              q[k] = pack_bf16x2(x.x, x.y);
            }
            store_16(dst + c, q, wide);
          }
        }
      }
    }
  }
  // TMEM stores in flight complete before TMEM is released.
  tmem_st_wait();
  if (!ok) raise_status(p, &sb.abort, kStatusTimeout);
}

// -------------------------------------------------------------------- kernel
template <int D, int BLK, int MODE, bool kPaired>
__global__ void __launch_bounds__(512, 1)
    attn_duo_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
                    const __grid_constant__ CUtensorMap mapV, const AttnParams p) {
  using C = DuoCfg<D, kPaired>;
  using Sh = DuoShared<C::kRing, BLK, MODE>;
  static_assert(sizeof(Sh) <= C::kStateBytes, "shared state");
  static_assert(C::kThreads == 512, "launch bounds");
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t* q_tiles = smem;
  uint8_t* kv = smem + 2 * C::kTile;
  Sh& sb = *reinterpret_cast<Sh*>(kv + C::kKVBytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (smem_u32(smem) & 1023u) {  // the swizzled tiles need it; never seen
    if (threadIdx.x == 0) atomicOr(p.status, kStatusTimeout);
    return;
  }
  if (threadIdx.x == 0) {
    sb.abort = 0;
    sb.beat[0] = sb.beat[1] = 0;
    sb.stage.next = 0;
    for (int i = 0; i < C::kRing; ++i) {
      mbar_init(&sb.full[i], 1);
      mbar_init(&sb.empty[i], 2);  // both streams
    }
    for (int s = 0; s < 2; ++s) {
      for (int i = 0; i < kDuoSlots; ++i) {
        mbar_init(&sb.sched_full[s][i], 1);
        mbar_init(&sb.sched_empty[s][i], 5);  // four softmax warps and the stream's product issuer
      }
      mbar_init(&sb.k_full[s][0], 1);
      mbar_init(&sb.k_full[s][1], 1);
      mbar_init(&sb.v_full[s][0], 1);
      mbar_init(&sb.v_full[s][1], 1);
      mbar_init(&sb.v_free[s], 1);
      mbar_init(&sb.q_full[s], 1);
      mbar_init(&sb.s_full[s], 1);
      mbar_init(&sb.p_full[s], 4);
      mbar_init(&sb.o_full[s], 1);
      mbar_init(&sb.epi[s], 4);
      mbar_init(&sb.done[s], 1);
    }
    for (int i = 0; i < Sh::Stage::kSlots; ++i) {
      mbar_init(&sb.stage.full[i], 1);
      mbar_init(&sb.stage.empty[i], 1);
    }
    fence_mbar_init();
  }
  if (warp == C::kProducerWarp && lane == 0) {
    tma_prefetch_map(&mapQ);
    tma_prefetch_map(&mapK);
    tma_prefetch_map(&mapV);
  }
  if (warp == C::kMmaWarp) {
    tmem_alloc(&sb.tmem_base, 512);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = sb.tmem_base;
  // As in attn_kernel: only idx and counts may be read before the previous
  // kernel of the stream has completed (the stager reads them, and the
  // producers wait before their first copy).
  if (warp < 8 || warp == C::kMmaWarp || warp == C::kMmaWarp + 1 || warp == C::kWatchWarp) griddep_wait();
  if (threadIdx.x == 0) griddep_launch_dependents();

  if (warp < 8) {
    warpgroup_reg_inc<C::kRegsSoftmax>();
    duo_softmax<D, BLK, MODE>(p, warp >> 2, tmem, sb);
  } else {
    warpgroup_reg_dec<C::kRegsOther>();
    if (warp == C::kProducerWarp || (warp == C::kProducerWarp1 && !kPaired)) {
      if constexpr (kPaired) {
        duo_producer_paired<D, BLK, MODE>(&mapK, &mapV, p, kv, sb);
      } else {
        duo_producer<D, BLK, MODE>(&mapK, &mapV, p, warp == C::kProducerWarp ? 0 : 1, kv, sb);
      }
    } else if (warp == C::kMmaWarp || warp == C::kMmaWarp + 1) {
      duo_mma<D, kPaired>(&mapQ, p, warp - C::kMmaWarp, tmem, q_tiles, kv, sb);
    } else if (warp == C::kStageWarp) {
      duo_stager<D, BLK, MODE>(p, sb);
    } else if (warp == C::kWatchWarp) {
      if (lane == 0) duo_watchdog(p, sb);
    }
  }

  __syncwarp();
  tc_fence_before_sync();
  __syncthreads();
  if (warp == C::kMmaWarp) {
    __syncwarp();
    tc_fence_after_sync();
    tmem_dealloc(tmem, 512);
  }
}

template <int D, int BLK, int MODE, bool kPaired>
cudaError_t launch_duo_instance(const AttnLaunch& L) {
  using C = DuoCfg<D, kPaired>;
  return launch_dependent<attn_duo_kernel<D, BLK, MODE, kPaired>>(L.grid, C::kThreads, C::kSmem, L.stream, L.mapQ, L.mapK, L.mapV, L.p);
}

// The dense variants are always paired (L.p.pair), sparse where two heads
// share a support.
template <int D, int BLK>
cudaError_t launch_duo_for_block(int mode, const AttnLaunch& L) {
  if (mode == kDenseMass) return launch_duo_instance<D, BLK, kDenseMass, true>(L);
  return L.p.pair != kPairNone ? launch_duo_instance<D, BLK, kSparse, true>(L)
                               : launch_duo_instance<D, BLK, kSparse, false>(L);
}

template <int D>
cudaError_t launch_duo_for_dim(int block, int mode, const AttnLaunch& L) {
  if (mode == kDense) return launch_duo_instance<D, 128, kDense, true>(L);
  return block == 128 ? launch_duo_for_block<D, 128>(mode, L)
         : block == 64 ? launch_duo_for_block<D, 64>(mode, L)
                       : launch_duo_for_block<D, 32>(mode, L);
}

}  // namespace wise
