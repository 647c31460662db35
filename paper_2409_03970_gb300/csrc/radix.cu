// Large plain sorts by digit: least-significant-digit-first passes of 8 bits
// (4 passes for 32-bit keys, 8 for 64-bit keys), each one stable scatter of
// the whole array.
//
// A merge sort of n keys moves the array 1 + log2(n / tile) times (15 at
// 2^28); the digit passes move it 4 times after one read for the histograms,
// whatever the key distribution.  The result is the same: the stable order
// by key is unique.
//
//   radix_histogram_kernel   counts every digit of every key at once;
//   radix_pass_kernel        one digit.  Each CTA takes a tile of the array in
//                            order (a ticket), counts its digits, publishes
//                            the counts, ranks its keys stably in shared
//                            memory and looks back over the tiles before it
//                            for where its keys go (the single-pass prefix
//                            scheme of Merrill and Garland, "Single-pass
//                            Parallel Prefix Scan with Decoupled Look-back",
//                            2016, applied to digit counts by Adinets and
//                            Merrill, "Onesweep", 2022).
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <string>
#include <type_traits>

#include "nsort.h"
#include "launch.h"
#include "nsort_internal.h"
#include "sort_device.cuh"
#include "tma_device.cuh"

namespace nsort {

namespace {

constexpr int BINS = 256;

// The order-preserving key map with the type chosen at run time by two
// masks: to = b ^ ((b >> 31 & arith) | flip).
template <typename K>
struct KeyMap {
  K arith, flip;
};

template <typename K>
__device__ __forceinline__ K map_in(K b, KeyMap<K> m) {
  if constexpr (sizeof(K) == 4)
    return b ^ (((K)((int32_t)b >> 31) & m.arith) | m.flip);
  else
    return b ^ (((K)((int64_t)b >> 63) & m.arith) | m.flip);
}

template <typename K>
__device__ __forceinline__ K map_out(K k, KeyMap<K> m) {
  if constexpr (sizeof(K) == 4)
    return k ^ (((K)((int32_t)~k >> 31) & m.arith) | m.flip);
  else
    return k ^ (((K)((int64_t)~k >> 63) & m.arith) | m.flip);
}

template <typename K>
KeyMap<K> key_map(int dt) {
  const K top = K(1) << (8 * sizeof(K) - 1);
  if (dt == DT_F32 || dt == DT_F64) return {~K(0), top};
  if (dt == DT_I32 || dt == DT_I64) return {K(0), top};
  return {K(0), K(0)};
}

// ---- histograms ------------------------------------------------------------

// Counts the 8-bit digits of every (mapped) key: hist[d][b] += ....  Each lane
// group counts in its own copy of the counters (COPIES of them, copy = lane
// mod COPIES, the copies of one counter in different banks), so that equal
// digits of a warp do not queue up on one address.  Also sets the passes'
// look-back words to "no entry" and the status word to NSORT_OK.
template <typename K, int NT, int COPIES>
__global__ void __launch_bounds__(NT) radix_histogram_kernel(const K *__restrict__ in, int64_t n,
                                                             KeyMap<K> map, uint32_t *hist,
                                                             uint32_t *state, int64_t state_words,
                                                             int *status) {
  constexpr int D = sizeof(K);
  extern __shared__ uint32_t rh_cnt[];   // [D][BINS][COPIES]
  const int tid = threadIdx.x;
  for (int i = tid; i < D * BINS * COPIES; i += NT) rh_cnt[i] = 0;
  const int64_t gtid = (int64_t)blockIdx.x * NT + tid;
  const int64_t gsize = (int64_t)gridDim.x * NT;
  for (int64_t i = gtid; i < state_words; i += gsize) state[i] = 0xFFFFFFFFu;
  if (gtid == 0) *status = NSORT_OK;
  __syncthreads();
  uint32_t *mine = rh_cnt + (tid & (COPIES - 1));
  auto count = [&](K raw) {
    const K k = map_in(raw, map);
#pragma unroll
    for (int d = 0; d < D; ++d)
      atomicAdd(mine + (d * BINS + (int)((k >> (8 * d)) & 0xFF)) * COPIES, 1u);
  };
  // 128-bit loads between the first and the last 16-byte boundary
  constexpr int EPV = 16 / sizeof(K);
  const int64_t mis = (int64_t)(((16 - (reinterpret_cast<uintptr_t>(in) & 15)) & 15) / sizeof(K));
  const int64_t head = mis < n ? mis : n;
  const int64_t vecs = (n - head) / EPV;
  const uint4 *v = reinterpret_cast<const uint4 *>(in + head);
  auto count4 = [&](uint4 q) {
    if constexpr (EPV == 4) {
      count(q.x);
      count(q.y);
      count(q.z);
      count(q.w);
    } else {
      count(((K)q.y << (4 * sizeof(K))) | q.x);
      count(((K)q.w << (4 * sizeof(K))) | q.z);
    }
  };
  constexpr int U = 4;   // loads in flight per thread
  int64_t i = gtid;
  for (; i + (U - 1) * gsize < vecs; i += U * gsize) {
    uint4 q[U];
#pragma unroll
    for (int u = 0; u < U; ++u) q[u] = __ldg(v + i + u * gsize);
#pragma unroll
    for (int u = 0; u < U; ++u) count4(q[u]);
  }
  for (; i < vecs; i += gsize) count4(__ldg(v + i));
  if (gtid < head) count(__ldg(in + gtid));
  const int64_t tail0 = head + vecs * EPV;
  if (gtid < n - tail0) count(__ldg(in + tail0 + gtid));
  __syncthreads();
  for (int b = tid; b < D * BINS; b += NT) {
    uint32_t sum = 0;
#pragma unroll
    for (int c = 0; c < COPIES; ++c) sum += rh_cnt[b * COPIES + ((c + tid) & (COPIES - 1))];
    if (sum) atomicAdd(hist + b, sum);
  }
}

// ---- one digit pass ----------------------------------------------------------

// Look-back word of (tile, digit): bit 31 the pass's parity, bit 30 set when
// the count is that of every tile up to this one (and of every smaller
// digit), else it is the tile's own, bits 29..0 the count.  A word of the
// other parity is no entry yet: the histogram kernel fills the words with
// ones (parity 1, the pass before the first) and every pass overwrites all
// of them.
constexpr uint32_t LB_INCL = 0x40000000u;
constexpr uint32_t LB_COUNT = 0x3FFFFFFFu;

__device__ __forceinline__ uint32_t load_relaxed(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void store_relaxed(uint32_t *p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Whether a wait that began at t0 (0: begins now) has lasted two seconds.
__device__ __forceinline__ bool gave_up(uint64_t &t0) {
  const uint64_t now = global_ns();
  if (!t0) t0 = now;
  return now - t0 > 2000000000ull;
}

// Shared memory: counters | staged keys (or payloads).
template <typename K, int NT, int IPT>
constexpr size_t radix_smem() {
  return (size_t)(NT / 16) * BINS * 4 + (size_t)(NT * IPT + NT * IPT / 512) * sizeof(K);
}

// Where position e of the tile is staged.  One word of padding per 512: in
// free order a tile of one digit gives every lane its own 512 consecutive
// positions, which would all start on one bank.
__device__ __forceinline__ uint32_t staged(uint32_t e) { return e + (e >> 9); }

struct NoValue {};

// One digit pass over keys (V = NoValue) or over pairs with payload word V.
// A tile is NT * IPT keys in chunks of 16 IPT: the first halves of the warps
// take the first NT / 32 chunks, the second halves the others, lane l of a
// half-warp key 16 i + l of the chunk at step i.
//
// Stable ranking.  Every half-warp has its own 256 counters, one word per
// digit: position << 16 | mask of lanes.  At each step the 16 lanes add
// their lane bits to their digits' words (one shared atomic), read the words
// back (the mask now holds every lane with the same digit) and take position
// + (mask bits below the own lane); the highest lane of each digit stores
// the word with the position moved on and the mask cleared.  A shared atomic
// costs as much as a shared load on this chip (2.6 against 2.4 cycles per
// warp on random digits), while matching a warp's digits by match.any costs
// 62 cycles and by eight ballots 24, against the 11.6 cycles in which HBM
// delivers and takes back 32 keys.
//
// Ranking where order is free.  Keys without payloads need to stay in order
// only if they differ in the lower digits, by which the array is sorted
// already.  A tile whose first and last keys agree in them (every tile of
// the first pass, nearly every one of the second) is ranked in any order:
// one counter per digit and lane (lanes mod NT / 16), so that no two lanes
// of a warp meet on an address or a bank, and one atomic per key.
//
// What bounds it (ncu at 2^26 uniform u32 keys): the shared-memory pipe in
// the stable passes (26 wavefronts for 32 keys, 80% of the pipe's peak; 197
// and 211 us), and in the free-order passes (15 wavefronts, 60%; 165 us)
// the latency of the phases of the two tiles an SM holds at a time.  A pass
// over 2^28 keys takes 0.70 ms on average, 3.1 TB/s of keys; 2^28 keys sort
// in 2.98 ms against 6.42 ms by merge passes, 2^27 f32 pairs in 2.49 against
// 7.19 ms, 3.0e7 pairs with 64-bit payloads in 1.00 against 2.03 ms, 2.0e7
// int64 keys in 0.88 against 1.07 ms.  Tried and slower at 2^28 keys: CTAs
// that stay for several tiles and load the next one early (3.0 to 5.2 ms:
// tickets taken early delay the counts that later tiles wait for), one CTA
// that scans all tiles' counts (4.35 ms), 32 tiles a look-back step (3.48).
template <typename K, typename V, int NT, int IPT, bool FIRST, bool LAST>
__global__ void __launch_bounds__(NT, 2) radix_pass_kernel(
    const K *__restrict__ src, const V *__restrict__ vsrc, K *__restrict__ dst,
    V *__restrict__ vdst, uint32_t n, int shift, KeyMap<K> map,
    const uint32_t *__restrict__ hist, uint32_t *state, uint32_t parity, uint32_t *ticket,
    int *status) {
  constexpr bool PAIRS = !std::is_same<V, NoValue>::value;
  constexpr int TILE = NT * IPT;
  constexpr int COPIES = NT / 16;        // counters per digit
  constexpr int WARPS = NT / 32;
  static_assert(NT == 2 * BINS && WARPS == 16, "two threads scan a digit's 32 counters");
  static_assert(TILE <= 32768, "positions take 15 bits of a counter");
  extern __shared__ __align__(16) unsigned char rp_smem[];
  // counters: word (warp * 256 + digit) * 2 + half (stable), digit * COPIES
  // + lane mod COPIES (free order)
  uint32_t *cnt = reinterpret_cast<uint32_t *>(rp_smem);
  K *stage = reinterpret_cast<K *>(rp_smem + (size_t)COPIES * BINS * 4);
  __shared__ uint32_t gbase[BINS];
  __shared__ uint32_t warp_sums[WARPS];
  __shared__ uint32_t tile_base[BINS], tile_total[BINS];
  __shared__ uint32_t tile_sh;
  __shared__ K ends[2];                  // the tile's first and last key
  pdl_wait();      // the previous kernel of the stream has finished writing
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const int warp = tid >> 5;
  const int hl = lane & 15;
  const uint32_t e0 = (uint32_t)(((lane >> 4) * WARPS + warp) * (16 * IPT) + hl);
  const K low = (K(1) << shift) - 1;     // the digits that are sorted already
  uint32_t sel = 0x4440u | (uint32_t)(shift >> 3 & 3);
  auto digit = [&](K k) {
    uint32_t w;
    if constexpr (sizeof(K) == 8) w = shift & 32 ? (uint32_t)(k >> 32) : (uint32_t)k;
    else w = k;
    return __byte_perm(w, 0u, sel);
  };
  if (tid == 0) tile_sh = atomicAdd(ticket, 1u);
  {
    uint4 *c4 = reinterpret_cast<uint4 *>(cnt);
#pragma unroll
    for (int i = 0; i < COPIES * BINS / 4 / NT; ++i) c4[tid + NT * i] = make_uint4(0, 0, 0, 0);
  }
  __syncthreads();
  // the sum of x over the digits below this thread's, for threads (digit
  // tid >> 1) that hold x in pairs; every thread of the CTA calls it
  auto sum_below = [&](uint32_t x) {
    uint32_t y = x;
#pragma unroll
    for (int o = 2; o < 32; o <<= 1) {
      const uint32_t z = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += z;
    }
    if (lane == 31) warp_sums[warp] = y;
    __syncthreads();
    return __reduce_add_sync(0xffffffffu, lane < warp ? warp_sums[lane] : 0u) + y - x;
  };
  const uint32_t tile = tile_sh;
  const uint32_t base = tile * (uint32_t)TILE;
  const uint32_t count = n - base < (uint32_t)TILE ? n - base : (uint32_t)TILE;
  K r[IPT];
  {
    const K *p = src + base + e0;
    if (count == TILE) {
#pragma unroll
      for (int i = 0; i < IPT; ++i) r[i] = __ldg(p + 16 * i);
    } else {
#pragma unroll
      for (int i = 0; i < IPT; ++i) r[i] = e0 + 16 * i < count ? __ldg(p + 16 * i) : K(0);
    }
  }
  if constexpr (PAIRS) {   // the payloads are loaded much later: bring them to L2, a line a thread
    constexpr uint32_t LINE = 128 / sizeof(V);
#pragma unroll
    for (uint32_t i = 0; i < TILE / LINE / NT; ++i) {
      const uint32_t e = (tid + NT * i) * LINE;
      if (e < count)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(vsrc + base + e));
    }
  }
  if (FIRST) {
#pragma unroll
    for (int i = 0; i < IPT; ++i) r[i] = map_in(r[i], map);
  }
  if (count != TILE) {   // padding: the largest key, behind every real one
#pragma unroll
    for (int i = 0; i < IPT; ++i)
      if (e0 + 16 * i >= count) r[i] = ~K(0);
  }
  if (tid == 0) ends[0] = r[0];
  if (tid == NT - 1) ends[1] = r[IPT - 1];
  __syncthreads();   // the counters are clear
  const bool free_order = !PAIRS && count == TILE && !((ends[0] ^ ends[1]) & low);
  // where this thread's counter of a digit is: mycnt + digit * dstride
  uint32_t *mycnt =
      free_order ? cnt + (lane & (COPIES - 1)) : cnt + warp * 2 * BINS + (lane >> 4);
  const uint32_t dstride = free_order ? COPIES : 2;
#pragma unroll
  for (int i = 0; i < IPT; ++i) atomicAdd(mycnt + dstride * digit(r[i]), 1u);
  __syncthreads();
  // counts -> positions in the tile: threads 2d and 2d + 1 take 16 of digit
  // d's counters each: those of the warps' first or second halves, or (free
  // order, so in any order) 16 copies, starting at another one in every
  // thread so that no two of a warp meet on a bank
  const int d = tid >> 1;
  auto counter = [&](int j) {
    return free_order ? cnt + d * COPIES + ((d & (COPIES - 1)) ^ ((tid & 1) * 16) ^ j)
                      : cnt + j * 2 * BINS + tid;
  };
  uint32_t own = 0;
#pragma unroll 8
  for (int j = 0; j < 16; ++j) own += *counter(j);
  const uint32_t other = __shfl_xor_sync(0xffffffffu, own, 1);
  const uint32_t total = own + other;
  if (!(tid & 1) && tile) store_relaxed(state + (size_t)tile * BINS + d, parity | total);
  const uint32_t tbase = sum_below(total);   // where the digit starts in the tile
  if (!(tid & 1)) {
    tile_base[d] = tbase;
    tile_total[d] = total;
  }
  {
    uint32_t run = tbase + (tid & 1 ? other : 0u);
    const int sh = free_order ? 0 : 16;
#pragma unroll 8
    for (int j = 0; j < 16; ++j) {
      uint32_t *c = counter(j);
      const uint32_t v = *c;
      *c = run << sh;
      run += v;
    }
  }
  __syncthreads();
  // rank and stage (the digits are extracted anew: kept from the counting
  // they would cost a register per key)
  asm volatile("" : "+r"(sel));
  [[maybe_unused]] uint32_t pos2[PAIRS ? IPT / 2 : 1];   // pairs: two positions a word
  const uint32_t below = (1u << hl) - 1u;
  auto rank_stable = [&](K k) {
    uint32_t *w = mycnt + 2 * digit(k);
    atomicAdd(w, 1u << hl);
    __syncwarp();
    const uint32_t v = *(volatile uint32_t *)w;
    const uint32_t pos = (v >> 16) + __popc(v & below);
    __syncwarp();
    if (((v & 0xFFFFu) >> hl) == 1u) *(volatile uint32_t *)w = (pos + 1u) << 16;
    __syncwarp();
    return pos;
  };
  if constexpr (PAIRS) {
#pragma unroll
    for (int i = 0; i < IPT; ++i) {
      const uint32_t pos = rank_stable(r[i]);
      stage[staged(pos)] = r[i];
      if (i & 1) {
        pos2[i / 2] |= pos << 16;
        asm volatile("" : "+r"(pos2[i / 2]));   // (kept packed)
      } else {
        pos2[i / 2] = pos;
      }
    }
  } else {
    if (free_order) {
#pragma unroll
      for (int i = 0; i < IPT; ++i)
        stage[staged(atomicAdd(mycnt + COPIES * digit(r[i]), 1u))] = r[i];
    } else {
      // the keys of this warp may be order-free even if the tile's are not
      const K f = __shfl_sync(0xffffffffu, r[0], lane & 16) & low;
      const K l = __shfl_sync(0xffffffffu, r[IPT - 1], lane | 15) & low;
      if (__all_sync(0xffffffffu, f == l)) {
#pragma unroll
        for (int i = 0; i < IPT; ++i)
          stage[staged(atomicAdd(mycnt + 2 * digit(r[i]), 1u << 16) >> 16)] = r[i];
      } else {
#pragma unroll
        for (int i = 0; i < IPT; ++i) stage[staged(rank_stable(r[i]))] = r[i];
      }
    }
  }
  // where the tile's keys go: thread d looks back over the counts of digit d
  // in the tiles before this one, LOOK at a time.  Words before tile 0's are
  // read too (other parts of the scratch) but not used: tile 0's count
  // covers every tile up to it.
  int flags = 0;   // 1: a digit's keys would go out of range, 2: no answer
  uint32_t excl = 0;
  if (tile == 0) excl = sum_below(hist[d]);   // (of digit tid >> 1)
  if (tile == 0 && !(tid & 1)) gbase[d] = excl;
  if (tile == 0) __syncthreads();
  if (tid < BINS) {
    uint32_t *word = state + (size_t)tile * BINS + tid;
    if (tile == 0) {
      excl = gbase[tid];
    } else {
      constexpr int LOOK = 8;
      const uint32_t *p = word;
      uint64_t t0 = 0;
      bool done = false;
      do {
        uint32_t v[LOOK];
#pragma unroll
        for (int j = 0; j < LOOK; ++j) v[j] = load_relaxed(p - (j + 1) * BINS);
        int used = 0;
#pragma unroll
        for (int j = 0; j < LOOK; ++j) {
          if ((v[j] ^ parity) & 0x80000000u) break;   // no entry yet: read again from here
          excl += v[j] & LB_COUNT;
          ++used;
          if (v[j] & LB_INCL) {
            done = true;
            break;
          }
        }
        p -= used * BINS;
        if (!used && gave_up(t0)) {
          flags = 2;
          break;
        }
      } while (!done);
    }
    const uint32_t t = tile_total[tid];
    store_relaxed(word, parity | LB_INCL | ((excl + t) & LB_COUNT));
    gbase[tid] = excl - tile_base[tid];
    // holds for every digit unless the keys changed while they were sorted
    if (excl + t > n + (tid == BINS - 1 ? TILE - count : 0)) flags |= 1;
  }
  const bool fault = __syncthreads_or(flags);
  if (fault && __syncthreads_or(flags & 2)) {
    if (tid == 0) atomicExch(status, (int)NSORT_ETIMEOUT);
    return;
  }
  const bool checked = fault || count != TILE;
  [[maybe_unused]] uint32_t dig4[PAIRS ? IPT / 4 : 1];   // pairs: four digits a word
  if constexpr (PAIRS) {
#pragma unroll
    for (int i = 0; i < IPT; ++i) {
      const uint32_t e = (uint32_t)(tid + NT * i);
      const K k = stage[staged(e)];
      const uint32_t dg = digit(k);
      const uint32_t at = gbase[dg] + e;
      if (!checked || (e < count && at < n)) dst[at] = LAST ? map_out(k, map) : k;
      if (i & 3) dig4[i / 4] |= dg << (8 * (i & 3));
      else dig4[i / 4] = dg;
      if (i % 4 == 3) asm volatile("" : "+r"(dig4[i / 4]));   // (kept packed)
    }
  } else if (!checked) {
#pragma unroll 8
    for (int i = 0; i < IPT; ++i) {
      const uint32_t e = (uint32_t)(tid + NT * i);
      const K k = stage[staged(e)];
      dst[gbase[digit(k)] + e] = LAST ? map_out(k, map) : k;
    }
  } else {
#pragma unroll 1
    for (int i = 0; i < IPT; ++i) {
      const uint32_t e = (uint32_t)(tid + NT * i);
      const K k = stage[staged(e)];
      const uint32_t at = gbase[digit(k)] + e;
      if (e < count && at < n) dst[at] = LAST ? map_out(k, map) : k;
    }
  }
  if constexpr (PAIRS) {
    // the payloads take the keys' places in the staging buffer, as many
    // positions at a time as fit
    constexpr int ROUNDS = sizeof(V) / sizeof(K);
    constexpr int RT = TILE / ROUNDS;
    V *vstage = reinterpret_cast<V *>(stage);
    const V *p = vsrc + base + e0;
#pragma unroll
    for (int q = 0; q < ROUNDS; ++q) {
      __syncthreads();   // the staging buffer has been read
      constexpr int VB = 32 / sizeof(V);   // loads in flight: what the registers hold
#pragma unroll
      for (int i0 = 0; i0 < IPT; i0 += VB) {
#pragma unroll
        for (int i = i0; i < i0 + VB; ++i) {
          const uint32_t pos = (pos2[i / 2] >> (16 * (i & 1))) & 0xFFFFu;
          if ((ROUNDS == 1 || (int)(pos / RT) == q) && e0 + 16 * i < count)
            vstage[staged(pos - q * RT)] = __ldg(p + 16 * i);
        }
        asm volatile("" ::: "memory");
      }
      __syncthreads();
#pragma unroll
      for (int i = 0; i < IPT / ROUNDS; ++i) {
        const int j = i + q * (IPT / ROUNDS);
        const uint32_t e = (uint32_t)(tid + NT * j);
        const uint32_t at = gbase[(dig4[j / 4] >> (8 * (j & 3))) & 0xFFu] + e;
        if (!checked || (e < count && at < n)) vdst[at] = vstage[staged(e - q * RT)];
      }
    }
  }
}

// Scratch of a digit sort inside a merge plan's splitter and sample arrays.
struct RadixLayout {
  size_t hist_off, ticket_off, state_off, end;
  int64_t tiles;
};

RadixLayout radix_layout(const Plan &p, int key_bytes, int tile) {
  RadixLayout l;
  l.tiles = (p.n + tile - 1) / tile;
  l.hist_off = p.split_off;
  l.ticket_off = l.hist_off + (size_t)key_bytes * BINS * 4;
  l.state_off = l.ticket_off + 256;
  l.end = l.state_off + (size_t)l.tiles * BINS * 4;
  return l;
}

template <typename K, typename V>
struct RadixShape {
  static constexpr int NT = 512;
  static constexpr int IPT = sizeof(K) == 8 ? 16 : 32;
  static constexpr int TILE = NT * IPT;
  static constexpr size_t SMEM = radix_smem<K, NT, IPT>();
};

constexpr int HIST_NT = 1024;
template <typename K>
constexpr int hist_copies() { return sizeof(K) == 8 ? 16 : 32; }
template <typename K>
constexpr size_t hist_smem() { return sizeof(K) * BINS * hist_copies<K>() * 4; }

// Opts the kernels of a key and payload type in to their shared memory, once
// per device, and finds the device's number of SMs.
template <typename K, typename V>
int radix_setup(int *sms) {
  using S = RadixShape<K, V>;
  static std::atomic<int> cached[64];
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 64 && (*sms = cached[dev].load()) > 0) return NSORT_OK;
  const void *fns[3] = {(const void *)radix_pass_kernel<K, V, S::NT, S::IPT, true, false>,
                        (const void *)radix_pass_kernel<K, V, S::NT, S::IPT, false, false>,
                        (const void *)radix_pass_kernel<K, V, S::NT, S::IPT, false, true>};
  for (const void *f : fns) {
    if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM) !=
            cudaSuccess ||
        cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, 100) != cudaSuccess)
      return NSORT_ECUDA;
  }
  if (cudaFuncSetAttribute(radix_histogram_kernel<K, HIST_NT, hist_copies<K>()>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)hist_smem<K>()) != cudaSuccess ||
      cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return NSORT_ECUDA;
  if (dev < 64) cached[dev].store(*sms);
  return NSORT_OK;
}

template <typename K, typename V>
int radix_sort_typed(const Plan &p, const K *in, const V *vin, K *out, V *vout, int dt, void *tmp,
                     cudaStream_t st) {
  using S = RadixShape<K, V>;
  int sms = 0;
  if (radix_setup<K, V>(&sms) != NSORT_OK) {
    set_last_error(std::string("radix set-up: ") + cudaGetErrorString(cudaGetLastError()));
    return NSORT_ECUDA;
  }
  const RadixLayout l = radix_layout(p, sizeof(K), S::TILE);
  char *t = static_cast<char *>(tmp);
  uint32_t *hist = reinterpret_cast<uint32_t *>(t + l.hist_off);
  uint32_t *ticket = reinterpret_cast<uint32_t *>(t + l.ticket_off);
  uint32_t *state = reinterpret_cast<uint32_t *>(t + l.state_off);
  int *status = reinterpret_cast<int *>(t + p.status_off);
  K *buf = reinterpret_cast<K *>(t + p.keys_off);
  V *vbuf = reinterpret_cast<V *>(t + p.vals_off);
  const KeyMap<K> map = key_map<K>(dt);
  cudaError_t e = cudaMemsetAsync(hist, 0, l.state_off - l.hist_off, st);
  if (e == cudaSuccess) {
    TraceScope tr(TK_RADIX_HIST, st);
    radix_histogram_kernel<K, HIST_NT, hist_copies<K>()><<<sms, HIST_NT, hist_smem<K>(), st>>>(
        in, p.n, map, hist, state, l.tiles * BINS, status);
  }
  const K *src = in;
  const V *vsrc = vin;
  constexpr int D = sizeof(K);
  for (int d = 0; d < D; ++d) {
    K *dst = (d & 1) ? out : buf;
    V *vdst = (d & 1) ? vout : vbuf;
    TraceScope tr(TK_RADIX_PASS, st);
    const uint32_t parity = (d & 1) ? 0x80000000u : 0u;
    const uint32_t *h = hist + d * BINS;
#define NSORT_RP(F, L)                                                                      \
  launch_pdl(radix_pass_kernel<K, V, S::NT, S::IPT, F, L>, (unsigned)l.tiles, S::NT, S::SMEM, st, src, vsrc, \
             dst, vdst, (uint32_t)p.n, 8 * d, map, h, state, parity, ticket + d, \
             status)
    if (d == 0) NSORT_RP(true, false);
    else if (d == D - 1) NSORT_RP(false, true);
    else NSORT_RP(false, false);
#undef NSORT_RP
    src = dst;
    vsrc = vdst;
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e == cudaSuccess) return NSORT_OK;
  set_last_error(std::string("radix pass: ") + cudaGetErrorString(e));
  return NSORT_ECUDA;
}

}  // namespace

// Whether a plan is sorted by digits: from the size on from which the counts
// of its tiles and the histograms always fit in the scratch that the merge
// passes would use for splitters and samples (the scratch of a size is the
// same either way), and while counts fit in 30 bits.  At that size it is the
// faster of the two already: 53 against 75 us for 2^21 u32 keys, 73 against
// 145 us for as many pairs, 117 against 184 us with 64-bit payloads, 122
// against 153 us for as many int64 keys.
bool radix_fits(const Plan &p, bool pairs, int key_bytes) {
  const int tile = key_bytes == 8 ? RadixShape<uint64_t, NoValue>::TILE
                                  : RadixShape<uint32_t, NoValue>::TILE;
  const int64_t least = pairs ? 9 << 17 : (key_bytes == 8 ? 15 << 17 : 17 << 17);
  return p.n >= least && p.n < (int64_t(1) << 30) &&
         radix_layout(p, key_bytes, tile).end <= p.total;
}

int radix_sort_keys(const Plan &p, const uint32_t *in, uint32_t *out, int dt, void *tmp,
                    cudaStream_t st) {
  return radix_sort_typed<uint32_t, NoValue>(p, in, nullptr, out, nullptr, dt, tmp, st);
}

int radix_sort_keys64(const Plan &p, const uint64_t *in, uint64_t *out, int dt, void *tmp,
                      cudaStream_t st) {
  return radix_sort_typed<uint64_t, NoValue>(p, in, nullptr, out, nullptr, dt, tmp, st);
}

int radix_sort_pairs(const Plan &p, const uint32_t *in, const uint32_t *vin, uint32_t *out,
                     uint32_t *vout, int dt, void *tmp, cudaStream_t st) {
  return radix_sort_typed<uint32_t, uint32_t>(p, in, vin, out, vout, dt, tmp, st);
}

int radix_sort_pairs64(const Plan &p, const uint32_t *in, const uint64_t *vin, uint32_t *out,
                       uint64_t *vout, int dt, void *tmp, cudaStream_t st) {
  return radix_sort_typed<uint32_t, uint64_t>(p, in, vin, out, vout, dt, tmp, st);
}

}  // namespace nsort
