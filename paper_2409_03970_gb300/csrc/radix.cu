// Plain sorts by digit: least-significant-digit-first passes of 8 bits (4
// passes for 32-bit keys, 8 for 64-bit keys), each one stable scatter of the
// whole array.
//
// A merge sort of n keys moves the array 1 + log2(n / tile) times (15 at
// 2^28); the digit passes move it 4 times after one read for the histograms,
// whatever the key distribution.  The result is the same: the stable order
// by key is unique.
//
//   radix_cluster_kernel     small sorts: all digits, by one cluster;
//   radix_histogram_kernel   else counts every digit of every key at once, and
//   radix_pass_kernel        takes one digit.  Each CTA takes a tile of the
//                            array in order (a ticket), counts its digits,
//                            publishes the counts, ranks its keys stably in
//                            shared memory and finds from the counts of the
//                            tiles before it where its keys go: by looking
//                            back (the single-pass prefix scheme of Merrill
//                            and Garland, "Single-pass Parallel Prefix Scan
//                            with Decoupled Look-back", 2016, applied to
//                            digit counts by Adinets and Merrill, "Onesweep",
//                            2022), or, for few tiles, by adding them all up.
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <string>
#include <type_traits>

#include "nsort.h"
#include "nsort_testing.h"
#include "launch.h"
#include "nsort_internal.h"
#include "sort_device.cuh"
#include "tma_device.cuh"

namespace nsort {

namespace {

constexpr int BINS = 256;
constexpr int WAIT_US = 2000000;   // limit of a pass's wait for other tiles

// Sets the histograms and the tickets to zero.  A kernel and not a memset,
// since kernels can be launched before their predecessors end: us, memset and
// plain launch of the histograms / this: 2^20 keys 44.8 / 39.3, 3.0e6 66.0 /
// 62.6, 200,003 pairs 35.4 / 30.8, 8.0e6 keys 131 / 125.5.  It does not release
// the histogram kernel early: the CTAs of that would crowd on the SMs that the
// last pass of a sort before leaves first (3.0e6: 74.7).
__global__ void radix_init_kernel(uint32_t *words, int n) {
  pdl_wait();
  for (int i = threadIdx.x; i < n; i += blockDim.x) words[i] = 0;
}

// ---- histograms ------------------------------------------------------------

// Counts the 8-bit digits of every (mapped) key: hist[d][b] += ....  Each lane
// group counts in its own copy of the counters (COPIES of them, copy = lane
// mod COPIES, the copies of one counter in different banks), so that equal
// digits of a warp do not queue up on one address.  Also sets the passes'
// look-back words to "no entry", the status word to NSORT_OK and the word behind
// it to the limit of the passes' waits.
// SMALL: the first pass may start to wait early (and take its tickets, which
// are zero by then: after pdl_wait).
template <typename K, int NT, int COPIES, bool SMALL>
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
  pdl_wait();
  for (int64_t i = gtid; i < state_words; i += gsize) state[i] = 0xFFFFFFFFu;
  if (gtid == 0) {
    status[0] = NSORT_OK;
    status[1] = WAIT_US;
  }
  if (SMALL) pdl_trigger();
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
// digit), else it is the tile's own, bits 29..0 the count.  Bits 30..0 all set: a
// tile up to this one gave up waiting, and there is no count (2^30 - 1 as a
// count says that no key of the digit is left in later tiles).  A word of the
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
__device__ __forceinline__ uint4 load_relaxed4(const uint4 *p) {
  uint4 v;
  asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p)
               : "memory");
  return v;
}
__device__ __forceinline__ void store_relaxed(uint32_t *p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Who writes what a kernel reads: no one in the kernel's life (the read-only
// path); the kernel before it, which may still be writing when this one starts
// (plain loads, not moved over the wait for it; ld.global.cg there costs 2-4%
// of a wave sort); or this kernel's other CTAs (loads from L2).
enum Writer { NOBODY, PREDECESSOR, THIS_KERNEL };
template <Writer W>
__device__ __forceinline__ uint32_t load_from(const uint32_t *p) {
  if constexpr (W == NOBODY) return __ldg(p);
  if constexpr (W == THIS_KERNEL) return __ldcg(p);
  uint32_t v;
  asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
template <Writer W>
__device__ __forceinline__ uint64_t load_from(const uint64_t *p) {
  if constexpr (W == NOBODY) return __ldg(p);
  if constexpr (W == THIS_KERNEL) return __ldcg(p);
  uint64_t v;
  asm volatile("ld.global.u64 %0, [%1];" : "=l"(v) : "l"(p));
  return v;
}

// Whether a wait that began at t0 (0: begins now) has lasted as many
// microseconds as the word behind the status word says.  (Read there, by a wait
// that has to wait: as an argument of the passes it costs some of them a
// register that they don't have.)
__device__ __forceinline__ bool gave_up(uint64_t &t0, const int *status) {
  const uint64_t now = global_ns();
  if (!t0) t0 = now;
  return now - t0 > load_relaxed(reinterpret_cast<const uint32_t *>(status) + 1) * 1000ull;
}

struct NoValue {};

constexpr int NT = 512;           // threads of a CTA
constexpr int WARPS = NT / 32;
constexpr int COPIES = 32;        // counters per digit: half-warps, or lanes
static_assert(NT == 2 * BINS && COPIES == 2 * WARPS, "two threads scan a digit's counters");

// Shared memory: counters | staged keys (or payloads).
template <typename K, int IPT>
constexpr size_t tile_smem() {
  return (size_t)COPIES * BINS * 4 + (size_t)(NT * IPT + NT * IPT / 512) * sizeof(K);
}

// Where position e of the tile is staged.  One word of padding per 512: in
// free order a tile of one digit gives every lane its own 512 consecutive
// positions, which would all start on one bank.
__device__ __forceinline__ uint32_t staged(uint32_t e) { return e + (e >> 9); }

// One tile's share of one digit pass, by one CTA: IPT keys per thread,
// TILE = 512 IPT in all, in chunks of 16 IPT: the first halves of the warps
// take the first 16 chunks, the second halves the others, lane l of a
// half-warp key 16 i + l of its chunk at step i.
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
// already.  A full tile whose first and last keys agree in them (every one of
// the first pass, nearly every one of the second) is ranked in any order:
// one counter per digit and lane, so that no two lanes of a warp meet on an
// address or a bank, and one atomic per key.
template <typename K, typename V, int IPT>
struct DigitTile {
  static constexpr bool PAIRS = !std::is_same<V, NoValue>::value;
  static constexpr int TILE = NT * IPT;
  static_assert(TILE <= 32768 && IPT % 4 == 0, "positions take 15 bits of a counter");
  // registers that last: pairs keep two positions a word, four digits a word
  static constexpr int NPOS = PAIRS ? IPT / 2 : 1, NDIG = PAIRS ? IPT / 4 : 1;

  struct Shared {
    uint32_t gbase[BINS];        // position of digit d's first key - its place in the tile
    uint32_t warp_sums[WARPS];
    uint32_t tile_base[BINS], tile_total[BINS];
    uint32_t tile;
    K ends[2];                   // the tile's first and last key
  };

  // counters: word (warp * 256 + digit) * 2 + half (stable), digit * 32 +
  // lane (free order)
  uint32_t *cnt;
  K *stage;
  Shared &sh;
  const int tid, lane, warp;
  const uint32_t e0;             // the thread's first key in the tile
  uint32_t sel;                  // byte of the digit
  bool upper;                    // 64-bit keys: the digit is in the upper word
  K low;                         // the digits that are sorted already
  bool free_order;
  uint32_t count;                // keys in the tile

  __device__ __forceinline__ DigitTile(unsigned char *smem, Shared &s)
      : cnt(reinterpret_cast<uint32_t *>(smem)),
        stage(reinterpret_cast<K *>(smem + (size_t)COPIES * BINS * 4)),
        sh(s),
        tid(threadIdx.x),
        lane(threadIdx.x & 31),
        warp(threadIdx.x >> 5),
        e0((uint32_t)(((threadIdx.x >> 4 & 1) * WARPS + (threadIdx.x >> 5)) * (16 * IPT) +
                      (threadIdx.x & 15))) {}

  __device__ __forceinline__ void set_digit(int shift) {
    sel = 0x4440u | (uint32_t)(shift >> 3 & 3);
    upper = shift & 32;
    low = (K(1) << shift) - 1;
  }
  __device__ __forceinline__ uint32_t digit(K k) const {
    uint32_t w;
    if constexpr (sizeof(K) == 8) w = upper ? (uint32_t)(k >> 32) : (uint32_t)k;
    else w = k;
    return __byte_perm(w, 0u, sel);
  }

  __device__ __forceinline__ void clear() {
    uint4 *c4 = reinterpret_cast<uint4 *>(cnt);
#pragma unroll
    for (int i = 0; i < COPIES * BINS / 4 / NT; ++i) c4[tid + NT * i] = make_uint4(0, 0, 0, 0);
  }

  // The tile's keys from p.
  template <Writer FROM>
  __device__ __forceinline__ void load(const K *p, K (&r)[IPT]) const {
    p += e0;
    if (count == TILE) {
#pragma unroll
      for (int i = 0; i < IPT; ++i) r[i] = load_from<FROM>(p + 16 * i);
    } else {
#pragma unroll
      for (int i = 0; i < IPT; ++i)
        r[i] = e0 + 16 * i < count ? load_from<FROM>(p + 16 * i) : K(0);
    }
  }
  // padding: the largest key, behind every real one
  __device__ __forceinline__ void pad(K (&r)[IPT]) const {
    if (count != TILE) {
#pragma unroll
      for (int i = 0; i < IPT; ++i)
        if (e0 + 16 * i >= count) r[i] = ~K(0);
    }
  }

  __device__ __forceinline__ uint32_t *my_counters() const {
    return free_order ? cnt + lane : cnt + warp * 2 * BINS + (lane >> 4);
  }

  // Counts the digits.  CLEAR: the counters were cleared before the caller's
  // last barrier; FIRST: no digit is sorted yet, so that order is free.
  template <bool CLEAR, bool FIRST>
  __device__ __forceinline__ void count_digits(const K (&r)[IPT]) {
    if constexpr (PAIRS || FIRST) {
      free_order = !PAIRS && count == TILE;
      if (!CLEAR) __syncthreads();
    } else {
      if (tid == 0) sh.ends[0] = r[0];
      if (tid == NT - 1) sh.ends[1] = r[IPT - 1];
      __syncthreads();   // (and the counters are clear)
      free_order = count == TILE && !((sh.ends[0] ^ sh.ends[1]) & low);
    }
    uint32_t *mine = my_counters();
    const uint32_t stride = free_order ? COPIES : 2;
#pragma unroll
    for (int i = 0; i < IPT; ++i) atomicAdd(mine + stride * digit(r[i]), 1u);
    __syncthreads();
  }

  // Threads 2d and 2d + 1 take 16 of digit d's counters each: those of the
  // warps' first or second halves, or (free order, so in any order) 16
  // lanes', starting at another one in every thread so that no two of a warp
  // meet on a bank.
  __device__ __forceinline__ uint32_t *counter(int j) const {
    const int d = tid >> 1;
    return free_order ? cnt + d * COPIES + ((d & (COPIES - 1)) ^ ((tid & 1) * 16) ^ j)
                      : cnt + j * 2 * BINS + tid;
  }
  // Whether the 16 counters stay in registers between half_count and
  // place_counters, two a word (a half-warp or a lane counts at most 512
  // keys).  Where the registers allow it (2.0e7 int64 keys 829 -> 805 us, 2^27
  // pairs 2.48 -> 2.43 ms); 32-bit keys and 64-bit payloads read them again
  // (2^28 u32 keys 2.78 -> 2.85 ms with them kept).
  static constexpr bool KEEP = sizeof(K) == 8 || (PAIRS && sizeof(V) == 4);
  static constexpr int NKEPT = KEEP ? 8 : 1;
  // This thread's half of digit tid >> 1's count.
  __device__ __forceinline__ uint32_t half_count(uint32_t (&kept)[NKEPT]) const {
    uint32_t own = 0;
    if constexpr (KEEP) {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint32_t a = *counter(2 * j), b = *counter(2 * j + 1);
        kept[j] = a | b << 16;
        own += a + b;
      }
    } else {
#pragma unroll 8
      for (int j = 0; j < 16; ++j) own += *counter(j);
    }
    return own;
  }

  // The sum of x over the digits below this thread's, for threads (digit
  // tid >> 1) that hold x in pairs; every thread of the CTA calls it.  A
  // barrier must lie between two calls.
  __device__ __forceinline__ uint32_t sum_below(uint32_t x) {
    uint32_t y = x;
#pragma unroll
    for (int o = 2; o < 32; o <<= 1) {
      const uint32_t z = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += z;
    }
    if (lane == 31) sh.warp_sums[warp] = y;
    __syncthreads();
    return __reduce_add_sync(0xffffffffu, lane < warp ? sh.warp_sums[lane] : 0u) + y - x;
  }

  // Counts -> positions in the tile, given the digit's place in it and what
  // of its count precedes this thread's half.
  __device__ __forceinline__ void place_counters(uint32_t run,
                                                 const uint32_t (&kept)[NKEPT]) const {
    const int up = free_order ? 0 : 16;
    if constexpr (KEEP) {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        *counter(2 * j) = run << up;
        run += kept[j] & 0xFFFFu;
        *counter(2 * j + 1) = run << up;
        run += kept[j] >> 16;
      }
    } else {
#pragma unroll 8
      for (int j = 0; j < 16; ++j) {
        uint32_t *c = counter(j);
        const uint32_t v = *c;
        *c = run << up;
        run += v;
      }
    }
    __syncthreads();
  }

  __device__ __forceinline__ uint32_t rank_stable(uint32_t *mine, K k) const {
    const int hl = lane & 15;
    uint32_t *w = mine + 2 * digit(k);
    atomicAdd(w, 1u << hl);
    __syncwarp();
    const uint32_t v = *(volatile uint32_t *)w;
    const uint32_t pos = (v >> 16) + __popc(v & ((1u << hl) - 1u));
    __syncwarp();
    if (((v & 0xFFFFu) >> hl) == 1u) *(volatile uint32_t *)w = (pos + 1u) << 16;
    __syncwarp();
    return pos;
  }

  // Ranks the thread's keys I0 .. I1 - 1 and stages them in order (the digits
  // are extracted anew: kept from the counting they would cost a register
  // per key).  FREE_PARTIAL: a partial tile's warps may rank in free order too
  // (64-bit look-back passes, with one such tile in hundreds, leave that out:
  // 2^27 int64 keys 4.89 -> 4.86 ms, 4.0e6 206.7 -> 204.5 us).
  template <int I0 = 0, int I1 = IPT, bool FREE_PARTIAL = true>
  __device__ __forceinline__ void rank(const K (&r)[IPT], uint32_t (&pos2)[NPOS]) {
    asm volatile("" : "+r"(sel));
    uint32_t *mine = my_counters();
    if constexpr (PAIRS) {
#pragma unroll
      for (int i = I0; i < I1; ++i) {
        const uint32_t pos = rank_stable(mine, r[i]);
        stage[staged(pos)] = r[i];
        if (i & 1) {
          pos2[i / 2] |= pos << 16;
          asm volatile("" : "+r"(pos2[i / 2]));   // (kept packed)
        } else {
          pos2[i / 2] = pos;
        }
      }
    } else if (free_order) {
#pragma unroll
      for (int i = I0; i < I1; ++i)
        stage[staged(atomicAdd(mine + COPIES * digit(r[i]), 1u))] = r[i];
    } else {
      // the keys of this warp may be order-free even if the tile's are not
      const K f = __shfl_sync(0xffffffffu, r[0], lane & 16) & low;
      const K l = __shfl_sync(0xffffffffu, r[IPT - 1], lane | 15) & low;
      if ((FREE_PARTIAL || count == TILE) && __all_sync(0xffffffffu, f == l)) {
        if (!FREE_PARTIAL || count == TILE) {
#pragma unroll
          for (int i = I0; i < I1; ++i)
            stage[staged(atomicAdd(mine + 2 * digit(r[i]), 1u << 16) >> 16)] = r[i];
        } else {
          // Padding takes no part.  It has the largest digit throughout, and
          // the lanes of one atomic are served in no specified order, so that
          // it could take the place of a key; its own places, all from `count`
          // on, stay empty.  (Ranked with the keys, all of it on one counter,
          // it also took longer: 4.0e6 u32 keys 83.3 -> 78.3 us, 1.2e6 int64
          // 87.9 -> 83.4.)
#pragma unroll
          for (int i = I0; i < I1; ++i)
            if (e0 + 16 * i < count)
              stage[staged(atomicAdd(mine + 2 * digit(r[i]), 1u << 16) >> 16)] = r[i];
        }
      } else {
#pragma unroll
        for (int i = I0; i < I1; ++i) stage[staged(rank_stable(mine, r[i]))] = r[i];
      }
    }
  }

  // Brings the payloads, which are loaded much later, to L2: a line a thread.
  __device__ __forceinline__ void prefetch(const V *p) const {
    if constexpr (PAIRS) {
      constexpr uint32_t LINE = 128 / sizeof(V);
#pragma unroll
      for (uint32_t l = 0; l < (TILE + LINE * NT - 1) / (LINE * NT); ++l) {
        const uint32_t e = (tid + NT * l) * LINE;
        if (e < count) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + e));
      }
    }
  }

  // Writes the staged keys to dst[gbase[digit] + position], mapped by out.
  // `checked`: positions from `count` on, or beyond n, are left out.
  template <bool MAP>
  __device__ __forceinline__ void write_keys(K *dst, uint32_t n, bool checked, KeyMap<K> out,
                                             uint32_t (&dig4)[NDIG]) const {
    if constexpr (PAIRS) {
#pragma unroll
      for (int i = 0; i < IPT; ++i) {
        const uint32_t e = (uint32_t)(tid + NT * i);
        if (i % 8 == 0) asm volatile("" : "+l"(dst)::"memory");   // (bounds the registers in use)
        const K k = stage[staged(e)];
        const uint32_t dg = digit(k);
        const uint32_t at = sh.gbase[dg] + e;
        if (!checked || (e < count && at < n)) dst[at] = MAP ? map_out(k, out) : k;
        if (i & 3) dig4[i / 4] |= dg << (8 * (i & 3));
        else dig4[i / 4] = dg;
        if (i % 4 == 3) asm volatile("" : "+r"(dig4[i / 4]));   // (kept packed)
      }
    } else if (!checked) {
#pragma unroll(IPT < 8 ? IPT : 8)
      for (int i = 0; i < IPT; ++i) {
        const uint32_t e = (uint32_t)(tid + NT * i);
        const K k = stage[staged(e)];
        dst[sh.gbase[digit(k)] + e] = MAP ? map_out(k, out) : k;
      }
    } else {
#pragma unroll 4
      for (int i = 0; i < IPT; ++i) {
        const uint32_t e = (uint32_t)(tid + NT * i);
        const K k = stage[staged(e)];
        const uint32_t at = sh.gbase[digit(k)] + e;
        if (e < count && at < n) dst[at] = MAP ? map_out(k, out) : k;
      }
    }
  }

  // The payloads, from p, take the keys' places in the staging buffer, as
  // many positions at a time as fit, and follow them.
  template <Writer FROM>
  __device__ __forceinline__ void move_values(const V *p, V *dst, uint32_t n, bool checked,
                                              const uint32_t (&pos2)[NPOS],
                                              const uint32_t (&dig4)[NDIG]) const {
    if constexpr (PAIRS) {
      constexpr int ROUNDS = sizeof(V) / sizeof(K);
      constexpr int RT = TILE / ROUNDS;
      constexpr int VB = sizeof(V) == 8 || IPT % 8 ? 4 : 8;   // loads in flight
      static_assert(IPT % VB == 0, "whole batches");
      V *vstage = reinterpret_cast<V *>(stage);
      p += e0;
#pragma unroll
      for (int q = 0; q < ROUNDS; ++q) {
        __syncthreads();   // the staging buffer has been read
        asm volatile("" : "+l"(p));   // (no addresses kept from round to round)
#pragma unroll
        for (int i0 = 0; i0 < IPT; i0 += VB) {
#pragma unroll
          for (int i = i0; i < i0 + VB; ++i) {
            const uint32_t pos = (pos2[i / 2] >> (16 * (i & 1))) & 0xFFFFu;
            if ((ROUNDS == 1 || (int)(pos / RT) == q) && e0 + 16 * i < count)
              vstage[staged(pos - q * RT)] = load_from<FROM>(p + 16 * i);
          }
          asm volatile("" ::: "memory");
        }
        __syncthreads();
        asm volatile("" : "+l"(dst));
#pragma unroll
        for (int i = 0; i < IPT / ROUNDS; ++i) {
          const int j = i + q * (IPT / ROUNDS);
          const uint32_t e = (uint32_t)(tid + NT * j);
          const uint32_t at = sh.gbase[(dig4[j / 4] >> (8 * (j & 3))) & 0xFFu] + e;
          if (!checked || (e < count && at < n)) dst[at] = vstage[staged(e - q * RT)];
        }
      }
    }
  }
};

__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// The word at shared address p of CTA c of the cluster.
__device__ __forceinline__ uint32_t load_of_cta(const uint32_t *p, uint32_t c) {
  uint32_t v;
  asm volatile(
      "{\n\t.reg .b32 a;\n\tmapa.shared::cluster.u32 a, %1, %2;\n\t"
      "ld.shared::cluster.u32 %0, [a];\n\t}"
      : "=r"(v)
      : "r"(smem_addr(p)), "r"(c)
      : "memory");
  return v;
}

// ---- one digit pass, one tile a CTA ------------------------------------------

// WAVE = false: thread d looks back over the counts of digit d in the tiles
// before this one (32-bit words, one per digit), as in the single-pass scans
// named above.  WAVE = true, for sorts of so few tiles that all of them run
// at once: every tile adds up the counts of all tiles before it, read in
// parallel (16-bit halves, two digits a word); a look-back would have to walk
// over all of them, since no tile is done before the others start.  CL > 1:
// a cluster of CL CTAs shares an entry of the counts (CL tiles in a row),
// which leaves room in the scratch for short tiles: the CTAs exchange their
// counts through distributed shared memory.  A wave pass is alive while the
// pass before it still writes (pdl_trigger), so it reads what that one and the
// histogram kernel write by loads for that (Writer); a look-back pass starts
// when its predecessor has ended, and may take the read-only path.
//
// What bounds it (ncu at 2^26 uniform u32 keys): the LSU data pipe in the
// stable passes (20-22 shared-memory wavefronts for 32 keys beside the
// scattered stores, 82-85% of the pipe's peak; 193 and 207 us), and in the
// free-order passes (11 wavefronts, 67-69%; 149-151 us) the latency of the
// phases of the two tiles an SM holds at a time.  A pass
// over 2^28 keys takes 0.65 ms on average, 3.3 TB/s of keys; 2^28 keys sort
// in 2.78 ms against 6.42 ms by merge passes, 2^27 f32 pairs in 2.43 against
// 7.19 ms, 3.0e7 pairs with 64-bit payloads in 0.96 against 2.03 ms, 2.0e7
// int64 keys in 0.81 against 1.07 ms.  Tried and slower at 2^28 keys: CTAs
// that stay for several tiles and load the next one early (2.9 to 5.2 ms:
// tickets taken early delay the counts that later tiles wait for), one CTA
// that scans all tiles' counts (4.35 ms), 32 tiles a look-back step (3.48),
// the look-back's first loads among the ranking (2.80).
//
// In a walk each CTA also asks L2 for the keys of the tile that starts about
// when this one ends.  Two tiles an SM run at once, so AHEAD tiles on is well
// before it runs and well within L2: 2^28 keys take 3.00 ms without, 2.96 with
// 20 tiles, 2.80 with 50, 2.79 with 76 to 304, 2.93 with 608 (40 MB ahead, in
// L2 beside the scattered writes).
constexpr uint32_t AHEAD = 76;   // tiles: a quarter of the 304 that run at once on 152 SMs
template <typename K, typename V, int IPT, bool FIRST, bool LAST, bool WAVE, int CL = 1>
__global__ void __launch_bounds__(NT, 2) radix_pass_kernel(
    const K *src, const V *vsrc, K *__restrict__ dst, V *__restrict__ vdst, uint32_t n, int shift,
    KeyMap<K> map_i, KeyMap<K> map_o, const uint32_t *hist, uint32_t *state, uint32_t parity,
    uint32_t *ticket, int *status) {
  using T = DigitTile<K, V, IPT>;
  extern __shared__ __align__(16) unsigned char rp_smem[];
  __shared__ typename T::Shared sh;
  T t(rp_smem, sh);
  t.set_digit(shift);
  const int tid = t.tid;
  // (the tickets were set to zero before the histogram kernel ran)
  uint32_t rank = 0;
  if constexpr (CL > 1) rank = cluster_rank();
  if (tid == 0 && rank == 0) sh.tile = atomicAdd(ticket, 1u);
  t.clear();
  uint32_t tile;   // the cluster's turn
  if constexpr (CL > 1) {
    cluster_arrive();
    cluster_wait();
    tile = load_of_cta(&sh.tile, 0);
  } else {
    __syncthreads();
    tile = sh.tile;
  }
  pdl_wait();      // the previous kernel of the stream has finished writing
  if constexpr (WAVE) pdl_trigger();   // the next pass may start to wait for this one
  const uint32_t base = (tile * CL + rank) * (uint32_t)T::TILE;
  t.count = base >= n ? 0u : (n - base < (uint32_t)T::TILE ? n - base : (uint32_t)T::TILE);
  const uint32_t count = t.count;
  K r[IPT];
  t.template load<WAVE ? PREDECESSOR : NOBODY>(src + base, r);
  // (WAVE) the digit's count in the array, asked for ahead of its use: at once
  // in the short tiles of clusters (200,003 u32 keys 28.6 -> 27.5 us), else
  // after the counting, where it keeps a register for less long (2.3e6 int64
  // keys 138.6 us, 141 at once)
  [[maybe_unused]] uint32_t digit_total = 0;
  if constexpr (WAVE && CL > 1) digit_total = load_from<PREDECESSOR>(hist + (tid >> 1));
  t.prefetch(vsrc + base);
  if constexpr (!WAVE) {   // the keys of the tile that starts when this one ends
    constexpr uint32_t LINE = 128 / sizeof(K);
    const uint32_t e = base + AHEAD * T::TILE + tid * LINE;
    static_assert(T::TILE == NT * LINE, "a line a thread");
    if (e < n) asm volatile("prefetch.global.L2 [%0];" ::"l"(src + e));
  }
  if (FIRST) {
#pragma unroll
    for (int i = 0; i < IPT; ++i) r[i] = map_in(r[i], map_i);
  }
  t.pad(r);
  t.template count_digits<true, FIRST && !LAST>(r);   // (WAVE: FIRST and LAST are set in all passes)
  const int d = tid >> 1;
  uint32_t kept[T::NKEPT];
  const uint32_t own = t.half_count(kept);
  const uint32_t other = __shfl_xor_sync(0xffffffffu, own, 1);
  const uint32_t total = own + other;
  const uint32_t flip = parity | parity >> 16;   // (WAVE) both halves' parity bits
  auto publish = [&](uint32_t c) {   // the count of an entry's tiles
    if constexpr (WAVE) {
      const uint32_t next = __shfl_down_sync(0xffffffffu, c, 2);
      if (!(tid & 3))
        store_relaxed(state + (size_t)tile * (BINS / 2) + (d >> 1), (c | next << 16) ^ flip);
    } else if (!(tid & 1) && tile) {
      store_relaxed(state + (size_t)tile * BINS + d, parity | c);
    }
  };
  if constexpr (CL == 1) publish(total);
  if (!(tid & 1)) sh.tile_total[d] = total;
  if constexpr (CL > 1) cluster_arrive();   // the count is there for the other CTAs
  if constexpr (WAVE && CL == 1) digit_total = load_from<PREDECESSOR>(hist + d);
  const uint32_t tbase = t.sum_below(total);   // where the digit starts in the tile
  if (!(tid & 1)) sh.tile_base[d] = tbase;
  t.place_counters(tbase + (tid & 1 ? other : 0u), kept);
  [[maybe_unused]] uint32_t excl0 = 0;   // (WAVE) all smaller digits, and the cluster's lower ranks
  if constexpr (WAVE) excl0 = t.sum_below(digit_total);
  if constexpr (CL > 1) {
    cluster_wait();
    uint32_t all = 0, lower = 0;
#pragma unroll
    for (int j = 0; j < CL / 2; ++j) {
      const uint32_t c = (tid & 1) * (CL / 2) + j;
      const uint32_t v = load_of_cta(&sh.tile_total[d], c);
      all += v;
      lower += c < rank ? v : 0u;
    }
    all += __shfl_xor_sync(0xffffffffu, all, 1);
    excl0 += lower + __shfl_xor_sync(0xffffffffu, lower, 1);
    if (rank == 0) publish(all);
    cluster_arrive();   // (waited for before the CTA ends: its counts have been read)
  }
  uint32_t pos2[T::NPOS];
  int flags = 0;   // 1: a digit's keys would go out of range, 2: no answer
  if constexpr (WAVE) {
    // Where the tile's keys go: warp w adds up the counts of tiles w, w + 16,
    // ..., lane l digits 8 l .. 8 l + 7; the warps' sums are added up through
    // the counters' memory.  The first loads run under the end of the ranking.
    uint32_t acc[8] = {};
    const uint4 *counts = reinterpret_cast<const uint4 *>(state) + t.lane;
    constexpr int LOADS = 4;
    uint4 v[LOADS];
    auto load_counts = [&](uint32_t q0) {
#pragma unroll
      for (int j = 0; j < LOADS; ++j) {
        const uint32_t q = q0 + WARPS * j;
        v[j] = q < tile ? load_relaxed4(counts + q * (BINS / 8)) : make_uint4(flip, flip, flip, flip);
      }
    };
    constexpr int HEAD = IPT / 8 * 4;   // (an even number: positions are kept in pairs)
    t.template rank<0, HEAD>(r, pos2);
    load_counts(t.warp);
    t.template rank<HEAD, IPT>(r, pos2);
    for (uint32_t q0 = t.warp; q0 < tile; q0 += LOADS * WARPS) {
      if (q0 != t.warp) load_counts(q0);
#pragma unroll
      for (int j = 0; j < LOADS; ++j) {
        uint64_t t0 = 0;
        for (;;) {
          uint4 x = v[j];
          x.x ^= flip; x.y ^= flip; x.z ^= flip; x.w ^= flip;
          if (!((x.x | x.y | x.z | x.w) & 0x80008000u)) {
            acc[0] += x.x & 0xFFFFu; acc[1] += x.x >> 16;
            acc[2] += x.y & 0xFFFFu; acc[3] += x.y >> 16;
            acc[4] += x.z & 0xFFFFu; acc[5] += x.z >> 16;
            acc[6] += x.w & 0xFFFFu; acc[7] += x.w >> 16;
            break;
          }
          if (flags || gave_up(t0, status)) {
            flags = 2;
            break;
          }
          v[j] = load_relaxed4(counts + (q0 + WARPS * j) * (BINS / 8));   // not there yet
        }
      }
    }
    __syncthreads();   // the counters are no longer used
    uint4 *sums = reinterpret_cast<uint4 *>(t.cnt) + t.warp * (BINS / 4) + t.lane * 2;
    sums[0] = make_uint4(acc[0], acc[1], acc[2], acc[3]);
    sums[1] = make_uint4(acc[4], acc[5], acc[6], acc[7]);
    __syncthreads();
    uint32_t x = 0;
#pragma unroll
    for (int j = 0; j < WARPS / 2; ++j) x += t.cnt[((tid & 1) * (WARPS / 2) + j) * BINS + d];
    const uint32_t excl = excl0 + x + __shfl_xor_sync(0xffffffffu, x, 1);
    if (!(tid & 1)) sh.gbase[d] = excl - tbase;
    if (excl + total > n + (d == BINS - 1 ? T::TILE - count : 0)) flags |= 1;
  } else {
    t.template rank<0, IPT, sizeof(K) == 4>(r, pos2);
    // where the tile's keys go
    uint32_t excl = 0;
    if (tile == 0) {   // the digit's first position: all keys of smaller digits
      excl = t.sum_below(hist[d]);
      if (!(tid & 1)) sh.gbase[d] = excl;
      __syncthreads();
    }
    if (tid < BINS) {
      uint32_t *word = state + (size_t)tile * BINS + tid;
      if (tile == 0) {
        excl = sh.gbase[tid];
      } else {
        // LOOK tiles at a time.  Words before tile 0's are read too (other
        // parts of the scratch) but not used: tile 0's count covers every
        // tile up to it.
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
          if (!used && gave_up(t0, status)) {
            excl = LB_COUNT;   // there is no sum, which later tiles have to see as well
            flags = 2;
            break;
          }
        } while (!done);
      }
      const uint32_t c = sh.tile_total[tid];
      store_relaxed(word, parity | LB_INCL | min(excl + c, LB_COUNT));
      sh.gbase[tid] = excl - sh.tile_base[tid];
      // holds for every digit unless a tile before gave up, or the keys changed
      // while they were sorted
      if (excl + c > n + (tid == BINS - 1 ? T::TILE - count : 0)) flags |= excl >= LB_COUNT ? 2 : 1;
    }
  }
  const bool fault = __syncthreads_or(flags);
  if (fault && __syncthreads_or(flags & 2)) {
    if (tid == 0) atomicExch(status, (int)NSORT_ETIMEOUT);
    if constexpr (CL > 1) cluster_wait();
    return;
  }
  const bool checked = fault || count != T::TILE;
  uint32_t dig4[T::NDIG];
  t.template write_keys<LAST>(dst, n, checked, map_o, dig4);
  t.template move_values<WAVE ? PREDECESSOR : NOBODY>(vsrc + base, vdst, n, checked, pos2, dig4);
  if constexpr (CL > 1) cluster_wait();
}

// ---- all digits of a small sort in one launch ------------------------------

// One cluster of CTAS CTAs sorts up to CTAS tiles: every CTA keeps its place
// in the array, and in each pass the CTAs exchange their digit counts through
// distributed shared memory and scatter to the other buffer (L2 holds both).
// Two cluster barriers a pass take the place of a launch, and no histogram
// or look-back is needed.
//
// The stream's next kernel may start (and wait) from the last scatter on.
// From the start on, each of a queue of such sorts let in the next, whose 16
// CTAs took 16 SMs each from other streams while they waited: beside a queue
// of 60,000-pair sorts, four sorts of 200,003 keys on another stream took 294
// us, now 116, as alone (191 beside the merge sorts); the queue itself got
// faster too (60,000 pairs 25.6 -> 25.1 us, 17,000 keys 17.5 -> 17.1, 100,000
// 29.0 -> 27.1).
template <typename K, typename V, int IPT, int CTAS>
__global__ void __launch_bounds__(NT, 1) radix_cluster_kernel(
    const K *in, const V *vin, K *out, V *vout, K *buf, V *vbuf, uint32_t n, KeyMap<K> map,
    int *status) {
  using T = DigitTile<K, V, IPT>;
  extern __shared__ __align__(16) unsigned char rc_smem[];
  __shared__ typename T::Shared sh;
  T t(rc_smem, sh);
  const int tid = t.tid, d = tid >> 1;
  const uint32_t rank = cluster_rank();
  const uint32_t base = rank * (uint32_t)T::TILE;
  t.count = base >= n ? 0u : (n - base < (uint32_t)T::TILE ? n - base : (uint32_t)T::TILE);
  pdl_wait();
  if (rank == 0 && tid == 0) *status = NSORT_OK;
  const K *src = in;
  const V *vsrc = vin;
#pragma unroll 1
  for (int dg = 0; dg < (int)sizeof(K); ++dg) {
    K *dst = dg & 1 ? out : buf;
    V *vdst = dg & 1 ? vout : vbuf;
    t.set_digit(8 * dg);
    t.clear();
    K r[IPT];
    t.template load<THIS_KERNEL>(src + base, r);
    t.prefetch(vsrc + base);
    if (dg == 0) {
#pragma unroll
      for (int i = 0; i < IPT; ++i) r[i] = map_in(r[i], map);
    }
    t.pad(r);
    t.template count_digits<false, false>(r);
    uint32_t kept[T::NKEPT];
    const uint32_t own = t.half_count(kept);
    const uint32_t other = __shfl_xor_sync(0xffffffffu, own, 1);
    if (!(tid & 1)) sh.tile_total[d] = own + other;
    const uint32_t tbase = t.sum_below(own + other);
    t.place_counters(tbase + (tid & 1 ? other : 0u), kept);
    cluster_arrive();   // this CTA's counts are there
    uint32_t pos2[T::NPOS];
    t.rank(r, pos2);
    cluster_wait();     // and so are the other CTAs'
    uint32_t all = 0, before = 0;
#pragma unroll
    for (int j = 0; j < CTAS / 2; ++j) {
      const uint32_t c = (tid & 1) * (CTAS / 2) + j;
      const uint32_t v = load_of_cta(&sh.tile_total[d], c);
      all += v;
      before += c < rank ? v : 0u;
    }
    all += __shfl_xor_sync(0xffffffffu, all, 1);
    before += __shfl_xor_sync(0xffffffffu, before, 1);
    const uint32_t start = t.sum_below(all);
    if (!(tid & 1)) sh.gbase[d] = start + before - tbase;
    __syncthreads();
    const bool last = dg == (int)sizeof(K) - 1;
    if (last) pdl_trigger();
    const KeyMap<K> map_o = {last ? map.arith : K(0), last ? map.flip : K(0)};
    uint32_t dig4[T::NDIG];
    // (checked throughout: the positions come from keys that were read again)
    t.template write_keys<true>(dst, n, true, map_o, dig4);
    t.template move_values<THIS_KERNEL>(vsrc + base, vdst, n, true, pos2, dig4);
    src = dst;
    vsrc = vdst;
    cluster_arrive();   // the pass is written, and no CTA reads another's counts any more
    cluster_wait();
  }
}

// ---- host side -----------------------------------------------------------------

// Scratch of a digit sort inside a merge plan's splitter and sample arrays.
struct RadixLayout {
  size_t hist_off, ticket_off, state_off, end;
  int64_t tiles;
};

RadixLayout radix_layout(const Plan &p, int key_bytes, int tile, bool wave) {
  RadixLayout l;
  l.tiles = (p.n + tile - 1) / tile;
  l.hist_off = p.split_off;
  l.ticket_off = l.hist_off + (size_t)key_bytes * BINS * 4;
  l.state_off = l.ticket_off + 256;
  l.end = l.state_off + (size_t)l.tiles * BINS * (wave ? 2 : 4);
  return l;
}

// Keys per thread of the passes of a large sort: 16384 keys or pairs, 8192
// 64-bit keys a tile, the smallest whose 32-bit counts fit in the scratch.
template <typename K>
constexpr int large_ipt() { return sizeof(K) == 8 ? 16 : 32; }

// The histogram kernel: a copy of the counters per lane (64-bit keys: for
// every other lane) in large sorts; small ones take fewer, to clear and add
// up.
constexpr int HIST_NT = 1024, HIST_SMALL_NT = 512;
template <typename K, bool SMALL>
constexpr int hist_copies() { return (sizeof(K) == 8 ? 16 : 32) / (SMALL ? 8 : 1); }
template <typename K, bool SMALL>
constexpr size_t hist_smem() { return sizeof(K) * BINS * hist_copies<K, SMALL>() * 4; }

// Keys per thread of the wave passes' tiles, while they all run at once (two
// CTAs per SM): the shortest in clusters of four (32-bit keys), else those of
// one CTA whose counts fit in the scratch, else the large sorts'.
constexpr int WAVE_CL = 4, WAVE_CL_IPT = 8;
template <typename K>
constexpr int wave_ipt() { return sizeof(K) == 8 ? 12 : 20; }

constexpr int CLUSTER = 16;   // CTAs (more than 8 need the non-portable size)

// Opts a kernel in to its shared memory.
template <typename F>
bool opt_in(F *kernel, size_t smem) {
  return cudaFuncSetAttribute((const void *)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)smem) == cudaSuccess &&
         cudaFuncSetAttribute((const void *)kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                              100) == cudaSuccess;
}

template <typename K, typename V, int IPT>
bool opt_in_cluster(cudaLaunchConfig_t *cfg, int *clusters) {
  auto kernel = radix_cluster_kernel<K, V, IPT, CLUSTER>;
  cfg->dynamicSmemBytes = tile_smem<K, IPT>();
  return opt_in(kernel, tile_smem<K, IPT>()) &&
         cudaFuncSetAttribute((const void *)kernel, cudaFuncAttributeNonPortableClusterSizeAllowed,
                              1) == cudaSuccess &&
         cudaOccupancyMaxActiveClusters(clusters, kernel, cfg) == cudaSuccess;
}

// What the device offers: how many clusters of WAVE_CL CTAs of the passes run
// at once << 16 | SMs << 1 | whether a cluster of CLUSTER CTAs fits; found, and
// the kernels of a key and payload type opted in, once per device.
template <typename K, typename V>
int radix_setup(int *sms, bool *cluster, int *wave_clusters) {
  static std::atomic<int> cached[64];
  int dev = 0, c = 0;
  cudaGetDevice(&dev);
  if (dev >= 64 || (c = cached[dev].load()) == 0) {
    constexpr int LI = large_ipt<K>(), WI = wave_ipt<K>();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CLUSTER);
    cfg.blockDim = dim3(NT);
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = CLUSTER;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int least = sizeof(K) == 8 ? 0 : 1, k = 0, wave = 0;
    if (!opt_in(radix_pass_kernel<K, V, LI, true, false, false>, tile_smem<K, LI>()) ||
        !opt_in(radix_pass_kernel<K, V, LI, false, false, false>, tile_smem<K, LI>()) ||
        !opt_in(radix_pass_kernel<K, V, LI, false, true, false>, tile_smem<K, LI>()) ||
        !opt_in(radix_pass_kernel<K, V, LI, true, true, true>, tile_smem<K, LI>()) ||
        !opt_in(radix_pass_kernel<K, V, WI, true, true, true>, tile_smem<K, WI>()) ||
        !opt_in(radix_histogram_kernel<K, HIST_NT, hist_copies<K, false>(), false>,
                hist_smem<K, false>()) ||
        !opt_in(radix_histogram_kernel<K, HIST_SMALL_NT, hist_copies<K, true>(), true>,
                hist_smem<K, true>()) ||
        cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      return NSORT_ECUDA;
    if constexpr (sizeof(K) == 4) {
      if (!opt_in(radix_pass_kernel<K, V, WAVE_CL_IPT, true, true, true, WAVE_CL>,
                  tile_smem<K, WAVE_CL_IPT>()))
        return NSORT_ECUDA;
      if (!opt_in_cluster<K, V, 4>(&cfg, &k)) return NSORT_ECUDA;
      least = k < least ? k : least;
      if (!opt_in_cluster<K, V, 8>(&cfg, &k)) return NSORT_ECUDA;
      least = k < least ? k : least;
      if (!opt_in_cluster<K, V, 16>(&cfg, &k)) return NSORT_ECUDA;
      least = k < least ? k : least;
      cfg.gridDim = dim3(WAVE_CL);
      cfg.dynamicSmemBytes = tile_smem<K, WAVE_CL_IPT>();
      attr.val.clusterDim.x = WAVE_CL;
      if (cudaOccupancyMaxActiveClusters(
              &wave, radix_pass_kernel<K, V, WAVE_CL_IPT, true, true, true, WAVE_CL>, &cfg) !=
          cudaSuccess)
        return NSORT_ECUDA;
    }
    c = wave << 16 | *sms << 1 | (least > 0 ? 1 : 0);
    if (dev < 64) cached[dev].store(c);
  }
  *sms = c >> 1 & 0x7FFF;
  *cluster = c & 1;
  *wave_clusters = c >> 16;
  return NSORT_OK;
}

int radix_status(cudaError_t e, const char *what) {
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e == cudaSuccess) return NSORT_OK;
  set_last_error(std::string(what) + ": " + cudaGetErrorString(e));
  return NSORT_ECUDA;
}

template <typename K, typename V, int IPT>
void launch_cluster(const Plan &p, const K *in, const V *vin, K *out, V *vout, int dt, char *t,
                    cudaStream_t st) {
  TraceScope tr(TK_RADIX_CLUSTER, st);
  launch_pdl<CLUSTER>(radix_cluster_kernel<K, V, IPT, CLUSTER>, CLUSTER, NT, tile_smem<K, IPT>(),
                      st, in, vin, out, vout, reinterpret_cast<K *>(t + p.keys_off),
                      reinterpret_cast<V *>(t + p.vals_off), (uint32_t)p.n, key_map<K>(dt),
                      reinterpret_cast<int *>(t + p.status_off));
}

template <typename K, typename V, int IPT, bool WAVE, int CL>
int radix_passes(const Plan &p, const RadixLayout &l, int sms, const K *in, const V *vin, K *out,
                 V *vout, int dt, char *t, cudaStream_t st) {
  uint32_t *hist = reinterpret_cast<uint32_t *>(t + l.hist_off);
  uint32_t *ticket = reinterpret_cast<uint32_t *>(t + l.ticket_off);
  uint32_t *state = reinterpret_cast<uint32_t *>(t + l.state_off);
  int *status = reinterpret_cast<int *>(t + p.status_off);
  K *buf = reinterpret_cast<K *>(t + p.keys_off);
  V *vbuf = reinterpret_cast<V *>(t + p.vals_off);
  const KeyMap<K> map = key_map<K>(dt), none = {K(0), K(0)};
  {
    TraceScope tr(TK_RADIX_HIST, st);
    launch_pdl(radix_init_kernel, 1, 1024, 0, st, hist, (int)((l.state_off - l.hist_off) / 4));
    const int64_t words = (int64_t)(l.end - l.state_off) / 4;
    if constexpr (WAVE)
      launch_pdl(radix_histogram_kernel<K, HIST_SMALL_NT, hist_copies<K, true>(), true>, sms,
                 HIST_SMALL_NT, hist_smem<K, true>(), st, in, p.n, map, hist, state, words, status);
    else
      launch_pdl(radix_histogram_kernel<K, HIST_NT, hist_copies<K, false>(), false>, sms, HIST_NT,
                 hist_smem<K, false>(), st, in, p.n, map, hist, state, words, status);
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
    const KeyMap<K> map_i = d == 0 ? map : none, map_o = d == D - 1 ? map : none;
#define NSORT_RP(F, L)                                                                          \
  launch_pdl<CL>(radix_pass_kernel<K, V, IPT, F, L, WAVE, CL>, (unsigned)l.tiles * CL, NT,      \
                 tile_smem<K, IPT>(), st, src, vsrc, dst, vdst, (uint32_t)p.n, 8 * d, map_i,    \
                 map_o, h, state, parity, ticket + d, status)
    // (few tiles: one kernel maps in every pass, by empty masks in the middle)
    if constexpr (WAVE) NSORT_RP(true, true);
    else if (d == 0) NSORT_RP(true, false);
    else if (d == D - 1) NSORT_RP(false, true);
    else NSORT_RP(false, false);
#undef NSORT_RP
    src = dst;
    vsrc = vdst;
  }
  return radix_status(cudaSuccess, "radix pass");
}

// Sorts a plan's keys by digits if there is a way to (*sorted).  The scratch of
// a size is that of the merge sort; which way is taken goes by what fits in
// it and by how many tiles the device runs at once.  us, merge passes against
// digits, u32 keys / f32 pairs / pairs with 64-bit payloads:
//   one cluster (up to 2^16, or 2^17 where the next does not fit):
//     17,000: 28 / 40 / 43 -> 17 / 20 / 22;  65,000: 42 / 53 / 55 -> 22 / 26 / 31
//   wave passes in clusters of four (4096-key tiles, as many as run at once:
//   74 on 152 SMs, 1.2 million keys; with all 76, two SMs' worth of which wait
//   for others to end, 1.22e6 u32 keys took 61 us, 40 the next way):
//     200,003: 47 / 60 / 63 -> 29 / 31 / 36;  2^20: 63 / 80 / 108 -> 39 / 44 / 52
//   wave passes of one CTA (10240- or 16384-key tiles: 5.0 million):
//     3.0e6: 127 / 210 / 249 -> 64 / 80 / 122
//   look-back passes beyond.
template <typename K, typename V>
int radix_sort_typed(const Plan &p, bool *sorted, const K *in, const V *vin, K *out, V *vout,
                     int dt, void *tmp, cudaStream_t st) {
  constexpr int LI = large_ipt<K>(), WI = wave_ipt<K>();
  *sorted = false;
  if (p.n >= (int64_t(1) << 30)) return NSORT_OK;   // (counts take 30 bits)
  // 64-bit keys take eight passes, which the merge passes beat, on sorted keys
  // at least, outside two ranges; beyond them digits are 2-4% slower on sorted
  // keys up to 2.0e6 and 10-18% faster on others, which the host can't tell
  // apart.  The lines lie where they do on 152 SMs: 5 << 17 is 0.70 of a
  // 6144-key tile on each of them, 9 << 17 0.95 of an 8192-key one.  int64,
  // uniform / sorted, merges -> digits:
  //   5.0e5: 60 / 55 -> 64 / 64;  6.6e5 (5 << 17): 77 / 69 -> 64 / 64;
  //   9.3e5: 81 / 72 -> 70 / 70;  then a larger tile: 9.5e5: 83 / 73 -> 80 / 79,
  //   1.1e6: 92 / 81 -> 82 / 82;  1.18e6 (9 << 17): 106 / 90 -> 84 / 83;
  //   then two tiles an SM: 1.3e6: 120 / 104 -> 108 / 107,
  //   2.0e6: 149 / 128 -> 132 / 131;  4.0e6: 256 / 217 -> 206 / 205.
  if (sizeof(K) == 8 && p.n < 5 << 17) return NSORT_OK;
  int sms = 0, wave_clusters = 0;
  bool cluster = false;
  if (radix_setup<K, V>(&sms, &cluster, &wave_clusters) != NSORT_OK)
    return radix_status(cudaGetLastError(), "radix set-up");
  if (sizeof(K) == 8 && p.n > (int64_t)sms * NT * WI && p.n < 9 << 17) return NSORT_OK;
  char *t = static_cast<char *>(tmp);
  RadixLayout l;
  if constexpr (sizeof(K) == 4) {
    l = radix_layout(p, sizeof(K), NT * WAVE_CL_IPT * WAVE_CL, true);
    const bool wave_fits = l.end <= p.total && l.tiles <= wave_clusters;
    const int64_t each = (p.n + CLUSTER * NT - 1) / (CLUSTER * NT);
    if (cluster && (each <= 8 || (each <= 16 && !wave_fits))) {
      *sorted = true;
      if (each <= 4) launch_cluster<K, V, 4>(p, in, vin, out, vout, dt, t, st);
      else if (each <= 8) launch_cluster<K, V, 8>(p, in, vin, out, vout, dt, t, st);
      else launch_cluster<K, V, 16>(p, in, vin, out, vout, dt, t, st);
      return radix_status(cudaSuccess, "radix cluster");
    }
    if (wave_fits) {
      *sorted = true;
      return radix_passes<K, V, WAVE_CL_IPT, true, WAVE_CL>(p, l, sms, in, vin, out, vout, dt, t,
                                                            st);
    }
  }
  if constexpr (std::is_same_v<V, NoValue>) {
    // Keys alone: rather one large tile on each SM than two small ones on some
    // and one on others, which the pass would wait for (u32, two small / one
    // large: 1.6e6: 58.7 / 52.8, 2.4e6: 63.4 / 58.9; int64: 1.2e6: 105 / 88).  A tile's payloads take
    // longer than that saves: 2.4e6 pairs 78.8 / 81.7, 64-bit payloads 116 / 129.
    l = radix_layout(p, sizeof(K), NT * LI, true);
    if (l.end <= p.total && l.tiles <= sms && p.n > (int64_t)sms * NT * WI) {
      *sorted = true;
      return radix_passes<K, V, LI, true, 1>(p, l, sms, in, vin, out, vout, dt, t, st);
    }
  }
  l = radix_layout(p, sizeof(K), NT * WI, true);
  if (l.end <= p.total && l.tiles <= 2 * sms) {
    *sorted = true;
    return radix_passes<K, V, WI, true, 1>(p, l, sms, in, vin, out, vout, dt, t, st);
  }
  l = radix_layout(p, sizeof(K), NT * LI, true);
  if (l.end <= p.total && l.tiles <= 2 * sms) {
    *sorted = true;
    return radix_passes<K, V, LI, true, 1>(p, l, sms, in, vin, out, vout, dt, t, st);
  }
  l = radix_layout(p, sizeof(K), NT * LI, false);
  if (l.end <= p.total) {
    *sorted = true;
    return radix_passes<K, V, LI, false, 1>(p, l, sms, in, vin, out, vout, dt, t, st);
  }
  return NSORT_OK;
}

// Self-test of a pass's wait for other tiles' counts: the pass's turns 1 and 2
// in a launch each, over a scratch where turn 0 never publishes any.  tmp:
// status words and limits of the two | destination | keys | histogram, ticket |
// counts.
__global__ void selftest_waits_kernel(int *status, uint32_t *ticket, int limit_us) {
  for (int turn = 0; turn < 2; ++turn) {
    status[2 * turn] = NSORT_OK;
    status[2 * turn + 1] = limit_us;
  }
  *ticket = 1;
}
template <int IPT, bool WAVE, int CL>
void selftest_waits(char *tmp, int limit_us, cudaStream_t st) {
  constexpr size_t TURN = NT * IPT * CL, N = 3 * TURN;
  constexpr size_t DST = 256, SRC = DST + N * 4, HIST = SRC + N * 4, TICKET = HIST + BINS * 4,
                   STATE = TICKET + 256, END = STATE + 3 * BINS * 4;
  static_assert(END <= NSORT_SELFTEST_DIGIT_BYTES, "fits");
  int *status = reinterpret_cast<int *>(tmp);
  uint32_t *ticket = reinterpret_cast<uint32_t *>(tmp + TICKET);
  cudaMemsetAsync(tmp + DST, 0xA5, N * 4, st);
  cudaMemsetAsync(tmp + SRC, 0, STATE - SRC, st);   // keys of one digit
  cudaMemsetAsync(tmp + STATE, 0xFF, END - STATE, st);
  selftest_waits_kernel<<<1, 1, 0, st>>>(status, ticket, limit_us);
  const KeyMap<uint32_t> none = {0u, 0u};
  const NoValue *vsrc = nullptr;
  NoValue *vdst = nullptr;
  for (int turn = 0; turn < 2; ++turn)
    launch_pdl<CL>(radix_pass_kernel<uint32_t, NoValue, IPT, WAVE, WAVE, WAVE, CL>, CL, NT,
                   tile_smem<uint32_t, IPT>(), st, reinterpret_cast<const uint32_t *>(tmp + SRC),
                   vsrc, reinterpret_cast<uint32_t *>(tmp + DST), vdst, (uint32_t)N, 0, none, none,
                   reinterpret_cast<const uint32_t *>(tmp + HIST),
                   reinterpret_cast<uint32_t *>(tmp + STATE), 0u, ticket, status + 2 * turn);
}

}  // namespace

extern "C" int nsort_selftest_digit_waits(int which, void *d_tmp, size_t tmp_bytes,
                                          uint32_t limit_us, void *stream) {
  if (which < 0 || which > 2 || limit_us > (uint32_t)WAIT_US || !d_tmp || tmp_bytes < NSORT_SELFTEST_DIGIT_BYTES ||
      (reinterpret_cast<uintptr_t>(d_tmp) & 255))
    return NSORT_EINVAL;
  int sms = 0, wave_clusters = 0;
  bool cluster = false;
  if (radix_setup<uint32_t, NoValue>(&sms, &cluster, &wave_clusters) != NSORT_OK)
    return radix_status(cudaGetLastError(), "radix set-up");
  char *t = static_cast<char *>(d_tmp);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (which == 0) selftest_waits<large_ipt<uint32_t>(), false, 1>(t, (int)limit_us, st);
  else if (which == 1) selftest_waits<wave_ipt<uint32_t>(), true, 1>(t, (int)limit_us, st);
  else selftest_waits<WAVE_CL_IPT, true, WAVE_CL>(t, (int)limit_us, st);
  return radix_status(cudaSuccess, "nsort_selftest_digit_waits");
}

int radix_sort_keys(const Plan &p, bool *sorted, const uint32_t *in, uint32_t *out, int dt,
                    void *tmp, cudaStream_t st) {
  return radix_sort_typed<uint32_t, NoValue>(p, sorted, in, nullptr, out, nullptr, dt, tmp, st);
}

int radix_sort_keys64(const Plan &p, bool *sorted, const uint64_t *in, uint64_t *out, int dt,
                      void *tmp, cudaStream_t st) {
  return radix_sort_typed<uint64_t, NoValue>(p, sorted, in, nullptr, out, nullptr, dt, tmp, st);
}

int radix_sort_pairs(const Plan &p, bool *sorted, const uint32_t *in, const uint32_t *vin,
                     uint32_t *out, uint32_t *vout, int dt, void *tmp, cudaStream_t st) {
  return radix_sort_typed<uint32_t, uint32_t>(p, sorted, in, vin, out, vout, dt, tmp, st);
}

int radix_sort_pairs64(const Plan &p, bool *sorted, const uint32_t *in, const uint64_t *vin,
                       uint32_t *out, uint64_t *vout, int dt, void *tmp, cudaStream_t st) {
  return radix_sort_typed<uint32_t, uint64_t>(p, sorted, in, vin, out, vout, dt, tmp, st);
}

}  // namespace nsort
