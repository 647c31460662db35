// nsort_segmented: many independent arrays sorted in one batch.
//
// Segments are binned by length on the device:
//   tiny   L <= W_t          one thread sorts the segment in registers with
//                            the W_t-input network (W_t = 8 or 16);
//   small  L <= 32 * IPT     one warp: column sort of IPT keys per lane and
//                            the warp flip merger (IPT = 8 or 16);
//   medium L <= 16 NT        keys: a group of 1, 2, 4 or 8 warps per segment
//                            (at most 1024 keys a warp), as many groups as fit
//                            a CTA; pairs: one CTA;
//   large  L >  16 NT        tile sorts of the segment's TILE-key tiles
//                            (level 0; keys take 32 per thread, TILE = 32 NT,
//                            pairs 16, TILE = 16 NT), then one merge level per
//                            doubling of the run length.
// A persistent kernel takes the level-0 tiles and the medium, small and tiny
// segments from a queue (one atomic counter):
// [level-0 tiles of all large segments][medium][small batches][tiny batches].
// The merge levels then run as the plain sort's bulk-copy merge passes over
// lists of merge tiles (launch_segmented_level): level k merges, in every
// segment with at least k levels, its runs of TILE * 2^(k-1) keys pairwise.
// Every step is stream-ordered, with no host synchronisation, so a batch can
// be captured into a CUDA graph: the host launches as many levels as the
// longest possible segment could need, and levels past the batch's longest
// segment find no tiles.
//
// The tunables (block size NT, tiny network width W_t, small-bin IPT, CTAs
// per SM) come from nsort_segmented_set_config, fed by the autotuner.
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <mutex>
#include <string>
#include <type_traits>

#include "nsort.h"
#include "launch.h"
#include "nsort_internal.h"
#include "sort_device.cuh"
#include "tma_device.cuh"

namespace nsort {
namespace seg {

constexpr int MAXLV = 40;          // merge levels a segment can need (2^40 keys / 4096)
constexpr int MIN_TILE = 256 * 16; // smallest tile over the configurations
constexpr int CLASSES = 4;         // medium segments of at most 1024 << c keys (pairs: all in 0)

struct Ctrl {
  int status;                          // NSORT_OK, NSORT_EINVAL (offsets), NSORT_ETIMEOUT
  int max_level;
  unsigned long long next_item;        // queue head
  unsigned long long n_tiny, n_small, n_medium[CLASSES];
  unsigned long long bucket_tiles[MAXLV + 1];   // tiles of large segments needing b levels
  unsigned long long bucket_base[MAXLV + 2];    // exclusive prefix of bucket_tiles
  unsigned long long q_medium[CLASSES], q_small, q_tiny, q_total;   // first items
  unsigned long long lvl_count[MAXLV + 2];      // merge tiles of level k (launch_segmented_level)
};

struct Params {
  const uint32_t *kin;
  uint32_t *kout;
  const uint32_t *vin;   // nullptr: keys only
  uint32_t *vout;
  uint32_t *ktmp;
  uint32_t *vtmp;
  const int64_t *off;
  int64_t nseg;
  int64_t n;
  Ctrl *ctrl;
  // Every segment is in one list only, so each array of nseg entries holds
  // two lists, one from either end: tiny and medium class 0, small and
  // medium class 1, medium classes 2 and 3.
  int *tiny_list;
  int *small_list;
  int *medium_list;
  int64_t *slot_base;    // large segment -> first slot of its tiles
  int *owner;            // slot -> large segment
  KeyMap<uint32_t> map;  // of the batch's type
  int dt;
  int tile;              // keys per level-0 tile: NT * 32 (keys) or NT * 16 (pairs)
  int mt;                // longest medium segment: NT * 16
  int nt;
  int tiny_w;            // 8 or 16
  int small_ipt;         // 8 or 16
};

__device__ __forceinline__ int ceil_log2(int64_t x) {
  int p = 0;
  while ((int64_t(1) << p) < x) ++p;
  return p;
}

// Entry i of medium class c's list.
__device__ __forceinline__ int *medium_entry(const Params &p, int c, unsigned long long i) {
  if (c == 0) return p.tiny_list + (p.nseg - 1 - (int64_t)i);
  if (c == 1) return p.small_list + (p.nseg - 1 - (int64_t)i);
  if (c == 2) return p.medium_list + i;
  return p.medium_list + (p.nseg - 1 - (int64_t)i);
}

// ---- set-up kernels ----------------------------------------------------------

// Clears the control block (a kernel and not a memset: it can be launched
// before its predecessors end, as in the digit sorts).
__global__ void seg_init_kernel(Ctrl *c) {
  static_assert(sizeof(Ctrl) % sizeof(unsigned long long) == 0, "whole words");
  pdl_wait();
  unsigned long long *w = reinterpret_cast<unsigned long long *>(c);
  for (unsigned i = threadIdx.x; i < sizeof(Ctrl) / sizeof(*w); i += blockDim.x) w[i] = 0;
}

// Bins the segments by length (the lists' order is of no matter).  A CTA adds up
// its own segments in shared memory and takes its places with one atomic add a
// list: an add a segment, all to a few addresses, took 16.9 us for 100,000 of
// them.  us in all, with the clearing kernel, before / now: 100,000 segments of
// up to 1000 keys 224 / 212, of up to 65,536 5463 / 5446; 100 of up to 64 16.2 /
// 14.2.
constexpr int BIN_NT = 256;
__global__ void __launch_bounds__(BIN_NT) seg_classify_kernel(Params p) {
  constexpr int LISTS = 2 + CLASSES;   // tiny, small, medium classes
  __shared__ unsigned count[LISTS];
  __shared__ unsigned long long base[LISTS];
  __shared__ unsigned long long tiles[MAXLV + 1], tile_base[MAXLV + 1];
  const int tid = threadIdx.x;
  if (tid < LISTS) count[tid] = 0;
  if (tid <= MAXLV) tiles[tid] = 0;
  __syncthreads();
  pdl_wait();      // the previous kernel of the stream has finished writing
  Ctrl *c = p.ctrl;
  const int64_t s = (int64_t)blockIdx.x * BIN_NT + tid;
  int list = -1, bucket = -1;
  unsigned at = 0;                    // place among the CTA's entries of the list
  unsigned long long slot = 0;        // or first slot among the CTA's of the bucket
  if (s < p.nseg) {
    const int64_t o0 = p.off[s], o1 = p.off[s + 1];
    const bool bad = o0 < 0 || o1 < o0 || o1 > p.n || (s == 0 && o0 != 0) ||
                     (s == p.nseg - 1 && o1 != p.n);
    const int64_t L = bad ? 0 : o1 - o0;
    if (bad) {
      atomicExch(&c->status, (int)NSORT_EINVAL);
    } else if (L > p.mt) {
      const int64_t T = (L + p.tile - 1) / p.tile;
      bucket = ceil_log2(T);
      slot = atomicAdd(&tiles[bucket], (unsigned long long)T);
    } else if (L > 0) {
      if (L <= p.tiny_w) {
        list = 0;
      } else if (L <= 32 * p.small_ipt) {
        list = 1;
      } else {
        list = 2;
        if (!p.vin)
          while ((1024 << (list - 2)) < L) ++list;   // (L <= 8192)
      }
      at = atomicAdd(&count[list], 1u);
    }
  }
  __syncthreads();
  if (tid < LISTS && count[tid]) {
    unsigned long long *n = tid == 0 ? &c->n_tiny : tid == 1 ? &c->n_small : &c->n_medium[tid - 2];
    base[tid] = atomicAdd(n, (unsigned long long)count[tid]);
  }
  if (tid <= MAXLV && tiles[tid]) tile_base[tid] = atomicAdd(&c->bucket_tiles[tid], tiles[tid]);
  __syncthreads();
  if (bucket >= 0) p.slot_base[s] = (int64_t)(tile_base[bucket] + slot);
  if (list == 0) p.tiny_list[base[0] + at] = (int)s;
  if (list == 1) p.small_list[base[1] + at] = (int)s;
  if (list >= 2) *medium_entry(p, list - 2, base[list] + at) = (int)s;
}

// Lays out the work queue (one warp).
__global__ void seg_plan_kernel(Params p) {
  pdl_wait();      // the previous kernel of the stream has finished writing
  Ctrl *c = p.ctrl;
  const int lane = threadIdx.x;
  if (c->status != NSORT_OK) {
    if (lane == 0) c->q_total = 0;
    return;
  }
  // exclusive prefix of the buckets' tiles, lanes taking buckets l and 32 + l
  const unsigned long long t0 = c->bucket_tiles[lane];
  const unsigned long long t1 = 32 + lane <= MAXLV ? c->bucket_tiles[32 + lane] : 0;
  unsigned long long s0 = t0, s1 = t1;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long x0 = __shfl_up_sync(0xffffffffu, s0, o);
    const unsigned long long x1 = __shfl_up_sync(0xffffffffu, s1, o);
    if (lane >= o) {
      s0 += x0;
      s1 += x1;
    }
  }
  s1 += __shfl_sync(0xffffffffu, s0, 31);
  c->bucket_base[lane] = s0 - t0;
  if (32 + lane <= MAXLV + 1) c->bucket_base[32 + lane] = s1 - t1;
  const unsigned m0 = __ballot_sync(0xffffffffu, t0 != 0), m1 = __ballot_sync(0xffffffffu, t1 != 0);
  unsigned long long base = __shfl_sync(0xffffffffu, s1, 31);
  if (lane) return;
  const unsigned long long warps = p.nt / 32;
  for (int k = CLASSES - 1; k >= 0; --k) {   // the longest first
    c->q_medium[k] = base;
    const unsigned long long per = p.vin ? 1 : warps >> k;   // segments an item
    base += (c->n_medium[k] + per - 1) / per;
  }
  c->q_small = base;
  c->q_tiny = c->q_small + (c->n_small + warps - 1) / warps;
  c->q_total = c->q_tiny + (c->n_tiny + p.nt - 1) / p.nt;
  c->max_level = m1 ? 63 - __clz(m1) : (m0 ? 31 - __clz(m0) : 0);
}

// Gives each large segment its global slot range and records the owner of
// every slot: a lane per segment, the warp together for each large one.
__global__ void seg_owner_kernel(Params p) {
  pdl_wait();      // the previous kernel of the stream has finished writing
  const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  if (p.ctrl->status != NSORT_OK) return;
  const int64_t L = w < p.nseg ? p.off[w + 1] - p.off[w] : 0;
  const bool large = L > p.mt;
  int64_t T = 0, g = 0;
  if (large) {
    T = (L + p.tile - 1) / p.tile;
    g = (int64_t)p.ctrl->bucket_base[ceil_log2(T)] + p.slot_base[w];
    p.slot_base[w] = g;
  }
  for (unsigned m = __ballot_sync(0xffffffffu, large); m; m &= m - 1) {
    const int l = __ffs(m) - 1;
    const int64_t Tl = __shfl_sync(0xffffffffu, T, l), gl = __shfl_sync(0xffffffffu, g, l);
    for (int64_t i = lane; i < Tl; i += 32) p.owner[gl + i] = (int)(w - lane + l);
  }
}

// ---- the persistent kernel ------------------------------------------------




template <typename K>
__device__ __forceinline__ K make_elem(uint32_t key, int pos) {
  if (sizeof(K) == 8) return (K)(((uint64_t)key << 32) | (uint32_t)pos);
  return (K)key;
}
template <typename K>
__device__ __forceinline__ uint32_t elem_key(K e) {
  return sizeof(K) == 8 ? (uint32_t)((uint64_t)e >> 32) : (uint32_t)e;
}
template <typename K>
__device__ __forceinline__ int elem_pos(K e) {
  return (int)((uint64_t)e & 0xFFFFu);
}

// Tile sort with an active size m (a multiple of 512, up to NT*16): only
// the first m/16 threads hold data; all threads take part in the barriers.
// On return thread t (< m/16) holds sorted elements [16t, 16t + 16).  The
// last run of a level may be short or have no partner (it stays as it is).
template <int NT, typename K>
__device__ __forceinline__ void sort_tile_dyn(K (&r)[16], K *s, int m) {
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const int e0 = tid * 16;
  if (e0 < m) {   // whole warps: m is a multiple of 512
    column_sort16(r);
    warp_merge<16>(r, lane);
  }
  if (m == 512) return;
  if (e0 < m) {
#pragma unroll
    for (int k = 0; k < 16; ++k) s[pidx<K>(e0 + k)] = r[k];
  }
  int unused[16];
#pragma unroll 1
  for (int run = 512; run < m; run <<= 1) {
    __syncthreads();
    const int g0 = e0 & ~(2 * run - 1);
    const int nb = m - g0 - run < run ? m - g0 - run : run;   // of the pair's second run
    if (e0 < m && nb > 0) {
      const int diag = e0 - g0;
      const int ai = merge_path_smem(s, g0, run, g0 + run, nb, diag);
      serial_merge<16, false>(s, g0 + ai, g0 + run, g0 + run + diag - ai, g0 + run + nb, r, unused);
    }
    if (2 * run < m) {
      __syncthreads();
      if (e0 < m) {
#pragma unroll
        for (int k = 0; k < 16; ++k) s[pidx<K>(e0 + k)] = r[k];
      }
    }
  }
}

struct Best32Columns {
  template <typename K>
  __device__ __forceinline__ static void sort(K (&r)[32]) { column_sort_net<NET_BEST, 32>(r); }
};

// What a group of warps sorts: kept in shared memory while it does, since the
// 32 keys a thread holds leave no registers for it.
struct GroupJob {
  const uint32_t *in;
  uint32_t *out;
  const uint32_t *vin;   // pairs: the payloads
  uint32_t *vout;
  int count;      // 1 .. 1024 per warp of the group (pairs: 512)
  int map;        // whether the keys are mapped back
};

// Sorts job[g], as group g of W warps of the CTA (sort_group).  Every
// thread of the group calls it, after thread 0 of the group wrote the job.
// Bound by the integer ALU pipe like the plain tile sort.  A segment costs
// as many warps as it fills (whole 16384-key tiles and power-of-two blocks
// sorted 1.2 keys of padding per 4 of log-uniform lengths), and segments of
// less than a CTA's keys share one: 5.9e8 keys in 100,000 segments up to
// 65536 long take 4.32 ms here, 5.54 before, 3.8 at the rate of the plain
// tile sort; 30,000 segments up to 20,000 long 557 us in all, 790 before.
template <int W>
__device__ __forceinline__ void group_sort(const Params &p, void *smem, GroupJob *job, int g) {
  uint32_t *s = static_cast<uint32_t *>(smem) + g * (W * group_warp_words(32));
  const int tid = threadIdx.x & (32 * W - 1);
  auto bar = [&] {
    if constexpr (W == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(32 * W) : "memory");
  };
  volatile GroupJob *j = job + g;
  bar();
  const int c0 = (tid >> 5) * 1024 + (tid & 31);   // a warp loads and stores 1024 keys in a row
  uint32_t r[32];
  int aw;   // warps that hold keys
  {
    const int left = j->count - c0;
    const uint32_t *in = j->in + c0;
    aw = (j->count + 1023) >> 10;
#pragma unroll
    for (int k = 0; k < 32; ++k) r[k] = 32 * k < left ? map_in(in[32 * k], p.map) : 0xFFFFFFFFu;
  }
  sort_group<32, W, Best32Columns>(r, s, tid, aw, bar);
  // thread t holds keys [32t, 32t + 32): staged in shared memory (padded,
  // conflict-free both ways) so that the global stores are coalesced
  // whatever the segment's alignment
  bar();   // every thread is done reading s in the last merge level
  if ((tid >> 5) < aw) {
    const int pb = pidx<uint32_t>(tid * 32);
    const KeyMap<uint32_t> map = j->map ? p.map : KeyMap<uint32_t>{0u, 0u};
#pragma unroll
    for (int k = 0; k < 32; ++k) s[pb + k] = map_out(r[k], map);
  }
  bar();
  const int left = j->count - c0;
  uint32_t *out = j->out + c0;
  const uint32_t *from = s + pidx<uint32_t>(c0);
#pragma unroll
  for (int k = 0; k < 32; ++k)
    if (32 * k < left) out[32 * k] = from[33 * k];
}

// Sorts job[0], pairs, by the whole CTA: composites of key and position, 16 a
// thread, by as many warps as hold pairs; the payloads wait in shared memory
// and are taken by position.
template <int NT>
__device__ __forceinline__ void pairs_sort(const Params &p, void *smem, volatile GroupJob *j) {
  uint64_t *s = static_cast<uint64_t *>(smem);
  uint32_t *sv = reinterpret_cast<uint32_t *>(s + merge_smem_len<uint64_t>(NT * 16, 16));
  const int tid = threadIdx.x;
  const int c0 = (tid >> 5) * 512 + (tid & 31);   // a warp loads and stores 512 pairs in a row
  __syncthreads();   // the job is there
  uint64_t r[16];
  int m;   // pairs sorted: whole warps
  {
    const int left = j->count - c0;
    const uint32_t *in = j->in + c0, *vin = j->vin + c0;
    uint32_t *to = sv + pidx<uint32_t>(c0);
    m = (j->count + 511) & ~511;
#pragma unroll
    for (int k = 0; k < 16; ++k)
      r[k] = 32 * k < left ? make_elem<uint64_t>(map_in(in[32 * k], p.map), c0 + 32 * k) : ~0ull;
#pragma unroll
    for (int k = 0; k < 16; ++k)
      if (32 * k < left) to[33 * k] = vin[32 * k];
  }
  sort_tile_dyn<NT>(r, s, m);
  // thread t holds pairs [16t, 16t + 16): staged (padded) so that the global
  // stores are coalesced whatever the segment's alignment
  __syncthreads();   // s is no longer read, the payloads are all there
  uint32_t *sk = reinterpret_cast<uint32_t *>(s);
  uint32_t *so = sk + padded_len<uint32_t>(NT * 16);
  static_assert(2 * padded_len<uint32_t>(NT * 16) <= 2 * merge_smem_len<uint64_t>(NT * 16, 16),
                "keys and payloads fit where the composites were");
  if (tid * 16 < m) {
    const KeyMap<uint32_t> map = j->map ? p.map : KeyMap<uint32_t>{0u, 0u};
    const int pb = pidx<uint32_t>(tid * 16);   // one pad block holds all 16
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      sk[pb + k] = map_out(elem_key(r[k]), map);
      so[pb + k] = sv[pidx<uint32_t>(elem_pos(r[k]) & (NT * 16 - 1))];
    }
  }
  __syncthreads();
  const int left = j->count - c0;
  uint32_t *out = j->out + c0, *vout = j->vout + c0;
  const int pf = pidx<uint32_t>(c0);
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    if (32 * k < left) {
      out[32 * k] = sk[pf + 33 * k];
      vout[32 * k] = so[pf + 33 * k];
    }
  }
}

// The medium segments of class C (at most 1024 << C keys) of one item: one
// per group of 1 << C warps.
template <int NT, int C>
__device__ __forceinline__ void medium_item(const Params &p, void *smem, GroupJob *job,
                                            unsigned long long item) {
  constexpr int W = 1 << C;
  const int g = threadIdx.x / (32 * W);
  const unsigned long long idx = item * (NT / (32 * W)) + g;
  if (idx < p.ctrl->n_medium[C]) {   // the same in all of the group
    if (!(threadIdx.x & (32 * W - 1))) {
      const int sid = *medium_entry(p, C, idx);
      const int64_t off = p.off[sid];
      job[g] = {p.kin + off, p.kout + off, nullptr, nullptr, (int)(p.off[sid + 1] - off), 1};
    }
    group_sort<W>(p, smem, job, g);
  }
}

// One warp sorts one segment of at most 32*IPT elements.
template <int IPT, bool PAIRS>
__device__ void warp_sort_segment(const Params &p, int64_t sid) {
  using K = typename std::conditional<PAIRS, uint64_t, uint32_t>::type;
  const int lane = threadIdx.x & 31;
  const int64_t off = p.off[sid];
  const int L = (int)(p.off[sid + 1] - off);
  K r[IPT];
#pragma unroll
  for (int k = 0; k < IPT; ++k) {
    const int e = lane + 32 * k;
    r[k] = e < L ? make_elem<K>(map_in(p.kin[off + e], p.map), e) : (K)~(K)0;
  }
  column_sort(r);
  warp_merge<IPT>(r, lane);
  uint32_t vo[IPT];
  const int e0 = lane * IPT;
  if (PAIRS) {
#pragma unroll
    for (int k = 0; k < IPT; ++k) vo[k] = e0 + k < L ? p.vin[off + elem_pos(r[k])] : 0u;
    __syncwarp();
  }
#pragma unroll
  for (int k = 0; k < IPT; ++k) {
    if (e0 + k < L) {
      p.kout[off + e0 + k] = map_out(elem_key(r[k]), p.map);
      if (PAIRS) p.vout[off + e0 + k] = vo[k];
    }
  }
}

// One thread sorts one segment of at most W elements.
template <int W, bool PAIRS>
__device__ void thread_sort_segment(const Params &p, int64_t sid) {
  using K = typename std::conditional<PAIRS, uint64_t, uint32_t>::type;
  const int64_t off = p.off[sid];
  const int L = (int)(p.off[sid + 1] - off);
  K r[W];
#pragma unroll
  for (int k = 0; k < W; ++k)
    r[k] = k < L ? make_elem<K>(map_in(p.kin[off + k], p.map), k) : (K)~(K)0;
  column_sort(r);
  uint32_t vo[W];
  if (PAIRS) {
#pragma unroll
    for (int k = 0; k < W; ++k) vo[k] = k < L ? p.vin[off + elem_pos(r[k])] : 0u;
  }
#pragma unroll
  for (int k = 0; k < W; ++k) {
    if (k < L) {
      p.kout[off + k] = map_out(elem_key(r[k]), p.map);
      if (PAIRS) p.vout[off + k] = vo[k];
    }
  }
}

// MINB: CTAs per SM that the registers are bounded for.  Two for keys and for
// large batches of pairs (4.4e7 pairs in 30,000 segments: 1107 against 1261
// us with one); one where the pairs fill no more than a tile per SM, when a
// tile's own time counts (100 segments of up to 65536 pairs: 109 against 119).
template <int NT, bool PAIRS, int MINB>
__global__ void __launch_bounds__(NT, MINB) seg_sort_kernel(Params p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned long long item_sh;
  // The queue's bin boundaries live in shared memory and are read per item:
  // held in registers for the whole loop they would cost the tile sorts
  // (at 2 CTAs of 512 threads, 64 registers a thread) registers they need.
  __shared__ unsigned long long q_sh[CLASSES + 3];   // medium classes, small, tiny, total
  __shared__ GroupJob job[PAIRS ? 1 : NT / 32];
  pdl_wait();      // the previous kernel of the stream has finished writing
  const int tid = threadIdx.x;
  Ctrl *c = p.ctrl;
  if (tid < CLASSES) q_sh[tid] = c->q_medium[tid];
  if (tid == 0) {
    q_sh[CLASSES] = c->q_small;
    q_sh[CLASSES + 1] = c->q_tiny;
    q_sh[CLASSES + 2] = c->q_total;
  }
  // Few items: the first half of the grid takes them all, about one CTA per
  // SM, rather than two on some SMs and none on others.
  if (2 * blockIdx.x >= gridDim.x && 2 * c->q_total <= gridDim.x) return;
  for (;;) {
    if (tid == 0) item_sh = atomicAdd(&c->next_item, 1ull);
    __syncthreads();
    const unsigned long long item = item_sh;
    const unsigned long long q_small = q_sh[CLASSES], q_tiny = q_sh[CLASSES + 1],
                             q_total = q_sh[CLASSES + 2];
    __syncthreads();
    if (item >= q_total) break;
    if (item < q_sh[CLASSES - 1]) {
      // level 0: tile sort of one tile of a large segment (the whole sort,
      // key map included, when the segment fits one tile)
      if (tid == 0) {
        const int sid = p.owner[item];
        const int64_t t = (int64_t)item - p.slot_base[sid];
        const int64_t off = p.off[sid];
        const int64_t L = p.off[sid + 1] - off;
        const int P = ceil_log2((L + p.tile - 1) / p.tile);
        const int64_t b0 = t * p.tile, at = off + b0;
        const bool tmp = P & 1;
        job[0] = {p.kin + at, (tmp ? p.ktmp : p.kout) + at, PAIRS ? p.vin + at : nullptr,
                  PAIRS ? (tmp ? p.vtmp : p.vout) + at : nullptr,
                  (int)(L - b0 < p.tile ? L - b0 : p.tile), P == 0};
      }
      if constexpr (PAIRS) pairs_sort<NT>(p, smem_raw, job);
      else group_sort<NT / 32>(p, smem_raw, job, 0);
    } else if (item < q_small) {
      if constexpr (PAIRS) {
        if (tid == 0) {
          const int sid = *medium_entry(p, 0, item - q_sh[0]);
          const int64_t off = p.off[sid];
          job[0] = {p.kin + off, p.kout + off, p.vin + off, p.vout + off,
                    (int)(p.off[sid + 1] - off), 1};
        }
        pairs_sort<NT>(p, smem_raw, job);
      } else {
        if (NT == 512 && item < q_sh[2]) medium_item<512, 3>(p, smem_raw, job, item - q_sh[3]);
        else if (item < q_sh[1]) medium_item<NT, 2>(p, smem_raw, job, item - q_sh[2]);
        else if (item < q_sh[0]) medium_item<NT, 1>(p, smem_raw, job, item - q_sh[1]);
        else medium_item<NT, 0>(p, smem_raw, job, item - q_sh[0]);
      }
    } else if (item < q_tiny) {
      const unsigned long long idx = (item - q_small) * (NT / 32) + (tid >> 5);
      if (idx < c->n_small) {
        const int sid = p.small_list[idx];
        if (p.small_ipt == 8) warp_sort_segment<8, PAIRS>(p, sid);
        else warp_sort_segment<16, PAIRS>(p, sid);
      }
    } else {
      const unsigned long long idx = (item - q_tiny) * NT + tid;
      if (idx < c->n_tiny) {
        const int sid = p.tiny_list[idx];
        if (p.tiny_w == 8) thread_sort_segment<8, PAIRS>(p, sid);
        else thread_sort_segment<16, PAIRS>(p, sid);
      }
    }
  }
}

// ---- host side -------------------------------------------------------------

struct Layout {
  size_t ctrl, keys, vals, tiny, small, medium, slot, owner, tile_seg, desc, total;
  int64_t max_tiles;   // merge tiles one level can have
};

Layout layout(uint64_t n, uint64_t nseg, bool pairs) {
  Layout l{};
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o = align_up(o + bytes, 256);
    return at;
  };
  l.ctrl = take(sizeof(Ctrl));
  l.keys = take(n * 4);
  l.vals = pairs ? take(n * 4) : 0;
  l.tiny = take(nseg * 4);
  l.small = take(nseg * 4);
  l.medium = take(nseg * 4);
  l.slot = take(nseg * 8);
  l.owner = take((2 * (n / MIN_TILE) + 2) * 4);
  // a segment of L keys has at most L / merge tile + (pairs of runs) + 1
  // merge tiles in a level, and at most L / MIN_TILE / 2 + 1 pairs of runs
  l.max_tiles = (int64_t)(n / (uint64_t)seg_merge_tile(pairs) + n / MIN_TILE + 2 * nseg + 16);
  l.tile_seg = take((size_t)l.max_tiles * 8);
  l.desc = take((size_t)l.max_tiles * seg_tile_desc_bytes());
  l.total = o;
  return l;
}

std::mutex g_cfg_mu;
nsort_seg_config g_cfg = {512, 16, 16, 0};

template <int NT, bool PAIRS>
size_t smem_bytes() {
  if (PAIRS)
    return sizeof(uint64_t) * merge_smem_len<uint64_t>(NT * 16, 16) +
           sizeof(uint32_t) * padded_len<uint32_t>(NT * 16);
  return sizeof(uint32_t) * (NT / 32) * group_warp_words(32);
}

template <int NT, bool PAIRS, int MINB>
int launch_sort(const Params &p, int blocks_per_sm, cudaStream_t st) {
  const size_t smem = smem_bytes<NT, PAIRS>();
  int dev = 0, sms = 0, occ = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaFuncSetAttribute(seg_sort_kernel<NT, PAIRS, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)smem) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, seg_sort_kernel<NT, PAIRS, MINB>, NT,
                                                    smem) !=
          cudaSuccess) {
    set_last_error(std::string("nsort_segmented set-up: ") + cudaGetErrorString(cudaGetLastError()));
    return NSORT_ECUDA;
  }
  if (occ < 1) occ = 1;
  const int per_sm = blocks_per_sm > 0 && blocks_per_sm < occ ? blocks_per_sm : occ;
  TraceScope tr(TK_SEG_SORT, st);
  launch_pdl(seg_sort_kernel<NT, PAIRS, MINB>, (unsigned)(sms * per_sm), NT, smem, st, p);
  return NSORT_OK;
}

}  // namespace seg

size_t segmented_temp_bytes(int kind, uint64_t n, uint64_t nseg) {
  if (kind != NSORT_KIND_SEGMENTED && kind != NSORT_KIND_SEGMENTED_PAIRS) return 0;
  return seg::layout(n, nseg, kind == NSORT_KIND_SEGMENTED_PAIRS).total;
}

}  // namespace nsort

using namespace nsort;

extern "C" int nsort_segmented_set_config(const nsort_seg_config *cfg) {
  if (!cfg) return NSORT_EINVAL;
  if ((cfg->block_threads != 256 && cfg->block_threads != 512) ||
      (cfg->tiny_width != 8 && cfg->tiny_width != 16) ||
      (cfg->small_ipt != 8 && cfg->small_ipt != 16) || cfg->blocks_per_sm < 0)
    return NSORT_EINVAL;
  std::lock_guard<std::mutex> lk(seg::g_cfg_mu);
  seg::g_cfg = *cfg;
  return NSORT_OK;
}

extern "C" int nsort_segmented_get_config(nsort_seg_config *cfg) {
  if (!cfg) return NSORT_EINVAL;
  std::lock_guard<std::mutex> lk(seg::g_cfg_mu);
  *cfg = seg::g_cfg;
  return NSORT_OK;
}

namespace nsort {

int segmented_impl(const void *d_keys_in, void *d_keys_out, const uint32_t *d_vals_in,
                   uint32_t *d_vals_out, const int64_t *d_offsets, uint64_t nseg, uint64_t n,
                   int dtype, void *d_tmp, size_t tmp_bytes, void *stream, uint64_t max_seg_len) {
  if (dtype != NSORT_U32 && dtype != NSORT_I32 && dtype != NSORT_F32) return NSORT_EINVAL;
  if (n > MAX_KEYS || nseg >= (uint64_t(1) << 31)) return NSORT_EINVAL;
  if ((d_vals_in == nullptr) != (d_vals_out == nullptr)) return NSORT_EINVAL;
  if (nseg == 0) return n == 0 ? NSORT_OK : NSORT_EINVAL;
  if (!d_offsets || (n > 0 && (!d_keys_in || !d_keys_out))) return NSORT_EINVAL;
  const uintptr_t al = reinterpret_cast<uintptr_t>(d_keys_in) |
                       reinterpret_cast<uintptr_t>(d_keys_out) |
                       reinterpret_cast<uintptr_t>(d_vals_in) |
                       reinterpret_cast<uintptr_t>(d_vals_out);
  if ((al & 3) || (reinterpret_cast<uintptr_t>(d_offsets) & 7)) return NSORT_EINVAL;
  const bool pairs = d_vals_in != nullptr;
  const seg::Layout l = seg::layout(n, nseg, pairs);
  if (!d_tmp || tmp_bytes < l.total) return NSORT_ENOMEM;
  if (reinterpret_cast<uintptr_t>(d_tmp) & 255) return NSORT_EINVAL;
  nsort_seg_config cfg;
  {
    std::lock_guard<std::mutex> lk(seg::g_cfg_mu);
    cfg = seg::g_cfg;
  }
  char *t = static_cast<char *>(d_tmp);
  seg::Params p;
  p.kin = static_cast<const uint32_t *>(d_keys_in);
  p.kout = static_cast<uint32_t *>(d_keys_out);
  p.vin = d_vals_in;
  p.vout = d_vals_out;
  p.ktmp = reinterpret_cast<uint32_t *>(t + l.keys);
  p.vtmp = pairs ? reinterpret_cast<uint32_t *>(t + l.vals) : nullptr;
  p.off = d_offsets;
  p.nseg = (int64_t)nseg;
  p.n = (int64_t)n;
  p.ctrl = reinterpret_cast<seg::Ctrl *>(t + l.ctrl);
  p.tiny_list = reinterpret_cast<int *>(t + l.tiny);
  p.small_list = reinterpret_cast<int *>(t + l.small);
  p.medium_list = reinterpret_cast<int *>(t + l.medium);
  p.slot_base = reinterpret_cast<int64_t *>(t + l.slot);
  p.owner = reinterpret_cast<int *>(t + l.owner);
  p.map = key_map<uint32_t>(dtype);
  p.dt = dtype;
  p.nt = cfg.block_threads;
  p.mt = cfg.block_threads * 16;
  p.tile = pairs ? p.mt : cfg.block_threads * 32;
  p.tiny_w = cfg.tiny_width;
  p.small_ipt = cfg.small_ipt;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const unsigned cblocks = (unsigned)((nseg + seg::BIN_NT - 1) / seg::BIN_NT);
  {
    TraceScope tr(TK_SEG_BIN, st);
    launch_pdl(seg::seg_init_kernel, 1, 128, 0, st, p.ctrl);
    launch_pdl(seg::seg_classify_kernel, cblocks, seg::BIN_NT, 0, st, p);
    launch_pdl(seg::seg_plan_kernel, 1, 32, 0, st, p);
    launch_pdl(seg::seg_owner_kernel, cblocks, seg::BIN_NT, 0, st, p);
  }
  int rc;
  const int per_sm = cfg.blocks_per_sm;
  int dev = 0, sms = 0;
  if (pairs && (cudaGetDevice(&dev) != cudaSuccess ||
                cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)) {
    set_last_error(std::string("nsort_segmented set-up: ") + cudaGetErrorString(cudaGetLastError()));
    return NSORT_ECUDA;
  }
  if (!pairs)
    rc = p.nt == 512 ? seg::launch_sort<512, false, 2>(p, per_sm, st)
                     : seg::launch_sort<256, false, 2>(p, per_sm, st);
  else if (p.nt == 512)
    rc = n <= (uint64_t)sms * p.tile ? seg::launch_sort<512, true, 1>(p, per_sm, st)
                                     : seg::launch_sort<512, true, 2>(p, per_sm, st);
  else
    rc = seg::launch_sort<256, true, 2>(p, per_sm, st);
  if (rc != NSORT_OK) return rc;
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_last_error(std::string("nsort_segmented: ") + cudaGetErrorString(e));
    return NSORT_ECUDA;
  }
  // the merge levels: as many as a segment of max_seg_len keys would need
  // (the host does not know the batch's longest segment; later levels find
  // no tiles)
  const uint64_t longest = max_seg_len < n ? max_seg_len : n;
  const int64_t tiles0 = ((int64_t)longest + p.tile - 1) / p.tile;
  int levels = 0;
  while ((int64_t(1) << levels) < tiles0) ++levels;
  SegLevelArgs a;
  a.off = d_offsets;
  a.nseg = (int64_t)nseg;
  a.n = (int64_t)n;
  a.min_len = p.mt;
  a.tile = p.tile;
  a.dt = dtype;
  a.kout = p.kout;
  a.ktmp = p.ktmp;
  a.vout = pairs ? p.vout : nullptr;
  a.vtmp = pairs ? p.vtmp : nullptr;
  a.status = &p.ctrl->status;
  a.max_level = &p.ctrl->max_level;
  a.tile_seg = reinterpret_cast<int64_t *>(t + l.tile_seg);
  a.desc = t + l.desc;
  a.max_tiles = l.max_tiles;
  for (int k = 1; k <= levels && k <= seg::MAXLV; ++k) {
    a.k = k;
    a.count = &p.ctrl->lvl_count[k];
    rc = launch_segmented_level(a, st);
    if (rc != NSORT_OK) return rc;
  }
  return NSORT_OK;
}

}  // namespace nsort

extern "C" int nsort_segmented(const void *d_keys_in, void *d_keys_out, const uint32_t *d_vals_in,
                               uint32_t *d_vals_out, const int64_t *d_offsets, uint64_t nseg,
                               uint64_t n, int dtype, void *d_tmp, size_t tmp_bytes,
                               void *stream) {
  return segmented_impl(d_keys_in, d_keys_out, d_vals_in, d_vals_out, d_offsets, nseg, n, dtype,
                        d_tmp, tmp_bytes, stream, n);
}

