// Plain sorts of at most one tile: one CTA, by the warps that the keys fill.
//
// Such a sort takes as long as one SM takes for it, so its size decides the
// shape: 8 keys a thread while latency counts, 32 where the SM's integer
// pipe does.  us for n keys (u32, back to back in a graph), before / now:
//   512: 2.2 / 2.1 (32 threads x 16);       1000: 4.9 / 3.5 (128 x 8);
//   2000: 5.4 / 4.8 (256 x 8);              4096: 12.6 / 7.3 (512 x 8);
//   6000: 13.5 / 10.9 (1024 x 8);           7000: 14.4 / 12.0 (256 x 32);
//   10,000: 23.7 / 16.2, 16384: 20.4 / 20.9 (512 x 32).
// 8192 keys, all of 512 x 16, keep the block sort with constant bounds (11.5;
// 12.2 at 256 x 32).  Pairs, which all took 512 x 16: 1000: 25 / 6.6 (128 x 8),
// 4096: 29 / 15.7 (512 x 8), 8192: 27.2 / 26.6 (512 x 16).  64-bit keys, all
// 256 x 16 before: 1000: 12.6 / 5.5 (128 x 8), 4096: 13.0 / 13.2 (256 x 16).
// (The larger shapes were one of 512 x 16 up to 8192 and one of 512 x 32
// above, all of whose threads worked whatever n was.)
//
// They are dependent launches that let the stream's next kernel be launched
// (and wait) as soon as they start, so that sorts that follow one another
// don't pay for a launch each: 1000 keys 6.2 -> 4.6 us a call, back to back,
// 1000 64-bit keys 8.4 -> 5.7, 500 pairs 8.4 -> 5.7, 10,000 keys 18.7 -> 16.5.
// (So calls gain where a graph of them does not: 16384 keys 23.1 -> 20.7, 4096
// 64-bit keys 15.0 -> 13.5, with the shapes.)  Those that wait take an SM each;
// beside a queue of them another stream's sorts took at most 9% longer than alone.
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

#include "nsort.h"
#include "launch.h"
#include "nsort_internal.h"
#include "sort_device.cuh"
#include "tma_device.cuh"

namespace nsort {

namespace {

struct Columns {
  template <typename K, int W>
  __device__ __forceinline__ static void sort(K (&r)[W]) { column_sort_net<NET_BEST, W>(r); }
};

struct CtaBarrier {
  __device__ __forceinline__ void operator()() const { __syncthreads(); }
};

// Thread t's IPT consecutive words, 128 bits at a time where that is allowed.
template <int IPT, typename K>
__device__ __forceinline__ void store_words(const K (&o)[IPT], K *out, int n) {
  const int e0 = threadIdx.x * IPT;
  constexpr int EPV = 16 / sizeof(K);
  if (e0 + IPT <= n && !(reinterpret_cast<uintptr_t>(out) & 15)) {
#pragma unroll
    for (int q = 0; q < IPT / EPV; ++q) {
      uint4 v;
      if constexpr (EPV == 4)
        v = make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
      else
        v = make_uint4((uint32_t)o[2 * q], (uint32_t)(o[2 * q] >> 32), (uint32_t)o[2 * q + 1],
                       (uint32_t)(o[2 * q + 1] >> 32));
      reinterpret_cast<uint4 *>(out + e0)[q] = v;
    }
  } else {
#pragma unroll
    for (int k = 0; k < IPT; ++k)
      if (e0 + k < n) out[e0 + k] = o[k];
  }
}

// n keys (at most 32 W IPT) by one CTA of W warps.  in may equal out: every
// key is read before the first barrier, or, when one warp holds them all,
// before its first shuffle.  FULL: n = 32 W IPT, with every bound of the
// merges a constant.
template <int W, int IPT, typename K, bool FULL = false>
__global__ void __launch_bounds__(32 * W) small_keys_kernel(const K *in, K *out, int n,
                                                            KeyMap<K> map) {
  extern __shared__ __align__(16) unsigned char sk_smem[];   // W * group_warp_words<K>(IPT) keys
  pdl_trigger();
  pdl_wait();
  const int tid = threadIdx.x;
  const int c0 = (tid >> 5) * (32 * IPT) + (tid & 31);   // a warp loads 32 IPT keys in a row
  K r[IPT];
  constexpr int EPV = 16 / sizeof(K);
  if (c0 - (tid & 31) + 32 * IPT <= n && !(reinterpret_cast<uintptr_t>(in) & 15)) {
    const uint4 *p = reinterpret_cast<const uint4 *>(in) + (c0 - (tid & 31)) / EPV + (tid & 31);
#pragma unroll
    for (int q = 0; q < IPT / EPV; ++q) {   // a full warp: in any order, 128 bits a load
      const uint4 v = p[32 * q];
      if constexpr (EPV == 4) {
        r[4 * q] = v.x;
        r[4 * q + 1] = v.y;
        r[4 * q + 2] = v.z;
        r[4 * q + 3] = v.w;
      } else {
        r[2 * q] = (K)v.y << (4 * sizeof(K)) | v.x;
        r[2 * q + 1] = (K)v.w << (4 * sizeof(K)) | v.z;
      }
    }
    if (map.flip) {   // (not for unsigned keys)
#pragma unroll
      for (int k = 0; k < IPT; ++k) r[k] = map_in(r[k], map);
    }
  } else {
#pragma unroll
    for (int k = 0; k < IPT; ++k) r[k] = c0 + 32 * k < n ? map_in(in[c0 + 32 * k], map) : ~K(0);
  }
  K *s = reinterpret_cast<K *>(sk_smem);
  if constexpr (FULL)
    sort_tile_in_block<32 * W, IPT, Columns>(r, s);
  else
    sort_group<IPT, W, Columns>(r, s, tid, (n + 32 * IPT - 1) / (32 * IPT), CtaBarrier());
  if (map.flip) {
#pragma unroll
    for (int k = 0; k < IPT; ++k) r[k] = map_out(r[k], map);
  }
  store_words<IPT>(r, out, n);
}

// n pairs: composites of key and position (distinct, so their order is the
// stable one); the payloads wait in shared memory and are taken by position.
template <int W, int IPT, typename V>
__global__ void __launch_bounds__(32 * W) small_pairs_kernel(const uint32_t *kin, const V *vin,
                                                             uint32_t *kout, V *vout, int n,
                                                             KeyMap<uint32_t> map) {
  extern __shared__ __align__(16) unsigned char sp_smem[];
  pdl_trigger();
  pdl_wait();
  uint64_t *s = reinterpret_cast<uint64_t *>(sp_smem);
  V *sv = reinterpret_cast<V *>(s + W * group_warp_words<uint64_t>(IPT));   // 32 W IPT payloads
  const int tid = threadIdx.x;
  const int c0 = (tid >> 5) * (32 * IPT) + (tid & 31);
  uint64_t r[IPT];
#pragma unroll
  for (int k = 0; k < IPT; ++k) {
    const int e = c0 + 32 * k;
    r[k] = e < n ? ((uint64_t)map_in(kin[e], map) << 32) | (uint32_t)e : ~0ull;
    if (e < n) sv[e] = vin[e];
  }
  const int aw = (n + 32 * IPT - 1) / (32 * IPT);
  sort_group<IPT, W, Columns>(r, s, tid, aw, CtaBarrier());
  if (aw == 1) __syncwarp();   // (else the merges' barriers lie between)
  uint32_t ko[IPT];
  V vo[IPT];
#pragma unroll
  for (int k = 0; k < IPT; ++k) {
    ko[k] = map_out((uint32_t)(r[k] >> 32), map);
    const uint32_t e = (uint32_t)r[k];
    vo[k] = e < (uint32_t)n ? sv[e] : V(0);
  }
  store_words<IPT>(ko, kout, n);
  store_words<IPT>(vo, vout, n);
}

// Opts a kernel (one per instantiation) in to its shared memory, once per
// device.
template <auto KERNEL>
bool opt_in(size_t smem) {
  if (smem <= 48 * 1024) return true;
  static std::atomic<uint64_t> done_mask{0};
  int dev = 0;
  cudaGetDevice(&dev);
  const uint64_t bit = dev < 64 ? (uint64_t(1) << dev) : 0;
  if (bit && (done_mask.load() & bit)) return true;
  if (cudaFuncSetAttribute((const void *)KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)smem) != cudaSuccess)
    return false;
  done_mask.fetch_or(bit);
  return true;
}

template <int W, int IPT, bool FULL = false, typename K>
void launch_keys(const K *in, K *out, int n, int dt, cudaStream_t st) {
  constexpr size_t smem = sizeof(K) * W * group_warp_words<K>(IPT);
  static_assert(W * group_warp_words<K>(IPT) >= block_smem_len<K>(32 * W, IPT), "FULL fits too");
  if (opt_in<small_keys_kernel<W, IPT, K, FULL>>(smem))
    launch_pdl(small_keys_kernel<W, IPT, K, FULL>, 1, 32 * W, smem, st, in, out, n, key_map<K>(dt));
}

template <int W, int IPT, typename V>
void launch_pairs(const uint32_t *kin, const V *vin, uint32_t *kout, V *vout, int n, int dt,
                  cudaStream_t st) {
  constexpr size_t smem = sizeof(uint64_t) * W * group_warp_words<uint64_t>(IPT) +
                          sizeof(V) * 32 * W * IPT;
  if (opt_in<small_pairs_kernel<W, IPT, V>>(smem))
    launch_pdl(small_pairs_kernel<W, IPT, V>, 1, 32 * W, smem, st, kin, vin, kout, vout, n,
               key_map<uint32_t>(dt));
}

template <typename V>
void small_pairs(const uint32_t *kin, const V *vin, uint32_t *kout, V *vout, int n, int dt,
                 cudaStream_t st) {
  if (n <= 256) launch_pairs<1, 8>(kin, vin, kout, vout, n, dt, st);
  else if (n <= 1024) launch_pairs<4, 8>(kin, vin, kout, vout, n, dt, st);
  else if (n <= 2048) launch_pairs<8, 8>(kin, vin, kout, vout, n, dt, st);
  else if (n <= 4096) launch_pairs<16, 8>(kin, vin, kout, vout, n, dt, st);
  else launch_pairs<16, 16>(kin, vin, kout, vout, n, dt, st);
}

}  // namespace

void small_sort_keys(const uint32_t *in, uint32_t *out, int n, int dt, cudaStream_t st) {
  if (n <= 512) launch_keys<1, 16>(in, out, n, dt, st);
  else if (n <= 1024) launch_keys<4, 8>(in, out, n, dt, st);
  else if (n <= 2048) launch_keys<8, 8>(in, out, n, dt, st);
  else if (n <= 4096) launch_keys<16, 8>(in, out, n, dt, st);
  else if (n <= 6144) launch_keys<32, 8>(in, out, n, dt, st);
  else if (n < 8192) launch_keys<8, 32>(in, out, n, dt, st);
  else if (n == 8192) launch_keys<16, 16, true>(in, out, n, dt, st);
  else launch_keys<16, 32>(in, out, n, dt, st);
}

void small_sort_keys64(const uint64_t *in, uint64_t *out, int n, int dt, cudaStream_t st) {
  if (n <= 256) launch_keys<1, 8>(in, out, n, dt, st);
  else if (n <= 1024) launch_keys<4, 8>(in, out, n, dt, st);
  else if (n <= 2048) launch_keys<8, 8>(in, out, n, dt, st);
  else if (n <= 3072) launch_keys<16, 8>(in, out, n, dt, st);
  else launch_keys<8, 16>(in, out, n, dt, st);
}

void small_sort_pairs(const uint32_t *kin, const uint32_t *vin, uint32_t *kout, uint32_t *vout,
                      int n, int dt, cudaStream_t st) {
  small_pairs(kin, vin, kout, vout, n, dt, st);
}

void small_sort_pairs64(const uint32_t *kin, const uint64_t *vin, uint32_t *kout, uint64_t *vout,
                        int n, int dt, cudaStream_t st) {
  small_pairs(kin, vin, kout, vout, n, dt, st);
}

}  // namespace nsort
