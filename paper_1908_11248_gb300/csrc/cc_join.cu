// Join of two children sorted by bag mapping and trial (Section 3.1, join rule).
//
// The rule combines entries of equal (phi, trial): C = C' | C'' whenever C' and C'' share exactly
// the bag's colours, counts multiplied and equal results summed.  With both children sorted by
// (phi, trial) the entries concerned are two contiguous ranges, and every result has the same
// (phi, trial), so a group is one warp's work from the first read to the last write: its results
// are accumulated in shared memory, one 64-bit sum per set of private colours (a colour of the
// bag is in every set), and leave in increasing order.  The output is dense and sorted like
// the children, so a join or a grouped introduce above it needs no sort.
//
// Steps: the groups of table a are listed (count, scan, write); one thread per group finds its
// range in table b by a binary search (one dependent load after another, so a thread per group
// and not a warp: up to 2048 searches an SM, some 310 000 on 152 of them, hide each other); a warp
// per group counts its results, a scan places them, a second pass writes them.
//
// What bounds it: per group the pair tests (|A| x |B| / 32 warp steps with the records in
// registers) and the clearing and scanning of 2^(k-b) sums (3.3 with 1.0 million entries into 4.8:
// the counting pass 0.17 ms and the writing one 0.24, SM throughput 58 and 67 %, DRAM 6 %), and the
// searches (0.03 ms, 17 of 27 cycles between a warp's instructions on dependent loads).  The hash join it
// replaces walks one chain of dependent loads per probe thread and inserts every pair into a
// global hash table.  The three joins of the 9-vertex tree A of Fig. 1
// (Barabasi-Albert n = 20000, m = 4; 4 trials; 10.7, 14.4 and 29.6 million entries in): 52.3 ms
// through hash tables, 5.8 ms here, 1.8 of it the sorts of children that come unsorted.
// Sums for more than kJoinBits private colours do not fit a warp's share of shared memory, and
// for few entries the sorts and launches cost more than the chains: those joins stay with the
// hash tables (cc_kernels.cu).
#include <algorithm>
#include <cstdint>

#include "cc_device.cuh"
#include "cc_internal.h"

namespace cc {
namespace {

using namespace dev;

constexpr int kJoinWarps = 4;

// first record of the sorted table [lo, hi) whose (slots, trial) is not before q
template <typename K>
__device__ __forceinline__ u64 group_bound(const Slot<K> *s, u64 lo, u64 hi, const SortSpec &sp,
                                           K q) {
  while (lo < hi) {
    const u64 mid = (lo + hi) >> 1;
    K km;
    u64 c;
    load_slot(s, mid, km, c);
    if (sort_key<K>(km, sp) < q) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// end of the run of records equal to s[lo] in everything but the colour set (k bits)
template <typename K>
__device__ __forceinline__ u64 group_end(const Slot<K> *s, u64 lo, u64 n, int k, K g) {
  u64 step = 1, in = lo;  // s[in] is in the run
  K key;
  u64 c;
  while (in + step < n) {
    load_slot(s, in + step, key, c);
    if ((key >> k) != g) break;
    in += step;
    step <<= 1;
  }
  u64 hi = in + step < n ? in + step : n;  // the first one outside is in (in, hi]
  while (in + 1 < hi) {
    const u64 mid = (in + hi) >> 1;
    load_slot(s, mid, key, c);
    if ((key >> k) == g) in = mid;
    else hi = mid;
  }
  return in + 1;
}

// the private colours of a set as a dense index: the bits of `bag` taken out
__device__ __forceinline__ uint32_t squeeze(uint32_t set, uint32_t bag) {
  while (bag) {
    const int p = 31 - __clz(bag);
    const uint32_t low = (1u << p) - 1u;
    set = (set & low) | ((set >> 1) & ~low);
    bag &= low;
  }
  return set;
}
__device__ __forceinline__ uint32_t unsqueeze(uint32_t idx, uint32_t bag) {
  for (uint32_t rest = bag; rest; rest &= rest - 1) {
    const uint32_t low = (rest & (~rest + 1u)) - 1u;
    idx = (idx & low) | ((idx & ~low) << 1);
  }
  return idx | bag;
}

template <typename K>
__device__ __forceinline__ bool starts_group(const Slot<K> *s, u64 i, int k) {
  if (i == 0) return true;
  K a, b;
  u64 c;
  load_slot(s, i, a, c);
  load_slot(s, i - 1, b, c);
  return (a >> k) != (b >> k);
}

// groups of table a starting in each block's contiguous range, to blk[block]
template <typename K>
__global__ void __launch_bounds__(256) join_heads_count_kernel(JoinGroupArgs a, u64 *blk) {
  __shared__ u64 s_red[8];
  const Slot<K> *ta = reinterpret_cast<const Slot<K> *>(a.a.slots);
  const u64 n = block_run_failed(a.err) ? 0 : table_bound<K>(a.a);
  const u64 G = gridDim.x, per = (n + G - 1) / G;
  const u64 lo = blockIdx.x * per, hi = min(n, lo + per);
  u64 heads = 0;
  for (u64 i = lo + threadIdx.x; i < hi; i += 256) heads += starts_group(ta, i, a.L.k);
  heads = block_sum<256>(heads, s_red);
  if (threadIdx.x == 0) blk[blockIdx.x] = heads;
}

__global__ void __launch_bounds__(1024) join_heads_scan_kernel(u64 *blk, int G, u64 *groups) {
  block_scan_array(blk, blk + G, (u64)G, groups);
}

// their first records, in order
template <typename K>
__global__ void __launch_bounds__(256) join_heads_list_kernel(JoinGroupArgs a, const u64 *blk) {
  __shared__ int s_wc[8];
  const Slot<K> *ta = reinterpret_cast<const Slot<K> *>(a.a.slots);
  const u64 n = block_run_failed(a.err) ? 0 : table_bound<K>(a.a);
  const u64 G = gridDim.x, per = (n + G - 1) / G;
  const u64 lo = blockIdx.x * per, hi = min(n, lo + per);
  u64 at = blk[G + blockIdx.x];
  for (u64 base = lo; base < hi; base += 256) {
    const u64 i = base + threadIdx.x;
    const bool head = i < hi && starts_group(ta, i, a.L.k);
    int tot;
    const int rank = block_flag_rank<256>(head, s_wc, tot);
    if (head) a.first[at + rank] = i;
    at += (u64)tot;
  }
}

// each group's range in table b (a group holds at most 2^(k-b) records: one per colour set)
template <typename K>
__global__ void __launch_bounds__(256) join_match_kernel(JoinGroupArgs a) {
  const Slot<K> *ta = reinterpret_cast<const Slot<K> *>(a.a.slots);
  const Slot<K> *tb = reinterpret_cast<const Slot<K> *>(a.b.slots);
  const u64 nb = block_run_failed(a.err) ? 0 : table_bound<K>(a.b);
  const u64 groups = *a.groups;
  for (u64 g = blockIdx.x * 256ull + threadIdx.x; g < groups; g += gridDim.x * 256ull) {
    K key, kb;
    u64 c;
    load_slot(ta, a.first[g], key, c);
    const u64 lo = group_bound(tb, 0, nb, a.sp, sort_key<K>(key, a.sp));
    unsigned len = 0;
    if (lo < nb) {
      load_slot(tb, lo, kb, c);
      if ((kb >> a.L.k) == (key >> a.L.k))
        len = (unsigned)(group_end(tb, lo, nb, a.L.k, key >> a.L.k) - lo);
    }
    a.blo[g] = lo;
    a.blen[g] = len;
  }
}

// the pairs of entries that share a group (the exact run's, for the plan; in the kernel above the sum
// would cost half of the searches in flight)
template <typename K>
__global__ void __launch_bounds__(256) join_tested_kernel(JoinGroupArgs a) {
  __shared__ u64 s_red[8];
  const u64 groups = block_run_failed(a.err) ? 0 : *a.groups, na = table_bound<K>(a.a);
  u64 tested = 0;
  for (u64 g = blockIdx.x * 256ull + threadIdx.x; g < groups; g += gridDim.x * 256ull)
    tested += ((g + 1 < groups ? a.first[g + 1] : na) - a.first[g]) * a.blen[g];
  tested = block_sum<256>(tested, s_red);
  if (threadIdx.x == 0 && tested) atomicAdd(a.tested, tested);
  if (blockIdx.x == 0 && threadIdx.x == 0) *a.n_groups = groups;
}

// MODE 0: the number of results of every group to cnt; MODE 1: the results themselves at the
// offsets made from those counts; MODE 2: as 0, and the matching pairs (their count costs the
// first pass a twentieth, so they are counted once, when a plan wants them).
template <typename K, int MODE>
__global__ void __launch_bounds__(32 * kJoinWarps) join_group_kernel(JoinGroupArgs a) {
  extern __shared__ u64 s_dyn[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int k = a.L.k;
  const unsigned m = 1u << (k - a.bag), words = m > 32 ? m / 32 : 1;
  constexpr bool WRITE = MODE == 1;
  u64 *acc = s_dyn + (size_t)w * m;  // WRITE
  unsigned *bits = reinterpret_cast<unsigned *>(s_dyn + (WRITE ? (size_t)kJoinWarps * m : 0)) +
                   (size_t)w * words;
  const Slot<K> *ta = reinterpret_cast<const Slot<K> *>(a.a.slots);
  const Slot<K> *tb = reinterpret_cast<const Slot<K> *>(a.b.slots);
  Slot<K> *out = reinterpret_cast<Slot<K> *>(a.out.slots);
  const bool failed = warp_run_failed(a.err);
  const u64 na = failed ? 0 : table_bound<K>(a.a);
  const u64 groups = failed ? 0 : *a.groups;
  const u64 warps = (u64)gridDim.x * kJoinWarps;
  const uint32_t cmask = (uint32_t)((1ull << k) - 1ull);
  bool full = false;
  unsigned hits = 0;  // MODE 2: pairs of this lane
  for (u64 base = ((u64)blockIdx.x * kJoinWarps + w) * 32; base < groups; base += warps * 32) {
    const u64 g = base + lane;
    u64 af = 0, ae = 0, bf = 0;
    unsigned bl = 0;
    if (g < groups) {
      af = a.first[g];
      ae = g + 1 < groups ? a.first[g + 1] : na;
      bf = a.blo[g];
      bl = a.blen[g];
      if (!WRITE && bl == 0) a.cnt[g] = 0;
    }
    for (unsigned todo = __ballot_sync(0xffffffffu, bl != 0); todo; todo &= todo - 1) {
      const int l = __ffs(todo) - 1;
      const u64 a0 = __shfl_sync(0xffffffffu, af, l), a1 = __shfl_sync(0xffffffffu, ae, l);
      const u64 b0 = __shfl_sync(0xffffffffu, bf, l);
      const u64 b1 = b0 + __shfl_sync(0xffffffffu, bl, l);
      K gkey;  // the group's mapping and trial
      u64 gc;
      load_slot(ta, a0, gkey, gc);
      uint32_t bagc = 0;
      if (lane < a.bag)
        bagc = 1u << a.G.colors[(u64)key_trial(gkey, a.L) * (u64)a.G.n +
                                (u64)key_slot(gkey, a.L, lane)];
      bagc = __reduce_or_sync(0xffffffffu, bagc);
      for (unsigned j = lane; j < words; j += 32) bits[j] = 0;
      if (WRITE)
        for (unsigned j = lane; j < m; j += 32) acc[j] = 0;
      __syncwarp();
      for (u64 x0 = a0; x0 < a1; x0 += 32) {
        const u64 x = x0 + lane;
        uint32_t ca = ~0u;  // lanes without a record match nothing
        u64 c1 = 0;
        if (x < a1) {
          K kx;
          load_slot(ta, x, kx, c1);
          ca = squeeze((uint32_t)kx & cmask, bagc);
        }
        for (u64 y0 = b0; y0 < b1; y0 += 32) {
          const u64 y = y0 + lane;
          uint32_t cb = 0;
          u64 c2 = 0;
          if (y < b1) {
            K ky;
            load_slot(tb, y, ky, c2);
            cb = squeeze((uint32_t)ky & cmask, bagc);
          }
          const int ny = b1 - y0 < 32 ? (int)(b1 - y0) : 32;
          for (int j = 0; j < ny; ++j) {
            const uint32_t cj = __shfl_sync(0xffffffffu, cb, j);
            const u64 dj = WRITE ? __shfl_sync(0xffffffffu, c2, j) : 0;
            if (ca != ~0u && (ca & cj) == 0) {
              const uint32_t s = ca | cj;
              atomicOr(&bits[s >> 5], 1u << (s & 31));
              if (WRITE) atomicAdd(&acc[s], c1 * dj);
              if (MODE == 2) ++hits;
            }
          }
        }
      }
      __syncwarp();
      if (!WRITE) {
        unsigned n = 0;
        for (unsigned j = lane; j < words; j += 32) n += __popc(bits[j]);
        n = __reduce_add_sync(0xffffffffu, n);
        if (lane == 0) a.cnt[base + l] = n;
      } else {
        u64 pos = a.off[base + l];
        for (unsigned j0 = 0; j0 < words; ++j0) {
          const unsigned word = bits[j0];
          if (!word) continue;
          const u64 at = pos + __popc(word & lt);
          if (word >> lane & 1u) {
            const uint32_t s = j0 * 32 + lane;
            if (at < a.out.cap)
              store_slot(out, at, (gkey & ~(K)cmask) | (K)unsqueeze(s, bagc), acc[s]);
            else
              full = true;
          }
          pos += __popc(word);
        }
      }
      __syncwarp();  // the sums are cleared for the next group
    }
  }
  if (MODE == 2) {
    u64 all = hits;
    for (int o = 16; o > 0; o >>= 1) all += __shfl_down_sync(0xffffffffu, all, o);
    if (lane == 0 && all) atomicAdd(a.pairs, all);
  }
  if (full) atomicOr(a.err, kErrOverflow);
}

size_t join_smem(int mode, int private_colours) {
  const size_t m = size_t(1) << private_colours, words = m > 32 ? m / 32 : 1;
  return kJoinWarps * ((mode == 1 ? m * sizeof(u64) : 0) + words * sizeof(unsigned));
}

}  // namespace

int prepare_join_kernels() {
  const int bytes = (int)join_smem(1, kJoinBits);
  return (int)cudaFuncSetAttribute(join_group_kernel<u64, 1>,
                                   cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) |
         (int)cudaFuncSetAttribute(join_group_kernel<u128, 1>,
                                   cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

int launch_join_match(cudaStream_t s, const DevInfo &d, int kw, const JoinGroupArgs &a,
                      unsigned long long *blk) {
  const int G = sort_grid(d);
#define CC_JM(K)                                                                     \
  join_heads_count_kernel<K><<<G, 256, 0, s>>>(a, blk);                              \
  join_heads_scan_kernel<<<1, 1024, 0, s>>>(blk, G, a.groups);                       \
  join_heads_list_kernel<K><<<G, 256, 0, s>>>(a, blk);                               \
  join_match_kernel<K><<<G, 256, 0, s>>>(a)
  if (kw == 1) {
    CC_JM(u64);
  } else {
    CC_JM(u128);
  }
#undef CC_JM
  return (int)cudaGetLastError();
}

int launch_join_tested(cudaStream_t s, const DevInfo &d, int kw, const JoinGroupArgs &a) {
  if (kw == 1) join_tested_kernel<u64><<<sort_grid(d), 256, 0, s>>>(a);
  else join_tested_kernel<u128><<<sort_grid(d), 256, 0, s>>>(a);
  return (int)cudaGetLastError();
}

int launch_join_groups(cudaStream_t s, const DevInfo &d, int kw, int mode,
                       const JoinGroupArgs &a) {
  const size_t smem = join_smem(mode, a.L.k - a.bag);
  // resident blocks: at most 2048 threads and 227 KB of shared memory an SM
  const int per_sm = std::max(1, std::min(2048 / (32 * kJoinWarps),
                                          (int)(220 * 1024 / (smem + 1024))));
  const int grid = d.sms * per_sm;
#define CC_JG(K, M) join_group_kernel<K, M><<<grid, 32 * kJoinWarps, smem, s>>>(a)
  if (kw == 1) {
    if (mode == 0) CC_JG(u64, 0);
    else if (mode == 1) CC_JG(u64, 1);
    else CC_JG(u64, 2);
  } else {
    if (mode == 0) CC_JG(u128, 0);
    else if (mode == 1) CC_JG(u128, 1);
    else CC_JG(u128, 2);
  }
#undef CC_JG
  return (int)cudaGetLastError();
}

}  // namespace cc
