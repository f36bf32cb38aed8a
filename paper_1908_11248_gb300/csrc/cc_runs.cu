// Introduce run by run, for many colourings at once.
//
// All trials share the host graph, so whether a vertex v may extend a mapping phi is the same in
// all of them up to the colours.  A child table sorted by mapping holds a run of entries, one per
// (trial, colour set), for every phi.  This file works on (run, candidate) pairs instead of
// entries: the pairs are listed with the number of entries each yields; when the parent forgets
// a vertex they are sorted by the mapping that is left (one 16-byte record a pair, the slots'
// bits only), and every pair's entries are written where they belong in the result, which is then
// sorted without any of its own records having moved.  A mapping that several pairs lead to can
// have equal entries: those pairs' entries go to a side buffer that is sorted and reduced as any
// forget's records are, and follow the others in the result (two sorted regions; every run of
// equal mappings lies in one of them).
//
// Why: the passes of a record sort move every entry six or seven times at half of HBM bandwidth.
// With T trials a pair stands for up to T entries (41 of them in the first forget of the 2x4 grid
// with 64 colourings, 20 in the 3x3 grid's with 32), and the entries of a run are read as four
// bytes each (trial and colour set) from L2.  What is left is the write of the result.
// Introduce, sort and reduce of the first forget of the 3x3 grid (Erdos-Renyi, n = 100 000, degree
// 10, 32 colourings; 221 million entries of 11 million pairs): 3.1 + 16.7 + 2.7 ms entry by entry,
// 4.4 ms here.  Of the three big ones of the 2x4 grid (Barabasi-Albert, n = 20 000, 64 colourings;
// 159, 154 and 90 million entries): 40 ms entry by entry, 11 here.
//
// Entries nobody reads.  When the vertex above the forget has every F-neighbour of the forgotten
// one among its own (the opposite corner of a 4-cycle, IntroArgs::twin), a mapping that only one
// pair leads to has no candidate there: that candidate could have been the forgotten vertex's
// image, and the mapping would have a second pair.  A run that keeps no tables counts the entries of
// such pairs and does not write them (`drop`): the 2x4 grid with 64 colourings 20.0 to 18.3 ms, with
// 13 (n = 4999) 3.62 to 3.53.
//
// Below a join the result's order saves a sort of its own.  With fewer than kRunYield entries a
// pair, a pair's record is no smaller than what it stands for; where most mappings have several
// origins (a forget that leaves one vertex) most entries would be sorted in the side buffer after
// all: the entry kernels take those nodes, and those of fewer than kRunTrials trials below a forget
// or above a leaf.  An exact run, which knows neither, goes by what the runs' lengths and random
// colours let it expect, before any pair is listed; what it has counted it also writes.  The
// 9-vertex tree (Barabasi-Albert, n = 20 000, 4 colourings), whose stored introduces yield 15 to
// 100 entries a pair: 8.5 to 7.8 ms a run; a batch of partial k-trees with 4 colourings is the same
// with the line at 4 trials as at 8 (9.07 and 8.99 ms).
#include <algorithm>
#include <cstdint>

#include "cc_device.cuh"
#include "cc_internal.h"

namespace cc {
namespace {

using namespace dev;

// colT[v * T + t] = colors[t * n + v]: the trials of one vertex side by side
__global__ void __launch_bounds__(256) runs_colours_kernel(const uint8_t *colors, int n, int T,
                                                           uint8_t *colT) {
  __shared__ uint8_t s[32][33];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  for (int v0 = blockIdx.x * 32; v0 < n; v0 += gridDim.x * 32)
    for (int t0 = 0; t0 < T; t0 += 32) {
      for (int r = y; r < 32; r += 8)
        if (t0 + r < T && v0 + x < n) s[r][x] = colors[(u64)(t0 + r) * (u64)n + (u64)(v0 + x)];
      __syncthreads();
      for (int r = y; r < 32; r += 8)
        if (v0 + r < n && t0 + x < T) colT[(u64)(v0 + r) * (u64)T + (u64)(t0 + x)] = s[x][r];
      __syncthreads();
    }
}

// the bag slots of a key, from bit 0
template <typename K>
__device__ __forceinline__ u64 phi_bits(K key, const RunsArgs &a) {
  return (u64)(key >> a.L.k) & ((1ull << (a.b_in * a.L.nb)) - 1ull);
}

template <typename K>
__device__ __forceinline__ bool starts_run(const Slot<K> *s, u64 i, const RunsArgs &a) {
  if (i == 0) return true;
  K x, y;
  u64 c;
  load_slot(s, i, x, c);
  load_slot(s, i - 1, y, c);
  return phi_bits(x, a) != phi_bits(y, a);
}

template <typename K>
__device__ __forceinline__ u64 child_bound(const RunsArgs &a) {
  return table_bound<K>(a.child);
}

// runs of the child starting in each block's range, to blk[block]
template <typename K>
__global__ void __launch_bounds__(256) runs_count_kernel(RunsArgs a, u64 *blk) {
  __shared__ u64 s_red[8];
  const Slot<K> *in = reinterpret_cast<const Slot<K> *>(a.child.slots);
  const u64 n = block_run_failed(a.err) ? 0 : child_bound<K>(a);
  const u64 G = gridDim.x, per = (n + G - 1) / G;
  const u64 lo = blockIdx.x * per, hi = min(n, lo + per);
  u64 heads = 0;
  for (u64 i = lo + threadIdx.x; i < hi; i += 256) heads += starts_run(in, i, a);
  heads = block_sum<256>(heads, s_red);
  if (threadIdx.x == 0) blk[blockIdx.x] = heads;
}

__global__ void __launch_bounds__(1024) runs_scan_kernel(u64 *blk, int G, u64 *total) {
  block_scan_array(blk, blk + G, (u64)G, total);
}

// their first entries, and every entry's trial and colour set in four bytes
template <typename K>
__global__ void __launch_bounds__(256) runs_list_kernel(RunsArgs a, const u64 *blk) {
  __shared__ int s_wc[8];
  const Slot<K> *in = reinterpret_cast<const Slot<K> *>(a.child.slots);
  const u64 n = block_run_failed(a.err) ? 0 : child_bound<K>(a);
  const u64 G = gridDim.x, per = (n + G - 1) / G;
  const u64 lo = blockIdx.x * per, hi = min(n, lo + per);
  u64 at = blk[G + blockIdx.x];
  for (u64 base = lo; base < hi; base += 256) {
    const u64 i = base + threadIdx.x;
    bool head = false;
    if (i < hi) {
      K key;
      u64 c;
      load_slot(in, i, key, c);
      a.packed[i] = (unsigned)key_trial(key, a.L) << a.L.k | key_mask(key, a.L);
      head = starts_run(in, i, a);
    }
    int tot;
    const int rank = block_flag_rank<256>(head, s_wc, tot);
    if (head && at + rank < a.run_cap) a.first[at + rank] = i;
    at += (u64)tot;
  }
}

__device__ __forceinline__ u64 run_count(const RunsArgs &a) { return min(*a.n_runs, a.run_cap); }

// a leaf's run (one host vertex) exists if the vertex passes the leaf's filters
__device__ __forceinline__ bool leaf_ok(const RunsArgs &a, int v) {
  return (a.leaf_degF == 0 || a.G.deg8[v] >= a.leaf_degF) &&
         (!a.G.allow || (a.G.allow[v] & a.leaf_ubit));
}

// candidates of every run (the neighbours of its anchor's image), and in all the candidates of its
// entries, the most entries there can be
template <typename K>
__global__ void __launch_bounds__(256) runs_degree_kernel(RunsArgs a) {
  __shared__ u64 s_red[8];
  const Slot<K> *in = reinterpret_cast<const Slot<K> *>(a.child.slots);
  const bool failed = block_run_failed(a.err);
  const u64 runs = failed ? 0 : run_count(a);
  const u64 n_in = a.leaf || failed ? 0 : child_bound<K>(a);
  u64 most = 0;
  for (u64 r = blockIdx.x * 256ull + threadIdx.x; r < runs; r += gridDim.x * 256ull) {
    unsigned d = 0;
    int w = (int)r;
    if (!a.leaf) {
      K key;
      u64 c;
      if (a.anchor >= 0) {
        load_slot(in, a.first[r], key, c);
        w = key_slot(key, a.L, a.anchor);
      }
    }
    if (!a.leaf || leaf_ok(a, w))
      d = a.anchor < 0 ? (unsigned)a.G.n : (unsigned)(a.G.row_ptr[w + 1] - a.G.row_ptr[w]);
    a.deg[r] = d;
    most += d * (a.leaf ? (u64)a.trials : (r + 1 < runs ? a.first[r + 1] : n_in) - a.first[r]);
  }
  most = block_sum<256>(most, s_red);
  if (threadIdx.x == 0 && most) atomicAdd(a.n_most, most);
}

// One thread a pair: its record (the mapping it leads to with a marker bit above, its slot and
// the number of entries it yields), or a hole.
template <typename K>
__global__ void __launch_bounds__(256) runs_pairs_kernel(RunsArgs a) {
  __shared__ u64 s_red[8];
  const Slot<K> *in = reinterpret_cast<const Slot<K> *>(a.child.slots);
  Slot<u64> *recs = reinterpret_cast<Slot<u64> *>(a.recs);
  const bool failed = block_run_failed(a.err);
  const u64 runs = failed ? 0 : run_count(a);
  const u64 pairs = failed ? 0 : min(*a.n_slots, a.pair_cap);
  const u64 n_in = a.leaf || failed ? 0 : child_bound<K>(a);
  const int T = a.trials, k = a.L.k, nb = a.L.nb;
  const uint32_t cmask = (uint32_t)((1ull << k) - 1ull);
  const u64 vm = (1ull << nb) - 1ull;
  u64 valid = 0, total = 0;
  for (u64 j = blockIdx.x * 256ull + threadIdx.x; j < pairs; j += gridDim.x * 256ull) {
    u64 lo = 0, hi = runs;  // the last run whose first slot is not beyond j
    while (lo + 1 < hi) {
      const u64 mid = (lo + hi) >> 1;
      if (a.off[mid] <= j) lo = mid;
      else hi = mid;
    }
    const u64 r = lo;
    u64 phi = r, e0 = 0, e1 = (u64)T;
    if (!a.leaf) {
      K key;
      u64 c;
      e0 = a.first[r];
      e1 = r + 1 < runs ? a.first[r + 1] : n_in;
      load_slot(in, e0, key, c);
      phi = phi_bits(key, a);
    }
    int v = (int)(j - a.off[r]);
    if (a.anchor >= 0) v = __ldg(a.G.col + a.G.row_ptr[(int)(phi >> (a.anchor * nb) & vm)] + v);
    unsigned cnt = 0;
    if ((a.degF == 0 || a.G.deg8[v] >= a.degF) && (!a.G.allow || (a.G.allow[v] & a.ubit))) {
      const uint8_t *cv = a.colT + (u64)v * (u64)T;
      if (a.leaf) {
        const uint8_t *cr = a.colT + r * (u64)T;
        for (int t = 0; t < T; ++t) cnt += cv[t] != cr[t];
      } else {
#pragma unroll 8
        for (u64 e = e0; e < e1; ++e) {  // (unrolled: the loads of eight entries overlap)
          const uint32_t pk = __ldg(a.packed + e);
          cnt += !((pk & cmask) >> __ldg(cv + (pk >> k)) & 1u);
        }
      }
    }
    u64 key = 0;
    if (cnt) {  // v inserted as slot p, slot q taken out
      u64 f = phi;
      if (a.q != a.p) {
        const u64 low = (1ull << (a.p * nb)) - 1ull;
        f = (f & low) | (u64)(unsigned)v << (a.p * nb) | (f & ~low) << nb;
        if (a.q >= 0) {
          const u64 lq = (1ull << (a.q * nb)) - 1ull;
          f = (f & lq) | (f >> nb & ~lq);
        }
      }
      key = f | 1ull << (a.b_out * nb);
      ++valid;
      total += cnt;
    }
    store_slot(recs, j, key, j | (u64)cnt << 32);
    a.prow[j] = (unsigned)r;
    a.pv[j] = v;
  }
  valid = block_sum<256>(valid, s_red);
  if (threadIdx.x == 0 && valid) atomicAdd(a.n_pairs, valid);
  total = block_sum<256>(total, s_red);
  if (threadIdx.x == 0 && total) atomicAdd(a.n_total, total);
}

// pairs to write; a list with more than its room is not read at all (the run is repeated)
__device__ __forceinline__ u64 list_count(const RunsArgs &a, bool failed) {
  const u64 n = *a.n_list;
  return failed || n > a.list_cap ? 0 : n;
}

// The pair records of one window of 32: whether a lane's pair is the only one of its mapping
// (always, when nothing is forgotten).
__device__ __forceinline__ bool alone(const Slot<u64> *recs, u64 i, u64 n, u64 key, bool merge) {
  if (!merge) return true;
  u64 x, c;
  if (i > 0) {
    load_slot(recs, i - 1, x, c);
    if (x == key) return false;
  }
  if (i + 1 < n) {
    load_slot(recs, i + 1, x, c);
    if (x == key) return false;
  }
  return true;
}

// entries of every window of 32 pairs: those of pairs alone with their mapping, the others'
__global__ void __launch_bounds__(256) runs_windows_kernel(RunsArgs a) {
  const int lane = threadIdx.x & 31;
  const Slot<u64> *list = reinterpret_cast<const Slot<u64> *>(a.list);
  const u64 n = list_count(a, *a.err != 0);
  const u64 windows = (a.list_cap + 31) / 32, warps = (u64)gridDim.x * 8;
  for (u64 w = blockIdx.x * 8ull + (threadIdx.x >> 5); w < windows; w += warps) {
    const u64 i = w * 32 + lane;
    unsigned one = 0, more = 0;
    if (i < n) {
      u64 key, c;
      load_slot(list, i, key, c);
      if (key) (alone(list, i, n, key, a.merge) ? one : more) = (unsigned)(c >> 32);
    }
    one = __reduce_add_sync(0xffffffffu, one);
    more = __reduce_add_sync(0xffffffffu, more);
    if (lane == 0) {
      a.win_one[w] = one;
      a.win_more[w] = more;
    }
  }
}

// Writes the entries of the listed pairs: a warp takes 32 pairs, and 32 entries of their runs a
// step, of one run or (short runs) of several laid end to end; as the offsets are exact, its
// results are one stretch of the output (and one of the side buffer).
constexpr int kRunLong = 20;  // entries a run from which pairs are written one after the other

template <typename K>
__global__ void __launch_bounds__(256, 5) runs_write_kernel(RunsArgs a) {
  const Slot<K> *in = reinterpret_cast<const Slot<K> *>(a.child.slots);
  Slot<K> *out = reinterpret_cast<Slot<K> *>(a.out.slots);
  Slot<K> *side = reinterpret_cast<Slot<K> *>(a.side);
  const Slot<u64> *list = reinterpret_cast<const Slot<u64> *>(a.list);
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const bool failed = warp_run_failed(a.err);
  const u64 n = list_count(a, failed);
  const u64 runs = failed ? 0 : run_count(a);
  const u64 n_in = a.leaf || failed ? 0 : child_bound<K>(a);
  const u64 windows = (n + 31) / 32, warps = (u64)gridDim.x * 8;
  const int T = a.trials, k = a.L.k;
  const uint32_t cmask = (uint32_t)((1ull << k) - 1ull);
  const u64 marker = 1ull << (a.b_out * a.L.nb);
  bool full = false;
  for (u64 w = blockIdx.x * 8ull + (threadIdx.x >> 5); w < windows; w += warps) {
    const u64 i = w * 32 + lane;
    u64 key = 0, e0 = 0;
    int len = 0, v = 0;
    bool one = false;
    if (i < n) {
      u64 c;
      load_slot(list, i, key, c);
      one = key && alone(list, i, n, key, a.merge);
      if (key && !(one && a.drop)) {
        const u64 j = c & 0xffffffffull, r = a.prow[j];
        v = a.pv[j];
        if (a.leaf) {
          e0 = r;
          len = T;
        } else {
          e0 = a.first[r];
          len = (int)((r + 1 < runs ? a.first[r + 1] : n_in) - e0);
        }
      }
    }
    const unsigned ones = __ballot_sync(0xffffffffu, one);
    const u64 phi = key & (marker - 1ull);
    int incl = len;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const int excl = incl - len, total = __shfl_sync(0xffffffffu, incl, 31);
    u64 at = a.off_one[w], at2 = a.off_more[w];
    // one step: the lane's entry, if any, of a pair (its run's entries from oe on; leaf vertex oe)
    auto step = [&](bool have, u64 oe, int x, u64 ophi, int ov, bool mine) {
      uint32_t t = 0, m = 0;
      bool ok = false;
      u64 e = 0;
      if (have) {
        if (a.leaf) {
          t = (uint32_t)x;
          m = 1u << a.colT[oe * (u64)T + t];
        } else {
          e = oe + (u64)x;
          const uint32_t pk = __ldg(a.packed + e);
          t = pk >> k;
          m = pk & cmask;
        }
        const uint32_t c = 1u << a.colT[(u64)ov * (u64)T + t];
        ok = !(m & c);
        m |= c;
      }
      const unsigned b1 = __ballot_sync(0xffffffffu, ok && mine);
      const unsigned b2 = __ballot_sync(0xffffffffu, ok && !mine);
      if (ok) {
        K okey = (K)ophi << k | (K)m;
        if (a.L.tb) okey |= (K)t << a.L.tpos;
        u64 c = 1;
        if (!a.ones) {
          K ignored;
          load_slot(in, e, ignored, c);
        }
        const u64 pos = mine ? at + __popc(b1 & lt) : at2 + __popc(b2 & lt);
        if (pos < (mine ? a.out.cap : a.side_cap)) store_slot(mine ? out : side, pos, okey, c);
        else full = true;
      }
      at += __popc(b1);
      at2 += __popc(b2);
    };
    if (total >= 32 * kRunLong) {  // long runs: one pair after the other, 32 of its entries a step
      for (unsigned todo = __ballot_sync(0xffffffffu, len > 0); todo; todo &= todo - 1) {
        const int l = __ffs(todo) - 1;
        const u64 oe = __shfl_sync(0xffffffffu, e0, l), ophi = __shfl_sync(0xffffffffu, phi, l);
        const int ol = __shfl_sync(0xffffffffu, len, l), ov = __shfl_sync(0xffffffffu, v, l);
        const bool mine = ones >> l & 1u;
#pragma unroll 4
        for (int x0 = 0; x0 < ol; x0 += 32) step(x0 + lane < ol, oe, x0 + lane, ophi, ov, mine);
      }
      continue;
    }
    for (int x0 = 0; x0 < total; x0 += 32) {  // short ones end to end
      const int x = x0 + lane;
      int lo = 0, hi = 31;  // owner: smallest lane with incl > x
#pragma unroll
      for (int i5 = 0; i5 < 5; ++i5) {
        const int mid = (lo + hi) >> 1;
        const int y = __shfl_sync(0xffffffffu, incl, mid);
        if (y > x) hi = mid;
        else lo = mid + 1;
      }
      const u64 oe = __shfl_sync(0xffffffffu, e0, lo), ophi = __shfl_sync(0xffffffffu, phi, lo);
      const int ox = __shfl_sync(0xffffffffu, excl, lo), ov = __shfl_sync(0xffffffffu, v, lo);
      step(x < total, oe, x - ox, ophi, ov, ones >> lo & 1u);
    }
  }
  if (full) atomicOr(a.err, kErrOverflow);
}

// the merged side entries behind the others (with `drop` they are all there is, in place), and the
// sizes: |D_x| counts the entries before equal ones are merged
template <typename K>
__global__ void __launch_bounds__(256) runs_append_kernel(RunsArgs a, const void *merged,
                                                          const u64 *n_merged, u64 *size_x,
                                                          u64 *size_f) {
  const Slot<K> *in = reinterpret_cast<const Slot<K> *>(merged);
  Slot<K> *out = reinterpret_cast<Slot<K> *>(a.out.slots);
  const u64 n = *n_merged, at = *a.n_one;
  for (u64 i = blockIdx.x * 256ull + threadIdx.x; i < n && !a.drop; i += gridDim.x * 256ull) {
    K key;
    u64 c;
    load_slot(in, i, key, c);
    if (at + i < a.out.cap) store_slot(out, at + i, key, c);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *size_x = at + *a.n_more;
    *size_f = at + n;
    if (a.drop) *a.kept = n;
  }
}

}  // namespace

int launch_runs_colours(cudaStream_t s, const DevInfo &d, const uint8_t *colors, int n, int T,
                        uint8_t *colT) {
  if (n > 0) runs_colours_kernel<<<d.sms * 4, 256, 0, s>>>(colors, n, T, colT);
  return (int)cudaGetLastError();
}

int launch_runs_list(cudaStream_t s, const DevInfo &d, int kw, const RunsArgs &a,
                     unsigned long long *blk) {
  const int G = sort_grid(d);
  if (!a.leaf) {
    if (kw == 1) runs_count_kernel<u64><<<G, 256, 0, s>>>(a, blk);
    else runs_count_kernel<u128><<<G, 256, 0, s>>>(a, blk);
    runs_scan_kernel<<<1, 1024, 0, s>>>(blk, G, a.n_runs);
    if (kw == 1) runs_list_kernel<u64><<<G, 256, 0, s>>>(a, blk);
    else runs_list_kernel<u128><<<G, 256, 0, s>>>(a, blk);
  }
  if (kw == 1) runs_degree_kernel<u64><<<G, 256, 0, s>>>(a);
  else runs_degree_kernel<u128><<<G, 256, 0, s>>>(a);
  return (int)cudaGetLastError();
}

int launch_runs_pairs(cudaStream_t s, const DevInfo &d, int kw, const RunsArgs &a) {
  if (kw == 1) runs_pairs_kernel<u64><<<sort_grid(d), 256, 0, s>>>(a);
  else runs_pairs_kernel<u128><<<sort_grid(d), 256, 0, s>>>(a);
  return (int)cudaGetLastError();
}

int launch_runs_windows(cudaStream_t s, const DevInfo &d, const RunsArgs &a) {
  runs_windows_kernel<<<sort_grid(d), 256, 0, s>>>(a);
  return (int)cudaGetLastError();
}

int launch_runs_write(cudaStream_t s, const DevInfo &d, int kw, const RunsArgs &a) {
  if (kw == 1) runs_write_kernel<u64><<<d.sms * 10, 256, 0, s>>>(a);
  else runs_write_kernel<u128><<<d.sms * 10, 256, 0, s>>>(a);
  return (int)cudaGetLastError();
}

int launch_runs_append(cudaStream_t s, const DevInfo &d, int kw, const RunsArgs &a,
                       const void *merged, const unsigned long long *n_merged,
                       unsigned long long *size_x, unsigned long long *size_f) {
  if (kw == 1)
    runs_append_kernel<u64><<<d.sms * 2, 256, 0, s>>>(a, merged, n_merged, size_x, size_f);
  else
    runs_append_kernel<u128><<<d.sms * 2, 256, 0, s>>>(a, merged, n_merged, size_x, size_f);
  return (int)cudaGetLastError();
}

}  // namespace cc
