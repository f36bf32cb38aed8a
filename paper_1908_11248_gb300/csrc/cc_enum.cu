// Result reconstruction (Section 4) on the device.
//
// The paper's R(x, M) walks the nice decomposition from the root, asking each node's child
// table how a (mapping, colour set) pair arose, and glues the answers.  Here the same walk is
// breadth-first over the nodes in pre-order: a state is (trial, colour set C still to account
// for, stack of colour sets owed to the second children of enclosing joins, partial map Phi).
// Taking a state through node x (next node in pre-order is x's first child, or, after a leaf,
// the second child of the innermost pending join; a kernel covers one forget or join and the
// introduces and leaves before it):
//   forget u    : one state per vertex v with (Phi + u->v restricted to the child bag, C) in
//                 the child table; Phi(u) = v
//   introduce u : C loses the colour of Phi(u)
//   join        : one state per split C = C' | C'' with C' & C'' the bag's colours, (phi, C') in
//                 the first child's table and (phi, C'') in the second's; C'' is pushed
//   leaf        : pops the next colour set (or, at the last leaf, the state is a full embedding)
// Every state is extendable to at least one embedding, so the state count never exceeds the
// final number of embeddings.  The union over trials is then sorted lexicographically and
// repeats are dropped: as table records (cc_sort.cu) when a row is at most kMaxBag vertices and
// 127 bits, five sorted passes and three reduce kernels for 40 bits instead of four kernels a
// byte of every column; else by an LSD radix sort of row indices over the columns.
//
// Membership "(t, phi, C) in D_y" is answered per table layout: a leaf table is indexed by
// (t, v); hashed tables are probed; sorted tables are binary-searched in their sort order; an
// introduce node, whose table need not be stored, is resolved by checking its rule (colour,
// degree filter, adjacency to the bag neighbours) and descending to its child.
#include <cstdint>

#include "cc_device.cuh"
#include "cc_internal.h"

namespace cc {
namespace {

using namespace dev;

__device__ __forceinline__ int colour_of(const GraphDev &G, int t, int v) {
  return G.colors[(u64)t * (u64)G.n + (u64)v];
}

template <typename SK, typename K>
__device__ bool sorted_contains(const Slot<K> *s, u64 first, u64 count, const SortSpec &sp,
                                K key) {
  const SK q = sort_key<SK>(key, sp);
  u64 lo = first, hi = count;
  while (lo < hi) {
    const u64 mid = (lo + hi) >> 1;
    K km;
    u64 c;
    load_slot(s, mid, km, c);
    const SK sm = sort_key<SK>(km, sp);
    if (sm < q) lo = mid + 1;
    else hi = mid;
  }
  if (lo >= count) return false;
  K kl;
  u64 c;
  load_slot(s, lo, kl, c);
  return kl == key;
}

template <typename K>
__device__ bool member(const EnumArgs &a, int y, K key) {
  for (int depth = 0; depth < 2 * kMaxBag + 8; ++depth) {
    const EnumNode &nd = a.nodes[y];
    if (nd.type == 1) {  // introduce: check its rule, then look in the child
      const int v = key_slot(key, a.L, nd.p);
      const int cv = colour_of(a.G, key_trial(key, a.L), v);
      if (!((key_mask(key, a.L) >> cv) & 1u)) return false;
      if (nd.degF && a.G.row_ptr[v + 1] - a.G.row_ptr[v] < nd.degF) return false;
      if (a.G.allow && !((a.G.allow[v] >> nd.vertex) & 1u)) return false;
      const K k2 = key_remove(key, a.L, nd.p) & ~((K)1 << cv);
      for (int j = 0; j < nd.nnb; ++j)
        if (!adjacent(a.G, key_slot(k2, a.L, nd.nb_slot[j]), v)) return false;
      key = k2;
      y = nd.child0;
      continue;
    }
    const Slot<K> *s = reinterpret_cast<const Slot<K> *>(nd.slots);
    if (nd.type == 0) {  // leaf: record (t, v) sits at t * n + v
      const u64 idx = (u64)key_trial(key, a.L) * (u64)a.G.n + (u64)key_slot(key, a.L, 0);
      K kk;
      u64 c;
      load_slot(s, idx, kk, c);
      return kk == key;
    }
    if (nd.hashed) return hash_find(s, nd.cap, key) >= 0;
    if (nd.sorted) {
      const bool narrow = nd.spec.bits + nd.spec.hbits <= 64;
      for (u64 lo = 0, hi = nd.split;; lo = hi, hi = nd.count) {
        if (narrow ? sorted_contains<u64>(s, lo, hi, nd.spec, key)
                   : sorted_contains<u128>(s, lo, hi, nd.spec, key))
          return true;
        if (hi == nd.count) return false;
      }
    }
    return false;
  }
  return false;
}

template <typename K>
__device__ __forceinline__ K key_of(const EnumArgs &a, const EnumNode &nd, int t, uint32_t C,
                                    const int *phi) {
  K key = (K)C;
  for (int s = 0; s < nd.b; ++s) key |= (K)(unsigned)phi[nd.bag[s]] << (a.L.k + s * a.L.nb);
  if (a.L.tb) key |= (K)(unsigned)t << a.L.tpos;
  return key;
}

// state layout: [0] trial, [1] colour set, [2] stack depth, [3, 3+D) stack, [3+D, 3+D+nF) Phi
//
// One warp a state, its candidates (vertices of a forget, colour splits of a join) over the
// lanes.  A table membership test is a chain of dependent loads (row pointers, a binary search or
// a hash probe), so a step is bound by how many of those chains are in flight: with one thread
// per state the first forget, one state over every host vertex, ran them all in sequence.
// MODE 2 appends to the output from one cursor (a warp takes the places of its valid candidates
// by one atomic add), so the tables are probed once and the host need not know how many states
// there are; MODEs 0 and 1 are the count and write passes for when only exact room is left.
// Measured: colour, DP and the first 100 000 of 325 000 embeddings of the path on four vertices
// (Erdos-Renyi, n = 1999, degree 12), 12.55 ms with a thread per state in two passes (11.8 ms of
// it in these kernels), 0.77 ms now; all 4000 five-cycles of a 200-vertex graph, 1.98 to 0.66 ms.
constexpr int kEnumWarps = 8;

template <typename K, int MODE>
__global__ void __launch_bounds__(32 * kEnumWarps) enum_step_kernel(EnumArgs a) {
  __shared__ int s_phi[kEnumWarps][32];
  __shared__ unsigned s_binom[33 * 33];  // binomials, for a join
  const EnumNode &nd = a.nodes[a.x];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  if (nd.type == 3) {  // row i of Pascal's triangle by thread i; C(32, 16) fits 32 bits
    if (threadIdx.x < 33) {
      u64 c = 1;
      for (int j = 0; j < 33; ++j) {
        s_binom[threadIdx.x * 33 + j] = j <= (int)threadIdx.x ? (unsigned)c : 0u;
        c = j < (int)threadIdx.x ? c * (u64)(threadIdx.x - j) / (u64)(j + 1) : 0;
      }
    }
    __syncthreads();
  }
  int *phi = s_phi[w];
  u64 n_in = a.n_in;
  if (a.n_dev) n_in = min(*a.n_dev, a.n_in);
  const u64 chunks = (u64)a.chunks, items = n_in * chunks;
  const u64 warps = (u64)gridDim.x * kEnumWarps;
  for (u64 item = (u64)blockIdx.x * kEnumWarps + w; item < items; item += warps) {
    const u64 i = item / chunks, part = item % chunks;
    const int *st = a.in + i * (u64)a.R;
    __syncwarp();  // the previous state's map is no longer read
    if (lane < a.nF) phi[lane] = st[3 + a.D + lane];
    __syncwarp();
    const int t = st[0];
    uint32_t C = (uint32_t)st[1];
    int sp = st[2];
    for (int j = a.u0; j < a.u1; ++j) {
      const EnumNode &un = a.nodes[a.pre[j]];
      if (un.type == 1) {  // introduce u: its colour leaves C
        C &= ~(1u << colour_of(a.G, t, phi[un.vertex]));
      } else if (sp > 0) {  // leaf: on to the second child of the innermost pending join
        --sp;
        C = (uint32_t)st[3 + sp];
      }
    }
    u64 made = 0;  // warp-uniform
    const u64 base = MODE == 1 ? a.off[i] : 0;
    // the lanes with `ok` emit a copy of this state with colour set C2 (push >= 0 pushes it on
    // the stack) and Phi(u) = v when u >= 0
    auto emit = [&](bool ok, uint32_t C2, long long push, int u, int v) {
      const unsigned bal = __ballot_sync(0xffffffffu, ok);
      if (!bal) return;
      if (MODE != 0) {
        u64 at = base + made;
        if (MODE == 2) {
          if (lane == 0) at = atomicAdd(a.cursor, (u64)__popc(bal));
          at = __shfl_sync(0xffffffffu, at, 0);
        }
        at += __popc(bal & lt);
        if (ok && (MODE == 1 || at < a.cap)) {
          int *o = a.out + at * (u64)a.R;
          o[0] = t;
          o[1] = (int)C2;
          o[2] = push >= 0 ? sp + 1 : sp;
          for (int j = 0; j < sp; ++j) o[3 + j] = st[3 + j];
          if (push >= 0) o[3 + sp] = (int)push;
          for (int f = 0; f < a.nF; ++f) o[3 + a.D + f] = phi[f];
          if (u >= 0) o[3 + a.D + u] = v;
        }
      }
      made += __popc(bal);
    };
    if (nd.type == 2) {  // forget u: every v completing (phi + u->v, C) in the child table
      const int u = nd.vertex;
      const EnumNode &ch = a.nodes[nd.child0];
      int best = INT_MAX, rs = 0;
      for (int j = 0; j < nd.nnb; ++j) {
        const int x = phi[nd.nb_slot[j]];  // F-vertex ids for forget nodes
        const int r0 = a.G.row_ptr[x], d = a.G.row_ptr[x + 1] - r0;
        if (d < best) {
          best = d;
          rs = r0;
        }
      }
      const int ncand = nd.nnb ? best : a.G.n;
      // the child's key with u's vertex left zero
      K kb = (K)C;
      int su = 0;
      for (int s = 0; s < ch.b; ++s) {
        if (ch.bag[s] == u) su = s;
        else kb |= (K)(unsigned)phi[ch.bag[s]] << (a.L.k + s * a.L.nb);
      }
      if (a.L.tb) kb |= (K)(unsigned)t << a.L.tpos;
      for (int j0 = (int)part * 32; j0 < ncand; j0 += 32 * (int)chunks) {
        const int j = j0 + lane;
        bool ok = false;
        int v = 0;
        if (j < ncand) {
          v = nd.nnb ? __ldg(a.G.col + rs + j) : j;
          ok = (C >> colour_of(a.G, t, v)) & 1u;
          if (ok) ok = member<K>(a, nd.child0, kb | ((K)(unsigned)v << (a.L.k + su * a.L.nb)));
        }
        emit(ok, C, -1, u, v);
      }
    } else {  // join: split the private colours between the children
      const EnumNode &y = a.nodes[nd.child0];
      const EnumNode &z = a.nodes[nd.child1];
      uint32_t bagc = 0;
      for (int s = 0; s < nd.b; ++s) bagc |= 1u << colour_of(a.G, t, phi[nd.bag[s]]);
      const uint32_t P = C & ~bagc;
      const int need = y.vstar - nd.b, nbits = __popc(P);
      if (need >= 0 && need <= nbits) {
        // subset number r of the C(nbits, need) subsets of P (combinatorial number system)
        const u64 subsets = s_binom[nbits * 33 + need];
        for (u64 r0 = part * 32; r0 < subsets; r0 += 32 * chunks) {
          const u64 r = r0 + lane;
          bool ok = false;
          uint32_t A = 0;
          if (r < subsets) {
            unsigned rest = (unsigned)r;
            int m = need;
            for (uint32_t q = P, pos = nbits; pos-- > 0 && m > 0;) {
              const int bit = 31 - __clz(q);
              const unsigned c = s_binom[pos * 33 + m];
              if (rest >= c) {
                rest -= c;
                --m;
                A |= 1u << bit;
              }
              q &= ~(1u << bit);
            }
            ok = member<K>(a, nd.child0, key_of<K>(a, y, t, bagc | A, phi)) &&
                 member<K>(a, nd.child1, key_of<K>(a, z, t, bagc | (P & ~A), phi));
          }
          emit(ok, bagc | A, (long long)(bagc | (P & ~A)), -1, 0);
        }
      }
    }
    if (MODE == 0 && lane == 0) a.cnt[i] = (unsigned)made;
  }
}

// root states: one per root entry (t, C)
template <typename K>
__global__ void enum_init_kernel(EnumArgs a, const void *root, u64 bound, unsigned long long *n) {
  const Slot<K> *s = reinterpret_cast<const Slot<K> *>(root);
  for (u64 i = blockIdx.x * (u64)blockDim.x + threadIdx.x; i < bound;
       i += (u64)gridDim.x * blockDim.x) {
    K key;
    u64 c;
    load_slot(s, i, key, c);
    if (key == 0) continue;
    const u64 pos = atomicAdd(n, 1ull);
    if (pos >= a.n_in) continue;  // capacity of the first state array
    int *o = a.out + pos * (u64)a.R;
    o[0] = key_trial(key, a.L);
    o[1] = (int)key_mask(key, a.L);
    o[2] = 0;
    for (int j = 3; j < a.R; ++j) o[j] = -1;
  }
}

// exclusive scan of n u32 values into u64 offsets; total at off[n]
__global__ void block_sums_kernel(const unsigned *v, u64 cap, const u64 *n_dev, u64 *sums) {
  const u64 n = n_dev ? min(*n_dev, cap) : cap, per = (n + gridDim.x - 1) / gridDim.x;
  const u64 lo = blockIdx.x * per, hi = min(n, lo + per);
  u64 s = 0;
  for (u64 i = lo + threadIdx.x; i < hi; i += blockDim.x) s += v[i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  __shared__ u64 w[32];
  if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    u64 t = 0;
    for (unsigned q = 0; q < blockDim.x / 32; ++q) t += w[q];
    sums[blockIdx.x] = t;
  }
}

__global__ void __launch_bounds__(1024) scan_small_kernel(u64 *v, int m, u64 *total) {
  block_scan_array(v, v, (u64)m, total);
}

// each block scans its range in chunks of blockDim (one block per range): warp shuffles and one
// pass over the 32 warp totals a chunk
__global__ void __launch_bounds__(1024) block_scan_kernel(const unsigned *v, u64 cap,
                                                          const u64 *n_dev, const u64 *sums,
                                                          u64 *off) {
  __shared__ u64 s_w[2][32];  // alternating, so that one barrier a chunk is enough
  const u64 n = n_dev ? min(*n_dev, cap) : cap, per = (n + gridDim.x - 1) / gridDim.x;
  const u64 lo = blockIdx.x * per, hi = min(n, lo + per);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  u64 run = sums[blockIdx.x];
  int flip = 0;
  for (u64 b = lo; b < hi; b += 1024, flip ^= 1) {
    const u64 i = b + threadIdx.x;
    const u64 own = i < hi ? v[i] : 0;
    u64 x = own;
    for (int o = 1; o < 32; o <<= 1) {
      const u64 y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_w[flip][w] = x;
    __syncthreads();
    u64 t = s_w[flip][lane];  // every warp scans the warp totals for itself
    const u64 mine = t;
    for (int o = 1; o < 32; o <<= 1) {
      const u64 y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    const u64 before = __shfl_sync(0xffffffffu, t - mine, w);
    if (i < hi) off[i] = run + before + x - own;
    run += __shfl_sync(0xffffffffu, t, 31);
  }
}

// ---- lexicographic sort of rows (LSD radix over columns, 8 bits per pass) -----------------
// perm holds row indices; a pass orders them stably by one byte of one column
__global__ void rows_hist_kernel(const int *rows, int nF, const unsigned *perm, u64 n, int col,
                                 int shift, u64 *hist) {
  __shared__ unsigned h[256];
  for (int d = threadIdx.x; d < 256; d += blockDim.x) h[d] = 0;
  __syncthreads();
  const u64 G = gridDim.x, chunk = (n + G - 1) / G;
  const u64 lo = blockIdx.x * chunk, hi = min(n, lo + chunk);
  for (u64 i = lo + threadIdx.x; i < hi; i += blockDim.x)
    atomicAdd(&h[((unsigned)rows[(u64)perm[i] * nF + col] >> shift) & 255u], 1u);
  __syncthreads();
  for (int d = threadIdx.x; d < 256; d += blockDim.x) hist[(u64)d * G + blockIdx.x] = h[d];
}

__global__ void __launch_bounds__(256) rows_row_scan_kernel(u64 *hist, int G) {
  __shared__ u64 s_w[8];
  __shared__ u64 s_carry;
  u64 *row = hist + (u64)blockIdx.x * G;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_carry = 0;
  __syncthreads();
  for (int base = 0; base < G; base += 256) {
    const int i = base + threadIdx.x;
    const u64 v = i < G ? row[i] : 0;
    u64 x = v;
    for (int o = 1; o < 32; o <<= 1) {
      u64 y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_w[w] = x;
    __syncthreads();
    u64 before = s_carry;
    for (int q = 0; q < w; ++q) before += s_w[q];
    if (i < G) row[i] = before + x - v;
    __syncthreads();
    if (threadIdx.x == 255) s_carry = before + x;
    __syncthreads();
  }
  if (threadIdx.x == 0) hist[(u64)256 * G + 256 + blockIdx.x] = s_carry;
}

__global__ void __launch_bounds__(256) rows_digit_base_kernel(u64 *hist, int G) {
  __shared__ u64 s_w[8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const u64 v = hist[(u64)256 * G + 256 + threadIdx.x];
  u64 x = v;
  for (int o = 1; o < 32; o <<= 1) {
    u64 y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_w[w] = x;
  __syncthreads();
  u64 before = 0;
  for (int q = 0; q < w; ++q) before += s_w[q];
  hist[(u64)256 * G + threadIdx.x] = before + x - v;
}

__global__ void __launch_bounds__(256) rows_scatter_kernel(const int *rows, int nF,
                                                           const unsigned *perm, u64 n, int col,
                                                           int shift, const u64 *off,
                                                           unsigned *out) {
  constexpr int W = 8;
  __shared__ unsigned s_wc[W][256];
  __shared__ unsigned s_run[256];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  s_run[tid] = 0;
  for (int x = 0; x < W; ++x) s_wc[x][tid] = 0;
  __syncthreads();
  const u64 G = gridDim.x, chunk = (n + G - 1) / G;
  const u64 lo = blockIdx.x * chunk, hi = min(n, lo + chunk);
  for (u64 base = lo; base < hi; base += 256) {
    const u64 i = base + tid;
    const bool valid = i < hi;
    const unsigned p = valid ? perm[i] : 0u;
    const int d = valid ? (int)(((unsigned)rows[(u64)p * nF + col] >> shift) & 255u) : 256 + lane;
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const int rank = __popc(peers & ((1u << lane) - 1u));
    if (valid && lane == __ffs(peers) - 1) s_wc[w][d] = __popc(peers);
    __syncthreads();
    unsigned acc = s_run[tid];
    for (int x = 0; x < W; ++x) {
      unsigned c = s_wc[x][tid];
      s_wc[x][tid] = acc;
      acc += c;
    }
    s_run[tid] = acc;
    __syncthreads();
    if (valid) out[off[(u64)d * G + blockIdx.x] + off[256 * G + d] + s_wc[w][d] + rank] = p;
    __syncthreads();
    for (int x = 0; x < W; ++x) s_wc[x][tid] = 0;
    __syncthreads();
  }
}

// each row (the images of F-vertices 0..nF-1) replaced by its vertex set in increasing order
__global__ void rows_canon_kernel(int *rows, int nF, u64 n) {
  for (u64 i = blockIdx.x * (u64)blockDim.x + threadIdx.x; i < n;
       i += (u64)gridDim.x * blockDim.x) {
    int *r = rows + i * (u64)nF;
    for (int a = 1; a < nF; ++a) {  // insertion sort, n_F <= 32
      const int v = r[a];
      int b = a - 1;
      while (b >= 0 && r[b] > v) {
        r[b + 1] = r[b];
        --b;
      }
      r[b + 1] = v;
    }
  }
}

// rows of the final states, and the identity permutation
__global__ void rows_extract_kernel(const int *states, u64 n, int R, int D, int nF, int *rows,
                                    unsigned *perm) {
  for (u64 i = blockIdx.x * (u64)blockDim.x + threadIdx.x; i < n;
       i += (u64)gridDim.x * blockDim.x) {
    for (int f = 0; f < nF; ++f) rows[i * nF + f] = states[i * (u64)R + 3 + D + f];
    perm[i] = (unsigned)i;
  }
}

// final states as records of a sortable table (rows_spec)
template <typename K>
__global__ void rows_pack_kernel(const int *states, u64 cap, const u64 *n_dev, int R, int D,
                                 int nF, int nb, int canon, Slot<K> *recs) {
  const u64 n = min(*n_dev, cap);
  for (u64 i = blockIdx.x * (u64)blockDim.x + threadIdx.x; i < n;
       i += (u64)gridDim.x * blockDim.x) {
    const int *p = states + i * (u64)R + 3 + D;
    int r[kMaxBag];
#pragma unroll
    for (int f = 0; f < kMaxBag; ++f) r[f] = f < nF ? p[f] : INT_MAX;
    if (canon) {  // the vertex set in increasing order (odd-even exchange over kMaxBag places)
#pragma unroll
      for (int round = 0; round < kMaxBag; ++round)
#pragma unroll
        for (int f = round & 1; f + 1 < kMaxBag; f += 2) {
          const int x = min(r[f], r[f + 1]), y = max(r[f], r[f + 1]);
          r[f] = x;
          r[f + 1] = y;
        }
    }
    K key = (K)1 << (nF * nb);
#pragma unroll
    for (int f = 0; f < kMaxBag; ++f)
      if (f < nF) key |= (K)(unsigned)r[f] << (f * nb);
    store_slot(recs, i, key, 1ull);
  }
}

template <typename K>
__global__ void rows_unpack_kernel(const Slot<K> *recs, const u64 *n_ptr, u64 limit, int nF,
                                   int nb, int *out) {
  const u64 n = min(*n_ptr, limit);
  for (u64 i = blockIdx.x * (u64)blockDim.x + threadIdx.x; i < n;
       i += (u64)gridDim.x * blockDim.x) {
    K key;
    u64 c;
    load_slot(recs, i, key, c);
    for (int f = 0; f < nF; ++f)
      out[i * nF + f] = (int)((key >> (f * nb)) & (K)((1ull << nb) - 1ull));
  }
}

// 1 where a row differs from its predecessor in sorted order
__global__ void rows_heads_kernel(const int *rows, int nF, const unsigned *perm, u64 n,
                                  unsigned *flag) {
  for (u64 i = blockIdx.x * (u64)blockDim.x + threadIdx.x; i < n;
       i += (u64)gridDim.x * blockDim.x) {
    unsigned h = 1;
    if (i > 0) {
      const int *a = rows + (u64)perm[i] * nF, *b = rows + (u64)perm[i - 1] * nF;
      h = 0;
      for (int f = 0; f < nF; ++f) h |= a[f] != b[f];
    }
    flag[i] = h;
  }
}

__global__ void rows_gather_kernel(const int *rows, int nF, const unsigned *perm, u64 n,
                                   const unsigned *flag, const u64 *off, u64 limit, int *out) {
  for (u64 i = blockIdx.x * (u64)blockDim.x + threadIdx.x; i < n;
       i += (u64)gridDim.x * blockDim.x) {
    if (!flag[i] || off[i] >= limit) continue;
    for (int f = 0; f < nF; ++f) out[off[i] * nF + f] = rows[(u64)perm[i] * nF + f];
  }
}

}  // namespace

static int enum_grid(const DevInfo &d) { return d.sms * 8; }

int launch_enum_init(cudaStream_t s, const DevInfo &d, int kw, const EnumArgs &a,
                     const void *root, unsigned long long bound, unsigned long long *n) {
  if (kw == 1) enum_init_kernel<u64><<<d.sms, 256, 0, s>>>(a, root, bound, n);
  else enum_init_kernel<u128><<<d.sms, 256, 0, s>>>(a, root, bound, n);
  return (int)cudaGetLastError();
}

int launch_enum_step(cudaStream_t s, const DevInfo &d, int kw, int mode, const EnumArgs &a) {
  if (a.n_in == 0) return 0;
  const int block = 32 * kEnumWarps;
  // no more warps than there can be (state, chunk) items
  const u64 want = (a.n_in * (u64)a.chunks + kEnumWarps - 1) / kEnumWarps;
  const int grid = (int)(want < (u64)enum_grid(d) ? want : (u64)enum_grid(d));
#define CC_STEP(K)                                                   \
  if (mode == 0) enum_step_kernel<K, 0><<<grid, block, 0, s>>>(a);   \
  else if (mode == 1) enum_step_kernel<K, 1><<<grid, block, 0, s>>>(a); \
  else enum_step_kernel<K, 2><<<grid, block, 0, s>>>(a)
  if (kw == 1) {
    CC_STEP(u64);
  } else {
    CC_STEP(u128);
  }
#undef CC_STEP
  return (int)cudaGetLastError();
}

SortSpec rows_spec(int nF, int nb) {
  SortSpec sp{};
  sp.L.nb = nb;
  sp.L.tpos = nF * nb;
  sp.b = nF;
  sp.nsl = nF;
  for (int f = 0; f < nF; ++f) sp.order[f] = f;
  sp.bits = nF * nb;
  return sp;
}

int launch_rows_pack(cudaStream_t s, const DevInfo &d, int kw, const int *states,
                     unsigned long long n, const unsigned long long *n_dev, int R, int D,
                     int nF, int nb, int canon, void *recs) {
  if (n == 0) return 0;
  const int grid = d.sms * 4;
  if (kw == 1)
    rows_pack_kernel<u64><<<grid, 256, 0, s>>>(states, n, n_dev, R, D, nF, nb, canon,
                                             (Slot<u64> *)recs);
  else
    rows_pack_kernel<u128><<<grid, 256, 0, s>>>(states, n, n_dev, R, D, nF, nb, canon,
                                             (Slot<u128> *)recs);
  return (int)cudaGetLastError();
}

int launch_rows_unpack(cudaStream_t s, const DevInfo &d, int kw, const void *recs,
                       const unsigned long long *n, unsigned long long limit, int nF, int nb,
                       int *out) {
  if (limit == 0) return 0;
  const int grid = d.sms * 4;
  if (kw == 1)
    rows_unpack_kernel<u64><<<grid, 256, 0, s>>>((const Slot<u64> *)recs, n, limit, nF, nb, out);
  else
    rows_unpack_kernel<u128><<<grid, 256, 0, s>>>((const Slot<u128> *)recs, n, limit, nF, nb, out);
  return (int)cudaGetLastError();
}

size_t scan_scratch_words(const DevInfo &d) { return (size_t)d.sms * 2 + 2; }

int launch_scan_u32(cudaStream_t s, const DevInfo &d, const unsigned *v, unsigned long long n,
                    unsigned long long *off, unsigned long long *scratch,
                    const unsigned long long *n_dev, unsigned long long *total) {
  const int nb = d.sms * 2;  // scratch: block sums
  if (!total) total = off + n;
  if (n == 0) return (int)cudaMemsetAsync(total, 0, sizeof(u64), s);
  block_sums_kernel<<<nb, 256, 0, s>>>(v, n, n_dev, scratch);
  scan_small_kernel<<<1, 1024, 0, s>>>(scratch, nb, total);
  block_scan_kernel<<<nb, 1024, 0, s>>>(v, n, n_dev, scratch, off);
  return (int)cudaGetLastError();
}

int launch_rows_canon(cudaStream_t s, const DevInfo &d, int *rows, int nF,
                      unsigned long long n) {
  if (n) rows_canon_kernel<<<d.sms * 4, 256, 0, s>>>(rows, nF, n);
  return (int)cudaGetLastError();
}

int launch_rows_extract(cudaStream_t s, const DevInfo &d, const int *states,
                        unsigned long long n, int R, int D, int nF, int *rows, unsigned *perm) {
  if (n) rows_extract_kernel<<<d.sms * 4, 256, 0, s>>>(states, n, R, D, nF, rows, perm);
  return (int)cudaGetLastError();
}

int launch_rows_sort(cudaStream_t s, const DevInfo &d, const int *rows, int nF, int nb,
                     unsigned long long n, unsigned *perm, unsigned *tmp, unsigned long long *hist,
                     unsigned **result) {
  const int G = d.sms * 2;
  unsigned *in = perm, *out = tmp;
  if (n > 1) {
    for (int col = nF - 1; col >= 0; --col)
      for (int shift = 0; shift < nb; shift += 8) {
        rows_hist_kernel<<<G, 256, 0, s>>>(rows, nF, in, n, col, shift, hist);
        rows_row_scan_kernel<<<256, 256, 0, s>>>(hist, G);
        rows_digit_base_kernel<<<1, 256, 0, s>>>(hist, G);
        rows_scatter_kernel<<<G, 256, 0, s>>>(rows, nF, in, n, col, shift, hist, out);
        unsigned *t = in;
        in = out;
        out = t;
      }
  }
  *result = in;
  return (int)cudaGetLastError();
}

int launch_rows_heads(cudaStream_t s, const DevInfo &d, const int *rows, int nF,
                      const unsigned *perm, unsigned long long n, unsigned *flag) {
  if (n) rows_heads_kernel<<<d.sms * 4, 256, 0, s>>>(rows, nF, perm, n, flag);
  return (int)cudaGetLastError();
}

int launch_rows_gather(cudaStream_t s, const DevInfo &d, const int *rows, int nF,
                       const unsigned *perm, unsigned long long n, const unsigned *flag,
                       const unsigned long long *off, unsigned long long limit, int *out) {
  if (n && limit) rows_gather_kernel<<<d.sms * 4, 256, 0, s>>>(rows, nF, perm, n, flag, off, limit, out);
  return (int)cudaGetLastError();
}

}  // namespace cc
