// Cluster contraction (Sec. 4.1, "contract it"; contraction semantics, Sec. 3):
// every block of a labelling becomes one vertex, intra-block edges vanish and
// parallel edges between two blocks merge with summed weight.  Block ids are the
// ranks of the label values.  Steps: relabel (flag + scan), the optional correcting
// step, pre-merge per fine vertex (lp.cu), then one of
//   * the table (few clusters and many pairs): the pairs are added up in c x c sums, which are
//     read row by row into the coarse lists,
//   * the cluster merge: a counting sort of the pre-merged pairs by source cluster,
//     then a warp per cluster of at most kMergeMax pairs (registers, or a bitonic sort
//     in shared memory), a block per cluster of at most kMergeBlockMax, and one radix
//     sort for all larger ("giant") clusters together; each writes its distinct
//     targets in ascending order at the front of its segment,
//   * pair build, LSD radix sort on (cid v, cid u) and a run reduction (when the giant
//     clusters hold more than half of the pairs).
#include <limits.h>

#include <algorithm>
#include <type_traits>

#include "kernels.cuh"
#include "prims.cuh"
#include "regvisit.cuh"

namespace vc {

__global__ void mark_labels_k(const int32_t* __restrict__ lab, int64_t n, int32_t* __restrict__ flags) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    if (lab[v] >= 0) flags[lab[v]] = 1;  // label -1: the vertex is dropped (batches)
}

__global__ void apply_rank_k(const int32_t* __restrict__ lab, int64_t n, const int32_t* __restrict__ rank,
                             int32_t* __restrict__ cid) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    cid[v] = lab[v] >= 0 ? rank[lab[v]] : -1;
}

void relabel(const int32_t* lab, int64_t n, int32_t* cid, ContractScratch& cs, int* c_dev, cudaStream_t s) {
  VC_CUDA(cudaMemsetAsync(cs.flags, 0, sizeof(int32_t) * n, s));
  int grid = grid_for(n, 256, kSMs * 8);
  mark_labels_k<<<grid, 256, 0, s>>>(lab, n, cs.flags);
  count_launch();
  VC_CHECK_LAUNCH();
  exclusive_scan<int, int>(cs.flags, cs.rank, n, c_dev, cs.scan_scr32, s);
  apply_rank_k<<<grid, 256, 0, s>>>(lab, n, cs.rank, cid);
  count_launch();
  VC_CHECK_LAUNCH();
}

// W lanes per fine vertex copy its pre-merged list into the contiguous pair arrays: a
// thread per vertex where lists are short (two entries on average on clustered graphs),
// wider groups where they run up to the degree (unclustered graphs).
template <int W>
__global__ void build_pairs_k(int64_t n, const int64_t* __restrict__ off, const int32_t* __restrict__ cid,
                              const int32_t* __restrict__ cnt, const long long* __restrict__ pos, PairOut in,
                              int bits, unsigned long long* __restrict__ keys, long long* __restrict__ vals,
                              LongLists longs) {
  const int lane = threadIdx.x & (W - 1);
  const int64_t groups = (int64_t)gridDim.x * (blockDim.x / W);
  for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / W; v < n; v += groups) {
    const int k = cnt[v];
    if (k == 0) continue;
    const int64_t src = off[v];
    const long long dst = pos[v];
    if (longs.item && k > kLongList) {
      if (lane == 0) longs.push((int32_t)v, dst);
      continue;
    }
    const unsigned long long hi = (unsigned long long)cid[v] << bits;
    for (int j = lane; j < k; j += W) {
      int32_t kk;
      long long x;
      in.get(v, src, j, &kk, &x);
      keys[dst + j] = hi | (unsigned long long)(uint32_t)kk;
      vals[dst + j] = x;
    }
  }
}

// The lists build_pairs_k left out.
__global__ void build_pairs_long_k(const int64_t* __restrict__ off, const int32_t* __restrict__ cid,
                                   const int32_t* __restrict__ cnt, PairOut in, int bits,
                                   unsigned long long* __restrict__ keys, long long* __restrict__ vals,
                                   LongLists longs) {
  const int n = *longs.n;
  const GridShare G(n);
  for (int i = G.first; i < n; i += G.step) {
    const int32_t v = longs.item[i];
    const long long dst = longs.at[i];
    const int64_t src = off[v];
    const int k = cnt[v];
    const unsigned long long hi = (unsigned long long)cid[v] << bits;
    for (int64_t j = (int64_t)G.part * blockDim.x + threadIdx.x; j < k; j += (int64_t)G.parts * blockDim.x) {
      int32_t kk;
      long long x;
      in.get(v, src, (int)j, &kk, &x);
      keys[dst + j] = hi | (unsigned long long)(uint32_t)kk;
      vals[dst + j] = x;
    }
  }
}

void build_pairs(const GraphView& g, const int32_t* cid, const ContractScratch& cs, int bits, int64_t pairs,
                 const LongLists& longs, unsigned long long* keys, long long* vals, cudaStream_t s) {
  const PairOut in{cs.tmp_key, cs.tmp_val, cs.cmp_key, cs.cmp_val};
  if (pairs <= 2 * g.n)
    build_pairs_k<1><<<grid_for(g.n, 256, kSMs * 8), 256, 0, s>>>(g.n, g.off, cid, cs.cnt, cs.pos, in, bits, keys,
                                                                  vals, longs);
  else if (pairs <= 16 * g.n)
    build_pairs_k<8><<<grid_for(g.n, 32, kSMs * 16), 256, 0, s>>>(g.n, g.off, cid, cs.cnt, cs.pos, in, bits, keys,
                                                                  vals, longs);
  else
    build_pairs_k<32><<<grid_for(g.n, 8, kSMs * 16), 256, 0, s>>>(g.n, g.off, cid, cs.cnt, cs.pos, in, bits, keys,
                                                                  vals, longs);
  count_launch();
  if (longs.item) {
    build_pairs_long_k<<<kSMs * 4, 256, 0, s>>>(g.off, cid, cs.cnt, in, bits, keys, vals, longs);
    count_launch();
  }
  VC_CHECK_LAUNCH();
}

__global__ void run_heads_k(const unsigned long long* __restrict__ keys, int64_t m, int32_t* __restrict__ heads) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
    heads[i] = (i == 0 || keys[i] != keys[i - 1]) ? 1 : 0;
}

// Every element adds its value to its run's output: run index = (heads up to and
// including it) - 1 = hpos[i] + heads[i] - 1.  The lanes of a warp in one run add their
// sum once (runs can be long: a giant cluster's pairs to one target); cw must be zero.
// The run's head writes the target and source ids.
__global__ void run_reduce_k(const unsigned long long* __restrict__ keys, const long long* __restrict__ vals,
                             int64_t m, int bits, const int32_t* __restrict__ heads,
                             const long long* __restrict__ hpos, int32_t* __restrict__ cadj,
                             long long* __restrict__ cw, int32_t* __restrict__ cv) {
  const unsigned long long mask = (bits >= 64) ? ~0ULL : ((1ULL << bits) - 1ULL);
  const int lane = threadIdx.x & 31;
  for (int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~31LL; b < m;
       b += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = b + lane;
    const bool ok = i < m;
    const long long r = ok ? hpos[i] + heads[i] - 1 : -1 - lane;
    const long long x = ok ? vals[i] : 0;
    // runs are consecutive lanes: a segmented inclusive sum, added by each run's last lane
    long long sum = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, sum, o);
      const long long ry = __shfl_up_sync(0xffffffffu, r, o);
      if (lane >= o && ry == r) sum += y;
    }
    const long long rn = __shfl_down_sync(0xffffffffu, r, 1);
    if (ok && (lane == 31 || rn != r)) atomicAdd((unsigned long long*)(cw + r), (unsigned long long)sum);
    if (ok && heads[i]) {
      const unsigned long long k = keys[i];
      cadj[r] = (int32_t)(k & mask);
      cv[r] = (int32_t)(k >> bits);
    }
  }
}

// offsets from the source-vertex column of the (sorted) unique entries
__global__ void build_offsets_k(const int32_t* __restrict__ cv, const long long* __restrict__ nnz_dev,
                                int64_t c, int64_t* __restrict__ coff) {
  const long long m = *nnz_dev;
  const int64_t T = (int64_t)gridDim.x * blockDim.x;
  const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (m == 0) {
    for (int64_t x = t0; x <= c; x += T) coff[x] = 0;
    return;
  }
  for (int64_t j = t0; j <= m; j += T) {
    // entry j starts the lists of every vertex in (cv[j-1], cv[j]]
    int64_t lo = (j == 0) ? -1 : cv[j - 1];
    int64_t hi = (j == m) ? c : cv[j];
    for (int64_t x = lo + 1; x <= hi; ++x) coff[x] = j;
  }
}

void reduce_pairs(const unsigned long long* keys, const long long* vals, int64_t pairs, int bits,
                  int64_t c, int32_t* heads, long long* hpos, long long* scan_scr, int64_t* coff,
                  int32_t* cadj, long long* cw, int32_t* cv_tmp, long long* nnz_dev, cudaStream_t s) {
  int grid = grid_for(pairs, 256, kSMs * 8);
  if (pairs > 0) {
    run_heads_k<<<grid, 256, 0, s>>>(keys, pairs, heads);
    count_launch();
    VC_CHECK_LAUNCH();
  }
  exclusive_scan<int, long long>(heads, hpos, pairs, nnz_dev, scan_scr, s);
  if (pairs > 0) {
    VC_CUDA(cudaMemsetAsync(cw, 0, sizeof(long long) * pairs, s));
    run_reduce_k<<<grid, 256, 0, s>>>(keys, vals, pairs, bits, heads, hpos, cadj, cw, cv_tmp);
    count_launch();
    VC_CHECK_LAUNCH();
  }
  build_offsets_k<<<grid_for(pairs + c + 1, 256, kSMs * 8), 256, 0, s>>>(cv_tmp, nnz_dev, c, (int64_t*)coff);
  count_launch();
  VC_CHECK_LAUNCH();
}

// ---------------------------------------------------------------- merge in a table
// Few clusters and many pairs: the pairs are added up in a table of c x c sums (additions in
// L2 that return nothing), which is then read row by row into the coarse lists.  No pair is
// sorted or moved, and a cluster's size does not matter.  A sum of 0 is no entry, unless a
// pair of weight 0 or below went into it (inputs that nothing checked): those are noted in a
// bit per sum (zero, 32 columns a word).
__host__ __device__ inline int64_t table_words(int64_t c) { return (c + 31) >> 5; }

// W lanes per fine vertex add its pre-merged list to its cluster's row.
template <int W>
__global__ void __launch_bounds__(256) table_add_k(int64_t n, const int64_t* __restrict__ off,
                                                   const int32_t* __restrict__ cid, const int32_t* __restrict__ cnt,
                                                   PairOut in, int64_t c, long long* __restrict__ sums,
                                                   unsigned* __restrict__ zero) {
  const int lane = threadIdx.x & (W - 1);
  const int64_t groups = (int64_t)gridDim.x * (256 / W);
  for (int64_t v = ((int64_t)blockIdx.x * 256 + threadIdx.x) / W; v < n; v += groups) {
    const int32_t x = cid[v];
    const int k = x >= 0 ? cnt[v] : 0;
    if (k == 0) continue;
    const int64_t src = off[v], row = (int64_t)x * c;
#pragma unroll 4
    for (int j = lane; j < k; j += W) {
      int32_t key;
      long long w;
      in.get(v, src, j, &key, &w);
      atomicAdd((unsigned long long*)(sums + row + key), (unsigned long long)w);
      if (w <= 0) atomicOr(zero + x * table_words(c) + (key >> 5), 1u << (key & 31));
    }
  }
}

// A warp per row: f of each entry, and then of the row.
constexpr int kTableUnroll = 8;
template <typename F>
__device__ __forceinline__ void table_rows(int64_t c, const long long* sums, const unsigned* zero, F f) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < c; x += warps) {
    const long long* row = sums + x * c;
    const unsigned* zrow = zero + x * table_words(c);
    int64_t made = 0;
    for (int64_t b = 0; b < c; b += 32 * kTableUnroll) {
      long long w[kTableUnroll];
      unsigned z[kTableUnroll];
#pragma unroll
      for (int q = 0; q < kTableUnroll; ++q) {
        w[q] = b + 32 * q + lane < c ? row[b + 32 * q + lane] : 0;
        z[q] = b + 32 * q < c ? zrow[(b >> 5) + q] : 0;
      }
#pragma unroll
      for (int q = 0; q < kTableUnroll; ++q) {
        const bool in = w[q] != 0 || (z[q] >> lane & 1u);
        const unsigned bal = __ballot_sync(0xffffffffu, in);
        if (in) f(x, made + __popc(bal & ((1u << lane) - 1u)), b + 32 * q + lane, w[q]);
        made += __popc(bal);
      }
    }
    f(x, made);
  }
}
struct TableCount {
  int32_t* count;
  __device__ __forceinline__ void operator()(int64_t, int64_t, int64_t, long long) const {}
  __device__ __forceinline__ void operator()(int64_t x, int64_t made) const {
    if ((threadIdx.x & 31) == 0) count[x] = (int32_t)made;
  }
};
struct TableWrite {
  const int64_t* coff;
  int32_t* cadj;
  long long* cw;
  int32_t* csrc;
  __device__ __forceinline__ void operator()(int64_t x, int64_t i, int64_t y, long long w) const {
    const int64_t to = coff[x] + i;
    cadj[to] = (int32_t)y;
    cw[to] = w;
    csrc[to] = (int32_t)x;
  }
  __device__ __forceinline__ void operator()(int64_t, int64_t) const {}
};
template <typename F>
__global__ void __launch_bounds__(256) table_rows_k(int64_t c, const long long* __restrict__ sums,
                                                    const unsigned* __restrict__ zero, F f) {
  table_rows(c, sums, zero, f);
}

int64_t table_elems(int64_t c) { return c * c + (c * table_words(c) + 1) / 2; }
bool table_merge_fits(int64_t c, int64_t pairs) {
  return c > 0 && c <= (int64_t(1) << 30) && c * c <= 2 * pairs && pairs <= std::max<int64_t>(64 * c * c, 1 << 16);
}

void table_merge(const GraphView& g, const int32_t* cid, const ContractScratch& cs, int64_t c, int64_t pairs,
                 long long* sums, int32_t* ccount, int64_t* coff, int32_t* cadj, long long* cw, int32_t* csrc,
                 long long* nnz_dev, cudaStream_t s) {
  const PairOut in{cs.tmp_key, cs.tmp_val, cs.cmp_key, cs.cmp_val};
  VC_CUDA(cudaMemsetAsync(sums, 0, sizeof(long long) * table_elems(c), s));
  unsigned* zero = (unsigned*)(sums + c * c);
  if (pairs <= 2 * g.n)
    table_add_k<1><<<grid_for(g.n, 256, kSMs * 8), 256, 0, s>>>(g.n, g.off, cid, cs.cnt, in, c, sums, zero);
  else if (pairs <= 16 * g.n)
    table_add_k<8><<<grid_for(g.n, 32, kSMs * 16), 256, 0, s>>>(g.n, g.off, cid, cs.cnt, in, c, sums, zero);
  else
    table_add_k<32><<<grid_for(g.n, 8, kSMs * 16), 256, 0, s>>>(g.n, g.off, cid, cs.cnt, in, c, sums, zero);
  const int grid = grid_for(c, 8, kSMs * 8);
  table_rows_k<<<grid, 256, 0, s>>>(c, sums, zero, TableCount{ccount});
  exclusive_scan<int, long long>(ccount, (long long*)coff, c, (long long*)coff + c, cs.scan_scr, s, nullptr, nnz_dev);
  table_rows_k<<<grid, 256, 0, s>>>(c, sums, zero, TableWrite{coff, cadj, cw, csrc});
  count_launch(3);
  VC_CHECK_LAUNCH();
}

// ---------------------------------------------------------------- cluster merge
// Warp-level grouping of the lanes whose vertices share a cluster (consecutive
// vertices often do), so that one atomic per group and warp moves its counter.
// Returns the sum of k over the lane's group and the sum over the group's lower
// lanes; sk is the warp's 32-entry scratch.
__device__ __forceinline__ void group_sums(int32_t c, int k, int lane, int* sk, unsigned* peers_out, int* total,
                                           int* below) {
  const unsigned peers = __match_any_sync(0xffffffffu, c);
  sk[lane] = k;
  __syncwarp();
  int t = 0, b = 0;
  for (unsigned m = peers; m; m &= m - 1) {
    const int j = __ffs(m) - 1;
    t += sk[j];
    if (j < lane) b += sk[j];
  }
  __syncwarp();
  *peers_out = peers;
  *total = t;
  *below = b;
}

// The largest pairs-per-cluster count and the total, over ccount[0, n).
__global__ void __launch_bounds__(256) cluster_stats_k(int64_t n, const int32_t* __restrict__ ccount, int* maxt,
                                                       long long* pairs, int* ngiant, long long* gpairs) {
  __shared__ int s_max;
  __shared__ unsigned long long s_sum;
  if (threadIdx.x == 0) { s_max = 0; s_sum = 0; }
  __syncthreads();
  int top = 0;
  long long sum = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int x = ccount[i];
    top = max(top, x);
    sum += x;
    if (x > kMergeBlockMax) {  // rare
      atomicAdd(ngiant, 1);
      atomicAdd((unsigned long long*)gpairs, (unsigned long long)x);
    }
  }
  const unsigned wtop = __reduce_max_sync(0xffffffffu, (unsigned)top);
  const long long w = warp_sum(sum);
  if ((threadIdx.x & 31) == 0) {
    if (wtop) atomicMax(&s_max, (int)wtop);
    if (w) atomicAdd(&s_sum, (unsigned long long)w);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_max) atomicMax(maxt, s_max);
    if (s_sum) atomicAdd((unsigned long long*)pairs, s_sum);
  }
}

// The pieces of a warp copied with the lanes on consecutive entries: lane j brings a
// piece of len entries (0: none) read from src + i and written to dst + i (i < len);
// load(s) reads the entry at source index s and put(d, j, value) writes it at
// destination index d (j: the piece's lane).  kPieceUnroll entries per lane at a time,
// all loads before the stores, so that they are in flight together.  Long lists of a
// few lanes and short lists of many lanes keep every lane busy alike.
constexpr int kPieceUnroll = 4;
template <typename T, typename LOAD, typename PUT>
__device__ __forceinline__ void warp_pieces(int64_t len, int64_t src, int64_t dst, LOAD load, PUT put) {
  const int lane = threadIdx.x & 31;
  int64_t incl = len;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  const int64_t total = __shfl_sync(0xffffffffu, incl, 31);
  const int64_t excl = incl - len;  // where lane j's piece starts among the laid-out pieces
  for (int64_t p0 = 0; p0 < total; p0 += 32 * kPieceUnroll) {
    int jj[kPieceUnroll];
    int64_t sp[kPieceUnroll], dp[kPieceUnroll];
    T val[kPieceUnroll];
#pragma unroll
    for (int u = 0; u < kPieceUnroll; ++u) {
      const int64_t p = p0 + lane + 32 * u;
      // the piece holding place p: the last lane whose piece starts at or before p
      int j = 0;
#pragma unroll
      for (int step = 16; step > 0; step >>= 1) {
        const int t = j + step;
        const int64_t ex = __shfl_sync(0xffffffffu, excl, t & 31);
        if (t < 32 && ex <= p) j = t;
      }
      const int64_t i = p - __shfl_sync(0xffffffffu, excl, j);
      sp[u] = __shfl_sync(0xffffffffu, src, j) + i;
      dp[u] = __shfl_sync(0xffffffffu, dst, j) + i;
      jj[u] = p < total ? j : -1;
    }
#pragma unroll
    for (int u = 0; u < kPieceUnroll; ++u)
      if (jj[u] >= 0) val[u] = load(sp[u]);
#pragma unroll
    for (int u = 0; u < kPieceUnroll; ++u)
      if (jj[u] >= 0) put(dp[u], jj[u], val[u]);
  }
}

struct KeyVal {
  int32_t k;
  long long v;
};

// Counting-sort scatter: the pre-merged pairs of fine vertex v move, in one piece,
// into their cluster's segment (cursor = the segments' running write positions).
// Lists of more than kScatterWarpMin pairs are copied by the whole warp.
constexpr int kScatterWarpMin = 16;
__global__ void __launch_bounds__(256) cluster_scatter_k(int64_t n, const int64_t* __restrict__ off,
                                                         const int32_t* __restrict__ cid,
                                                         const int32_t* __restrict__ cnt, PairOut in,
                                                         long long* __restrict__ cursor, int32_t* __restrict__ seg_key,
                                                         long long* __restrict__ seg_val, LongLists longs) {
  __shared__ int s_k[8][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
    const int64_t v = base + lane;
    const int k = v < n ? cnt[v] : 0;
    const int32_t c = k > 0 ? cid[v] : -1;
    unsigned peers;
    int t, b;
    group_sums(c, k, lane, s_k[wid], &peers, &t, &b);
    const int leader = __ffs(peers) - 1;
    long long at = 0;
    if (c >= 0 && lane == leader) at = atomicAdd((unsigned long long*)&cursor[c], (unsigned long long)t);
    at = __shfl_sync(0xffffffffu, at, leader);
    const long long dst = at + b;
    if (c >= 0) {
      // the first kPairSlots pairs from the dense strip, all in flight at once
      int32_t kk[kPairSlots];
      long long vv[kPairSlots];
#pragma unroll
      for (int j = 0; j < kPairSlots; ++j)
        if (j < k) { kk[j] = in.ckey[v * kPairSlots + j]; vv[j] = in.cval[v * kPairSlots + j]; }
#pragma unroll
      for (int j = 0; j < kPairSlots; ++j)
        if (j < k) { seg_key[dst + j] = kk[j]; seg_val[dst + j] = vv[j]; }
      if (k > kPairSlots && k <= kScatterWarpMin) {  // short rest: this thread
        const int64_t src = off[v];
        for (int j = kPairSlots; j < k; ++j) {
          seg_key[dst + j] = in.tkey[src + j];
          seg_val[dst + j] = in.tval[src + j];
        }
      }
    }
    // the rest of the long lists, laid end to end over the lanes (coalesced); the longest by
    // cluster_scatter_long_k
    const bool whole = longs.item && k > kLongList;
    if (c >= 0 && whole) longs.push((int32_t)v, dst);
    const bool longl = c >= 0 && k > kScatterWarpMin && !whole;
    if (__any_sync(0xffffffffu, longl)) {
      warp_pieces<KeyVal>(
          longl ? (int64_t)(k - kPairSlots) : 0, longl ? off[v] + kPairSlots : 0, dst + kPairSlots,
          [&](int64_t at) { return KeyVal{in.tkey[at], in.tval[at]}; },
          [&](int64_t at, int, const KeyVal& kv) {
            seg_key[at] = kv.k;
            seg_val[at] = kv.v;
          });
    }
  }
}

// The rests of the lists cluster_scatter_k left out.
__global__ void cluster_scatter_long_k(const int64_t* __restrict__ off, const int32_t* __restrict__ cnt, PairOut in,
                                       int32_t* __restrict__ seg_key, long long* __restrict__ seg_val,
                                       LongLists longs) {
  const int n = *longs.n;
  const GridShare G(n);
  for (int i = G.first; i < n; i += G.step) {
    const int32_t v = longs.item[i];
    const long long dst = longs.at[i];
    const int64_t src = off[v];
    const int k = cnt[v];
    for (int64_t j = kPairSlots + (int64_t)G.part * blockDim.x + threadIdx.x; j < k;
         j += (int64_t)G.parts * blockDim.x) {
      seg_key[dst + j] = in.tkey[src + j];
      seg_val[dst + j] = in.tval[src + j];
    }
  }
}

// ---- sorting pairs by target: a bitonic network over packed elements (target << kIdxBits |
// place of the pair), E of them in the registers of each thread.  Element i = thread E + r,
// so that strides below E stay in a thread, strides up to 16 E are one shuffle and only a
// block's longest strides go through shared memory; the pairs' sums never move.
constexpr int kIdxBits = 12;  // places below kMergeBlockMax
static_assert((1 << kIdxBits) >= kMergeBlockMax, "a pair's place fits beside its target");
constexpr unsigned long long kSortPad = ~0ull;

__device__ __forceinline__ void sort_pair(unsigned long long& a, unsigned long long& b, bool up) {
  const unsigned long long lo = a < b ? a : b, hi = a < b ? b : a;
  a = up ? lo : hi;
  b = up ? hi : lo;
}

// The strides below E of merge level k; `up` for levels of at least E.
template <int E>
__device__ __forceinline__ void sort_inside(unsigned long long (&x)[E], int k, bool up) {
#pragma unroll
  for (int j = E / 2; j > 0; j >>= 1)
#pragma unroll
    for (int r = 0; r < E; ++r)
      if ((r & j) == 0 && j < k) sort_pair(x[r], x[r | j], k < E ? (r & k) == 0 : up);
}

// Sorts the T E elements of T threads (32: a warp, each warp for itself; more: the block, with
// T E elements of shared memory).
template <int E, int T>
__device__ __forceinline__ void sort_elements(unsigned long long (&x)[E], unsigned long long* sh) {
  const int t = T == 32 ? (threadIdx.x & 31) : threadIdx.x;
#pragma unroll
  for (int k = 2; k < E; k <<= 1) sort_inside<E>(x, k, true);
  if (E > 1) sort_inside<E>(x, E, (t & 1) == 0);
#pragma unroll 1
  for (int h = 2; h <= T; h <<= 1) {  // merge level h E
    const bool up = (t & h) == 0;
#pragma unroll 1
    for (int m = h >> 1; m > 0; m >>= 1) {  // stride m E
      const bool keep_low = ((t & m) == 0) == up;
      if (m >= 32) {
        __syncthreads();
#pragma unroll
        for (int r = 0; r < E; ++r) sh[r * T + t] = x[r];
        __syncthreads();
      }
#pragma unroll
      for (int r = 0; r < E; ++r) {
        const unsigned long long y = m >= 32 ? sh[r * T + (t ^ m)] : __shfl_xor_sync(0xffffffffu, x[r], m);
        x[r] = (y < x[r]) == keep_low ? y : x[r];
      }
    }
    sort_inside<E>(x, h * E, up);
  }
}

// Places of sorted elements in shared memory, padded so that threads writing their E
// consecutive elements meet no bank conflicts (4-byte and 8-byte elements).
__device__ __forceinline__ int pad4(int i) { return i + (i >> 5); }
__device__ __forceinline__ int pad8(int i) { return i + (i >> 4); }

// A warp per cluster of at most kMergeMax pairs, the distinct targets written back in
// ascending order at the front of the segment; dcount[c] = their number.  The pairs go
// into registers and the warp takes one step per distinct target (summing its
// weights) while targets are few; a cluster reaching kMergeWarpKeys targets is sorted
// instead, and every run head sums its run (a step per target costs slots x compares, which only pays while
// targets are few).  With sort_first (a contraction whose clusters are mostly one or
// two vertices: nearly every pair its own target) a cluster of at least kMergeSortMin
// pairs is sorted without walking first.  S slots per lane: clusters of at most
// kMergeSmall pairs with four, the others with sixteen, whose registers would halve the
// warps in flight for all.  With a list (list_n not null) only the listed clusters are
// visited (a sparse contraction leaves nearly all of them without pairs: 0.75 ms for
// 3.5 million empty clusters, 0.04 ms to list the others).
constexpr int kMergeWarpKeys = 32;
constexpr int kMergeSortMin = 12;
constexpr int kMergeSmall = 128;
constexpr int kMergeWarps = 4;

template <int S>
__global__ void __launch_bounds__(kMergeWarps * 32) cluster_merge_k(int64_t c, const long long* __restrict__ cbase,
                                                       int32_t* __restrict__ seg_key, long long* __restrict__ seg_val,
                                                       int32_t* __restrict__ dcount, bool sort_first,
                                                       const int32_t* __restrict__ list,
                                                       const int* __restrict__ list_n) {
  constexpr int kMax = 32 * S;
  __shared__ int32_t sk_all[kMergeWarps][kMax + S];
  __shared__ uint16_t si_all[kMergeWarps][kMax + S];
  __shared__ long long sv_all[kMergeWarps][kMax];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int32_t* sk = sk_all[wid];   // sorted targets (at pad4),
  uint16_t* si = si_all[wid];  // the places of their pairs,
  long long* sv = sv_all[wid]; // the pairs' sums by place
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  if (list_n) c = *list_n;
  for (int64_t xi = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; xi < c; xi += warps) {
    const int64_t x = list_n ? (int64_t)list[xi] : xi;
    const long long b = cbase[x];
    const int T = (int)(cbase[x + 1] - b);
    if (T > kMax) continue;  // another launch takes it
    RegList<long long, S> L;
    L.slots = (T + 31) >> 5;
    L.todo = 0;
#pragma unroll
    for (int r = 0; r < S; ++r) {
      const int i = lane + 32 * r;
      L.k[r] = -1;
      L.wt[r] = 0;
      if (32 * r < T && i < T) {  // 32 r < T is the same in every lane
        L.k[r] = seg_key[b + i];
        L.wt[r] = seg_val[b + i];
        L.todo |= 1u << r;
      }
    }
    bool walk = !sort_first || T < kMergeSortMin;
    if (walk && T >= kMergeSortMin) {
      // probe: the distinct targets among the first row's pairs (one match); a row more
      // than half distinct (a cluster of one or two vertices of a weakly clustered
      // graph, or a long run of an exact-step round) is sorted without walking first
      const bool use = lane < T;
      const unsigned long long tag =
          use ? (unsigned long long)(uint32_t)L.k[0] : (0xffffffff00000000ull | (unsigned long long)lane);
      const unsigned peers = __match_any_sync(0xffffffffu, tag);
      const int nd = __popc(__ballot_sync(0xffffffffu, use && (__ffs(peers) - 1) == lane));
      if (2 * nd > (T < 32 ? T : 32)) walk = false;
    }
    if (walk) {
      int made = 0;  // warp-uniform
      int32_t ok = INT_MAX;
      long long ov = 0;
      reg_visit<long long, long long, 32, S>(L, 0xffffffffu, [&](int32_t key, long long total) {
        if (lane == made) { ok = key; ov = total; }
        return ++made >= kMergeWarpKeys;
      });
      if (made < kMergeWarpKeys) {
        // lane i holds target i: its rank among the made targets places it
        int rank = 0;
        for (int j = 0; j < made; ++j) rank += __shfl_sync(0xffffffffu, ok, j) < ok;
        if (lane < made) {
          seg_key[b + rank] = ok;
          seg_val[b + rank] = ov;
        }
        if (lane == 0) dcount[x] = made;
        continue;
      }
    }
    if (sort_first) {
      // pairs already strictly ascending (one vertex's list over near-monotone ids)
      // stay where they are
      bool asc = true;
#pragma unroll
      for (int r = 0; r < S; ++r) {
        if (32 * r < T) {
          const int32_t up = __shfl_up_sync(0xffffffffu, L.k[r], 1);
          const int32_t wrap = r > 0 ? __shfl_sync(0xffffffffu, L.k[r > 0 ? r - 1 : 0], 31) : INT_MIN;
          const int i = lane + 32 * r;
          if (i < T && i > 0 && (lane ? up : wrap) >= L.k[r]) asc = false;
        }
      }
      if (__all_sync(0xffffffffu, asc)) {
        if (lane == 0) dcount[x] = T;
        continue;
      }
    }
    // many targets: sort the pairs
#pragma unroll
    for (int r = 0; r < S; ++r)
      if (32 * r < T && lane + 32 * r < T) sv[lane + 32 * r] = L.wt[r];
    auto sorted = [&](auto size) {
      constexpr int E = decltype(size)::value;
      unsigned long long e[E];
#pragma unroll
      for (int r = 0; r < E; ++r) {
        const int i = lane + 32 * r;
        e[r] = i < T ? ((unsigned long long)(uint32_t)L.k[r] << kIdxBits | (unsigned)i) : kSortPad;
      }
      sort_elements<E, 32>(e, nullptr);
#pragma unroll
      for (int r = 0; r < E; ++r) {
        const int i = pad4(lane * E + r);
        sk[i] = (int32_t)(e[r] >> kIdxBits);  // pads: beyond T
        si[i] = (uint16_t)(e[r] & ((1u << kIdxBits) - 1u));
      }
    };
    // T > kMergeSmall in the launch of the larger clusters
    if (2 * T <= kMax) sorted(std::integral_constant<int, S / 2>());
    else sorted(std::integral_constant<int, S>());
    __syncwarp();
    int out = 0;
    for (int c0 = 0; c0 < T; c0 += 32) {
      const int i = c0 + lane;
      const int32_t key = i < T ? sk[pad4(i)] : 0;
      const bool head = i < T && (i == 0 || sk[pad4(i - 1)] != key);
      long long sum = 0;
      if (head) {
        sum = sv[si[pad4(i)]];
        for (int j = i + 1; j < T && sk[pad4(j)] == key; ++j) sum += sv[si[pad4(j)]];
      }
      const unsigned bal = __ballot_sync(0xffffffffu, head);
      if (head) {
        const int at = out + __popc(bal & ((1u << lane) - 1u));
        seg_key[b + at] = key;
        seg_val[b + at] = sum;
      }
      out += __popc(bal);
    }
    if (lane == 0) dcount[x] = out;
    __syncwarp();
  }
}

// Clusters of kMergeMax < T <= kMergeBlockMax pairs: a block per cluster sorts the pairs by
// target (sort_elements, 4 to 16 elements per thread), then every run head sums its run; the
// distinct targets are written back in ascending order at the front of the segment.
// The clusters are the listed ones, list[0, *list_count).
constexpr int kMergeBlockSmem = (kMergeBlockMax + kMergeBlockMax / 16 + kMergeBlockMax) * 8;  // elements, sums

template <int E>
__device__ __forceinline__ int merge_block(long long b, int T, int32_t* __restrict__ seg_key,
                                           long long* __restrict__ seg_val, unsigned long long* se, long long* sv,
                                           int* s_warp) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  unsigned long long e[E];
#pragma unroll
  for (int r = 0; r < E; ++r) {
    const int i = tid + 256 * r;
    e[r] = i < T ? ((unsigned long long)(uint32_t)seg_key[b + i] << kIdxBits | (unsigned)i) : kSortPad;
    if (i < T) sv[i] = seg_val[b + i];
  }
  sort_elements<E, 256>(e, se);
  __syncthreads();
#pragma unroll
  for (int r = 0; r < E; ++r) se[pad8(tid * E + r)] = e[r];
  __syncthreads();
  // run heads among this thread's consecutive elements, numbered by a block scan
  const unsigned long long before0 = tid ? se[pad8(tid * E - 1)] >> kIdxBits : ~0ull;
  unsigned heads = 0;
#pragma unroll
  for (int r = 0; r < E; ++r) {
    const unsigned long long key = e[r] >> kIdxBits, prev = r ? e[r ? r - 1 : 0] >> kIdxBits : before0;
    if (e[r] != kSortPad && key != prev) heads |= 1u << r;
  }
  const int cnt = __popc(heads);
  int inc = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) s_warp[wid] = inc;
  __syncthreads();
  int before = 0, total = 0;
  for (int w2 = 0; w2 < 8; ++w2) {
    if (w2 < wid) before += s_warp[w2];
    total += s_warp[w2];
  }
  int at = before + inc - cnt;
  // the sorted copy and the sums are in shared memory, so the segment can be overwritten
  for (unsigned m = heads; m; m &= m - 1u) {
    const int i = tid * E + __ffs(m) - 1;
    const unsigned long long x = se[pad8(i)], key = x >> kIdxBits;
    long long sum = sv[x & ((1u << kIdxBits) - 1u)];
    for (int j = i + 1; j < T; ++j) {
      const unsigned long long y = se[pad8(j)];
      if (y >> kIdxBits != key) break;
      sum += sv[y & ((1u << kIdxBits) - 1u)];
    }
    seg_key[b + at] = (int32_t)key;
    seg_val[b + at] = sum;
    ++at;
  }
  return total;
}

__global__ void __launch_bounds__(256) cluster_merge_block_k(const long long* __restrict__ cbase,
                                                             int32_t* __restrict__ seg_key,
                                                             long long* __restrict__ seg_val,
                                                             int32_t* __restrict__ dcount,
                                                             const int32_t* __restrict__ list,
                                                             const int* __restrict__ list_count) {
  extern __shared__ __align__(16) unsigned char mb_dyn[];
  unsigned long long* se = (unsigned long long*)mb_dyn;
  long long* sv = (long long*)(se + kMergeBlockMax + kMergeBlockMax / 16);
  __shared__ int s_warp[8];
  const int total = *list_count;
  for (int xi = blockIdx.x; xi < total; xi += gridDim.x) {
    const int32_t x = list[xi];
    const long long b = cbase[x];
    const int T = (int)(cbase[x + 1] - b);  // kMergeMax < T <= kMergeBlockMax
    int d;
    if (T <= 1024) d = merge_block<4>(b, T, seg_key, seg_val, se, sv, s_warp);
    else if (T <= 2048) d = merge_block<8>(b, T, seg_key, seg_val, se, sv, s_warp);
    else d = merge_block<16>(b, T, seg_key, seg_val, se, sv, s_warp);
    if (threadIdx.x == 0) dcount[x] = d;
    __syncthreads();
  }
}

// The sorted distinct targets of every cluster, copied from the front of its segment
// to coff[c].
// Clusters with skip[x] != 0 (skip may be null) are left out (their lists are written
// by the sparse contraction's copy).
__global__ void __launch_bounds__(256) cluster_place_k(int64_t c, const long long* __restrict__ cbase,
                                                       const int64_t* __restrict__ coff,
                                                       const int32_t* __restrict__ seg_key,
                                                       const long long* __restrict__ seg_val,
                                                       int32_t* __restrict__ cadj, long long* __restrict__ cw,
                                                       int32_t* __restrict__ csrc,
                                                       const unsigned char* __restrict__ skip, LongLists longs) {
  // 32 clusters per warp step, their lists laid end to end over the lanes
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t x0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); x0 < c; x0 += stride) {
    const int64_t x = x0 + lane;
    const bool take = x < c && !(skip && skip[x]);
    const long long b = take ? cbase[x] : 0;
    const int64_t o = take ? coff[x] : 0;
    int64_t D = take ? coff[x + 1] - o : 0;
    if (longs.item && D > kLongList) {
      longs.push((int32_t)x, o);
      D = 0;
    }
    warp_pieces<KeyVal>(
        D, b, o, [&](int64_t at) { return KeyVal{seg_key[at], seg_val[at]}; },
        [&](int64_t at, int j, const KeyVal& kv) {
          cadj[at] = kv.k;
          cw[at] = kv.v;
          csrc[at] = (int32_t)(x0 + j);
        });
  }
}

// The lists cluster_place_k left out.
__global__ void cluster_place_long_k(const long long* __restrict__ cbase, const int64_t* __restrict__ coff,
                                     const int32_t* __restrict__ seg_key, const long long* __restrict__ seg_val,
                                     int32_t* __restrict__ cadj, long long* __restrict__ cw,
                                     int32_t* __restrict__ csrc, LongLists longs) {
  const int n = *longs.n;
  const GridShare G(n);
  for (int i = G.first; i < n; i += G.step) {
    const int32_t x = longs.item[i];
    const long long b = cbase[x];
    const int64_t o = longs.at[i], D = coff[x + 1] - o;
    for (int64_t j = (int64_t)G.part * blockDim.x + threadIdx.x; j < D; j += (int64_t)G.parts * blockDim.x) {
      cadj[o + j] = seg_key[b + j];
      cw[o + j] = seg_val[b + j];
      csrc[o + j] = x;
    }
  }
}

// ---------------------------------------------------------------- sparse contraction
// Contractions in which most vertices keep their own id as label, alone in their cluster
// (Padberg-Rinaldi passes and exact-step rounds by union-find roots, label-propagation
// levels that merge few vertices), on a graph with strictly increasing lists.  The
// cluster id of such a "lone" vertex is the rank of its own id among the labels, so lone
// neighbours keep their order and stay distinct under the renumbering.  The coarse list of
// a lone vertex is its fine list renumbered, except for the few entries that point into
// the other ("merged") clusters: those may repeat a target and sit out of order.
// A warp per lone vertex sums them per target in shared memory and merges the distinct
// ones into the renumbered list -- one pass to count the coarse degree, one to write.  Only
// the members of merged groups (and lone vertices with more than kScMaxM such entries) go
// through the pre-merge and the cluster merge.
constexpr int kScMaxM = 32;  // entries into merged groups per lone vertex

// mflag[cid[v]] = 1 for every v not labelled by its own id (its cluster has another
// member, or its label is another vertex's id); a plain store of 1 from any number of
// threads.
__global__ void sc_merged_k(int64_t n, const int32_t* __restrict__ lab, const int32_t* __restrict__ cid,
                            unsigned char* __restrict__ mflag) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    if (lab[v] != (int32_t)v) mflag[cid[v]] = 1;
}

// cidm[u] = cid[u], with the sign bit set when u's group is merged: one gather per entry
// gives both.
__global__ void sc_pack_k(int64_t n, const int32_t* __restrict__ cid, const unsigned char* __restrict__ mflag,
                          int32_t* __restrict__ cidm) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t x = cid[v];
    cidm[v] = mflag[x] ? (int32_t)((uint32_t)x | 0x80000000u) : x;
  }
}

constexpr int kScUnroll = 4;  // rows of 32 entries in flight per warp

// The entries of lone vertex v's list that point into merged groups, collected row by
// row in the warp's shared arrays mk and (kWeights) mw (at most kScMaxM kept; the return
// value counts them all).
template <bool kWeights, typename WT>
__device__ __forceinline__ int sc_collect(int64_t beg, int64_t end, int lane, const int32_t* __restrict__ adj,
                                          const WT* __restrict__ w, const int32_t* __restrict__ cidm, int32_t* mk,
                                          long long* mw) {
  int nm = 0;
  for (int64_t b = beg; b < end; b += 32 * kScUnroll) {
    int32_t u[kScUnroll], k[kScUnroll];
#pragma unroll
    for (int q = 0; q < kScUnroll; ++q) {
      const int64_t e = b + 32 * q + lane;
      u[q] = e < end ? __ldg(adj + e) : -1;
    }
#pragma unroll
    for (int q = 0; q < kScUnroll; ++q) k[q] = u[q] >= 0 ? __ldg(cidm + u[q]) : 0;
    bool any = false;
#pragma unroll
    for (int q = 0; q < kScUnroll; ++q) any |= k[q] < 0;
    if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll
    for (int q = 0; q < kScUnroll; ++q) {
      const bool m = k[q] < 0;
      const unsigned bal = __ballot_sync(0xffffffffu, m);
      if (m) {
        const int at = nm + __popc(bal & ((1u << lane) - 1u));
        if (at < kScMaxM) {
          mk[at] = k[q] & 0x7fffffff;
          if (kWeights) mw[at] = ldw(w, b + 32 * q + lane);
        }
      }
      nm += __popc(bal);
    }
  }
  __syncwarp();
  return nm;
}

// A contraction that merges few vertices touches few lists: the neighbours of the merged
// groups' members (every edge is in both lists: GraphView::symmetric), found from the
// members' own.  They are marked so (touched) while at most a sixteenth of the vertices
// disappears, and pass 1 then reads only those lists; otherwise it reads every list.  Planted
// 8 x 2^20, 392 million entries: 1.25 ms a pass over every list, whatever the pass merged (one
// random gather per entry, at 0.8 of one per SM and cycle); 31.0 -> 17.2 ms for its 25
// contractions.  Below kScPushMin entries a pass costs less than the marking: whole planted
// runs by entries, with the marks and sc_copy_k and without both, 6.3 million 14.6 and 13.8 ms,
// 25 million 28.4 and 27.7, 50 million 60.6 and 60.7, 101 million 90.5 and 93.0, 201 million
// 173 and 177.  An eighth or a thirty-second of the vertices instead: the same within 1 %.
constexpr int64_t kScPushMin = int64_t(1) << 25;
__device__ __forceinline__ bool sc_few(int64_t n, const int* nclust) { return 16 * (n - __ldg(nclust)) <= n; }

__global__ void __launch_bounds__(256) sc_push_k(int64_t n, const int* __restrict__ nclust,
                                                 const int32_t* __restrict__ cidm, const int64_t* __restrict__ off,
                                                 const int32_t* __restrict__ adj,
                                                 unsigned char* __restrict__ touched, int32_t* __restrict__ longs,
                                                 int* __restrict__ nlong) {
  if (!sc_few(n, nclust)) return;
  const int lane = threadIdx.x & 31;
  for (int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~31LL; b < n;
       b += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = b + lane;
    for (unsigned m = __ballot_sync(0xffffffffu, v < n && cidm[v] < 0); m; m &= m - 1u) {
      const int64_t x = b + __ffs(m) - 1, beg = off[x], end = off[x + 1];
      if (end - beg > kLongList) {
        if (lane == 0) longs[atomicAdd(nlong, 1)] = (int32_t)x;
        continue;
      }
#pragma unroll 4
      for (int64_t e = beg + lane; e < end; e += 32) touched[__ldg(adj + e)] = 1;
    }
  }
}

// The lists sc_push_k left out (a hub's), shared by the blocks.
__global__ void __launch_bounds__(256) sc_push_long_k(const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
                                                      unsigned char* __restrict__ touched,
                                                      const int32_t* __restrict__ longs,
                                                      const int* __restrict__ nlong) {
  const int n = *nlong;
  const GridShare G(n);
  for (int i = G.first; i < n; i += G.step) {
    const int64_t beg = off[longs[i]], end = off[longs[i] + 1];
#pragma unroll 4
    for (int64_t e = beg + G.part * 256 + threadIdx.x; e < end; e += (int64_t)G.parts * 256)
      touched[__ldg(adj + e)] = 1;
  }
}

// Pass 1: the coarse degree of every lone vertex handled here (sdeg[v], else -1), and in
// dirty the vertices left to the pre-merge (1) and the lists with no entry into a merged
// group (2).  A warp per `per` vertices, the lists to read one after another: 32 where most
// are not read (touched), else 1.
__global__ void __launch_bounds__(256) sc_count_k(int64_t n, const int* __restrict__ nclust,
                                                  const int32_t* __restrict__ cidm, const int64_t* __restrict__ off,
                                                  const int32_t* __restrict__ adj,
                                                  const unsigned char* __restrict__ touched,
                                                  int32_t* __restrict__ sdeg, unsigned char* __restrict__ dirty,
                                                  int per) {
  __shared__ int32_t s_mk[8][kScMaxM];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const bool few = touched && sc_few(n, nclust);
  for (int64_t b = ((int64_t)blockIdx.x * 8 + wid) * per; b < n; b += (int64_t)gridDim.x * 8 * per) {
    const int64_t v = lane < per ? b + lane : n;
    int64_t beg = 0, end = 0;
    bool read = false;
    int32_t deg = -1;         // a member of a merged group
    unsigned char state = 1;
    if (v < n) {
      beg = off[v];
      end = off[v + 1];
      if (cidm[v] >= 0) {
        read = !few || touched[v];
        deg = (int32_t)(end - beg);
        state = 2;
      }
    }
    for (unsigned m = __ballot_sync(0xffffffffu, read); m; m &= m - 1u) {
      const int j = __ffs(m) - 1;
      const int64_t lb = __shfl_sync(0xffffffffu, beg, j), le = __shfl_sync(0xffffffffu, end, j);
      const int nm = sc_collect<false>(lb, le, lane, adj, (const UnitW*)nullptr, cidm, s_mk[wid], nullptr);
      int nd = nm;
      if (nm > 1 && nm <= kScMaxM) {  // the same in every lane
        const bool have = lane < nm;
        const int32_t key = have ? s_mk[wid][lane] : -1 - lane;
        const unsigned peers = __match_any_sync(0xffffffffu, key);
        nd = __popc(__ballot_sync(0xffffffffu, have && (__ffs(peers) - 1) == lane));
      }
      if (lane == j && nm > 0) {
        deg = nm > kScMaxM ? -1 : deg - nm + nd;
        state = nm > kScMaxM ? 1 : 0;
      }
      __syncwarp();
    }
    if (v < n) {
      sdeg[v] = deg;
      dirty[v] = state;
    }
  }
}

// Pass 2 of the lists with no entry into a merged group, where at most one vertex in 512
// disappears: most runs of 2^shift consecutive ids then lose none, and their new ids are the
// old ones less one offset.  The offsets of all runs (tab; -1: some id is gone) fit shared
// memory, and only entries into the other runs gather their new id.  What is left is a
// stream: 12 bytes read and 16 written per entry (392 million entries, 1800 of 4.4 million
// vertices gone: 3.5 ms -> 2.4 ms here and 0.4 ms in sc_write_k; 15,800 gone, over one in
// 512: too few whole runs).  From kScPushMin entries on (alone, whole planted runs: 25 million
// 28.3 against 27.7 ms, 101 million 92.6 against 93.0).  One vertex in 128 or in 2048 instead:
// within 1 % at 101 and 134 million entries.
constexpr int kScTab = 16384;  // runs at most
constexpr int kScCopyThreads = 512;
static int sc_shift(int64_t n) { return std::max(8, ceil_log2(n) - 14); }

__global__ void sc_table_k(int64_t n, int64_t c, int shift, const int32_t* __restrict__ rank,
                           int32_t* __restrict__ tab) {
  const int64_t runs = (n + (1LL << shift) - 1) >> shift;
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < runs; r += (int64_t)gridDim.x * blockDim.x) {
    const int64_t a = r << shift, z = (r + 1) << shift < n ? (r + 1) << shift : n;
    const int64_t ra = rank[a], rz = z < n ? (int64_t)rank[z] : c;
    tab[r] = rz - ra == z - a ? (int32_t)(a - ra) : -1;
  }
}

template <typename WT>
__global__ void __launch_bounds__(kScCopyThreads) sc_copy_k(int64_t n, int shift, const int32_t* __restrict__ tab,
                                                            const int32_t* __restrict__ cidm,
                                                            const int64_t* __restrict__ off,
                                                            const int32_t* __restrict__ adj,
                                                            const WT* __restrict__ w,
                                                            const unsigned char* __restrict__ dirty,
                                                            const int64_t* __restrict__ coff,
                                                            int32_t* __restrict__ cadj, long long* __restrict__ cw,
                                                            int32_t* __restrict__ csrc) {
  extern __shared__ int32_t s_tab[];
  const int lane = threadIdx.x & 31;
  const int runs = (int)((n + (1LL << shift) - 1) >> shift);
  for (int i = threadIdx.x; i < runs; i += kScCopyThreads) s_tab[i] = tab[i];
  __syncthreads();
  const int64_t warps = (int64_t)gridDim.x * (kScCopyThreads / 32);
  int64_t v = ((int64_t)blockIdx.x * kScCopyThreads + threadIdx.x) >> 5;
  if (v >= n) return;
  // the next list's header is read ahead
  int64_t beg = off[v], to = 0;
  int len = dirty[v] == 2 ? (int)(off[v + 1] - beg) : 0;  // a strictly increasing list: below 2^31 entries
  int32_t x = cidm[v];
  for (;;) {
    const int64_t vn = v + warps;
    int64_t nbeg = 0;
    int nlen = 0;
    int32_t xn = 0;
    if (vn < n) {
      nbeg = off[vn];
      nlen = dirty[vn] == 2 ? (int)(off[vn + 1] - nbeg) : 0;
      xn = cidm[vn];
    }
    if (len > 0) {
      to = coff[x];
      const int32_t* a = adj + beg;
      for (int b = lane; b - lane < len; b += 32 * kScUnroll) {
        int32_t u[kScUnroll];
        long long wt[kScUnroll];
#pragma unroll
        for (int q = 0; q < kScUnroll; ++q) {
          u[q] = b + 32 * q < len ? __ldg(a + b + 32 * q) : -1;
          wt[q] = b + 32 * q < len ? ldw(w, beg + b + 32 * q) : 0;
        }
#pragma unroll
        for (int q = 0; q < kScUnroll; ++q)
          if (u[q] >= 0) {
            const int32_t d = s_tab[u[q] >> shift];
            u[q] = d >= 0 ? u[q] - d : __ldg(cidm + u[q]) & 0x7fffffff;
          }
#pragma unroll
        for (int q = 0; q < kScUnroll; ++q)
          if (u[q] >= 0) {
            cadj[to + b + 32 * q] = u[q];
            cw[to + b + 32 * q] = wt[q];
            csrc[to + b + 32 * q] = x;
          }
      }
    }
    if (vn >= n) break;
    v = vn;
    beg = nbeg;
    len = nlen;
    x = xn;
  }
}

// Pass 2: the lists of the lone vertices counted in pass 1, at their coarse offsets.
// The coarse list merges two ascending sequences: the entries into lone vertices' clusters
// (in list order) and the nd distinct merged targets (sorted).  The warp gathers a chunk of
// kScChunk entries' new ids once, packs the lone ones into shared memory with their places,
// finds every target's place among them by one binary search per target, marks the places the
// targets take in the output as bits, and writes the output row by row: a bit count tells
// which target or which lone entry each place holds.  A list of one chunk (nearly all) is
// read once; a longer one is read once more beforehand for its merged entries.
// Planted 8 x 2^20 (392 million entries, 12 bytes read and 16 written each, a random gather
// each): 22 passes 79.0 -> 77.0 ms, 8 x 60,013: 20 passes 4.47 -> 4.16 ms against a version
// that gathered twice and searched and matched per entry; it waits on memory (DRAM 39 %, L1
// 56 %).  A copy of the unchanged lists in a kernel of its own with half the registers, and
// evict-first loads and stores, measured slower (80 and 85 ms).
constexpr int kScChunk = 512;

template <typename WT>
__global__ void __launch_bounds__(256) sc_write_k(int64_t n, const int32_t* __restrict__ cidm,
                                                  const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
                                                  const WT* __restrict__ w,
                                                  const unsigned char* __restrict__ dirty,
                                                  const int64_t* __restrict__ coff, int32_t* __restrict__ cadj,
                                                  long long* __restrict__ cw, int32_t* __restrict__ csrc,
                                                  bool copied) {
  __shared__ int32_t s_mk[8][kScMaxM];
  __shared__ long long s_mw[8][kScMaxM];
  __shared__ int32_t s_dk[8][kScMaxM];
  __shared__ long long s_dw[8][kScMaxM];
  __shared__ int32_t s_key[8][kScChunk];                     // lone entries of the chunk: new id,
  __shared__ uint16_t s_at[8][kScChunk];                     // place in the chunk
  __shared__ unsigned s_bits[8][(kScChunk + kScMaxM) / 32];  // output places held by targets
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned lower = (1u << lane) - 1u;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  int32_t *mk = s_mk[wid], *dk = s_dk[wid], *key = s_key[wid];
  long long *mw = s_mw[wid], *dw = s_dw[wid];
  uint16_t* at = s_at[wid];
  unsigned* bits = s_bits[wid];
  for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += warps) {
    const unsigned char state = dirty[v];
    if (state == 1 || (state == 2 && copied)) continue;  // the same in every lane
    const int64_t beg = off[v], end = off[v + 1];
    const int32_t x = cidm[v];  // lone: no sign bit
    int64_t o = coff[x];
    if (state == 2) {  // no entry into a merged cluster: the list renumbered in place
      for (int64_t b = beg; b < end; b += 32 * kScUnroll) {
        int32_t u[kScUnroll];
        long long wt[kScUnroll];
#pragma unroll
        for (int q = 0; q < kScUnroll; ++q) {
          const int64_t e = b + 32 * q + lane;
          u[q] = e < end ? __ldcs(adj + e) : -1;
          wt[q] = e < end ? ldw(w, e) : 0;
        }
#pragma unroll
        for (int q = 0; q < kScUnroll; ++q) u[q] = u[q] >= 0 ? __ldg(cidm + u[q]) & 0x7fffffff : -1;
#pragma unroll
        for (int q = 0; q < kScUnroll; ++q)
          if (u[q] >= 0) {
            const int64_t to = o + (b + 32 * q + lane - beg);
            cadj[to] = u[q];
            cw[to] = wt[q];
            csrc[to] = x;
          }
      }
      continue;
    }
    const bool one = end - beg <= kScChunk;
    int nm = one ? 0 : sc_collect<true>(beg, end, lane, adj, w, cidm, mk, mw);
    int nd = -1, td = 0;  // distinct targets (-1: not known yet), those written so far
    for (int64_t c0 = beg; c0 < end; c0 += kScChunk) {
      const int64_t c1 = c0 + kScChunk < end ? c0 + kScChunk : end;
      // the chunk's lone entries, packed in order (and, in a list of one chunk, the merged ones)
      int nl = 0;
      for (int64_t b = c0; b < c1; b += 32 * kScUnroll) {
        int32_t u[kScUnroll];
#pragma unroll
        for (int q = 0; q < kScUnroll; ++q) {
          const int64_t e = b + 32 * q + lane;
          u[q] = e < c1 ? __ldg(adj + e) : -1;
        }
        unsigned in = 0;
#pragma unroll
        for (int q = 0; q < kScUnroll; ++q) {
          if (u[q] >= 0) in |= 1u << q;
          u[q] = u[q] >= 0 ? __ldg(cidm + u[q]) : 0;
        }
#pragma unroll
        for (int q = 0; q < kScUnroll; ++q) {
          const bool lone = ((in >> q) & 1u) && u[q] >= 0;
          const bool m = one && u[q] < 0;
          const unsigned balL = __ballot_sync(0xffffffffu, lone);
          if (lone) {
            const int p = nl + __popc(balL & lower);
            key[p] = u[q];
            at[p] = (uint16_t)(b + 32 * q + lane - c0);
          }
          nl += __popc(balL);
          const unsigned balM = __ballot_sync(0xffffffffu, m);
          if (m) {  // at most kScMaxM: pass 1 left a list with more to the pre-merge
            const int p = nm + __popc(balM & lower);
            mk[p] = u[q] & 0x7fffffff;
            mw[p] = ldw(w, b + 32 * q + lane);
          }
          nm += __popc(balM);
        }
      }
      __syncwarp();
      if (nd < 0) {
        // distinct targets into merged groups: the lowest lane of each target sums it and
        // places it by its rank among the distinct targets
        const bool have = lane < nm;
        const int32_t k = have ? mk[lane] : -1 - lane;
        const unsigned peers = __match_any_sync(0xffffffffu, k);
        const bool first = have && (__ffs(peers) - 1) == lane;
        const unsigned firsts = __ballot_sync(0xffffffffu, first);
        nd = __popc(firsts);
        if (first) {
          long long sum = 0;
          for (unsigned m = peers; m; m &= m - 1u) sum += mw[__ffs(m) - 1];
          int rank = 0;
          for (unsigned m = firsts; m; m &= m - 1u) rank += mk[__ffs(m) - 1] < k;
          dk[rank] = k;
          dw[rank] = sum;
        }
        __syncwarp();
      }
      // the targets that belong here: those below the chunk's last lone entry, and in the last
      // chunk all that are left; td + 0, td + 1, ... in order
      const bool mine = lane >= td && lane < nd && (c1 == end || (nl > 0 && dk[lane] < key[nl - 1]));
      const int nt = __popc(__ballot_sync(0xffffffffu, mine));
      const int total = nl + nt;
      for (int r = lane; r < (total + 31) >> 5; r += 32) bits[r] = 0;
      __syncwarp();
      if (mine) {
        int lo = 0, hi = nl;  // the lone entries below the target
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (key[mid] < dk[lane]) lo = mid + 1;
          else hi = mid;
        }
        const int p = lo + lane - td;
        atomicOr(&bits[p >> 5], 1u << (p & 31));
      }
      __syncwarp();
      int tb = 0;  // targets in the rows before
      for (int r0 = 0; r0 < total; r0 += 32 * kScUnroll) {
        int32_t k[kScUnroll];
        long long wt[kScUnroll];
#pragma unroll
        for (int q = 0; q < kScUnroll; ++q) {
          const int p = r0 + 32 * q + lane;
          const unsigned m = r0 + 32 * q < total ? bits[(r0 >> 5) + q] : 0u;
          const int below = tb + __popc(m & lower);
          tb += __popc(m);
          k[q] = -1;
          if (p < total) {
            if ((m >> lane) & 1u) {
              k[q] = dk[td + below];
              wt[q] = dw[td + below];
            } else {
              k[q] = key[p - below];
              wt[q] = ldw(w, c0 + at[p - below]);
            }
          }
        }
#pragma unroll
        for (int q = 0; q < kScUnroll; ++q)
          if (k[q] >= 0) {
            const int64_t to = o + r0 + 32 * q + lane;
            cadj[to] = k[q];
            cw[to] = wt[q];
            csrc[to] = x;
          }
      }
      o += total;
      td += nt;
      __syncwarp();  // the chunk's arrays are filled again
    }
  }
}

// The vertices left to the pre-merge, listed (in no particular order); *count their number.
__global__ void sc_list_k(int64_t n, const unsigned char* __restrict__ dirty, int32_t* __restrict__ list,
                          int* __restrict__ count) {
  const int lane = threadIdx.x & 31;
  for (int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~31LL; b < n;
       b += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = b + lane;
    const bool d = v < n && dirty[v] == 1;
    const unsigned bal = __ballot_sync(0xffffffffu, d);
    int at = 0;
    if (lane == 0 && bal) at = atomicAdd(count, __popc(bal));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (d) list[at + __popc(bal & ((1u << lane) - 1u))] = (int32_t)v;
  }
}

// After the merge of the pre-merged clusters: the coarse degree of every cluster of a
// lone vertex handled here, and clean[x] marking those clusters.
__global__ void sc_clean_deg_k(int64_t n, const int32_t* __restrict__ sdeg, const int32_t* __restrict__ cid,
                               int32_t* __restrict__ ccount, unsigned char* __restrict__ clean) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    if (sdeg[v] < 0) continue;
    const int32_t x = cid[v];
    ccount[x] = sdeg[v];
    clean[x] = 1;
  }
}

template <typename F>
static void sc_by_weight(const GraphView& g, F f) {
  if (g.unit) f((const UnitW*)nullptr);
  else if (g.wbytes == 4) f((const int32_t*)g.w);
  else f((const long long*)g.w);
}

void sparse_mark(const GraphView& g, const int32_t* lab, const int32_t* cid, const int* nclust, unsigned char* mflag,
                 unsigned char* touched, int32_t* cidm, unsigned char* dirty, int32_t* sdeg, int32_t* list, int* count,
                 cudaStream_t s) {
  VC_CUDA(cudaMemsetAsync(mflag, 0, (size_t)g.n, s));
  VC_CUDA(cudaMemsetAsync(count, 0, sizeof(int), s));
  const int grid = grid_for(g.n, 256, kSMs * 8);
  sc_merged_k<<<grid, 256, 0, s>>>(g.n, lab, cid, mflag);
  sc_pack_k<<<grid, 256, 0, s>>>(g.n, cid, mflag, cidm);
  if (touched) {
    VC_CUDA(cudaMemsetAsync(touched, 0, (size_t)g.n, s));
    sc_push_k<<<grid, 256, 0, s>>>(g.n, nclust, cidm, g.off, g.adj, touched, list, count);
    sc_push_long_k<<<kSMs * 4, 256, 0, s>>>(g.off, g.adj, touched, list, count);
    VC_CUDA(cudaMemsetAsync(count, 0, sizeof(int), s));
    count_launch(2);
  }
  const int per = touched ? 32 : 1;
  sc_count_k<<<grid_for(g.n, 8 * per, kSMs * (touched ? 64 : 16)), 256, 0, s>>>(g.n, nclust, cidm, g.off, g.adj,
                                                                                touched, sdeg, dirty, per);
  sc_list_k<<<grid, 256, 0, s>>>(g.n, dirty, list, count);
  count_launch(4);
  VC_CHECK_LAUNCH();
}

bool sparse_touches(const GraphView& g) { return g.symmetric && g.nnz >= kScPushMin; }

static void sparse_finish_degrees(const GraphView& g, const int32_t* cid, const int32_t* sdeg, int32_t* ccount,
                                  unsigned char* clean, int64_t c, cudaStream_t s) {
  VC_CUDA(cudaMemsetAsync(clean, 0, (size_t)std::max<int64_t>(c, 1), s));
  sc_clean_deg_k<<<grid_for(g.n, 256, kSMs * 8), 256, 0, s>>>(g.n, sdeg, cid, ccount, clean);
  count_launch();
  VC_CHECK_LAUNCH();
}

static void sparse_copy(const GraphView& g, int64_t c, const SparseCtx& sp, const int64_t* coff, int32_t* cadj,
                        long long* cw, int32_t* csrc, cudaStream_t s) {
  const bool table = 512 * (g.n - c) <= g.n && g.nnz >= kScPushMin;
  const int shift = sc_shift(g.n), runs = (int)((g.n + (int64_t(1) << shift) - 1) >> shift);
  if (table) {
    sc_table_k<<<grid_for(runs, 256, kSMs), 256, 0, s>>>(g.n, c, shift, sp.rank, sp.tab);
    count_launch();
  }
  sc_by_weight(g, [&](auto wp) {
    using WT = std::remove_cv_t<std::remove_pointer_t<decltype(wp)>>;
    if (table) {
      set_smem(sc_copy_k<WT>, kScTab * sizeof(int32_t));
      sc_copy_k<WT><<<grid_for(g.n, kScCopyThreads / 32, kSMs * 8), kScCopyThreads, sizeof(int32_t) * runs, s>>>(
          g.n, shift, sp.tab, sp.cidm, g.off, g.adj, wp, sp.dirty, coff, cadj, cw, csrc);
      count_launch();
    }
    sc_write_k<WT><<<grid_for(g.n, 8, kSMs * 16), 256, 0, s>>>(g.n, sp.cidm, g.off, g.adj, wp, sp.dirty, coff, cadj,
                                                               cw, csrc, table);
  });
  count_launch();
  VC_CHECK_LAUNCH();
}

// ---------------------------------------------------------------- correcting step
// Sec. 4.1, "correcting algorithm" (fixMisplacedVertices of Algorithm 1), optional: in
// every cluster C of 2..lg vertices (lg = floor(log2 n)), d(C) = weight of the edges
// leaving C and, for a member v, d(C - v) = d(C) - c(v, V - C) + c(v, C - v); v is
// misplaced when d(C - v) < d(C), and each cluster gives up at most its misplaced
// vertex of smallest d(C - v) (ties: smallest id), which becomes a singleton with a
// cluster id after all others, in ascending vertex order.
__global__ void corr_size_k(int64_t n, const int32_t* __restrict__ cid, int* __restrict__ csize) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(&csize[cid[v]], 1);
}

__device__ __forceinline__ bool corr_small(int sz, int lg) { return sz >= 2 && sz <= lg; }

// Eight lanes per vertex of a small cluster: its weight to the outside and to the rest
// of its cluster; the outside weights sum into d(C).
template <typename WT>
__global__ void corr_sums_k(int64_t n, const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
                            const WT* __restrict__ w, const int32_t* __restrict__ cid,
                            const int* __restrict__ csize, int lg, long long* __restrict__ vout,
                            long long* __restrict__ vin, long long* __restrict__ dc) {
  constexpr int G = 8;
  const int lane = threadIdx.x & 31, glane = lane & (G - 1);
  const unsigned gmask = ((1u << G) - 1u) << (lane & ~(G - 1));
  const int64_t groups = (int64_t)gridDim.x * (blockDim.x / G);
  for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G; v < n; v += groups) {
    const int32_t C = cid[v];
    if (!corr_small(csize[C], lg)) continue;  // the same in the group's lanes
    long long o = 0, i = 0;
    for (int64_t e = off[v] + glane; e < off[v + 1]; e += G) {
      const long long x = ldw(w, e);
      if (cid[adj[e]] == C) i += x;
      else o += x;
    }
#pragma unroll
    for (int k = G / 2; k > 0; k >>= 1) {
      o += __shfl_xor_sync(gmask, o, k);
      i += __shfl_xor_sync(gmask, i, k);
    }
    if (glane == 0) {
      vout[v] = o;
      vin[v] = i;
      if (o) atomicAdd((unsigned long long*)&dc[C], (unsigned long long)o);
    }
  }
}

// pass 0: the smallest d(C - v) below d(C) per cluster; pass 1: the smallest id
// attaining it; pass 2: flag[v] = v leaves its cluster.
__global__ void corr_pick_k(int64_t n, const int32_t* __restrict__ cid, const int* __restrict__ csize, int lg,
                            const long long* __restrict__ vout, const long long* __restrict__ vin,
                            const long long* __restrict__ dc, long long* __restrict__ bestv,
                            int* __restrict__ bestid, int* __restrict__ flag, int pass) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t C = cid[v];
    const bool small = corr_small(csize[C], lg);
    if (pass == 2) {
      flag[v] = small && bestid[C] == (int)v ? 1 : 0;
      continue;
    }
    if (!small) continue;
    const long long without = dc[C] - vout[v] + vin[v];
    if (without >= dc[C]) continue;
    if (pass == 0) atomicMin(&bestv[C], without);
    else if (without == bestv[C]) atomicMin(&bestid[C], (int)v);
  }
}

__global__ void corr_apply_k(int64_t n, const int* __restrict__ flag, const int* __restrict__ rank,
                             const int* __restrict__ c_dev, int32_t* __restrict__ cid) {
  const int c = *c_dev;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    if (flag[v]) cid[v] = c + rank[v];
}

__global__ void corr_count_k(int* __restrict__ c_dev, const int* __restrict__ moved) { *c_dev += *moved; }

void correct_clusters(const GraphView& g, int32_t* cid, int* c_dev, const CorrectScratch& cs, cudaStream_t s) {
  const int64_t n = g.n;
  if (n < 4) return;  // no cluster of 2..floor(log2 n) vertices below 4 vertices
  int lg = 0;
  while ((int64_t(2) << lg) <= n) ++lg;
  VC_CUDA(cudaMemsetAsync(cs.csize, 0, sizeof(int) * n, s));
  VC_CUDA(cudaMemsetAsync(cs.dc, 0, sizeof(long long) * n, s));
  VC_CUDA(cudaMemsetAsync(cs.bestv, 0x7f, sizeof(long long) * n, s));  // above every d(C - v)
  VC_CUDA(cudaMemsetAsync(cs.bestid, 0x7f, sizeof(int) * n, s));       // above every vertex id
  const int grid = grid_for(n, 256, kSMs * 8);
  corr_size_k<<<grid, 256, 0, s>>>(n, cid, cs.csize);
  const int gs = grid_for(n, 32, kSMs * 16);
  if (g.unit)
    corr_sums_k<UnitW><<<gs, 256, 0, s>>>(n, g.off, g.adj, nullptr, cid, cs.csize, lg, cs.vout, cs.vin, cs.dc);
  else if (g.wbytes == 4)
    corr_sums_k<int32_t><<<gs, 256, 0, s>>>(n, g.off, g.adj, (const int32_t*)g.w, cid, cs.csize, lg, cs.vout,
                                            cs.vin, cs.dc);
  else
    corr_sums_k<long long><<<gs, 256, 0, s>>>(n, g.off, g.adj, (const long long*)g.w, cid, cs.csize, lg, cs.vout,
                                              cs.vin, cs.dc);
  for (int pass = 0; pass < 3; ++pass)
    corr_pick_k<<<grid, 256, 0, s>>>(n, cid, cs.csize, lg, cs.vout, cs.vin, cs.dc, cs.bestv, cs.bestid, cs.flag,
                                     pass);
  count_launch(5);
  VC_CHECK_LAUNCH();
  exclusive_scan<int, int>(cs.flag, cs.rank, n, cs.moved, cs.scan_scr32, s);
  corr_apply_k<<<grid, 256, 0, s>>>(n, cs.flag, cs.rank, c_dev, cid);
  corr_count_k<<<1, 1, 0, s>>>(c_dev, cs.moved);
  count_launch(2);
  VC_CHECK_LAUNCH();
}

// ---------------------------------------------------------------- giant clusters
__global__ void giant_list_k(int64_t c, const long long* __restrict__ cbase, int* __restrict__ gcount,
                             int32_t* __restrict__ glist, int32_t* __restrict__ gT) {
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < c; x += (int64_t)gridDim.x * blockDim.x) {
    const long long T = cbase[x + 1] - cbase[x];
    if (T > kMergeBlockMax) {
      const int j = atomicAdd(gcount, 1);
      glist[j] = (int32_t)x;
      gT[j] = (int32_t)T;
    }
  }
}

// The giant clusters' pairs, keyed (j << bits | target) for giant j.
__global__ void giant_gather_k(int ng, const int32_t* __restrict__ glist, const long long* __restrict__ gstart,
                               const long long* __restrict__ cbase, const int32_t* __restrict__ seg_key,
                               const long long* __restrict__ seg_val, int bits, unsigned long long* __restrict__ keys,
                               long long* __restrict__ vals) {
  const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, st = (int64_t)gridDim.x * blockDim.x;
  for (int j = 0; j < ng; ++j) {
    const long long b = cbase[glist[j]], o = gstart[j], T = gstart[j + 1] - o;
    for (int64_t e = t0; e < T; e += st) {
      keys[o + e] = ((unsigned long long)j << bits) | (unsigned long long)(uint32_t)seg_key[b + e];
      vals[o + e] = seg_val[b + e];
    }
  }
}

// Every run head of the sorted giant pairs sums its run and writes it at its rank within
// its cluster, at the front of the cluster's segment.
__global__ void giant_reduce_k(int64_t m, int bits, const unsigned long long* __restrict__ keys,
                               const long long* __restrict__ vals, const int32_t* __restrict__ heads,
                               const long long* __restrict__ hpos, const long long* __restrict__ gstart,
                               const int32_t* __restrict__ glist, const long long* __restrict__ cbase,
                               int32_t* __restrict__ seg_key, long long* __restrict__ seg_val) {
  const unsigned long long mask = (1ULL << bits) - 1ULL;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    if (!heads[i]) continue;
    const unsigned long long k = keys[i];
    long long sum = vals[i];
    for (int64_t q = i + 1; q < m && keys[q] == k; ++q) sum += vals[q];
    const int j = (int)(k >> bits);
    const long long at = cbase[glist[j]] + (hpos[i] - hpos[gstart[j]]);
    seg_key[at] = (int32_t)(k & mask);
    seg_val[at] = sum;
  }
}

__global__ void giant_count_k(int ng, const int32_t* __restrict__ glist, const long long* __restrict__ gstart,
                              const long long* __restrict__ hpos, int32_t* __restrict__ dcount) {
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < ng; j += gridDim.x * blockDim.x)
    dcount[glist[j]] = (int32_t)(hpos[gstart[j + 1]] - hpos[gstart[j]]);
}

static void giant_merge(GiantScratch G, int64_t c, const long long* cbase, int32_t* seg_key,
                        long long* seg_val, int32_t* dcount, long long* scan_scr, cudaStream_t s) {
  VC_CUDA(cudaMemsetAsync(G.gcount, 0, sizeof(int), s));
  giant_list_k<<<grid_for(c, 256, kSMs * 8), 256, 0, s>>>(c, cbase, G.gcount, G.glist, G.gT);
  count_launch();
  VC_CHECK_LAUNCH();
  exclusive_scan<int, long long>(G.gT, G.gstart, G.ngiant, G.gstart + G.ngiant, scan_scr, s);
  int bits = ceil_log2(c);
  if (bits < 1) bits = 1;
  int jbits = ceil_log2(G.ngiant);
  if (jbits < 1) jbits = 1;
  const int grid = grid_for(G.pairs, 256, kSMs * 8);
  giant_gather_k<<<grid, 256, 0, s>>>(G.ngiant, G.glist, G.gstart, cbase, seg_key, seg_val, bits, G.k0, G.v0);
  count_launch();
  VC_CHECK_LAUNCH();
  radix_sort_pairs(G.k0, G.v0, G.k1, G.v1, G.pairs, bits + jbits, G.hist, s);
  run_heads_k<<<grid, 256, 0, s>>>(G.k0, G.pairs, G.heads);
  count_launch();
  VC_CHECK_LAUNCH();
  exclusive_scan<int, long long>(G.heads, G.hpos, G.pairs, G.hpos + G.pairs, scan_scr, s);
  giant_reduce_k<<<grid, 256, 0, s>>>(G.pairs, bits, G.k0, G.v0, G.heads, G.hpos, G.gstart, G.glist, cbase, seg_key,
                                      seg_val);
  giant_count_k<<<grid_for(G.ngiant, 256, kSMs), 256, 0, s>>>(G.ngiant, G.glist, G.gstart, G.hpos, dcount);
  count_launch(2);
  VC_CHECK_LAUNCH();
}

void cluster_stats(int64_t n, const int32_t* ccount, int* maxt, long long* pairs, int* ngiant, long long* gpairs,
                   cudaStream_t s) {
  if (n <= 0) return;
  cluster_stats_k<<<grid_for(n, 256, kSMs * 4), 256, 0, s>>>(n, ccount, maxt, pairs, ngiant, gpairs);
  count_launch();
  VC_CHECK_LAUNCH();
}

__global__ void block_class_list_k(int64_t c, const long long* __restrict__ cbase, int32_t* __restrict__ list,
                                   int* __restrict__ count) {
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < c; x += (int64_t)gridDim.x * blockDim.x) {
    const long long T = cbase[x + 1] - cbase[x];
    if (T > kMergeMax && T <= kMergeBlockMax) list[atomicAdd(count, 1)] = (int32_t)x;
  }
}

// The clusters of lo + 1 to hi pairs.
__global__ void warp_class_list_k(int64_t c, const long long* __restrict__ cbase, int lo, int hi,
                                  int32_t* __restrict__ list, int* __restrict__ count) {
  const int lane = threadIdx.x & 31;
  for (int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~31LL; b < c;
       b += (int64_t)gridDim.x * blockDim.x) {
    const int64_t x = b + lane;
    const long long T = x < c ? cbase[x + 1] - cbase[x] : 0;
    const bool in = T > lo && T <= hi;
    const unsigned bal = __ballot_sync(0xffffffffu, in);
    int at = 0;
    if (lane == 0 && bal) at = atomicAdd(count, __popc(bal));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (in) list[at + __popc(bal & ((1u << lane) - 1u))] = (int32_t)x;
  }
}

void cluster_merge(const GraphView& g, const int32_t* cid, const ContractScratch& cs, int32_t* ccount, int64_t c,
                   long long* cbase, long long* cursor, int32_t* seg_key, long long* seg_val, int64_t* coff,
                   int32_t* cadj, long long* cw, int32_t* csrc, long long* nnz_dev, int maxt, bool sort_first,
                   const GiantScratch* giant, int32_t* blist, int* blist_n, const MergeLists& lists, cudaStream_t s,
                   const SparseCtx* sp,
                   const LongLists& longs) {
  exclusive_scan<int, long long>(ccount, cbase, c, cbase + c, cs.scan_scr, s, cursor);
  const int gv = grid_for(g.n, 256, kSMs * 8), gc = grid_for(c, kMergeWarps, kSMs * 32);
  const PairOut in{cs.tmp_key, cs.tmp_val, cs.cmp_key, cs.cmp_val};
  cluster_scatter_k<<<gv, 256, 0, s>>>(g.n, g.off, cid, cs.cnt, in, cursor, seg_key, seg_val, longs);
  if (longs.item) {
    cluster_scatter_long_k<<<kSMs * 4, 256, 0, s>>>(g.off, cs.cnt, in, seg_key, seg_val, longs);
    count_launch();
  }
  const int gl = grid_for(c, 256, kSMs * 8);
  if (sp) {
    warp_class_list_k<<<gl, 256, 0, s>>>(c, cbase, 0, kMergeSmall, lists.small, lists.n);
    count_launch();
  }
  cluster_merge_k<kMergeSmall / 32><<<gc, kMergeWarps * 32, 0, s>>>(
      c, cbase, seg_key, seg_val, ccount, sort_first, sp ? lists.small : nullptr, sp ? lists.n : nullptr);
  count_launch(2);
  if (maxt > kMergeSmall) {
    warp_class_list_k<<<gl, 256, 0, s>>>(c, cbase, kMergeSmall, kMergeMax, lists.large, lists.n + 1);
    cluster_merge_k<kMergeMax / 32><<<gc, kMergeWarps * 32, 0, s>>>(c, cbase, seg_key, seg_val, ccount, sort_first,
                                                                   lists.large, lists.n + 1);
    count_launch(2);
  }
  VC_CHECK_LAUNCH();
  if (maxt > kMergeMax) {
    // the clusters of kMergeMax < T <= kMergeBlockMax pairs listed first, so that the
    // blocks visit only them (blist: n ints no longer needed once the scatter ran; its count,
    // like the other lists' here, starts from zero)
    block_class_list_k<<<grid_for(c, 256, kSMs * 8), 256, 0, s>>>(c, cbase, blist, blist_n);
    set_smem(cluster_merge_block_k, kMergeBlockSmem);
    cluster_merge_block_k<<<kSMs * 3, 256, kMergeBlockSmem, s>>>(cbase, seg_key, seg_val, ccount, blist, blist_n);
    count_launch(2);
    VC_CHECK_LAUNCH();
  }
  if (giant && giant->ngiant > 0) giant_merge(*giant, c, cbase, seg_key, seg_val, ccount, cs.scan_scr, s);
  if (sp) sparse_finish_degrees(g, cid, sp->sdeg, ccount, sp->clean, c, s);
  exclusive_scan<int, long long>(ccount, (long long*)coff, c, (long long*)coff + c, cs.scan_scr, s, nullptr, nnz_dev);
  LongLists place = longs;
  if (longs.n) place.n = longs.n + 1;  // a count of its own, the items no longer needed
  cluster_place_k<<<grid_for(c, 256, kSMs * 8), 256, 0, s>>>(c, cbase, coff, seg_key, seg_val, cadj, cw, csrc,
                                                               sp ? sp->clean : nullptr, place);
  if (longs.item) {
    cluster_place_long_k<<<kSMs * 4, 256, 0, s>>>(cbase, coff, seg_key, seg_val, cadj, cw, csrc, place);
    count_launch();
  }
  count_launch();
  VC_CHECK_LAUNCH();
  if (sp) sparse_copy(g, c, *sp, coff, cadj, cw, csrc, s);
}

}  // namespace vc
