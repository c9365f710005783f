// Padberg-Rinaldi reductions (Lemma "Padberg-Rinaldi", Sec. 4.1) with lock-free
// union-find.  Pass A tests conditions 1 and 2, pass B conditions 3 and 4, as the
// two passes of one "run" (Sec. 4.1, "Exact Reductions by Padberg and Rinaldi").
// Condition 2 marks only the edge to the designated partner p(v) = argmax over
// neighbours of (c(v,u), -u), and conditions 3/4 are checked on mutual partner
// pairs; the union of the marked edges is contracted in one step.
#include <limits.h>

#include "kernels.cuh"

namespace vc {

// Union-find whose representative is the smallest id of the component: a root is
// only ever linked below a smaller root (CAS on a root's own entry), so the final
// root of a component is its minimum.  Path halving writes only ancestors.
__device__ __forceinline__ int uf_find(volatile int32_t* p, int x) {
  for (;;) {
    int px = p[x];
    if (px == x) return x;
    int ppx = p[px];
    if (ppx != px) p[x] = ppx;
    x = px;
  }
}

__device__ __forceinline__ void uf_unite(int32_t* p, int a, int b) {
  for (;;) {
    a = uf_find(p, a);
    b = uf_find(p, b);
    if (a == b) return;
    if (a < b) { int t = a; a = b; b = t; }
    if (atomicCAS(&p[a], a, b) == a) return;
  }
}

// A warp per vertex (kPartnerG lanes; 16, two vertices per warp, measured slower on
// the long lists of deep Padberg-Rinaldi levels); lists of more than kPartnerBlockMin
// entries (hubs that absorbed many vertices) take a block each in partners_long_k.
constexpr int kPartnerG = 32;
constexpr int64_t kPartnerBlockMin = 8192;

// Degree and designated partner of one list, folded into (s, bw, bu) (bu INT_MAX: none).
__device__ __forceinline__ void partner_fold(long long& s, long long& bw, int& bu, long long x, int u) {
  s += x;
  if (x > bw || (x == bw && u < bu)) { bw = x; bu = u; }
}

// With a list (list_n not null) only the listed vertices list[0, *list_n).
template <typename WT>
__global__ void partners_k(int64_t n, const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
                           const WT* __restrict__ w, int32_t* __restrict__ partner, long long* __restrict__ pw,
                           long long* __restrict__ deg, const int32_t* __restrict__ list,
                           const int* __restrict__ list_n) {
  constexpr int G = kPartnerG;
  const int lane = threadIdx.x & 31, glane = lane & (G - 1);
  const unsigned gmask = G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u) << (lane & ~(G - 1));
  const int64_t groups = (int64_t)gridDim.x * (blockDim.x / G);
  if (list_n) n = *list_n;
  for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G; i < n; i += groups) {
    const int64_t v = list_n ? (int64_t)list[i] : i;
    const int64_t beg = off[v], end = off[v + 1];
    if (end - beg > kPartnerBlockMin) continue;  // partners_long_k
    long long s = 0, bw = -1;
    int bu = INT_MAX;
    for (int64_t e = beg + glane; e < end; e += G) partner_fold(s, bw, bu, (long long)w[e], adj[e]);
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
      const long long os = __shfl_xor_sync(gmask, s, o);
      const long long ow = __shfl_xor_sync(gmask, bw, o);
      const int ou = __shfl_xor_sync(gmask, bu, o);
      s += os;
      if (ow > bw || (ow == bw && ou < bu)) { bw = ow; bu = ou; }
    }
    if (glane == 0) {
      deg[v] = s;
      partner[v] = bw < 0 ? -1 : bu;
      pw[v] = bw;
    }
  }
}

// The lists of more than kPartnerBlockMin entries: each block lists the long ones among
// 256 consecutive vertices (those flagged kListNew, where flags are given), then folds
// each of them with all its threads.
template <typename WT>
__global__ void __launch_bounds__(256) partners_long_k(int64_t n, const int64_t* __restrict__ off,
                                                       const int32_t* __restrict__ adj, const WT* __restrict__ w,
                                                       int32_t* __restrict__ partner, long long* __restrict__ pw,
                                                       long long* __restrict__ deg,
                                                       const unsigned char* __restrict__ flag) {
  __shared__ int32_t s_list[256];
  __shared__ int s_n;
  __shared__ long long s_s[8], s_bw[8];
  __shared__ int s_bu[8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int64_t base = (int64_t)blockIdx.x * 256; base < n; base += (int64_t)gridDim.x * 256) {
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const int64_t v0 = base + threadIdx.x;
    if (v0 < n && (!flag || (flag[v0] & kListNew)) && off[v0 + 1] - off[v0] > kPartnerBlockMin)
      s_list[atomicAdd(&s_n, 1)] = (int32_t)v0;
    __syncthreads();
    const int cnt = s_n;
    for (int i = 0; i < cnt; ++i) {
      const int32_t v = s_list[i];
      long long s = 0, bw = -1;
      int bu = INT_MAX;
      const int64_t end = off[v + 1];
      for (int64_t e0 = off[v] + threadIdx.x; e0 < end; e0 += 8 * 256) {  // eight entries in flight per thread
        long long x[8];
        int u[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int64_t e = e0 + 256 * q;
          x[q] = e < end ? (long long)w[e] : 0;
          u[q] = e < end ? adj[e] : -1;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (u[q] >= 0) partner_fold(s, bw, bu, x[q], u[q]);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const long long os = __shfl_xor_sync(0xffffffffu, s, o);
        const long long ow = __shfl_xor_sync(0xffffffffu, bw, o);
        const int ou = __shfl_xor_sync(0xffffffffu, bu, o);
        s += os;
        if (ow > bw || (ow == bw && ou < bu)) { bw = ow; bu = ou; }
      }
      if (lane == 0) { s_s[wid] = s; s_bw[wid] = bw; s_bu[wid] = bu; }
      __syncthreads();
      if (threadIdx.x == 0) {
        for (int k = 1; k < 8; ++k) {
          s += s_s[k];
          if (s_bw[k] > bw || (s_bw[k] == bw && s_bu[k] < bu)) { bw = s_bw[k]; bu = s_bu[k]; }
        }
        deg[v] = s;
        partner[v] = bw < 0 ? -1 : bu;
        pw[v] = bw;
      }
      __syncthreads();
    }
  }
}

void pr_partners(const GraphView& g, int32_t* partner, long long* pw, long long* deg, cudaStream_t s,
                 const int32_t* list, const int* list_n, const unsigned char* flag) {
  const int grid = grid_for(g.n, 256 / kPartnerG, kSMs * 16), gl = grid_for(g.n, 256, kSMs * 4);
  if (g.wbytes == 4) {
    partners_k<int32_t><<<grid, 256, 0, s>>>(g.n, g.off, g.adj, (const int32_t*)g.w, partner, pw, deg, list, list_n);
    partners_long_k<int32_t><<<gl, 256, 0, s>>>(g.n, g.off, g.adj, (const int32_t*)g.w, partner, pw, deg, flag);
  } else {
    partners_k<long long><<<grid, 256, 0, s>>>(g.n, g.off, g.adj, (const long long*)g.w, partner, pw, deg, list,
                                               list_n);
    partners_long_k<long long><<<gl, 256, 0, s>>>(g.n, g.off, g.adj, (const long long*)g.w, partner, pw, deg, flag);
  }
  count_launch(2);
  VC_CHECK_LAUNCH();
}

// ------------------------------------------------------------ unchanged lists
// A contraction that merges few vertices leaves most lists as they were but for the
// renumbering.  What such a list gave keeps: its vertex's degree, partner and partner weight;
// and an edge (a pair) both of whose lists are unchanged since a pass tested it with the same
// bound still fails that test, as the pass merged whatever passed.  flag[v] says what v's
// list is new for: kListNew (degree and partner, just now), kListA, kListB (a test of pass A,
// of pass B).

// From the old graph's vertices whose lists the sparse contraction copied unchanged (dirty
// 2): degree, partner and flags under the new ids (flag1 starts with every bit set).
__global__ void carry_k(int64_t n, const int32_t* __restrict__ cid, const int32_t* __restrict__ sdeg,
                        const unsigned char* __restrict__ dirty, const long long* __restrict__ deg0,
                        const int32_t* __restrict__ partner0, const long long* __restrict__ pw0,
                        const unsigned char* __restrict__ flag0, long long* __restrict__ deg1,
                        int32_t* __restrict__ partner1, long long* __restrict__ pw1,
                        unsigned char* __restrict__ flag1) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    if (sdeg[v] < 0 || dirty[v] != 2) continue;
    const int32_t x = cid[v], p = partner0[v];
    deg1[x] = deg0[v];
    partner1[x] = p < 0 ? -1 : cid[p];  // a neighbour, so alone in its cluster too
    pw1[x] = pw0[v];
    flag1[x] = flag0[v] & (kListA | kListB);
  }
}

// The vertices flagged with bit, listed (in no particular order), and the numbers of
// vertices flagged kListA and kListB.
__global__ void flag_list_k(int64_t n, const unsigned char* __restrict__ flag, int bit, int32_t* __restrict__ list,
                            int* __restrict__ count, int* __restrict__ nab) {
  const int lane = threadIdx.x & 31;
  int na = 0, nb = 0;
  for (int64_t b = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~31LL; b < n;
       b += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = b + lane;
    const int f = v < n ? flag[v] : 0;
    na += (f & kListA) != 0;
    nb += (f & kListB) != 0;
    const unsigned bal = __ballot_sync(0xffffffffu, (f & bit) != 0);
    int at = 0;
    if (lane == 0 && bal) at = atomicAdd(count, __popc(bal));
    at = __shfl_sync(0xffffffffu, at, 0);
    if (f & bit) list[at + __popc(bal & ((1u << lane) - 1u))] = (int32_t)v;
  }
  if (nab) {
    na = (int)__reduce_add_sync(0xffffffffu, (unsigned)na);
    nb = (int)__reduce_add_sync(0xffffffffu, (unsigned)nb);
    if (lane == 0 && na) atomicAdd(nab, na);
    if (lane == 0 && nb) atomicAdd(nab + 1, nb);
  }
}

__global__ void flag_clear_k(int64_t n, unsigned char* __restrict__ flag, int bit) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    flag[v] = (unsigned char)(flag[v] & ~bit);
}

void flag_clear(int64_t n, unsigned char* flag, int bit, cudaStream_t s) {
  flag_clear_k<<<grid_for(n, 256, kSMs * 8), 256, 0, s>>>(n, flag, bit);
  count_launch();
  VC_CHECK_LAUNCH();
}

void flag_list(int64_t n, const unsigned char* flag, int bit, int32_t* list, int* count, int* nab, cudaStream_t s) {
  VC_CUDA(cudaMemsetAsync(count, 0, sizeof(int), s));
  if (nab) VC_CUDA(cudaMemsetAsync(nab, 0, 2 * sizeof(int), s));
  flag_list_k<<<grid_for(n, 256, kSMs * 8), 256, 0, s>>>(n, flag, bit, list, count, nab);
  count_launch();
  VC_CHECK_LAUNCH();
}

void pr_carry(int64_t n, const int32_t* cid, const int32_t* sdeg, const unsigned char* dirty, const PrLists& from,
              const PrLists& to, int64_t c, cudaStream_t s) {
  VC_CUDA(cudaMemsetAsync(to.flag, kListNew | kListA | kListB, (size_t)c, s));
  carry_k<<<grid_for(n, 256, kSMs * 8), 256, 0, s>>>(n, cid, sdeg, dirty, from.deg, from.partner, from.pw, from.flag,
                                                     to.deg, to.partner, to.pw, to.flag);
  count_launch();
  VC_CHECK_LAUNCH();
}

__global__ void uf_init_k(int32_t* __restrict__ p, int64_t n) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    p[v] = (int32_t)v;
}

// Bound and activity of the graph vertex v belongs to (single graph: the run's bound).
__device__ __forceinline__ bool pr_graph(const BatchCtx& bc, const DevState* st, int64_t v, long long* lam) {
  if (!bc.gid) {
    *lam = st->lambda_hat;
    return true;
  }
  const int g = bc.gid[v];
  if (!bc.gact[g]) return false;
  *lam = bc.glam[g];
  return true;
}

// Condition 1 on every edge (once per undirected edge: u > v) and condition 2 on the
// designated-partner edge; both ends must have at least two distinct neighbours.
// Union-find finds are chains of dependent loads, so short lists take a thread each
// (all of them in flight at once) and only lists longer than kPrThreadMax a warp.
constexpr int kPrThreadMax = 64;

template <typename WT>
__global__ void pr_a_mark_thread_k(int64_t n, const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
                                   const WT* __restrict__ w, const int32_t* __restrict__ partner,
                                   const long long* __restrict__ pw, const long long* __restrict__ deg,
                                   const DevState* st, int32_t* parent, BatchCtx bc) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    long long lam;
    if (!pr_graph(bc, st, v, &lam)) continue;
    const int64_t beg = off[v], end = off[v + 1];
    if (end - beg < 2 || end - beg > kPrThreadMax) continue;
    for (int64_t e = beg; e < end; ++e) {
      const int u = adj[e];
      if (u > v && (long long)w[e] >= lam && off[u + 1] - off[u] >= 2) uf_unite(parent, (int)v, u);
    }
    const int p = partner[v];
    if (p >= 0 && off[p + 1] - off[p] >= 2 && deg[v] <= 2 * pw[v]) uf_unite(parent, (int)v, p);
  }
}

// Contracted graphs carry each entry's source, so every entry takes a thread.
// The entry count is the graph's last offset, read on the device (a host-side count
// may be an upper bound).
template <typename WT>
__global__ void pr_a_edge_k(int64_t n, const int32_t* __restrict__ src, const int64_t* __restrict__ off,
                            const int32_t* __restrict__ adj, const WT* __restrict__ w, const DevState* st,
                            int32_t* parent, BatchCtx bc) {
  const int64_t nnz = off[n];
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz; e += (int64_t)gridDim.x * blockDim.x) {
    const int v = src[e], u = adj[e];
    if (u <= v) continue;
    long long lam;
    if (!pr_graph(bc, st, v, &lam)) continue;
    if ((long long)w[e] < lam) continue;
    if (off[v + 1] - off[v] < 2 || off[u + 1] - off[u] < 2) continue;
    uf_unite(parent, v, u);
  }
}

// Union-find start for pass A on sorted lists: each vertex points at its smallest
// marked neighbour below it (or at itself).  Every such pointer is a union of a
// marked edge towards a smaller id, so this is a valid forest with min-id roots,
// shallow from the start; the per-entry pass then finds short paths.  A start is only a
// start: eight lanes per vertex look at the first 32 entries of its list, in four rows of
// eight, and a vertex without a marked neighbour among them stays its own.  Each further 32
// entries cost three dependent loads and the per-entry pass is no slower without them
// (planted 8 x 2^20, 12 passes: 9.7 ms with 1024 entries, 7.4 with 128, 3.8 with 32, the
// per-entry pass 11.0 to 11.5 ms each time; 2326 vertices of 1345 entries: 100, 16, 7 us).
constexpr int kInitMinG = 8;
constexpr int kInitMinRows = 4;
template <typename WT>
__global__ void uf_init_min_k(int64_t n, const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
                              const WT* __restrict__ w, const DevState* st, int32_t* __restrict__ parent,
                              BatchCtx bc) {
  constexpr int G = kInitMinG;
  const int lane = threadIdx.x & 31, glane = lane & (G - 1);
  const unsigned gmask = G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u) << (lane & ~(G - 1));
  const int64_t groups = (int64_t)gridDim.x * (blockDim.x / G);
  for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G; v < n; v += groups) {
    int32_t p = (int32_t)v;
    long long lam;
    const int64_t beg = off[v], end = off[v + 1];
    if (end - beg >= 2 && pr_graph(bc, st, v, &lam)) {
      // the rows in flight: ids, then the weights of the entries below v, then the list
      // lengths of the heavy ones
      int u[kInitMinRows];
      bool mk[kInitMinRows];
#pragma unroll
      for (int r = 0; r < kInitMinRows; ++r) {
        const int64_t e = beg + r * G + glane;
        u[r] = e < end ? adj[e] : INT_MAX;
      }
#pragma unroll
      for (int r = 0; r < kInitMinRows; ++r) mk[r] = u[r] < v && (long long)w[beg + r * G + glane] >= lam;
#pragma unroll
      for (int r = 0; r < kInitMinRows; ++r) mk[r] = mk[r] && off[u[r] + 1] - off[u[r]] >= 2;
#pragma unroll
      for (int r = 0; r < kInitMinRows; ++r) {
        const unsigned mb = __ballot_sync(gmask, mk[r]);
        if (mb) {  // sorted: the lowest marked lane holds the smallest marked neighbour
          p = __shfl_sync(gmask, u[r], __ffs(mb) - 1);
          break;
        }
      }
    }
    if (glane == 0) parent[v] = p;
  }
}

// Between the two: every vertex points at the root of its start, so that the per-entry pass
// walks one or two links.  Starts chain (on a graph whose ids follow its geometry over
// hundreds of links), and a walk per vertex shortens them once for all entries: RHG n = 2^22,
// two passes over the coarse graphs, 100 us -> 13 us here and 16 us in pr_a_edge_k.  From
// kShortenMin vertices on: chains of fewer cost less than the launch (a run with four passes
// on at most 2326 vertices: 2928 us without it, 2948 us with).  Whole runs without it and with
// it: RHG n = 2^17 (degree 64) 0.67 and 0.67 ms, 2^20 (64) 1.26 and 1.22, 2^21 (32) 1.79 and 1.73.
constexpr int64_t kShortenMin = 4096;
__global__ void uf_shorten_k(int32_t* parent, int64_t n) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
    parent[v] = uf_find(parent, (int)v);
}

__global__ void pr_a_partner_k(int64_t n, const int64_t* __restrict__ off, const int32_t* __restrict__ partner,
                               const long long* __restrict__ pw, const long long* __restrict__ deg,
                               const DevState* st, int32_t* parent, BatchCtx bc) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    long long lam;
    if (!pr_graph(bc, st, v, &lam)) continue;
    if (off[v + 1] - off[v] < 2) continue;
    const int p = partner[v];
    if (p >= 0 && off[p + 1] - off[p] >= 2 && deg[v] <= 2 * pw[v]) uf_unite(parent, (int)v, p);
  }
}

// Condition 1 on the entries of the listed vertices (a warp each), in both directions: an
// edge with a listed end is seen from there.
template <typename WT>
__global__ void pr_a_list_k(const int32_t* __restrict__ list, const int* __restrict__ list_n,
                            const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
                            const WT* __restrict__ w, const DevState* st, int32_t* parent) {
  const int lane = threadIdx.x & 31, n = *list_n;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  const long long lam = st->lambda_hat;
  for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += warps) {
    const int32_t v = list[i];
    const int64_t beg = off[v], end = off[v + 1];
    if (end - beg < 2) continue;
    for (int64_t e = beg + lane; e < end; e += 32) {
      if ((long long)w[e] < lam) continue;
      const int32_t u = adj[e];
      if (off[u + 1] - off[u] >= 2) uf_unite(parent, v, u);
    }
  }
}

template <typename WT>
__global__ void pr_a_mark_k(int64_t n, const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
                            const WT* __restrict__ w, const int32_t* __restrict__ partner,
                            const long long* __restrict__ pw, const long long* __restrict__ deg,
                            const DevState* st, int32_t* parent, BatchCtx bc) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += warps) {
    long long lam;
    if (!pr_graph(bc, st, v, &lam)) continue;
    const int64_t beg = off[v], end = off[v + 1];
    if (end - beg <= kPrThreadMax) continue;
    for (int64_t e = beg + lane; e < end; e += 32) {
      int u = adj[e];
      if (u > v && (long long)w[e] >= lam && off[u + 1] - off[u] >= 2) uf_unite(parent, (int)v, u);
    }
    if (lane == 0) {
      int p = partner[v];
      if (p >= 0 && off[p + 1] - off[p] >= 2 && deg[v] <= 2 * pw[v]) uf_unite(parent, (int)v, p);
    }
  }
}

__global__ void uf_flatten_k(int32_t* parent, int64_t n, int32_t* __restrict__ labels, int* changed, BatchCtx bc) {
  int any = 0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
    if (bc.gid && !bc.gact[bc.gid[v]]) continue;
    int r = uf_find(parent, (int)v);
    labels[v] = r;
    if (r != v) {
      any = 1;
      if (bc.gid) bc.gchanged[bc.gid[v]] = 1;
    }
  }
  if (__syncthreads_or(any) && threadIdx.x == 0 && changed) atomicOr(changed, 1);
}

void pr_pass_a(const GraphView& g, const int32_t* partner, const long long* pw, const long long* deg,
               const DevState* st, int32_t* parent, int32_t* labels, int* changed, cudaStream_t s,
               const BatchCtx* bcp) {
  BatchCtx bc = bcp ? *bcp : BatchCtx{};
  int grid1 = grid_for(g.n, 256, kSMs * 8);
  if (!g.src) uf_init_k<<<grid1, 256, 0, s>>>(parent, g.n);
  int grid = grid_for(g.n, 8, kSMs * 16);
  if (g.src) {  // contracted graph: sorted lists and entry sources
    const int ge = grid_for(g.nnz, 256, kSMs * 16);
    const int gi = grid_for(g.n, 256 / kInitMinG, kSMs * 16);
    if (g.wbytes == 4)
      uf_init_min_k<int32_t><<<gi, 256, 0, s>>>(g.n, g.off, g.adj, (const int32_t*)g.w, st, parent, bc);
    else
      uf_init_min_k<long long><<<gi, 256, 0, s>>>(g.n, g.off, g.adj, (const long long*)g.w, st, parent, bc);
    if (g.n >= kShortenMin) {
      uf_shorten_k<<<grid1, 256, 0, s>>>(parent, g.n);
      count_launch();
    }
    if (g.wbytes == 4)
      pr_a_edge_k<int32_t><<<ge, 256, 0, s>>>(g.n, g.src, g.off, g.adj, (const int32_t*)g.w, st, parent, bc);
    else
      pr_a_edge_k<long long><<<ge, 256, 0, s>>>(g.n, g.src, g.off, g.adj, (const long long*)g.w, st, parent, bc);
    pr_a_partner_k<<<grid1, 256, 0, s>>>(g.n, g.off, partner, pw, deg, st, parent, bc);
  } else if (g.wbytes == 4) {
    pr_a_mark_thread_k<int32_t><<<grid1, 256, 0, s>>>(g.n, g.off, g.adj, (const int32_t*)g.w, partner, pw, deg, st,
                                                      parent, bc);
    pr_a_mark_k<int32_t><<<grid, 256, 0, s>>>(g.n, g.off, g.adj, (const int32_t*)g.w, partner, pw, deg, st, parent, bc);
  } else {
    pr_a_mark_thread_k<long long><<<grid1, 256, 0, s>>>(g.n, g.off, g.adj, (const long long*)g.w, partner, pw, deg,
                                                        st, parent, bc);
    pr_a_mark_k<long long><<<grid, 256, 0, s>>>(g.n, g.off, g.adj, (const long long*)g.w, partner, pw, deg, st,
                                                parent, bc);
  }
  uf_flatten_k<<<grid1, 256, 0, s>>>(parent, g.n, labels, changed, bc);
  count_launch(4);
  VC_CHECK_LAUNCH();
}

void pr_pass_a_lists(const GraphView& g, const int32_t* partner, const long long* pw, const long long* deg,
                     const DevState* st, const int32_t* list, const int* list_n, int32_t* parent, int32_t* labels,
                     int* changed, cudaStream_t s) {
  const BatchCtx bc{};
  const int grid1 = grid_for(g.n, 256, kSMs * 8), grid = grid_for(g.n, 8, kSMs * 16);
  uf_init_k<<<grid1, 256, 0, s>>>(parent, g.n);
  if (g.wbytes == 4)
    pr_a_list_k<int32_t><<<grid, 256, 0, s>>>(list, list_n, g.off, g.adj, (const int32_t*)g.w, st, parent);
  else
    pr_a_list_k<long long><<<grid, 256, 0, s>>>(list, list_n, g.off, g.adj, (const long long*)g.w, st, parent);
  pr_a_partner_k<<<grid1, 256, 0, s>>>(g.n, g.off, partner, pw, deg, st, parent, bc);
  uf_flatten_k<<<grid1, 256, 0, s>>>(parent, g.n, labels, changed, bc);
  count_launch(4);
  VC_CHECK_LAUNCH();
}

// Conditions 3 and 4 on mutual partner pairs v < w = p(v), p(w) = v, through the
// common neighbourhood: the warp walks the shorter of the two lists and finds each entry
// in the longer one by binary search (a longer list of at most kPrBStage ids is first
// copied into the warp's shared memory, so the searches there wait on no global loads).
// Walking the shorter list keeps a pair of a hub and a small vertex as cheap as the
// small vertex's list.  With flags, only pairs with an end flagged kListB are tested.
constexpr int kPrBStage = 1024;
template <typename WT>
__global__ void __launch_bounds__(256) pr_b_k(int64_t n, const int64_t* __restrict__ off,
                                              const int32_t* __restrict__ adj, const WT* __restrict__ w,
                                              const int32_t* __restrict__ partner, const long long* __restrict__ pw,
                                              const long long* __restrict__ deg, const DevState* st,
                                              int32_t* __restrict__ labels, int* changed, BatchCtx bc,
                                              const unsigned char* __restrict__ flag, PrLong longs) {
  __shared__ int32_t s_list[8][kPrBStage];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int32_t* sl = s_list[wid];
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += warps) {
    long long lam;
    if (!pr_graph(bc, st, v, &lam)) continue;
    const int p = partner[v];
    if (p <= v || partner[p] != v) continue;
    if (flag && !((flag[v] | flag[p]) & kListB)) continue;
    const int64_t vb = off[v], ve = off[v + 1], pb = off[p], pe = off[p + 1];
    if (ve - vb < 2 || pe - pb < 2) continue;
    const long long cvw = pw[v], dv = deg[v], dp = deg[p];
    // walk list s, search list l (s the shorter; ties: walk v's)
    const bool swap = pe - pb < ve - vb;
    if (longs.v && (swap ? pe - pb : ve - vb) > kPrLongMin) {  // pr_b_long_k
      if (lane == 0) longs.v[atomicAdd(longs.n, 1)] = (int32_t)v;
      continue;
    }
    const int64_t sb = swap ? pb : vb, se = swap ? pe : ve, lb = swap ? vb : pb, le = swap ? ve : pe;
    const bool staged = le - lb <= kPrBStage;
    if (staged)
      for (int64_t i = lane; i < le - lb; i += 32) sl[i] = adj[lb + i];
    __syncwarp();
    bool pr3 = false;
    long long sum = 0;
    for (int64_t e = sb + lane; e < se; e += 32) {
      const int u = adj[e];
      int64_t lo = lb, hi = le;
      if (staged) {
        int l = 0, h = (int)(le - lb);
        while (l < h) {
          const int mid = (l + h) >> 1;
          if (sl[mid] < u) l = mid + 1;
          else h = mid;
        }
        lo = lb + l;
      } else {
        while (lo < hi) {
          int64_t mid = (lo + hi) >> 1;
          if (adj[mid] < u) lo = mid + 1;
          else hi = mid;
        }
      }
      if (lo < le && (staged ? sl[lo - lb] : adj[lo]) == u) {
        const long long cs = (long long)w[e], cl = (long long)w[lo];
        const long long cvu = swap ? cl : cs, cwu = swap ? cs : cl;  // c(v, u), c(p, u)
        if (dv <= 2 * (cvw + cvu) && dp <= 2 * (cvw + cwu)) pr3 = true;
        sum += cvu < cwu ? cvu : cwu;
      }
    }
    pr3 = __any_sync(0xffffffffu, pr3);
    sum = warp_sum(sum);
    if (lane == 0 && (pr3 || cvw + sum >= lam)) {
      labels[p] = (int32_t)v;
      if (changed) atomicOr(changed, 1);
      if (bc.gid) bc.gchanged[bc.gid[v]] = 1;
    }
    __syncwarp();  // the staged list is overwritten by the warp's next pair
  }
}

// The pairs pr_b_k left out (the shorter list's entries over the threads of the blocks that
// share the pair, a binary search of the longer one each); then the decision.
template <typename WT>
__global__ void __launch_bounds__(256) pr_b_long_k(const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
                                                   const WT* __restrict__ w, const int32_t* __restrict__ partner,
                                                   const long long* __restrict__ pw,
                                                   const long long* __restrict__ deg, PrLong longs) {
  const int n = *longs.n, lane = threadIdx.x & 31;
  const GridShare G(n);
  for (int i = G.first; i < n; i += G.step) {
    const int32_t v = longs.v[i], p = partner[v];
    const int64_t vb = off[v], ve = off[v + 1], pb = off[p], pe = off[p + 1];
    const long long cvw = pw[v], dv = deg[v], dp = deg[p];
    const bool swap = pe - pb < ve - vb;
    const int64_t sb = swap ? pb : vb, se = swap ? pe : ve, lb = swap ? vb : pb, le = swap ? ve : pe;
    bool pr3 = false;
    long long sum = 0;
    for (int64_t e = sb + (int64_t)G.part * blockDim.x + threadIdx.x; e < se; e += (int64_t)G.parts * blockDim.x) {
      const int u = adj[e];
      int64_t lo = lb, hi = le;
      while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (adj[mid] < u) lo = mid + 1;
        else hi = mid;
      }
      if (lo < le && adj[lo] == u) {
        const long long cs = (long long)w[e], cl = (long long)w[lo];
        const long long cvu = swap ? cl : cs, cwu = swap ? cs : cl;  // c(v, u), c(p, u)
        if (dv <= 2 * (cvw + cvu) && dp <= 2 * (cvw + cwu)) pr3 = true;
        sum += cvu < cwu ? cvu : cwu;
      }
    }
    pr3 = __any_sync(0xffffffffu, pr3);
    sum = warp_sum(sum);
    if (lane == 0) {
      if (pr3) atomicOr(longs.pr3 + i, 1);
      if (sum) atomicAdd(longs.sum + i, (unsigned long long)sum);
    }
  }
}

__global__ void pr_b_long_done_k(const int32_t* __restrict__ partner, const long long* __restrict__ pw,
                                 const DevState* st, int32_t* __restrict__ labels, int* changed, PrLong longs) {
  const int n = *longs.n;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int32_t v = longs.v[i];
    if (longs.pr3[i] || pw[v] + (long long)longs.sum[i] >= st->lambda_hat) {
      labels[partner[v]] = v;
      if (changed) atomicOr(changed, 1);
    }
  }
}

void pr_pass_b(const GraphView& g, const int32_t* partner, const long long* pw, const long long* deg,
               const DevState* st, int32_t* labels, int* changed, cudaStream_t s, const BatchCtx* bcp,
               const unsigned char* flag, const PrLong& longs) {
  BatchCtx bc = bcp ? *bcp : BatchCtx{};
  if (longs.v) {
    const int64_t cap = pr_long_cap(g.nnz);
    VC_CUDA(cudaMemsetAsync(longs.n, 0, sizeof(int), s));
    VC_CUDA(cudaMemsetAsync(longs.sum, 0, sizeof(unsigned long long) * cap, s));
    VC_CUDA(cudaMemsetAsync(longs.pr3, 0, sizeof(int) * cap, s));
  }
  if (!bc.gid) iota(labels, g.n, s);
  int grid = grid_for(g.n, 8, kSMs * 16);
  if (g.wbytes == 4)
    pr_b_k<int32_t><<<grid, 256, 0, s>>>(g.n, g.off, g.adj, (const int32_t*)g.w, partner, pw, deg, st, labels,
                                         changed, bc, flag, longs);
  else
    pr_b_k<long long><<<grid, 256, 0, s>>>(g.n, g.off, g.adj, (const long long*)g.w, partner, pw, deg, st, labels,
                                           changed, bc, flag, longs);
  count_launch();
  if (longs.v) {
    if (g.wbytes == 4)
      pr_b_long_k<int32_t><<<kSMs * 4, 256, 0, s>>>(g.off, g.adj, (const int32_t*)g.w, partner, pw, deg, longs);
    else
      pr_b_long_k<long long><<<kSMs * 4, 256, 0, s>>>(g.off, g.adj, (const long long*)g.w, partner, pw, deg, longs);
    pr_b_long_done_k<<<1, 256, 0, s>>>(partner, pw, st, labels, changed, longs);
    count_launch(2);
  }
  VC_CHECK_LAUNCH();
}

}  // namespace vc
