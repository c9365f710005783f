// Final exact step: the minimum-cut algorithm of Nagamochi, Ono and Ibaraki (Sec. 3,
// "The Minimum Cut Algorithm of Nagamochi, Ono and Ibaraki"; used on the kernel in
// Sec. 4.1, "Final Step", and Algorithm 1).  A round is a maximum-adjacency scan
// from vertex 0 that always visits the unvisited vertex of largest attachment r
// (ties: smallest id); when x is visited every unvisited neighbour y gets
// r(y) += c(x,y) and q(x,y) = r(y) bounds the smallest x-y cut from below, so every
// edge with q >= lambda-hat (fixed for the round) is contracted.  Rounds repeat on
// the contracted graph until one vertex is left, the bound following the minimum
// degree after each contraction.
#include <limits.h>

#include <algorithm>
#include <mutex>
#include <string>
#include <type_traits>
#include <utility>

#include "kernels.cuh"
#include "viecut.h"

namespace vc {

constexpr int kNoiThreads = 512;
constexpr int kNoiWarpMax = 32;  // kernels up to this size scan with one warp

__device__ __forceinline__ int sfind(volatile int* p, int x) {
  for (;;) {
    int px = p[x];
    if (px == x) return x;
    int ppx = p[px];
    if (ppx != px) p[x] = ppx;
    x = px;
  }
}

__device__ __forceinline__ void sunite(int* p, int a, int b) {
  for (;;) {
    a = sfind(p, a);
    b = sfind(p, b);
    if (a == b) return;
    if (a < b) { int t = a; a = b; b = t; }
    if (atomicCAS(&p[a], a, b) == a) return;
  }
}

// argmax of (r, -k) over unseen k < nk, by one warp
__device__ __forceinline__ int warp_argmax_unseen(const long long* r, const int* seen, int nk) {
  const int lane = threadIdx.x & 31;
  long long br = -1;
  int bx = INT_MAX;
  for (int k = lane; k < nk; k += 32)
    if (!seen[k]) {
      long long rv = r[k];
      if (rv > br || (rv == br && k < bx)) { br = rv; bx = k; }
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    long long orv = __shfl_xor_sync(0xffffffffu, br, o);
    int ox = __shfl_xor_sync(0xffffffffu, bx, o);
    if (orv > br || (orv == br && ox < bx)) { br = orv; bx = ox; }
  }
  return bx;
}

// ------------------------------------------------------------ a round as closures
// Call a vertex "low" when it is visited with attachment r < max(lambda-hat, 1).  When a
// low vertex u is visited every unvisited r is at most r(u), so no unvisited vertex has
// reached lambda-hat; the vertices visited after u up to the next low vertex are then
// exactly the closure of u: the smallest set R holding u such that every vertex outside R
// and outside the earlier runs has fewer than lambda-hat of weight into the vertices
// visited so far.  Adding a vertex only raises the weights into the set, so the closure
// does not depend on the order in which its vertices are added, and neither do the
// attachments of the vertices left afterwards; the next low vertex (the largest r, ties
// to the smallest id) is therefore the same as in the maximum-adjacency order.  The round
// unites every x, y with r(y) >= lambda-hat once x's edge is added; each such pair lies
// within one run, and every vertex of a run is joined to the vertex whose edge raised it
// to lambda-hat (visited inside the run), so the round's components are the runs and the
// union-find with smallest-id roots labels each run with its smallest id.
//
// So a round needs the exact order only to pick each run's first vertex (an argmax over
// the vertices not yet taken); a run then grows level by level, the block relaxing all
// vertices of a level at once, a warp per list (a level of few vertices splits its lists
// over the warps).  The time is a chain of dependent steps -- a level waits for its lists
// (one L2 access), its shared-memory additions and one barrier -- so what counts is the
// cost of a step: the state of the graph sits in shared memory (attachments, queue, list
// offsets), and r holds the attachment less lam = max(lambda-hat, 1): a vertex is taken
// exactly when its r is not negative (an untaken one stays below lam; a run's first vertex
// is raised to 0 when it is chosen), so that one addition tests, raises and takes, and
// the untaken vertex of largest attachment holds the largest r read as unsigned.
//
// A vertex is taken at most once whatever the weights, so the queue (n places) never
// overflows: a negative weight, which only an input that nothing checked can hold, counts as
// 0, so that r never falls; and on graphs whose sums may leave 64 bits (GraphView::wraps) a
// taken vertex is not added to any more, so that r cannot come back below 0 around the end of
// its range either (-lam plus one weight stays inside it).
//
// Measured (RHG n = 8191, average degree 32, unit weights: 612 runs, 2174 levels): 1.66 ms a
// round, about 1400 cycles a level (450 of them the lists' L2 access) and 1100 a choice,
// against 4.47 ms for one warp over the same state.  8 and 4 warps take 1.70 and 2.05 ms;
// lists prefetched into L1 when a vertex is first touched, the same time.
//
// Vertices are local ids of the graph [lo, lo + n).
struct NoiShared {
  int cnt[3];     // vertices taken in a level, by level modulo 3
  int runmin[2];  // smallest id of a run, by run modulo 2
  unsigned long long red_v[32];
  int red_i[32];
};

// The state in shared memory.  R = int serves graphs in which lam x entries stays below
// 2^31: weights are cut to lam (which crosses it as the weight itself does), so no sum
// wraps.  kOff: the list offsets are kept too (they are read from goff otherwise).
template <typename RT, typename OT, bool kOff>
struct ClosureSmem {
  using R = RT;
  using O = OT;
  static constexpr bool kBounds = false;
  R* r;  // 16-byte aligned, a multiple of 4 entries (0, as taken, past n)
  OT* soff;
  uint16_t* queue;
  const int64_t* goff;  // the graph's offsets
  int64_t e0;           // its first entry
  __device__ __forceinline__ void init(int n, R lam) const {
    const int T = blockDim.x;
    for (int k = threadIdx.x; k < ((n + 3) & ~3); k += T) r[k] = k < n ? -lam : 0;
    if (kOff)
      for (int k = threadIdx.x; k <= n; k += T) soff[k] = (OT)(goff[k] - e0);
  }
  __device__ __forceinline__ OT beg(int x) const { return kOff ? soff[x] : (OT)(__ldg(goff + x) - e0); }
  __device__ __forceinline__ OT end(int x) const { return kOff ? soff[x + 1] : (OT)(__ldg(goff + x + 1) - e0); }
};

// The state in global memory (graphs beyond the shared-memory size), read past the L1
// cache, which the atomic operations do not update.  cmax[c] bounds the unsigned values
// of chunk c's 32 vertices that are untaken from above (0: all taken).
struct ClosureGlobal {
  using R = long long;
  using O = int64_t;
  static constexpr bool kBounds = true;
  R* r;
  unsigned long long* cmax;
  int32_t* queue;
  const int64_t* goff;
  int64_t e0;
  __device__ __forceinline__ void init(int n, R lam) const {
    const int T = blockDim.x;
    for (int k = threadIdx.x; k < n; k += T) __stcg(r + k, -lam);
    for (int k = threadIdx.x; k < ((n + 31) >> 5); k += T) __stcg(cmax + k, (unsigned long long)-lam);
  }
  __device__ __forceinline__ int64_t beg(int x) const { return __ldg(goff + x) - e0; }
  __device__ __forceinline__ int64_t end(int x) const { return __ldg(goff + x + 1) - e0; }
};

__device__ __forceinline__ unsigned warp_max_r(unsigned x) { return __reduce_max_sync(0xffffffffu, x); }
__device__ __forceinline__ unsigned long long warp_max_r(unsigned long long x) {
  const unsigned hi = (unsigned)(x >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? (unsigned)x : 0u);
  return ((unsigned long long)mh << 32) | ml;
}

// The largest v of the block and the smallest i holding it (i >= 0), in every thread.
// One barrier; red_v and red_i may be written again after the next one.
template <int NW, typename R>
__device__ __forceinline__ int block_argmax(R v, int i, R* top, NoiShared& sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const R wv = warp_max_r(v);
  const unsigned wi = __reduce_min_sync(0xffffffffu, v == wv ? (unsigned)i : 0xffffffffu);
  if (lane == 0) {
    sh.red_v[wid] = wv;
    sh.red_i[wid] = (int)wi;
  }
  __syncthreads();
  const R bv = lane < NW ? (R)((volatile unsigned long long*)sh.red_v)[lane] : (R)0;
  const unsigned bi = lane < NW ? (unsigned)((volatile int*)sh.red_i)[lane] : 0xffffffffu;
  *top = warp_max_r(bv);
  return (int)__reduce_min_sync(0xffffffffu, bv == *top ? bi : 0xffffffffu);
}

// lam x entries (and the offsets) below 2^31: 32-bit values do not wrap.
__device__ __forceinline__ bool noi_fits32(long long lam, int64_t entries) {
  return lam < INT_MAX && entries < INT_MAX && (lam > 1 ? lam : 1) * entries < INT_MAX;
}

// Additions of either width (the 64-bit one is declared unsigned); the value before.  WRAPS:
// a value that is no longer negative stays as it is (each failed exchange is another's
// addition, so the loop ends).
template <bool WRAPS>
__device__ __forceinline__ int noi_add(int* p, int x) { return atomicAdd(p, x); }
template <bool WRAPS>
__device__ __forceinline__ long long noi_add(long long* p, long long x) {
  unsigned long long* q = (unsigned long long*)p;
  if constexpr (!WRAPS) return (long long)atomicAdd(q, (unsigned long long)x);
  unsigned long long old = atomicAdd(q, 0ull);
  while ((long long)old < 0) {
    const unsigned long long seen = atomicCAS(q, old, old + (unsigned long long)x);
    if (seen == old) break;
    old = seen;
  }
  return (long long)old;
}

constexpr int kNoiUnroll = 4;  // rows of a list in flight per warp while relaxing

// One round by a block of NW warps (a power of two), one graph at a time.  put(x, m)
// receives every vertex x with the smallest id m of its run.  Returns, in every thread,
// whether some run holds two or more vertices.  Ends with a barrier.
template <int NW, bool WRAPS = false, typename WT, typename ST, typename PUT>
__device__ __forceinline__ bool noi_closure_block(int32_t lo, int n, const int32_t* __restrict__ adj,
                                                  const WT* __restrict__ w, long long lam_in, const ST& S,
                                                  NoiShared& sh, PUT put) {
  using R = typename ST::R;
  using U = typename std::make_unsigned<R>::type;
  using OT = typename ST::O;
  using QT = typename std::remove_pointer<decltype(ST::queue)>::type;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const unsigned below = (1u << lane) - 1u;
  const R lam = (R)(lam_in > 1 ? lam_in : 1);  // weights >= 1: a first addition crosses any bound below 1
  const int64_t e0 = S.e0;
  S.init(n, lam);
  if (tid < 3) sh.cnt[tid] = 0;
  if (tid < 2) sh.runmin[tid] = INT_MAX;
  __syncthreads();
  int qt = 0, lev = 0, run = 0;  // taken so far, levels so far modulo 3, runs so far modulo 2
  bool unites = false;
  while (qt < n) {
    // the run's first vertex: the untaken vertex of largest r, ties to the smallest id
    int u;
    if constexpr (!ST::kBounds) {
      // every thread reads its vertices, four at a time; the best four again at the end
      U bv = 0, top;
      int bk = tid * 4;
      auto four = [&](int k, U* x) {
#pragma unroll
        for (int q = 0; q < (int)sizeof(R) / 4; ++q) ((uint4*)x)[q] = ((const uint4*)(S.r + k))[q];
      };
      for (int k = tid * 4; k < n; k += NW * 128) {
        U x[4];
        four(k, x);
        const U m = max(max(x[0], x[1]), max(x[2], x[3]));
        if (m > bv) { bv = m; bk = k; }
      }
      if (bv) {  // the first of the four (bk is in range: a thread without vertices has bv = 0)
        U x[4];
        four(bk, x);
        bk += x[0] == bv ? 0 : x[1] == bv ? 1 : x[2] == bv ? 2 : 3;
      }
      u = block_argmax<NW>(bv, bk, &top, sh);
    } else {
      // the chunk of largest bound (ties: the lower chunk), read exactly; a stale bound (its
      // vertex was taken) is lowered and the choice made again
      for (;;) {
        U bv = 0, top;
        int bc = 0;
        for (int c = tid; c < ((n + 31) >> 5); c += NW * 32) {
          const U m = __ldcg(S.cmax + c);
          if (m > bv) { bv = m; bc = c; }
        }
        const int uc = block_argmax<NW>(bv, bc, &top, sh), k = uc * 32 + lane;
        const R x = k < n ? __ldcg(S.r + k) : 0;
        const U rv = x < 0 ? (U)x : 0;
        const U best = warp_max_r(rv);
        u = uc * 32 + __ffs(__ballot_sync(0xffffffffu, rv == best)) - 1;
        if (best == top) break;
        __syncthreads();  // every warp has read the bounds and its copy of the choice
        if (tid == 0) __stcg(S.cmax + uc, best);
        __syncthreads();
      }
    }
    // every warp has read the values: the barrier of the choice lies between
    if (ST::kBounds) __syncthreads();
    if (tid == 0) {
      S.r[u] = 0;
      S.queue[qt] = (QT)u;
      sh.runmin[run ^ 1] = INT_MAX;  // the last run's, read before this run's first barrier
    }
    const int rs = qt;
    int qh = qt++;
    while (qh < qt) {
      const int cnt = qt - qh;
      int* got = &sh.cnt[lev];
      lev = lev == 2 ? 0 : lev + 1;
      if (tid == 0) sh.cnt[lev] = 0;  // last read two barriers ago
      // a warp per list, or (fewer lists than warps) P warps per list on interleaved rows
      const int lg = cnt >= NW ? 31 - __clz(NW) : 32 - __clz(cnt - 1);
      const int P = NW >> lg, part = wid >> lg;
      for (int i = wid & ((1 << lg) - 1); i < cnt; i += NW) {
        const int x = qh == rs ? u : (int)S.queue[qh + i];
        const OT beg = S.beg(x), len = S.end(x) - beg;
        const int32_t* a = adj + e0 + beg;
        for (OT row = (OT)part * 32; row < len; row += P * kNoiUnroll * 32) {
          int y[kNoiUnroll];
          R c[kNoiUnroll];
#pragma unroll
          for (int q = 0; q < kNoiUnroll; ++q) {
            const OT e = row + q * P * 32 + lane;
            y[q] = -1;
            c[q] = 0;
            if (e < len) {
              y[q] = __ldg(a + e) - lo;
              const long long x64 = ldw(w, e0 + beg + e);
              c[q] = x64 < 0 ? 0 : (sizeof(R) == 4 && x64 > (long long)lam) ? lam : (R)x64;
            }
          }
#pragma unroll
          for (int q = 0; q < kNoiUnroll; ++q) {
            if (row + q * P * 32 >= len) break;  // the same in every lane
            bool join = false;
            if (y[q] >= 0) {
              const R old = noi_add<WRAPS>(&S.r[y[q]], c[q]), now = (R)((U)old + (U)c[q]);
              join = old < 0 && now >= 0;  // the addition that crosses lam takes the vertex
              if constexpr (ST::kBounds)
                if ((old & now) < 0) atomicMax(&S.cmax[y[q] >> 5], (U)now);
            }
            const unsigned b = __ballot_sync(0xffffffffu, join);
            if (b) {
              int at = 0;
              if (lane == 0) at = atomicAdd(got, __popc(b));
              if (join) atomicMin(&sh.runmin[run], y[q]);
              at = qt + __shfl_sync(0xffffffffu, at, 0) + __popc(b & below);
              if (join) S.queue[at] = (QT)y[q];
            }
          }
        }
      }
      __syncthreads();
      qh = qt;
      qt += *(volatile int*)got;
    }
    if (qt - rs == 1) {
      if (tid == 0) put(u, u);
    } else {
      const int m = min(u, *(volatile int*)&sh.runmin[run]);
      for (int i = rs + tid; i < qt; i += NW * 32) put((int)S.queue[i], m);
      unites = true;
    }
    run ^= 1;
  }
  __syncthreads();
  return unites;
}

// Where one graph's exact-step results go: its bound, best-side kind, shape and
// trace (fields of DevState for single runs, per-graph arrays for batches).
struct NoiIO {
  long long* lam;
  int* best_kind;
  long long* n_out;
  long long* nnz_out;
  long long* dmin;
  long long* argmin;
  int* trace_len;
  TraceStep* trace;
  int trace_cap;
  int level;
};

// All rounds on one graph of n <= kDenseMax vertices, by one block.  The first round runs
// on the lists (a closure level touches its vertices' entries, not whole matrix rows), and
// the matrix that the later rounds work on is built from the lists for the contracted
// graph alone, which is several times smaller; it sits in the block's dynamic shared
// memory (scap entries at dyn) when it fits there, else in M0 / M1.
// The graph's vertices are [base, base + n) of the CSR (off points at its first row).
template <typename WT>
__device__ __forceinline__ void noi_dense_body(int n, const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
                                               const WT* __restrict__ w, int32_t base, long long* dyn, int scap,
                                               long long* M0, long long* M1, int32_t* curK, unsigned char* sideK,
                                               const NoiIO& io) {
  __shared__ __align__(16) long long r[kDenseMax];
  __shared__ int seen[kDenseMax];
  __shared__ int parent[kDenseMax];
  __shared__ int root[kDenseMax];
  __shared__ int rr[kDenseMax];
  __shared__ int wsum[kNoiThreads / 32];
  __shared__ long long red_d[kNoiThreads / 32];
  __shared__ int red_v[kNoiThreads / 32];
  __shared__ long long red_c[kNoiThreads / 32];
  __shared__ int s_stop, s_improved, s_nk2, s_arg, s_qt;
  __shared__ int64_t s_off[kDenseMax + 1];
  __shared__ uint16_t s_queue[kDenseMax];
  __shared__ NoiShared s_noi;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  constexpr int T = kNoiThreads;
  int nk = n;
  long long* M = nullptr;   // the current matrix (null: the first round, on the lists)
  long long* Mn = nullptr;  // where the next one goes
  for (int k = tid; k < n; k += T) curK[k] = k;
  __syncthreads();
  while (nk > 1) {
    const long long lam = *io.lam;
    if (!M) {
      const int64_t e0 = off[0];
      auto put = [&](int x, int m) { root[x] = m; };
      if (noi_fits32(lam, off[n] - e0)) {
        const ClosureSmem<int, int64_t, true> S{(int*)r, s_off, s_queue, off, e0};
        noi_closure_block<kNoiThreads / 32>(base, nk, adj, w, lam, S, s_noi, put);
      } else {
        const ClosureSmem<long long, int64_t, true> S{r, s_off, s_queue, off, e0};
        noi_closure_block<kNoiThreads / 32>(base, nk, adj, w, lam, S, s_noi, put);
      }
    } else {
    for (int k = tid; k < nk; k += T) { r[k] = 0; seen[k] = 0; parent[k] = k; }
    __syncthreads();
    if (nk <= kNoiWarpMax) {
      // small kernels: warp 0 alone runs the scan (no block barrier per step)
      if (wid == 0) {
        for (int step = 0; step < nk; ++step) {
          const int x = warp_argmax_unseen(r, seen, nk);
          __syncwarp();
          if (lane == 0) seen[x] = 1;
          __syncwarp();
          const long long* row = M + (int64_t)x * nk;
          for (int y = lane; y < nk; y += 32) {
            if (!seen[y]) {
              const long long c = row[y];
              if (c != 0) {
                const long long ry = r[y] + c;
                r[y] = ry;
                if (ry >= lam) sunite(parent, x, y);
              }
            }
          }
          __syncwarp();
        }
      }
      __syncthreads();
    } else {
      // the round as closures (see noi_closure_block above): each run's first vertex is the
      // untaken vertex of largest r (ties: smallest id); the run then grows level by
      // level, every thread relaxing matrix entries of the level's vertices, and takes
      // its smallest id as the label of all its vertices (rr holds the taken vertices)
      int qt = 0, qh = 0;
      while (qt < nk) {
        if (wid == 0) {
          const int x = warp_argmax_unseen(r, seen, nk);
          if (lane == 0) {
            rr[qt] = x;
            seen[x] = 1;
            s_qt = qt + 1;
          }
        }
        __syncthreads();
        const int rs = qt;
        qt = s_qt;
        while (qh < qt) {
          const int F = qt - qh;
          for (int idx = tid; idx < F * nk; idx += T) {
            const int f = idx / nk, y = idx - f * nk;
            if (seen[y]) continue;
            const long long c = M[(int64_t)rr[qh + f] * nk + y];
            if (c == 0) continue;
            const long long ry = (long long)atomicAdd((unsigned long long*)&r[y], (unsigned long long)c) + c;
            if (ry >= lam && (ry - c < lam || ry - c <= 0) && atomicExch(&seen[y], 1) == 0)
              rr[atomicAdd(&s_qt, 1)] = y;
          }
          __syncthreads();
          qh = qt;
          qt = s_qt;
          __syncthreads();  // every thread has read s_qt before the next level adds to it
        }
        int m = INT_MAX;
        for (int i = rs + tid; i < qt; i += T) m = rr[i] < m ? rr[i] : m;
        m = (int)__reduce_min_sync(0xffffffffu, (unsigned)m);
        if (lane == 0) red_v[wid] = m;
        __syncthreads();
        if (tid == 0) {
          for (int q = 1; q < T / 32; ++q) m = red_v[q] < m ? red_v[q] : m;
          s_arg = m;
        }
        __syncthreads();
        m = s_arg;
        for (int i = rs + tid; i < qt; i += T) root[rr[i]] = m;
        __syncthreads();
      }
    }
    if (nk <= kNoiWarpMax) {
      for (int k = tid; k < nk; k += T) root[k] = sfind(parent, k);
      __syncthreads();
    }
    }
    // roots -> ranks (every root is the minimum of its component)
    {
      int flag = (tid < nk && root[tid] == tid) ? 1 : 0;  // nk <= T
      int inc = flag;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      if (lane == 31) wsum[wid] = inc;
      __syncthreads();
      if (tid == 0) {
        int acc = 0;
        for (int q = 0; q < T / 32; ++q) { int t = wsum[q]; wsum[q] = acc; acc += t; }
        s_nk2 = acc;
      }
      __syncthreads();
      if (tid < nk) rr[tid] = wsum[wid] + inc - flag;
      __syncthreads();
    }
    const int nk2 = s_nk2;
    if (nk2 == nk) break;  // no contraction (cannot happen while lambda-hat <= min degree)
    // the next matrix: beside the current one, or over the one before it (which was larger)
    long long* prev = M;
    if (!M) Mn = nk2 * nk2 <= scap ? dyn : M0;
    else if (!Mn) Mn = nk2 * nk2 + (M == dyn ? nk * nk : 0) <= scap ? dyn + (M == dyn ? nk * nk : 0) : M1;
    for (int i = tid; i < nk2 * nk2; i += T) Mn[i] = 0;
    for (int k = tid; k < nk; k += T) parent[k] = rr[root[k]];  // every vertex's new id
    __syncthreads();
    if (!M) {
      // a warp per list
      for (int v = wid; v < nk; v += T / 32) {
        const int a = parent[v];
        for (int64_t e = off[v] + lane; e < off[v + 1]; e += 32) {
          const int b = parent[adj[e] - base];
          if (a != b) atomicAdd((unsigned long long*)&Mn[a * nk2 + b], (unsigned long long)w[e]);
        }
      }
    } else {
      for (int i = tid; i < nk * nk; i += T) {
        const long long c = M[i];
        if (c != 0) {
          const int a = parent[i / nk], b = parent[i % nk];
          if (a != b) atomicAdd((unsigned long long*)&Mn[a * nk2 + b], (unsigned long long)c);
        }
      }
    }
    for (int k = tid; k < n; k += T) curK[k] = parent[curK[k]];
    __syncthreads();
    M = Mn;
    Mn = prev;
    nk = nk2;
    // degrees, minimum with smallest argmin, and entry count of the contracted graph
    long long bd = LLONG_MAX, cnt = 0;
    int bv = INT_MAX;
    for (int a = tid; a < nk; a += T) {
      long long d = 0;
      const long long* row = M + (int64_t)a * nk;
      for (int b = 0; b < nk; ++b) {
        long long c = row[b];
        d += c;
        cnt += c != 0;
      }
      if (d < bd || (d == bd && a < bv)) { bd = d; bv = a; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      long long od = __shfl_xor_sync(0xffffffffu, bd, o);
      int ov = __shfl_xor_sync(0xffffffffu, bv, o);
      cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
      if (od < bd || (od == bd && ov < bv)) { bd = od; bv = ov; }
    }
    if (lane == 0) { red_d[wid] = bd; red_v[wid] = bv; red_c[wid] = cnt; }
    __syncthreads();
    if (tid == 0) {
      long long tot = 0;
      for (int q = 0; q < T / 32; ++q) {
        tot += red_c[q];
        if (red_d[q] < bd || (red_d[q] == bd && red_v[q] < bv)) { bd = red_d[q]; bv = red_v[q]; }
      }
      s_stop = 0;
      s_improved = 0;
      *io.n_out = nk;
      *io.nnz_out = tot;
      if (nk > 1) {
        *io.dmin = bd;
        *io.argmin = bv;
        if (bd < *io.lam) {
          *io.lam = bd;
          *io.best_kind = 2;
          s_improved = 1;
          s_arg = bv;
        }
        if (*io.lam == 0) s_stop = 1;
      }
      int i = *io.trace_len;
      if (i < io.trace_cap) io.trace[i] = TraceStep{4, io.level, (long long)nk, tot, *io.lam};
      *io.trace_len = i + 1;
    }
    __syncthreads();
    if (s_improved) {
      const int b = s_arg;
      for (int k = tid; k < n; k += T) sideK[k] = curK[k] == b ? 1 : 0;
    }
    __syncthreads();
    if (s_stop) break;
  }
}

template <typename WT>
__global__ void __launch_bounds__(kNoiThreads) noi_dense_k(int n, const int64_t* __restrict__ off,
                                                           const int32_t* __restrict__ adj, const WT* __restrict__ w,
                                                           long long* M0, long long* M1, int32_t* curK,
                                                           unsigned char* sideK, DevState* st, TraceStep* trace,
                                                           int trace_cap, int level, int scap) {
  extern __shared__ __align__(16) long long noi_dyn[];
  NoiIO io{&st->lambda_hat, &st->best_kind, &st->n, &st->nnz, &st->dmin, &st->argmin, &st->trace_len,
           trace, trace_cap, level};
  noi_dense_body<WT>(n, off, adj, w, 0, noi_dyn, scap, M0, M1, curK, sideK, io);
}

// Matrix entries in dynamic shared memory: a contracted graph of at most 150 vertices
// (beside the body's own arrays, below the 227 KB of a block).
constexpr int kNoiDenseSmem = 150 * 150;

template <typename WT>
static void noi_dense_launch(const GraphView& g, long long* M0, long long* M1, int32_t* curK, unsigned char* sideK,
                             DevState* st, TraceStep* trace, int trace_cap, int level, cudaStream_t s) {
  const int n = (int)g.n;
  const int scap = std::min(n * n, kNoiDenseSmem);
  set_smem(noi_dense_k<WT>, sizeof(long long) * kNoiDenseSmem);
  noi_dense_k<WT><<<1, kNoiThreads, sizeof(long long) * scap, s>>>(n, g.off, g.adj, (const WT*)g.w, M0, M1, curK,
                                                                   sideK, st, trace, trace_cap, level, scap);
  count_launch();
  VC_CHECK_LAUNCH();
}

void noi_dense(const GraphView& g, long long* M0, long long* M1, int32_t* curK, unsigned char* sideK,
               DevState* st, TraceStep* trace, int trace_cap, int level, cudaStream_t s) {
  if (g.wbytes == 4) noi_dense_launch<int32_t>(g, M0, M1, curK, sideK, st, trace, trace_cap, level, s);
  else noi_dense_launch<long long>(g, M0, M1, curK, sideK, st, trace, trace_cap, level, s);
}

// Batches: a persistent grid pulls the listed graphs; each block solves one at a time
// with its own matrices (mcap entries each; those of at most 60 vertices in the 28 KB of
// shared memory that four blocks per SM would leave each).
constexpr int kNoiDenseBatchSmem = 60 * 60;
template <typename WT>
__global__ void __launch_bounds__(kNoiThreads) noi_dense_batch_k(const int32_t* __restrict__ list, int count,
                                                                 const int64_t* __restrict__ off,
                                                                 const int32_t* __restrict__ adj,
                                                                 const WT* __restrict__ w, const long long* vbase,
                                                                 const long long* nv, long long* M, int64_t mcap,
                                                                 int32_t* curK, unsigned char* sideK, BatchNoi bn,
                                                                 int scap) {
  extern __shared__ __align__(16) long long noi_dyn[];
  long long* M0 = M + (int64_t)blockIdx.x * 2 * mcap;
  long long* M1 = M0 + mcap;
  int32_t* ck = curK + (int64_t)blockIdx.x * kDenseMax;
  for (int idx = blockIdx.x; idx < count; idx += gridDim.x) {
    const int g = list[idx];
    const int32_t base = (int32_t)vbase[g];
    NoiIO io{bn.lam + g, bn.best_kind + g, bn.n_out + g, bn.nnz_out + g, bn.dmin + g, bn.argmin + g,
             bn.trace_len + g, bn.trace + (int64_t)g * bn.trace_cap, bn.trace_cap, bn.level[g]};
    noi_dense_body<WT>((int)nv[g], off + base, adj, w, base, noi_dyn, scap, M0, M1, ck,
                       sideK + (int64_t)g * kDenseMax, io);
    __syncthreads();
  }
}

void noi_dense_batch(const GraphView& u, const int32_t* list, int count, const long long* vbase, const long long* nv,
                     long long* M, int64_t mcap, int blocks, int32_t* curK, unsigned char* sideK, const BatchNoi& bn,
                     cudaStream_t s) {
  if (count <= 0) return;
  const size_t smem = sizeof(long long) * kNoiDenseBatchSmem;
  if (u.wbytes == 4)
    noi_dense_batch_k<int32_t><<<blocks, kNoiThreads, smem, s>>>(list, count, u.off, u.adj, (const int32_t*)u.w, vbase,
                                                                 nv, M, mcap, curK, sideK, bn, kNoiDenseBatchSmem);
  else
    noi_dense_batch_k<long long><<<blocks, kNoiThreads, smem, s>>>(list, count, u.off, u.adj, (const long long*)u.w,
                                                                   vbase, nv, M, mcap, curK, sideK, bn,
                                                                   kNoiDenseBatchSmem);
  count_launch();
  VC_CHECK_LAUNCH();
}

// ------------------------------------------------------------ sparse single round
constexpr int kSparseThreads = 1024;

// One round on the vertices [lo, hi) (ids are global: r, seen, parent, labels are
// indexed by them); returns through *any whether something merged.
template <typename WT>
__device__ __forceinline__ void noi_round_body(int64_t lo, int64_t hi, const int64_t* __restrict__ off,
                                               const int32_t* __restrict__ adj, const WT* __restrict__ w,
                                               long long lam, long long* r, unsigned char* seen, int32_t* parent,
                                               int32_t* labels, int* any_out) {
  __shared__ long long red_r[kSparseThreads / 32];
  __shared__ long long red_x[kSparseThreads / 32];
  __shared__ long long s_x;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (int64_t k = lo + tid; k < hi; k += kSparseThreads) { r[k] = 0; seen[k] = 0; parent[k] = (int32_t)k; }
  __syncthreads();
  for (int64_t step = lo; step < hi; ++step) {
    long long br = -1, bx = LLONG_MAX;
    for (int64_t k = lo + tid; k < hi; k += kSparseThreads)
      if (!seen[k]) {
        long long rv = r[k];
        if (rv > br || (rv == br && k < bx)) { br = rv; bx = k; }
      }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      long long orv = __shfl_xor_sync(0xffffffffu, br, o);
      long long ox = __shfl_xor_sync(0xffffffffu, bx, o);
      if (orv > br || (orv == br && ox < bx)) { br = orv; bx = ox; }
    }
    if (lane == 0) { red_r[wid] = br; red_x[wid] = bx; }
    __syncthreads();
    if (tid == 0) {
      for (int q = 1; q < kSparseThreads / 32; ++q)
        if (red_r[q] > br || (red_r[q] == br && red_x[q] < bx)) { br = red_r[q]; bx = red_x[q]; }
      s_x = bx;
      seen[bx] = 1;
    }
    __syncthreads();
    const int64_t x = s_x;
    for (int64_t e = off[x] + tid; e < off[x + 1]; e += kSparseThreads) {
      const int y = adj[e];
      if (seen[y]) continue;
      const long long c = (long long)w[e];
      const long long ry = (long long)atomicAdd((unsigned long long*)&r[y], (unsigned long long)c) + c;
      if (ry >= lam) sunite(parent, (int)x, y);
    }
    __syncthreads();
  }
  int any = 0;
  for (int64_t k = lo + tid; k < hi; k += kSparseThreads) {
    int rt = sfind(parent, (int)k);
    labels[k] = rt;
    any |= rt != k;
  }
  if (__syncthreads_or(any) && tid == 0) atomicOr(any_out, 1);
  __syncthreads();
}

// ---- the same round as closures, a block per graph
// Shared memory of a graph of at most ncap vertices: 32-bit values, list offsets and
// queue, or 64-bit values and queue.  16,384 vertices take 160 KB of a block's 227.
constexpr int kNoiSmemRoundMaxN = 16384;
__host__ __device__ constexpr size_t noi_round_smem(int ncap) { return (size_t)((ncap + 3) & ~3) * 10 + 16; }

// The listed graphs (list null: the one graph of n1 vertices with bound st->lambda_hat),
// a block at a time each.  Graphs of at most ncap vertices keep their state in shared
// memory; the others in r (values at the vertex), cmax (chunk bounds) and queue.
template <typename WT, int NW, bool WRAPS>
__global__ void __launch_bounds__(NW * 32) noi_round_k(
    const int32_t* __restrict__ list, int count, int64_t n1, const DevState* st, const long long* __restrict__ vbase,
    const long long* __restrict__ nv, const long long* __restrict__ glam, const int64_t* __restrict__ off,
    const int32_t* __restrict__ adj, const WT* __restrict__ w, long long* r, unsigned long long* cmax,
    int32_t* queue, int32_t* __restrict__ labels, int* changed, int ncap) {
  extern __shared__ __align__(16) unsigned char noi_rs[];
  __shared__ NoiShared sh;
  for (int idx = blockIdx.x; idx < count; idx += gridDim.x) {
    const int g = list ? list[idx] : 0;
    const int64_t lo = list ? vbase[g] : 0;
    const int n = (int)(list ? nv[g] : n1);
    const long long lam = list ? glam[g] : st->lambda_hat;
    const int64_t* goff = off + lo;
    const int64_t e0 = goff[0];
    auto put = [&](int x, int m) { labels[lo + x] = (int32_t)(lo + m); };
    bool any;
    if (n > ncap) {
      const ClosureGlobal S{r + lo, cmax + lo, queue + lo, goff, e0};
      any = noi_closure_block<NW, WRAPS>((int32_t)lo, n, adj, w, lam, S, sh, put);
    } else if (noi_fits32(lam, goff[n] - e0)) {
      ClosureSmem<int, int32_t, true> S;
      S.r = (int*)noi_rs;
      S.soff = (int32_t*)(S.r + ((n + 3) & ~3));
      S.queue = (uint16_t*)(S.soff + n + 1);
      S.goff = goff;
      S.e0 = e0;
      any = noi_closure_block<NW, WRAPS>((int32_t)lo, n, adj, w, lam, S, sh, put);
    } else {
      ClosureSmem<long long, int64_t, false> S;
      S.r = (long long*)noi_rs;
      S.soff = nullptr;
      S.queue = (uint16_t*)(S.r + ((n + 3) & ~3));
      S.goff = goff;
      S.e0 = e0;
      any = noi_closure_block<NW, WRAPS>((int32_t)lo, n, adj, w, lam, S, sh, put);
    }
    if (any && threadIdx.x == 0) atomicOr(list ? changed + g : changed, 1);
  }
}

template <int NW, typename WT, bool WRAPS = false>
static void noi_round_launch(const GraphView& u, const int32_t* list, int count, const DevState* st,
                             const long long* vbase, const long long* nv, const long long* glam, long long* r,
                             int32_t* queue, int32_t* labels, int* changed, int ncap, cudaStream_t s) {
  set_smem(noi_round_k<WT, NW, WRAPS>, noi_round_smem(kNoiSmemRoundMaxN));
  noi_round_k<WT, NW, WRAPS><<<std::min(count, kSMs * 8), NW * 32, noi_round_smem(ncap), s>>>(
      list, count, u.n, st, vbase, nv, glam, u.off, u.adj, (const WT*)u.w, r, (unsigned long long*)r + u.n, queue,
      labels, changed, ncap);
  count_launch();
  VC_CHECK_LAUNCH();
}

template <int NW>
static void noi_round_by_weight(const GraphView& u, const int32_t* list, int count, const DevState* st,
                                const long long* vbase, const long long* nv, const long long* glam, long long* r,
                                int32_t* queue, int32_t* labels, int* changed, int ncap, cudaStream_t s) {
  if (u.unit)
    noi_round_launch<NW, UnitW>(u, list, count, st, vbase, nv, glam, r, queue, labels, changed, ncap, s);
  else if (u.wbytes == 4)
    noi_round_launch<NW, int32_t>(u, list, count, st, vbase, nv, glam, r, queue, labels, changed, ncap, s);
  else
    noi_round_launch<NW, long long>(u, list, count, st, vbase, nv, glam, r, queue, labels, changed, ncap, s);
}

void noi_round_sparse(const GraphView& g, const DevState* st, long long* r, int32_t* parent, int32_t* labels,
                      int* changed, cudaStream_t s) {
  // parent (n entries) holds the queue of taken vertices
  const int ncap = (int)std::min<int64_t>(g.n, kNoiSmemRoundMaxN);
  if (g.wraps)
    noi_round_launch<16, long long, true>(g, nullptr, 1, st, nullptr, nullptr, nullptr, r, parent, labels, changed,
                                          ncap, s);
  else
    noi_round_by_weight<16>(g, nullptr, 1, st, nullptr, nullptr, nullptr, r, parent, labels, changed, ncap, s);
}

void noi_round_batch(const GraphView& u, const int32_t* list, int count, const long long* vbase, const long long* nv,
                     const long long* glam, long long* r, int32_t* parent, int32_t* labels, int* gchanged, int cls,
                     cudaStream_t s) {
  if (count <= 0) return;
  // r holds noi_round_scratch(union size) entries: the values, then each graph's chunk
  // bounds at its own range; parent (union size) holds the queues
  const int ncap = std::min(noi_class_max(cls), kNoiSmemRoundMaxN);
  if (cls == kNoiClasses - 1)
    noi_round_by_weight<16>(u, list, count, nullptr, vbase, nv, glam, r, parent, labels, gchanged, ncap, s);
  else
    noi_round_by_weight<8>(u, list, count, nullptr, vbase, nv, glam, r, parent, labels, gchanged, ncap, s);
}

// ------------------------------------------------------- allocation-free round
// Scratch of viecut_noi_round_noalloc: r (int64), parent (int32) and seen (byte) for
// at most kNoAllocMaxN vertices, in one array that every device loading the library
// keeps until the process exits (about 0.8 MB).  Host code must not pass the array's
// name to a kernel: on the host it is only a stand-in; its device address comes from
// cudaGetSymbolAddress, looked up once per device.
constexpr int64_t kNoAllocMaxN = 1 << 16;
constexpr size_t kNoAllocBytes = (size_t)kNoAllocMaxN * (sizeof(long long) + sizeof(int32_t) + 1);
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

__global__ void __launch_bounds__(kSparseThreads) noi_round_noalloc_k(int64_t n, const int64_t* __restrict__ off,
                                                                      const int32_t* __restrict__ adj,
                                                                      const long long* __restrict__ w, long long lam,
                                                                      unsigned char* scratch, int32_t* labels,
                                                                      int32_t* changed) {
  long long* r = (long long*)scratch;
  int32_t* parent = (int32_t*)(scratch + (size_t)kNoAllocMaxN * sizeof(long long));
  unsigned char* seen = scratch + (size_t)kNoAllocMaxN * (sizeof(long long) + sizeof(int32_t));
  if (threadIdx.x == 0) *changed = 0;
  __syncthreads();
  // the body clears r, seen and parent for [0, n) before using them
  noi_round_body<long long>(0, n, off, adj, w, lam, r, seen, parent, labels, changed);
}

static unsigned char* noalloc_scratch_address() {
  static std::mutex mu;
  static unsigned char* addr[256] = {nullptr};
  int dev = 0;
  VC_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 256) throw Error{VIECUT_EINVAL, "device ordinal out of range"};
  std::lock_guard<std::mutex> lock(mu);
  if (!addr[dev]) {
    void* p = nullptr;
    VC_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
    addr[dev] = (unsigned char*)p;
  }
  return addr[dev];
}

void set_last_error(const std::string& msg);

}  // namespace vc

extern "C" int viecut_noi_round_noalloc(const int64_t* d_offsets, const int32_t* d_adj, const int64_t* d_weights,
                                        int64_t n, int64_t lambda_hat, int32_t* d_labels, int32_t* d_changed,
                                        void* stream) {
  try {
    if (n < 1 || n > vc::kNoAllocMaxN)
      throw vc::Error{VIECUT_EINVAL, "viecut_noi_round_noalloc: n = " + std::to_string(n) + " is outside [1, " +
                                         std::to_string(vc::kNoAllocMaxN) + "], the size of its static scratch"};
    // the host cannot see offsets[n], so a graph with edges cannot be told apart from an
    // edgeless one here: every array must be given
    if (!d_offsets || !d_adj || !d_weights || !d_labels || !d_changed)
      throw vc::Error{VIECUT_EINVAL, "viecut_noi_round_noalloc: null device pointer"};
    if (lambda_hat < 0) throw vc::Error{VIECUT_EINVAL, "lambda_hat must be >= 0"};
    unsigned char* scratch = vc::noalloc_scratch_address();
    vc::noi_round_noalloc_k<<<1, vc::kSparseThreads, 0, (cudaStream_t)stream>>>(
        n, d_offsets, d_adj, (const long long*)d_weights, lambda_hat, scratch, d_labels, d_changed);
    vc::count_launch();
    VC_CHECK_LAUNCH();
  } catch (const vc::Error& e) {
    vc::set_last_error(e.msg);
    return e.code;
  }
  return VIECUT_OK;
}
