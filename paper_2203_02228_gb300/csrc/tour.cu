// tour.cu -- the initial solution of Alg 2 (Sec. 4.3): nearest-neighbour
// tour from node 0 -- first unvisited candidate, else first unvisited backup
// entry, else the globally nearest unvisited node by (squared distance, id)
// -- improved by the local search with every node queued in tour order.
// Both steps are sequential by definition; each runs on one block.
//
// Also: small device self-test kernels (Philox, EUC_2D, roulette) that the
// tests call through the library to compare with their own expectations.
#include <climits>

#include "common.cuh"
#include "launch.h"
#include "ls.cuh"
#include "nearest.cuh"

namespace faco {

namespace {

// The walk is one warp's chain of dependent steps: the row of the current
// node, the visited bits of its candidates, the first free one.  A row costs
// an L2 round trip unless it is in L1 by then, and a prefetch of the
// candidates' rows, one step ahead, comes too late for half of them (L1 hit
// rate 48 %, 837 cycles a step).  So kNnHelpers more warps follow the walk
// and bring the rows two steps out into L1: they read the current node from
// shared memory and touch the rows of its candidates' candidates.  They only
// load: the walk never waits for them.  Set-up in ms at n = 5k / 20k / 100k /
// 200k with 0, 1, 3, 7 helpers: 9.2 / 36.8 / 208 / 485; 8.5 / 34.2 / 197 / 461; 8.5 /
// 34.1 / 196 / 460; 8.5 / 34.0 / 195 / 457.
constexpr int kNnHelpers = 3;

__device__ __forceinline__ void nn_helper(int n, const int32_t* cand, int k, const volatile int* cur) {
  const int lane = lane_id();
  const int part = ((threadIdx.x >> 5) - 1) * 2 + (lane >> 4);  // of a row's entries
  const int limit = n < (1 << 18) ? n * 4096 : 1 << 30;  // never reached: the walk ends first
  int last = -1;
  for (int spin = 0; spin < limit; ++spin) {
    const int u = *cur;
    if (u < 0) break;  // the walk is done
    if (u == last) {
      __nanosleep(40);
      continue;
    }
    last = u;
    for (int j = lane & 15; j < k; j += 16) {
      const int c = cand[(size_t)u * k + j];
      for (int e = part; e < k; e += 2 * kNnHelpers) prefetch_l1(cand + (size_t)cand[(size_t)c * k + e] * k);
    }
  }
}

__device__ __forceinline__ void nn_tour_body(const int2* xy, int n, const int32_t* cand, int k,
                                             const int32_t* backup, int bl, int32_t* route, uint32_t* vis,
                                             const Grid& g, const int32_t* cstart, const int4* recs,
                                             volatile int* cur) {
  const int lane = lane_id();
  const int words = (n + 31) >> 5;
  for (int i = lane; i < words; i += 32) vis[i] = 0;
  __syncwarp();
  if (lane == 0) {
    route[0] = 0;
    vis[0] = 1u;
    *cur = 0;
  }
  __syncwarp();
  int u = 0;
  int c = lane < k ? cand[lane] : -1;  // the row of u
  for (int i = 1; i < n; ++i) {
    int v = -1;
    {
      const bool ok = c >= 0 && !((vis[c >> 5] >> (c & 31)) & 1u);
      const unsigned bal = __ballot_sync(kFull, ok);
      if (bal) v = __shfl_sync(kFull, c, __ffs(bal) - 1);
    }
    for (int j0 = 0; v < 0 && j0 < bl; j0 += 32) {
      const int j = j0 + lane;
      const int c = j < bl ? backup[(size_t)u * bl + j] : -1;
      const bool ok = c >= 0 && !((vis[c >> 5] >> (c & 31)) & 1u);
      const unsigned bal = __ballot_sync(kFull, ok);
      if (bal) v = __shfl_sync(kFull, c, __ffs(bal) - 1);
    }
    if (v < 0) {
      // global nearest unvisited node: rings of grid cells, else a scan of
      // the visited words that skips full ones
      const int2 xu = xy[u];
      int h;
      v = ring_nearest(recs, g, cstart, xu, 24,
                       [&](const int4& P) { return ((vis[P.w >> 5] >> (P.w & 31)) & 1u) != 0; }, h);
    }
    if (v < 0) {
      const int2 xu = xy[u];
      uint64_t bk = ~0ull;
      int32_t bi = INT_MAX;
      for (int wi = lane; wi < words; wi += 32) {
        uint32_t fr = ~vis[wi];
        if (wi == words - 1 && (n & 31)) fr &= (1u << (n & 31)) - 1u;
        while (fr) {
          const int w = wi * 32 + __ffs(fr) - 1;
          fr &= fr - 1;
          const uint64_t m = sqdist(xu, xy[w]);
          if (m < bk || (m == bk && w < bi)) {
            bk = m;
            bi = w;
          }
        }
      }
      warp_min_key(bk, bi);
      v = (bi >= 0 && bi < n) ? bi : 0;  // bi is valid while a node is unvisited
    }
    u = v;
    c = lane < k ? cand[(size_t)u * k + lane] : -1;  // on its way while the step is written down
    if (lane == 0) {
      route[i] = v;
      vis[v >> 5] |= 1u << (v & 31);
      *cur = v;
    }
    __syncwarp();
  }
  if (lane == 0) *cur = -1;
}

constexpr int kNnThreads = 32 * (1 + kNnHelpers);

__global__ void __launch_bounds__(kNnThreads) k_nn_tour(const int2* xy, int n, const int32_t* cand, int k,
                                                        const int32_t* backup, int bl, int32_t* route,
                                                        uint32_t* vis_g, Grid g, const int32_t* cstart,
                                                        const int4* recs) {
  extern __shared__ uint32_t sv[];
  __shared__ int s_cur;
  if (threadIdx.x == 0) s_cur = 0;
  __syncthreads();
  if (threadIdx.x >= 32)
    nn_helper(n, cand, k, &s_cur);
  else
    nn_tour_body(xy, n, cand, k, backup, bl, route, vis_g ? vis_g : sv, g, cstart, recs, &s_cur);
}

// Batch: one block per colony, visited bits in shared memory.
__global__ void __launch_bounds__(kNnThreads) k_nn_tour_b(const Colony* cols, const ColonySetup* sets) {
  extern __shared__ uint32_t sv[];
  const Colony C = cols[blockIdx.x];
  const ColonySetup S = sets[blockIdx.x];
  __shared__ int s_cur;
  if (threadIdx.x == 0) s_cur = 0;
  __syncthreads();
  if (threadIdx.x >= 32)
    nn_helper(C.n, S.cand, C.k, &s_cur);
  else
    nn_tour_body(C.xy, C.n, S.cand, C.k, S.backup, C.bl, S.init_route, sv, C.grid, S.cell_start, S.cell_src, &s_cur);
}

// Window and block size (entries + 1 warps), set-up in ms at n = 5k / 20k /
// 100k / 200k: 11: 9.7 / 38.8 / 242 / 621; 15: 8.8 / 35.2 / 212 / 531; 19: 9.0 /
// 35.8 / 208 / 505; 23: 9.4 / 37.2 / 211 / 499; 31 (64 registers, spills): 10.3 /
// 41.2 / 229 / 526.  The tour positions stay in global memory: in shared memory
// (17 bits a node, up to 106k nodes) they took the L1 cache from everything
// else, 272 against 229 ms at n = 100k with 31 entries.
constexpr int kWin = 19;                       // entries, a warp each; the last warp keeps the queue
constexpr int kInitThreads = 32 * (kWin + 1);

// A reversed span of tour positions: i, i + 1, ..., i + L - 1 (cyclic).
struct Span {
  int i, L;
};

// The span that reversing the forward span i..j turns over: itself, or its
// complement when longer than n / 2.
__device__ __forceinline__ Span flip_span(int i, int j, int n) {
  int L = j - i;
  if (L < 0) L += n;
  L += 1;
  if (2 * L > n) return Span{j + 1 == n ? 0 : j + 1, n - L};
  return Span{i, L};
}

// Reverses a span with the whole block.  Every caller reaches it after a
// block barrier that follows the last write to the tour, and the next reader
// waits at one.
// Most spans are shorter than the block; on the long ones, bound by the
// latency of their loads, each thread keeps U swaps in flight (set-up at
// n = 200,000 505 -> 491 ms).
__device__ __forceinline__ void cta_reverse(ArrTour& T, Span sp) {
  constexpr int U = 4;
  const int n = T.n;
  int j = sp.i + sp.L - 1;
  if (j >= n) j -= n;
  const int half = sp.L >> 1;
  if (half <= kInitThreads) {
    const int t = threadIdx.x;
    if (t < half) {
      const int ia = wrapn(sp.i + t, n), ib = wrapn(j - t, n);
      const int va = T.route[ia], vb = T.route[ib];
      T.route[ia] = vb;
      T.route[ib] = va;
      T.pos[vb] = ia;
      T.pos[va] = ib;
    }
    return;
  }
#pragma unroll 1
  for (int t0 = threadIdx.x; t0 < half; t0 += U * kInitThreads) {
    int va[U], vb[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int t = t0 + u * kInitThreads;
      if (t < half) {
        va[u] = T.route[wrapn(sp.i + t, n)];
        vb[u] = T.route[wrapn(j - t, n)];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int t = t0 + u * kInitThreads;
      if (t < half) {
        const int ia = wrapn(sp.i + t, n), ib = wrapn(j - t, n);
        T.route[ia] = vb[u];
        T.route[ib] = va[u];
        T.pos[vb[u]] = ia;
        T.pos[va[u]] = ib;
      }
    }
  }
}

// The local search with every node queued (the initial tour), run by one
// block of kWin + 1 warps over a window of the next kWin queued nodes.  Each
// window entry keeps its evaluation -- the best move from its node on the
// tour as it was -- together with the tour positions that evaluation read
// (the node's, the next three and the previous one; each candidate's and its
// two neighbours').  A move reverses spans of positions; an entry whose
// positions meet none of them would evaluate to the same result, so it is
// kept, the others are dropped.  Each round pops entries in queue order up
// to and including the first one whose evaluation found a move, which is
// applied.  An evaluation runs only when an entry without one comes before
// the first improving entry (all entries without one are then evaluated, a
// warp each).  The pops, moves and queue are exactly those of popping one
// node at a time.
//
// Bound by the latency of a round, one move long: evaluation, decision,
// reversal.  So every warp takes the same decisions from the same shared
// values, in registers, with two block barriers per round (after the
// evaluations, after the reversal); a 2-opt move brings the positions of its
// ends along; entries to drop are found while the span is being reversed;
// and the queue's own work -- flags, log, pushes, reading nodes ahead into
// shared memory -- is left to the last warp, during the next round's
// evaluations.  Only with less than kAhead nodes queued does a round wait
// for it (sync_queue).  Set-up 14.1 -> 12.1 ms at n = 5,003 and 322 -> 302 ms at
// n = 100,000 against the form with six barriers per round and the queue's
// work between them.  Evaluating only the first 8 / 16 / 24 entries of the
// window without an evaluation: 408 / 330 / 316 ms against 318 (n = 100,000).
constexpr int kAhead = 96;   // queued nodes read ahead (a ring of 128)

template <bool TWO>
__device__ __forceinline__ void init_ls_body(ArrTour& T, int oropt, int verify, int init3, int32_t* queue, uint8_t* flags,
                                             int32_t* logb) {
  __shared__ int32_t s_gain[32];
  __shared__ int s_mv[32][8];
  __shared__ int2 s_ij[32];               // 2-opt: positions of the span's ends
  __shared__ int s_any[32];               // 1: the evaluation read beyond s_dep (3-opt scan): any move drops it
  __shared__ int s_dep[32][kMaxK + 1];    // [0]: its position, [1 + s]: candidate s's position
  __shared__ int s_inv[2][32];            // 1: the round's move drops the entry
  __shared__ int s_q[128];                // nodes of the queue by position modulo 128, from the head on
  __shared__ int s_pmv[8];                // the last warp's copy of that round's move
  __shared__ int s_qn, s_nlog;
  const int n = T.n, k = T.k;
  int32_t* route = T.route;
  LsEnv E{n, oropt, verify, queue, flags, logb};
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const bool keeper = w == kWin;
  for (int i = tid; i < n; i += blockDim.x) {
    const int x = route[i];
    queue[i] = x;
    flags[x] = 1;
  }
  __syncthreads();
  // the same on every thread: queue position of the head (counted from the
  // start, and modulo n), nodes queued (not counting pushes since the last
  // sync_queue), moves applied, entries of the window with an evaluation
  unsigned qa = 0;
  int qh = 0, qn = n, changes = 0, moves_round = 0, par = 0;
  unsigned have = 0;
  // the last warp: nodes queued, nodes logged, nodes read ahead, and the
  // round whose pops and pushes it has not done yet
  int kq = n, klog = 0, kld = 0, p_cnt = 0, p_np = 0, p_node = -1, p_qh = 0;
  auto keep_pending = [&]() {  // (last warp)
    if (p_cnt == 0) return;
    bool first_pop = false;
    if (lane < p_cnt) {
      const uint8_t f = flags[p_node];
      first_pop = !(f & 2);
      flags[p_node] = (uint8_t)((f & ~1) | 2);
    }
    const unsigned fb = __ballot_sync(kFull, first_pop);
    if (first_pop) logb[klog + __popc(fb & ((1u << lane) - 1u))] = p_node;
    klog += __popc(fb);
    kq -= p_cnt;
    __syncwarp();
    if (p_np > 0) kq = ls_push_warp(E, s_pmv, p_np, p_qh, kq);
    p_cnt = 0;
  };
  auto read_ahead = [&]() {  // (last warp) up to kAhead nodes from the head on
    const int upto = min(kAhead, kq);
    for (int o = kld; o < upto; o += 32) {
      if (o + lane < upto) {
        int idx = qh + o + lane;
        if (idx >= n) idx -= n;
        s_q[(qa + o + lane) & 127] = queue[idx];
      }
    }
    kld = max(kld, upto);
  };
  // every thread: the exact queue length, and the nodes ahead of it
  auto sync_queue = [&]() {
    if (keeper) {
      keep_pending();
      kld = 0;
      read_ahead();
      if (lane == 0) {
        s_qn = kq;
        s_nlog = klog;
      }
    }
    __syncthreads();
    qn = s_qn;
  };
  sync_queue();
  for (;;) {
    if (qn == 0 || changes >= n) {
      if (changes >= n || !verify || moves_round == 0) break;
      const int nl = s_nlog;  // verify round: queue again the nodes popped
      for (int i = tid; i < nl; i += blockDim.x) {
        const int x = logb[i];
        queue[i] = x;
        flags[x] = 1;
      }
      __syncthreads();
      qh = 0;
      moves_round = 0;
      have = 0;  // the queue changed: no evaluation carries over
      kq = nl;
      klog = 0;
      sync_queue();
      continue;
    }
    // window offset `lane` of every warp: its node and slot
    const int R = qn < kWin ? qn : kWin;
    const unsigned live = R == 32 ? kFull : ((1u << R) - 1u);
    const int slot = (qa + lane) & 31;
    const int node = lane < R ? s_q[(qa + lane) & 127] : -1;
    const unsigned bimp = __ballot_sync(kFull, ((have >> lane) & 1u) && s_gain[slot] > 0);
    const unsigned bmiss = live & ~have;
    const int f = bimp ? __ffs(bimp) - 1 : R;
    const bool eval = (bmiss & ((1u << f) - 1u)) != 0;  // an entry without an evaluation comes first
    if (keeper) {
      keep_pending();
      read_ahead();
    } else if (eval && ((bmiss >> w) & 1u)) {
      const int my_node = __shfl_sync(kFull, node, w);
      const int my_slot = (qa + w) & 31;
      int mv[8], mv3[6];
      const int32_t g = eval_both<TWO>(T, my_node, oropt != 0, mv);
      int64_t g3 = 0;
      // the 3-opt exchange only when neither 2-opt nor Or-opt improves
      // (g is the warp's reduction: the branch is warp-uniform)
      const bool try3 = init3 && g == 0;
      if (try3) g3 = eval_or3(T, my_node, mv3);
      if (lane < k) s_dep[my_slot][1 + lane] = T.pos_of(T.cand(my_node, lane));
      if (lane == 0) {
        s_dep[my_slot][0] = T.pos_of(my_node);
        if (g3 > 0) {
          s_gain[my_slot] = (int32_t)g3;
          for (int t = 0; t < 6; ++t) s_mv[my_slot][t] = mv3[t];
          s_mv[my_slot][7] = 2;
        } else {
          s_gain[my_slot] = g;
          if (g > 0) {
            for (int t = 0; t < 8; ++t) s_mv[my_slot][t] = mv[t];
            s_ij[my_slot] = make_int2(T.pos_of(mv[1]), T.pos_of(mv[2]));
          }
        }
        s_any[my_slot] = try3 ? 1 : 0;
      }
    }
    if (eval) {
      __syncthreads();
      have |= bmiss;
    }
    const unsigned bal = __ballot_sync(kFull, ((have >> lane) & 1u) && s_gain[slot] > 0);
    const int first = bal ? __ffs(bal) - 1 : R;
    const int cnt = bal ? first + 1 : R;  // queue entries popped this round
    if (keeper) {
      p_cnt = cnt;
      p_node = node;
      p_np = 0;
      p_qh = qh + cnt;
      if (p_qh >= n) p_qh -= n;
      kld -= cnt;
    }
    if (bal) {
      const int win = (qa + first) & 31;
      const int kind = s_mv[win][7];
      if (keeper) {
        p_np = kind == 0 ? 4 : 6;
        if (lane < 8) s_pmv[lane] = s_mv[win][lane];
        __syncwarp();
      }
      // the entry of window offset w: does a reversed position matter to it?
      const int ws = (qa + w) & 31;
      const bool mine = w > first && w < R && ((have >> w) & 1u);
      bool hit = mine && s_any[ws] != 0;
      const int dep = mine ? (lane < k ? s_dep[ws][1 + lane] : s_dep[ws][0]) : 0;
      const int dn = mine ? s_dep[ws][0] : 0;
      auto meets = [&](Span sp) {
        // a candidate's position and its two neighbours: dep - 1 .. dep + 1
        int d = dep + 1 - sp.i;
        if (d < 0) d += n;
        if (d >= n) d -= n;
        if (lane < k && d < sp.L + 2) hit = true;
        // the node's: dn - 1 .. dn + 3
        d = dn + 3 - sp.i;
        while (d < 0) d += n;
        while (d >= n) d -= n;
        if (d < sp.L + 4) hit = true;
      };
      if (kind == 0) {
        const int2 ij = s_ij[win];
        const Span sp = flip_span(ij.x, ij.y, n);
        if (mine) meets(sp);
        cta_reverse(T, sp);
      } else {
        // two or three edge exchanges {n1,n2},{n3,n4} -> {n1,n3},{n2,n4}
        //   Or-opt {p,a,e,q,u,v,kept}; 3-opt {a,t2,b,b',c,c'}:
        //   {a,t2},{b,b'} -> {a,b},{t2,b'}; {a,b},{c,c'} -> {a,c},{b,c'}; {a,c},{b',t2} -> {a,b'},{c,t2}
        const int* mv = s_mv[win];
        const int steps = kind == 1 ? (mv[6] ? 3 : 2) : 3;
        for (int st = 0; st < steps; ++st) {
          int n1, n2, n3, n4;
          if (kind == 1) {
            n1 = st == 2 ? mv[4] : mv[0];
            n2 = st == 0 ? mv[1] : (st == 1 ? mv[4] : mv[2]);
            n3 = st == 0 ? mv[4] : (st == 1 ? mv[3] : mv[1]);
            n4 = st == 1 ? mv[2] : mv[5];
          } else {
            n1 = mv[0];
            n2 = st == 0 ? mv[1] : (st == 1 ? mv[2] : mv[4]);
            n3 = st == 0 ? mv[2] : (st == 1 ? mv[4] : mv[3]);
            n4 = st == 0 ? mv[3] : (st == 1 ? mv[5] : mv[1]);
          }
          const bool fwd = T.succ(n1) == n2;
          const int i = T.pos_of(fwd ? n2 : n1), j = T.pos_of(fwd ? n3 : n4);
          __syncthreads();  // every thread has read the tour before a position moves
          const Span sp = flip_span(i, j, n);
          if (mine) meets(sp);
          cta_reverse(T, sp);
          if (st + 1 < steps) __syncthreads();
        }
      }
      const bool any = __any_sync(kFull, hit);
      if (lane == 0) s_inv[par][w] = any ? 1 : 0;
      ++changes;
      ++moves_round;
    }
    __syncthreads();  // the tour, s_inv and the nodes read ahead are there; s_gain and s_mv were read
    if (bal) {
      have &= ~__ballot_sync(kFull, lane < R && s_inv[par][lane] != 0);  // a warp each: entries below R
      par ^= 1;
    }
    have = cnt >= 32 ? 0u : have >> cnt;
    qa += cnt;
    qh += cnt;
    if (qh >= n) qh -= n;
    qn -= cnt;
    if (qn < kAhead) sync_queue();
  }
  __syncthreads();
  if (keeper) {
    keep_pending();
    if (lane == 0) {
      s_qn = kq;
      s_nlog = klog;
    }
  }
  __syncthreads();
  const int ql = s_qn, nl = s_nlog;
  for (int t = tid; t < ql; t += blockDim.x) {
    int i = qh + t;
    if (i >= n) i -= n;
    flags[queue[i]] = 0;
  }
  for (int i = tid; i < nl; i += blockDim.x) flags[logb[i]] = 0;
}

template <bool TWO>
__global__ void __launch_bounds__(kInitThreads) k_init_ls(const int2* xy, int n, const int32_t* cand,
                                                          const int32_t* dcand, int k, int oropt, int verify,
                                                          int init3, int32_t* route, int32_t* pos, int32_t* queue,
                                                          uint8_t* flags, int32_t* logb) {
  ArrTour T{n, k, route, pos, xy, cand, k, dcand};
  init_ls_body<TWO>(T, oropt, verify, init3, queue, flags, logb);
}

// Batch: one block per colony; positions of the initial tour in src_pos.
template <bool TWO>
__global__ void __launch_bounds__(kInitThreads) k_init_ls_b(const Colony* cols, const ColonySetup* sets) {
  const Colony C = cols[blockIdx.x];
  const ColonySetup S = sets[blockIdx.x];
  ArrTour T{C.n, C.k, S.init_route, C.src_pos, C.xy, S.cand, C.k, S.dcand};
  init_ls_body<TWO>(T, C.oropt, C.verify, C.init3, S.queue, S.flags, S.logb);
}

// what = 0: Philox draws   in: uint32 [count][4] = (idx, ant, iter, tag) -> out uint32
// what = 1: EUC_2D         in: int32 [count][4] = (x1, y1, x2, y2)       -> out int32
// what = 2: roulette       in: float [count][width + 1] (weights, u)     -> out int32
__global__ void k_tests(int what, const void* in, void* out, int count, int width, uint64_t seed) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  if (what == 0) {
    const uint32_t* a = static_cast<const uint32_t*>(in) + 4 * i;
    static_cast<uint32_t*>(out)[i] = draw(seed, a[0], a[1], a[2], a[3]);
  } else if (what == 1) {
    const int32_t* a = static_cast<const int32_t*>(in) + 4 * i;
    static_cast<int32_t*>(out)[i] = euc2d(make_int2(a[0], a[1]), make_int2(a[2], a[3]));
  } else {
    const float* a = static_cast<const float*>(in) + (size_t)(width + 1) * i;
    int r;
    if (width == 16) {
      float w[16];
      for (int s = 0; s < 16; ++s) w[s] = a[s];
      r = roulette<16>(w, a[16]);
    } else {
      float w[32];
      for (int s = 0; s < 32; ++s) w[s] = a[s];
      r = roulette<32>(w, a[32]);
    }
    static_cast<int32_t*>(out)[i] = r;
  }
}

// The initial search names nodes by their position in the nearest-
// neighbour tour: node i of the copies is route0[i], and a candidate list
// names its entries the same way.  Lists keep their order and coordinates
// their values, so every decision of the search is the same; what changes is
// where things lie in memory -- consecutive names are neighbours on the walk,
// so a node's coordinates, lists and tour neighbours share cache lines with
// those of the nodes around it.  One thread per list entry.
__global__ void k_relabel(const int32_t* __restrict__ route0, const int32_t* __restrict__ pos0,
                          const int2* __restrict__ xy, const int32_t* __restrict__ cand,
                          const int32_t* __restrict__ dcand, int n, int k, int2* __restrict__ xy_t,
                          int32_t* __restrict__ cand_t, int32_t* __restrict__ dcand_t,
                          int32_t* __restrict__ route_t, int32_t* __restrict__ pos_t) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (size_t)n * k) return;
  const int i = (int)(e / k), s = (int)(e - (size_t)i * k);
  const int u = route0[i];
  const int c = cand[(size_t)u * k + s];
  cand_t[e] = c >= 0 ? pos0[c] : c;
  dcand_t[e] = dcand[(size_t)u * k + s];
  if (s == 0) {
    xy_t[i] = xy[u];
    route_t[i] = i;
    pos_t[i] = i;
  }
}

// route[t] = route0[route_t[t]]: the searched tour back in node ids.
__global__ void k_unlabel(const int32_t* __restrict__ route0, const int32_t* __restrict__ route_t,
                          int32_t* __restrict__ route, int n) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) route[t] = route0[route_t[t]];
}

}  // namespace

cudaError_t launch_nn_tour(const int2* xy, int n, const int32_t* cand, int k, const int32_t* backup,
                           int bl, int32_t* route, uint32_t* vis_g, const Grid& g, const int32_t* cstart,
                           const int4* recs, cudaStream_t s) {
  const size_t smem = vis_g ? 0 : (size_t)((n + 31) >> 5) * sizeof(uint32_t);
  if (smem > 48 * 1024) {
    cudaError_t e = allow_dyn_smem(reinterpret_cast<const void*>(k_nn_tour), smem);
    if (e != cudaSuccess) return e;
  }
  k_nn_tour<<<1, kNnThreads, smem, s>>>(xy, n, cand, k, backup, bl, route, vis_g, g, cstart, recs);
  return cudaGetLastError();
}

cudaError_t launch_relabel(const int32_t* route0, const int32_t* pos0, const int2* xy, const int32_t* cand,
                           const int32_t* dcand, int n, int k, int2* xy_t, int32_t* cand_t, int32_t* dcand_t,
                           int32_t* route_t, int32_t* pos_t, cudaStream_t s) {
  const size_t e = (size_t)n * k;
  k_relabel<<<(unsigned)((e + 255) / 256), 256, 0, s>>>(route0, pos0, xy, cand, dcand, n, k, xy_t, cand_t, dcand_t,
                                                        route_t, pos_t);
  return cudaGetLastError();
}

cudaError_t launch_unlabel(const int32_t* route0, const int32_t* route_t, int32_t* route, int n, cudaStream_t s) {
  k_unlabel<<<(n + 255) / 256, 256, 0, s>>>(route0, route_t, route, n);
  return cudaGetLastError();
}

cudaError_t launch_init_ls(const int2* xy, int n, const int32_t* cand, const int32_t* dcand, int k, int oropt,
                           int verify, int init3, int32_t* route, int32_t* pos, int32_t* queue, uint8_t* flags,
                           int32_t* logb, cudaStream_t s) {
  if (k > 16)
    k_init_ls<true><<<1, kInitThreads, 0, s>>>(xy, n, cand, dcand, k, oropt, verify, init3, route, pos, queue, flags,
                                               logb);
  else
    k_init_ls<false><<<1, kInitThreads, 0, s>>>(xy, n, cand, dcand, k, oropt, verify, init3, route, pos, queue, flags,
                                                logb);
  return cudaGetLastError();
}

cudaError_t launch_init_tour_batch(const Colony* cols, const ColonySetup* sets, int count, int max_n, int kw,
                                   int stage, cudaStream_t s) {
  if (stage == 0) {
    const size_t smem = (size_t)((max_n + 31) >> 5) * sizeof(uint32_t);
    if (smem > 48 * 1024) {
      cudaError_t e = allow_dyn_smem(reinterpret_cast<const void*>(k_nn_tour_b), smem);
      if (e != cudaSuccess) return e;
    }
    k_nn_tour_b<<<count, kNnThreads, smem, s>>>(cols, sets);
  } else if (kw == 32) {
    k_init_ls_b<true><<<count, kInitThreads, 0, s>>>(cols, sets);
  } else {
    k_init_ls_b<false><<<count, kInitThreads, 0, s>>>(cols, sets);
  }
  return cudaGetLastError();
}

cudaError_t launch_test_kernels(int what, const void* in, void* out, int count, int width,
                                uint64_t seed, cudaStream_t s) {
  k_tests<<<(count + 127) / 128, 128, 0, s>>>(what, in, out, count, width, seed);
  return cudaGetLastError();
}

}  // namespace faco
