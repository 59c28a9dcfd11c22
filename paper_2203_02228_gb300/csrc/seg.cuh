// seg.cuh -- an ant's tour held as runs of the source solution.
//
// After focused construction (Alg 2) an ant's tour is a concatenation of a
// few runs of the source solution; the local search (Alg 3) then changes
// the tour by reversals.  Instead of materialising route[]/pos[] arrays of
// n entries per ant, a block keeps the tour as a table of segments in shared
// memory.  Nodes are named by their source position; the segments tile
// 0..n-1, so one sorted array of boundaries describes them all: boundary r
// is the first node lo[r] of segment r, which ends before lo[r + 1]
// (lo[S] = n).  Per boundary the table keeps
//   - br: the segment's map from node to tour position, base + q (bit 31
//     clear: the tour walks it upwards) or base - q (bit 31 set), modulo n;
//   - nb: the tour neighbours across the boundary, x = that of lo[r] outside
//     segment r, y = that of lo[r] - 1 outside segment r - 1.
// A tour neighbour is one search by node, then q + 1, q - 1 or a stored
// neighbour; no order by tour position is needed.  A reversal of positions
// i..j maps base to i + j - base and flips bit 31 in every segment inside
// the span, adds a boundary at each cut that falls inside a segment, drops
// the boundaries between segments that now continue each other, and sets the
// four neighbours of the two new edges -- exactly the array reversal.  Since
// a split part keeps its map and a merge keeps either part's, one pass that
// copies the table into its second buffer does all of it: segments may run
// across tour position 0, so no span is a special case.
// When the table is full the reversal reports failure and the search goes on
// on explicit arrays (same result, more memory traffic).
#pragma once

#include "common.cuh"
#include "ls.cuh"

namespace faco {

// A run as construction emits it: source positions [lo, lo + len), tour
// positions [off, off + len), walked downwards when rev.
struct Seg {
  int32_t lo, len, off, rev;
};

// Shared memory of a table of `cap` segments: two buffers of cap + 1
// boundaries, 16 bytes each.
constexpr size_t kSegBytes = 2 * (sizeof(int2) + 2 * sizeof(int32_t));
static_assert(kSegBytes == 2 * sizeof(Seg), "construction's list of runs takes one buffer's room");
__host__ __device__ constexpr size_t segtab_bytes(int cap) { return (size_t)(cap + 1) * kSegBytes; }

// Table capacity once the visited bits in front of a table of `cap`
// segments are free (the local search does not need them): the same
// shared memory, whole multiples of 32 segments added.
__host__ __device__ constexpr int segtab_cap_ls(size_t vis_bytes, int cap) {
  return cap + (int)((vis_bytes / kSegBytes) & ~(size_t)31);
}

// Construction's list of runs: the last cap * 16 bytes of the shared memory
// (`total` bytes) that holds the visited bits and a table of `cap` segments.
// It lies behind the visited bits, and behind buffer 0 of the larger table
// that the local search lays over both.
__device__ __forceinline__ Seg* segtab_runs(char* smem, size_t vis_bytes, int cap) {
  return reinterpret_cast<Seg*>(smem + vis_bytes + segtab_bytes(cap) - (size_t)cap * sizeof(Seg));
}

// One segment.
struct SegRec {
  int lo, hi, base, nlo, nhi;  // nlo, nhi: tour neighbours of lo and hi outside the segment
  bool rev;
  // the next node towards higher (else lower) source positions, or across
  // the segment's end
  __device__ __forceinline__ int step(int q, bool up) const {
    return up ? (q < hi ? q + 1 : nhi) : (q > lo ? q - 1 : nlo);
  }
  __device__ __forceinline__ bool inside(int q, bool up) const { return up ? q < hi : q > lo; }
  __device__ __forceinline__ int pos(int q, int n) const { return wrapn(rev ? base - q : base + q, n); }
};

// The table's current buffer, and the tour over it (nodes = source
// positions).  Taken anew after every reversal.
struct SegView {
  int n, k, kw, S;
  const int2* nb;
  const int32_t* lo;
  const int32_t* br;
  const int2* xy;       // coordinates by source position
  const int32_t* cn;    // candidate source positions by source position [n][kw]
  const int32_t* cd;    // their EUC_2D costs, same layout

  __device__ __forceinline__ int2 coord(int q) const { return xy[q]; }
  __device__ __forceinline__ int cand(int q, int s) const { return cn[(size_t)q * kw + s]; }
  __device__ __forceinline__ int cdist(int q, int s) const { return cd[(size_t)q * kw + s]; }

  // Segment of node q: the largest r with lo[r] <= q.
  __device__ __forceinline__ int locate(int q) const {
    int r = 0;
    for (int st = 1 << (31 - __clz(S)); st > 0; st >>= 1) {
      const int m = r + st;
      if (m < S && lo[m] <= q) r = m;
    }
    return r;
  }
  // The same by a whole warp for one (warp-uniform) node: each level
  // compares 32 boundaries spaced evenly over the remaining range, so a
  // table of up to 1,024 segments takes two shared-memory round trips
  // instead of ten dependent ones.
  __device__ __forceinline__ int locate_w(int q) const {
    const int lane = lane_id();
    int at = 0, len = S;  // the answer lies in [at, at + len); lo[at] <= q
    while (len > 1) {
      const int st = (len + 31) >> 5;
      const bool le = lane * st < len && lo[at + lane * st] <= q;
      const unsigned b = __ballot_sync(kFull, le);
      const int L = b ? 31 - __clz(b) : 0;
      at += L * st;
      len = min(st, len - L * st);
    }
    return at;
  }
  // Two of them level by level, so that their round trips overlap.
  __device__ __forceinline__ void locate2_w(int q1, int q2, int& r1, int& r2) const {
    const int lane = lane_id();
    int at1 = 0, at2 = 0, len = S;  // both ranges shrink alike, up to a shorter last part
    int len1 = S, len2 = S;
    while (len > 1) {
      const int st = (len + 31) >> 5, o = lane * st;
      const bool le1 = o < len1 && lo[at1 + o] <= q1, le2 = o < len2 && lo[at2 + o] <= q2;
      const unsigned b1 = __ballot_sync(kFull, le1), b2 = __ballot_sync(kFull, le2);
      const int L1 = b1 ? (31 - __clz(b1)) * st : 0, L2 = b2 ? (31 - __clz(b2)) * st : 0;
      at1 += L1;
      at2 += L2;
      len1 = min(st, len1 - L1);
      len2 = min(st, len2 - L2);
      len = st;
    }
    r1 = at1;
    r2 = at2;
  }
  __device__ __forceinline__ SegRec rec(int r) const {
    const int b = br[r];
    SegRec s;
    s.lo = lo[r];
    s.hi = lo[r + 1] - 1;
    s.nlo = nb[r].x;
    s.nhi = nb[r + 1].y;
    s.base = b & 0x7fffffff;
    s.rev = b < 0;
    return s;
  }
  // succ(q) when up, else pred(q): one lookup whatever the direction
  __device__ __forceinline__ int adj(int q, bool up) const {
    const SegRec s = rec(locate(q));
    return s.step(q, up != s.rev);
  }
  __device__ __forceinline__ void nbrs(int q, int& p, int& s) const {
    const SegRec g = rec(locate(q));
    p = g.step(q, g.rev);
    s = g.step(q, !g.rev);
  }
  // the predecessor and three successors of a warp-uniform node
  // (warp-collective); most often all in one segment
  __device__ __forceinline__ void walk(int a, int& p, int& s1, int& s2, int& s3) const {
    SegRec g = rec(locate_w(a));
    p = g.step(a, g.rev);
    int q = a;
    int s[3];
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const bool in = g.inside(q, !g.rev);
      q = g.step(q, !g.rev);
      s[t] = q;
      if (t < 2 && !in) g = rec(locate_w(q));
    }
    s1 = s[0];
    s2 = s[1];
    s3 = s[2];
  }
};

// Segments in the table and the buffer they are in: the same on every thread
// that changes the tour, kept in registers.
struct SegState {
  int S, cur;
};

// Tour over the segment table: what changes it.
struct SegTour {
  int n, k, kw;
  char* mem;            // buffers 0 and 1
  int cap;
  const int2* xy;
  const int32_t* cn;
  const int32_t* cd;

  __device__ __forceinline__ char* buffer(int which) const {
    return mem + (which ? (size_t)(cap + 1) * (kSegBytes / 2) : 0);
  }
  __device__ __forceinline__ SegView view(SegState st) const {
    const int m = cap + 1;
    char* b = buffer(st.cur);
    SegView v;
    v.n = n;
    v.k = k;
    v.kw = kw;
    v.S = st.S;
    v.nb = reinterpret_cast<const int2*>(b);
    v.lo = reinterpret_cast<const int32_t*>(b + (size_t)m * sizeof(int2));
    v.br = v.lo + m;
    v.xy = xy;
    v.cn = cn;
    v.cd = cd;
    return v;
  }

  // The table of construction's `S` runs (in tour order), with the whole
  // block: a thread per run finds its rank by counting.
  __device__ __forceinline__ SegState build(const Seg* runs, int S) const {
    const int m = cap + 1;
    char* b = buffer(0);
    int2* nb = reinterpret_cast<int2*>(b);
    int32_t* lo = reinterpret_cast<int32_t*>(b + (size_t)m * sizeof(int2));
    int32_t* br = lo + m;
    for (int id = threadIdx.x; id < S; id += blockDim.x) {
      const Seg s = runs[id];
      int r = 0;
      for (int o = 0; o < S; ++o) r += runs[o].lo < s.lo;
      const Seg pr = runs[id == 0 ? S - 1 : id - 1], nx = runs[id + 1 == S ? 0 : id + 1];
      const int hi = s.lo + s.len - 1;
      const int before = pr.rev ? pr.lo : pr.lo + pr.len - 1;   // last node of the run before
      const int after = nx.rev ? nx.lo + nx.len - 1 : nx.lo;    // first node of the run after
      lo[r] = s.lo;
      br[r] = s.rev ? (wrapn(s.off + hi, n) | (int)0x80000000) : wrapn(s.off - s.lo, n);
      nb[r].x = s.rev ? after : before;
      nb[r + 1].y = s.rev ? before : after;
    }
    if (threadIdx.x == 0) {
      nb[0].y = 0;  // no node before 0: never read
      nb[S].x = 0;
      lo[S] = n;
      br[S] = 0;
    }
    __syncthreads();
    return SegState{S, 0};
  }

  // Reverse the forward span x..y, or its complement when longer than n/2
  // (the array rule, entry for entry).  Returns the nodes reversed, or -1
  // when the table is full (then nothing has changed).  Run by the first nw
  // warps of the block (this one is warp w): each finds the span and the cuts
  // for itself, copies its share of the boundaries into the other buffer, and
  // has the new state; the new table may be read after a block barrier, which
  // also has to lie between two reversals.
  //
  // Bound by the latency of the search for x and y and of the copying pass,
  // one boundary per thread and 32 nw of them at a time: an ant's table holds
  // 80 to 600 segments.  Nothing orders the boundaries, so no warp waits for
  // another.  Of the slowest ants' time at n = 100,000 reversals took 2,120 us
  // of 4,870 with two orders of the table, 1,350 of 3,290 with one order and
  // one warp, 680 of 2,820 with the block's warps sharing the pass and the last
  // one doing the queue's work beside it.
  // Inlined, like everything else in the block kernel: it makes no calls.
  __device__ __forceinline__ int flip(SegState& st, int x, int y, int w, int nw) const {
    const int lane = lane_id();
    const SegView V = view(st);
    const int S = V.S;
    int rx, ry;
    V.locate2_w(x, y, rx, ry);
    const SegRec X = V.rec(rx), Y = V.rec(ry);
    const int px = X.step(x, X.rev), sy = Y.step(y, !Y.rev);  // pred x, succ y
    const bool inx = X.inside(x, X.rev), iny = Y.inside(y, !Y.rev);
    int i = X.pos(x, n);
    const int j = Y.pos(y, n);
    int L = j - i;
    if (L < 0) L += n;
    L += 1;
    int sum = i + j;  // a position t of the span goes to sum - t, whichever part is reversed
    if (sum >= n) sum -= n;
    if (2 * L > n) {
      i = (j + 1 == n) ? 0 : j + 1;
      L = n - L;
    }
    if (L <= 1) return L;
    if (S + 2 > cap) return -1;  // at most two boundaries more
    // the cut edges {px, x} and {y, sy} become {px, y} and {x, sy}: new
    // boundaries where a cut edge lies inside a segment; boundaries that go:
    // a new edge joins source neighbours q, q + 1 whose cut ends face each
    // other across boundary q + 1
    constexpr int kNone = INT_MAX;
    const int c1 = inx ? max(px, x) : kNone, c2 = iny ? max(y, sy) : kNone;
    auto joined = [&](int p, int pe, int q, int qe) {  // p was cut from pe, q from qe
      const int v = max(p, q);
      if (p - q != 1 && q - p != 1) return kNone;
      const int r = V.locate_w(v);
      const int2 e = make_int2(V.nb[r].x, V.nb[r].y);
      return V.lo[r] == v && e.x == (v == p ? pe : qe) && e.y == (v == p ? qe : pe) ? v : kNone;
    };
    const int m1 = joined(px, x, y, sy), m2 = joined(x, px, sy, y);
    // (boundaries of the new table) - (of the old one) below node v
    auto shift = [&](int v) { return (c1 < v) + (c2 < v) - (m1 < v) - (m2 < v); };
    // the map of a segment that contains node v, after the reversal
    auto turned = [&](int b, int v) {
      const int base = b & 0x7fffffff;
      int d = wrapn(b < 0 ? base - v : base + v, n) - i;
      if (d < 0) d += n;
      int nbase = sum - base;
      if (nbase < 0) nbase += n;
      return d < L ? nbase | (~b & (int)0x80000000) : b;
    };
    // the new tour neighbour of node o where the old one was e
    auto across = [&](int o, int e) {
      int t = e;
      t = (o == px) & (e == x) ? y : t;
      t = (o == x) & (e == px) ? sy : t;
      t = (o == y) & (e == sy) ? px : t;
      t = (o == sy) & (e == y) ? x : t;
      return t;
    };
    const int m = cap + 1;
    char* out = buffer(st.cur ^ 1);
    int2* nb2 = reinterpret_cast<int2*>(out);
    int32_t* lo2 = reinterpret_cast<int32_t*>(out + (size_t)m * sizeof(int2));
    int32_t* br2 = lo2 + m;
    for (int r = w * 32 + lane; r <= S; r += 32 * nw) {
      const int v = V.lo[r];
      const int b = V.br[r];
      const int2 e = V.nb[r];
      if (v != m1 && v != m2) {
        const int at = r + shift(v);
        lo2[at] = v;
        br2[at] = turned(b, v);
        nb2[at] = make_int2(across(v, e.x), across(v - 1, e.y));
      }
    }
    if (w == 0 && lane < 2) {  // the new boundaries: between px and x, between y and sy
      const bool one = lane == 0;
      const int p = one ? px : y, q = one ? x : sy;        // the cut edge
      const int tp = one ? y : px, tq = one ? sy : x;      // its ends' new neighbours
      const SegRec& G = one ? X : Y;
      if (one ? inx : iny) {
        const int v = max(p, q);
        const int at = (one ? rx : ry) + 1 + shift(v);
        lo2[at] = v;
        br2[at] = turned(G.base | (G.rev ? (int)0x80000000 : 0), v);
        nb2[at] = make_int2(v == p ? tp : tq, v == p ? tq : tp);
      }
    }
    st.S = S + (inx ? 1 : 0) + (iny ? 1 : 0) - (m1 != kNone) - (m2 != kNone);
    st.cur ^= 1;
    return L;
  }
};

// Warps that reverse.  Every one of them finds the span for itself, which
// costs issue slots of the other ants on the SM; iterations of 32 ants at
// n = 1k / 256 at 20k / 1,024 at 100k with 2, 3, 4, 5, 7 of them: 0.267 0.267
// 0.267 0.269 0.269 / 2.71 2.63 2.58 2.60 2.57 / 4.01 3.92 3.88 3.89 3.90 ms.
constexpr int kFlipWarps = 4;

// Shared scratch of the block search.
struct LsShared {
  int32_t gain[32];
  int mv[32][8];
  int qh, qn, nlog, changes, moves_round;
  int full;  // the table filled up: 4 * the move + 1 + exchanges of it that were done
  SegState tab;
  int64_t total, t_confirm, t_push;
};

// The block search's tour: a segment table ...
struct TableRep {
  static constexpr int kWarps = kFlipWarps;  // that apply a move, from warp 0 on
  const SegTour& T;
  SegState tab;  // the same on every thread

  __device__ __forceinline__ SegView view() const { return T.view(tab); }
  // {n1,n2},{n3,n4} -> {n1,n3},{n2,n4}; fwd: n2 is known to follow n1.  Below 0:
  // the table is full (nothing has changed)
  __device__ __forceinline__ int exchange(int n1, int n2, int n3, int n4, bool fwd, int w, LsStats& S) {
    if (!fwd) {
      const SegView V = T.view(tab);
      const SegRec g = V.rec(V.locate_w(n1));
      fwd = g.step(n1, !g.rev) == n2;
    }
    const int L = T.flip(tab, fwd ? n2 : n1, fwd ? n3 : n4, w, kWarps);
    S.flip += max(L, 0);
    return L;
  }
  __device__ __forceinline__ void post(LsShared& sh) const { sh.tab = tab; }
  __device__ __forceinline__ void fetch(const LsShared& sh, int w) {
    if (w >= kWarps) tab = sh.tab;  // (written again only after the next round's first barrier)
  }
};

// ... or, once that is full, arrays over source positions.
struct ArrayRep {
  static constexpr int kWarps = 1;
  ArrTour T;

  __device__ __forceinline__ const ArrTour& view() const { return T; }
  __device__ __forceinline__ int exchange(int n1, int n2, int n3, int n4, bool, int, LsStats& S) {
    (void)tour_move2(T, n1, n2, n3, n4, S);
    return 0;
  }
  __device__ __forceinline__ void post(LsShared&) const {}
  __device__ __forceinline__ void fetch(const LsShared&, int) {}
};

// The rounds of the block search, until the search ends or the table is full
// (sh.full).  In each, warp w evaluates the w-th queued node; entries are
// popped in queue order up to and including the first one whose evaluation
// found a move, which is applied.  Nothing changes the tour between the
// confirmed evaluations, so the result equals popping one node at a time.  The
// last warp does the queue's work -- pops, log, pushing the move's ends --
// while the others reverse.
template <bool TWO, class Rep>
__device__ __forceinline__ void ls_rounds(const LsEnv& E, Rep& rep, LsStats& S, LsShared& sh) {
  const int n = E.n, tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int W = blockDim.x >> 5;
  const bool keeper = w == W - 1;
  for (;;) {
    const int qh = sh.qh, qn = sh.qn;
    if (qn == 0 || sh.changes >= n || sh.full) {
      if (sh.full || sh.changes >= n || !E.verify || sh.moves_round == 0) break;
      const int nl = sh.nlog;  // verify round: queue again the nodes popped
      for (int i = tid; i < nl; i += blockDim.x) {
        const int x = E.logb[i];
        E.queue[i] = x;
        E.flags[x] = 1;
      }
      __syncthreads();
      if (tid == 0) {
        sh.qh = 0; sh.qn = nl; sh.nlog = 0; sh.moves_round = 0;
      }
      if (w == 0) S.verify++;
      __syncthreads();
      continue;
    }
    const int R = qn < W ? qn : W;
    const uint64_t t0 = (w == 0) ? global_ns() : 0;
    if (w < R) {
      int idx = qh + w;
      if (idx >= n) idx -= n;
      const int a = E.queue[idx];
      int mv[8];
      const int32_t g = eval_both<TWO>(rep.view(), a, E.oropt != 0, mv);
      if (lane == 0) {
        sh.gain[w] = g;
        if (g > 0)
          for (int t = 0; t < 8; ++t) sh.mv[w][t] = mv[t];
      }
    }
    __syncthreads();
    const unsigned bal = __ballot_sync(kFull, lane < R && sh.gain[lane] > 0);
    const int first = bal ? __ffs(bal) - 1 : R;
    const int cnt = bal ? first + 1 : R;  // queue entries popped this round
    const int* mv = sh.mv[bal ? first : 0];
    // a 2-opt move is one edge exchange, its first edge (mv[0], mv[1])
    // forward; an Or-opt move is two or three
    const bool two = mv[7] == 0;
    const int steps = bal ? (two ? 1 : (mv[6] ? 3 : 2)) : 0;
    if (keeper) {
      const uint64_t t1 = global_ns();
      int a = -1;
      bool first_pop = false;
      if (lane < cnt) {
        int idx = qh + lane;
        if (idx >= n) idx -= n;
        a = E.queue[idx];
        const uint8_t f = E.flags[a];
        first_pop = !(f & 2);
        E.flags[a] = (uint8_t)((f & ~1) | 2);
      }
      const unsigned fb = __ballot_sync(kFull, first_pop);
      const int nlog = sh.nlog;
      if (first_pop) E.logb[nlog + __popc(fb & ((1u << lane) - 1u))] = a;
      __syncwarp();
      int qh2 = qh + cnt;
      if (qh2 >= n) qh2 -= n;
      int qn2 = qn - cnt;
      const uint64_t t2 = global_ns();
      if (bal) qn2 = ls_push_warp(E, mv, two ? 4 : 6, qh2, qn2);
      if (lane == 0) {
        sh.t_confirm += (int64_t)(t2 - t1);
        sh.t_push += (int64_t)(global_ns() - t2);
        sh.nlog = nlog + __popc(fb);
        sh.qh = qh2;
        sh.qn = qn2;
        if (bal) {
          sh.total += sh.gain[first];
          sh.changes++;
          sh.moves_round++;
        }
      }
      for (int st = 1; st < steps; ++st) __syncthreads();
    } else {
      const uint64_t t1 = (w == 0) ? global_ns() : 0;
      S.t_eval += (int64_t)(t1 - t0);
      S.pops += cnt;
      int full = 0;
      for (int st = 0; st < steps; ++st) {
        if (st > 0) __syncthreads();
        const int n1 = st == 2 ? mv[4] : mv[0];
        const int n2 = st == 0 ? mv[1] : (st == 1 ? mv[4] : mv[2]);
        const int n3 = st == 0 ? (two ? mv[2] : mv[4]) : (st == 1 ? mv[3] : mv[1]);
        const int n4 = st == 0 ? (two ? mv[3] : mv[5]) : (st == 1 ? mv[2] : mv[5]);
        if (full || w >= Rep::kWarps) continue;
        const int L = rep.exchange(n1, n2, n3, n4, two, w, S);
        if (L < 0) full = 1 + st;
      }
      if (bal) {
        if (two)
          S.moves2++;
        else
          S.movesor++;
      }
      if (tid == 0) {
        rep.post(sh);
        if (full) sh.full = 4 * first + full;
        S.t_flip += (int64_t)(global_ns() - t1);
      }
    }
    __syncthreads();
    rep.fetch(sh, w);
  }
  __syncthreads();
}

// The search of ls_run by a block on one tour: ls_begin with the checklist,
// ls_rounds on the table, ls_end, each by every thread of the block.  When the
// rounds end with the table full (rare: the tables are sized for it not to),
// ls_to_arrays writes it out as arrays of source positions and applies the rest
// of the move that did not fit, and the rounds go on there with the same queue.
//
// (A launch lasts as long as its slowest ant, and an ant that one warp builds
// and searches again from the start takes several times as long as it had.
// Left to the array kernel instead, an iteration of 1,024 ants at n = 100,000
// took 36.6 ms with min_new_edges = 64 (53 ants' tables fill up) and 197 ms with
// 256 (963); going on takes 16.4 and 66.5 ms.  256 ants at n = 20,000 with
// 64-segment tables: 4.0 against 1.16 ms.)
__device__ __forceinline__ void ls_begin(const LsEnv& E, const int32_t* init, int ninit, LsShared& sh) {
  for (int i = threadIdx.x; i < ninit; i += blockDim.x) {
    const int x = init[i];
    E.queue[i] = x;
    E.flags[x] = 1;
  }
  if (threadIdx.x == 0) {
    sh.qh = 0; sh.qn = ninit; sh.nlog = 0; sh.changes = 0; sh.moves_round = 0; sh.full = 0;
    sh.total = 0; sh.t_confirm = 0; sh.t_push = 0;
  }
  __syncthreads();
}

// full: sh.full as the rounds left it; it is cleared.
__device__ __forceinline__ void ls_to_arrays(const SegView& V, ArrTour& T, int full, LsStats& S, LsShared& sh) {
  const int n = V.n, tid = threadIdx.x;
  const uint64_t t0 = tid == 0 ? global_ns() : 0;
  for (int r = 0; r < V.S; ++r) {
    const SegRec g = V.rec(r);
    for (int q = g.lo + tid; q <= g.hi; q += blockDim.x) {
      const int t = g.pos(q, n);
      T.route[t] = q;
      T.pos[q] = t;
    }
  }
  __syncthreads();
  if (tid < 32) {
    // an Or-opt move's exchanges from the one that did not fit on (ls.cuh: apply_or)
    const int* mv = sh.mv[full >> 2];
    const int done = (full & 3) - 1;
    if (mv[7] == 0) {
      (void)tour_move2(T, mv[0], mv[1], mv[2], mv[3], S);
    } else {
      if (done == 0) (void)tour_move2(T, mv[0], mv[1], mv[4], mv[5], S);
      if (done <= 1) (void)tour_move2(T, mv[0], mv[4], mv[3], mv[2], S);
      if (mv[6]) (void)tour_move2(T, mv[4], mv[2], mv[1], mv[5], S);
    }
  }
  if (tid == 0) {
    sh.full = 0;
    S.t_flip += (int64_t)(global_ns() - t0);
  }
  __syncthreads();
}

// Leaves the flags clean.  Returns the gain.
__device__ __forceinline__ int64_t ls_end(const LsEnv& E, LsStats& S, const LsShared& sh) {
  const int n = E.n, tid = threadIdx.x;
  const int qh = sh.qh, qn = sh.qn, nl = sh.nlog;
  for (int t = tid; t < qn; t += blockDim.x) {
    int i = qh + t;
    if (i >= n) i -= n;
    E.flags[E.queue[i]] = 0;
  }
  for (int i = tid; i < nl; i += blockDim.x) E.flags[E.logb[i]] = 0;
  S.t_confirm = sh.t_confirm;
  S.t_push = sh.t_push;
  __syncthreads();
  return sh.total;
}

}  // namespace faco
