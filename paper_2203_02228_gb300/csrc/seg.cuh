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
// When the table is full the reversal reports failure and the ant is redone
// on explicit arrays by the array kernel (same result, more memory traffic).
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
// boundaries, 16 bytes each, then the count and the buffer in use.
constexpr size_t kSegBytes = 2 * (sizeof(int2) + 2 * sizeof(int32_t));
static_assert(kSegBytes == 2 * sizeof(Seg), "construction's list of runs takes one buffer's room");
__host__ __device__ constexpr size_t segtab_bytes(int cap) { return (size_t)(cap + 1) * kSegBytes + 16; }

struct SegTab {
  char* mem;         // buffers 0 and 1
  int32_t* hdr;      // [0] segments, [1] buffer in use
  int cap;
};

__device__ __forceinline__ SegTab segtab_at(char* base, int cap) {
  SegTab T;
  T.mem = base;
  T.hdr = reinterpret_cast<int32_t*>(base + (size_t)(cap + 1) * kSegBytes);
  T.cap = cap;
  return T;
}

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

// Tour over the segment table: what changes it.
struct SegTour {
  int n, k, kw;
  SegTab T;
  const int2* xy;
  const int32_t* cn;
  const int32_t* cd;

  __device__ __forceinline__ char* buffer(int which) const {
    return T.mem + (which ? (size_t)(T.cap + 1) * (kSegBytes / 2) : 0);
  }
  __device__ __forceinline__ SegView view() const {
    const int m = T.cap + 1;
    char* b = buffer(T.hdr[1]);
    SegView v;
    v.n = n;
    v.k = k;
    v.kw = kw;
    v.S = T.hdr[0];
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
  __device__ __forceinline__ void build(const Seg* runs, int S) const {
    const int m = T.cap + 1;
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
    __syncthreads();  // the count and buffer number may lie in the runs' room
    if (threadIdx.x == 0) {
      T.hdr[0] = S;
      T.hdr[1] = 0;
    }
    __syncthreads();
  }

  // Reverse the forward span x..y, or its complement when longer than n/2
  // (the array rule, entry for entry).  Returns the nodes reversed, or -1
  // when the table is full.  One warp; V: the current view.
  //
  // Bound by the latency of one warp's dependent steps: the search for x and
  // y, the one for the nodes before and after them (only where a cut falls
  // on a boundary), and the copying pass, S / 32 independent steps.  (The
  // table it replaced kept an order by tour position beside the one by
  // source position, shifted both for every cut and merge, and cut segments
  // at position 0: with it the iteration of 1,024 ants at n = 100k took
  // 6.3 ms and 2,048 ants at n = 200k 8.6 ms, with this one 4.8 and 6.0 ms.)
  // Inlined, like everything else in the block kernel: it makes no calls.
  __device__ __forceinline__ int flip(const SegView& V, int x, int y) const {
    const int lane = lane_id();
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
    // at most two boundaries more: refuse before touching the table, which
    // then still holds the tour
    if (S + 2 > T.cap) return -1;
    int rp = rx, rs = ry;  // segments of px and sy
    bool revp = X.rev, revs = Y.rev;
    if (!inx || !iny) {
      V.locate2_w(px, sy, rp, rs);
      revp = V.br[rp] < 0;
      revs = V.br[rs] < 0;
    }
    // new boundaries where a cut edge lies inside a segment; boundaries that
    // go: the new edge {px, y} or {x, sy} joins source neighbours, each at the
    // end of its segment that faces the other
    constexpr int kNone = INT_MAX;
    const int c1 = inx ? max(px, x) : kNone, c2 = iny ? max(y, sy) : kNone;
    const int m1 = (revp != Y.rev && y - px == (revp ? -1 : 1)) ? max(px, y) : kNone;
    const int m2 = (X.rev != revs && sy - x == (X.rev ? 1 : -1)) ? max(x, sy) : kNone;
    // (boundaries of the new table) - (of the old one) below node v
    auto shift = [&](int v) { return (c1 < v) + (c2 < v) - (m1 < v) - (m2 < v); };
    // the map of a segment that contains node v, after the reversal
    auto turned = [&](int b, int v) {
      const int base = b & 0x7fffffff;
      int d = wrapn(b < 0 ? base - v : base + v, n) - i;
      if (d < 0) d += n;
      if (d >= L) return b;
      int nbase = sum - base;
      if (nbase < 0) nbase += n;
      return nbase | (~b & (int)0x80000000);
    };
    const int m = T.cap + 1, cur = T.hdr[1];
    char* out = buffer(cur ^ 1);
    int2* nb2 = reinterpret_cast<int2*>(out);
    int32_t* lo2 = reinterpret_cast<int32_t*>(out + (size_t)m * sizeof(int2));
    int32_t* br2 = lo2 + m;
#pragma unroll 2
    for (int r = lane; r <= S; r += 32) {
      const int v = V.lo[r];
      const int b = V.br[r];
      const int2 e = V.nb[r];
      if (v != m1 && v != m2) {
        const int w = r + shift(v);
        lo2[w] = v;
        br2[w] = turned(b, v);
        nb2[w] = e;
      }
    }
    __syncwarp();  // the neighbours below overwrite copied ones
    // lanes 0..3: the ends px, x, y, sy of the two cut edges get their new
    // neighbours y, sy, px, x, in the slot of the side that faced the cut
    if (lane < 4) {
      const bool first = lane < 2;  // an end of the cut {px, x}
      const int o = lane == 0 ? px : (lane == 1 ? x : (lane == 2 ? y : sy));
      const int to = lane == 0 ? y : (lane == 1 ? sy : (lane == 2 ? px : x));
      const bool hiside = lane == 0 ? !revp : (lane == 1 ? X.rev : (lane == 2 ? !Y.rev : revs));
      const int ro = lane == 0 ? rp : (lane == 1 ? rx : (lane == 2 ? ry : rs));
      const bool in = first ? inx : iny;
      const int v = hiside ? o + 1 : o;  // the boundary
      const int w = ro + ((in || hiside) ? 1 : 0) + shift(v);
      const bool gone = ((lane == 0 || lane == 2) ? m1 : m2) != kNone;
      if (!gone) {
        if (hiside)
          nb2[w].y = to;
        else
          nb2[w].x = to;
      }
      // lanes 1 and 2 also write the new boundary of their cut
      if (in && (lane == 1 || lane == 2)) {
        lo2[w] = v;
        br2[w] = turned((first ? X.base | (X.rev ? (int)0x80000000 : 0) : Y.base | (Y.rev ? (int)0x80000000 : 0)), v);
      }
    }
    if (lane == 0) {
      T.hdr[0] = S + (inx ? 1 : 0) + (iny ? 1 : 0) - (m1 != kNone) - (m2 != kNone);
      T.hdr[1] = cur ^ 1;
    }
    __syncwarp();
    return L;
  }
};

// Shared scratch of the block search.
struct LsShared {
  int32_t gain[32];
  int mv[32][8];
  int qh, qn, nlog, changes, moves_round, fail;
  int64_t total;
};

// The search of ls_run by a block of W warps on one tour: each round, warp w
// evaluates the w-th queued node; entries are popped in queue order up to
// and including the first one whose evaluation found a move, which warp 0
// applies.  Nothing changes the tour between the confirmed evaluations, so
// the result equals popping one node at a time.  Must be called by every
// thread of the block.  Returns the gain, or -1 when the table filled up
// (flags are left clean either way; the caller has the ant redone on arrays).
template <bool TWO>
__device__ __forceinline__ int64_t ls_run_block(const LsEnv& E, const SegTour& T, const int32_t* init, int ninit,
                                                LsStats& S, LsShared& sh) {
  const int n = E.n, tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int W = blockDim.x >> 5;
  for (int i = tid; i < ninit; i += blockDim.x) {
    const int x = init[i];
    E.queue[i] = x;
    E.flags[x] = 1;
  }
  if (tid == 0) {
    sh.qh = 0; sh.qn = ninit; sh.nlog = 0; sh.changes = 0; sh.moves_round = 0; sh.fail = 0;
    sh.total = 0;
  }
  __syncthreads();
  for (;;) {
    const int qh = sh.qh, qn = sh.qn;
    if (qn == 0 || sh.changes >= n || sh.fail) {
      if (sh.fail || sh.changes >= n || !E.verify || sh.moves_round == 0) break;
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
      const int32_t g = eval_both<TWO>(T.view(), a, E.oropt != 0, mv);
      if (lane == 0) {
        sh.gain[w] = g;
        if (g > 0)
          for (int t = 0; t < 8; ++t) sh.mv[w][t] = mv[t];
      }
    }
    __syncthreads();
    if (w == 0) {
      const uint64_t t1 = global_ns();
      S.t_eval += (int64_t)(t1 - t0);
      const unsigned bal = __ballot_sync(kFull, lane < R && sh.gain[lane] > 0);
      const int first = bal ? __ffs(bal) - 1 : R;
      const int cnt = bal ? first + 1 : R;  // queue entries popped this round
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
      if (first_pop) E.logb[sh.nlog + __popc(fb & ((1u << lane) - 1u))] = a;
      S.pops += cnt;
      __syncwarp();
      int qh2 = qh + cnt;
      if (qh2 >= n) qh2 -= n;
      int qn2 = qn - cnt;
      const uint64_t t2 = global_ns();
      S.t_confirm += (int64_t)(t2 - t1);
      if (bal) {  // apply the first move found, queue its endpoints
        const int* mv = sh.mv[first];
        const bool two = mv[7] == 0;
        // a 2-opt move is one edge exchange, its first edge (mv[0], mv[1])
        // forward; an Or-opt move is two or three
        const int steps = two ? 1 : (mv[6] ? 3 : 2);
        for (int st = 0; st < steps; ++st) {
          const int n1 = st == 2 ? mv[4] : mv[0];
          const int n2 = st == 0 ? mv[1] : (st == 1 ? mv[4] : mv[2]);
          const int n3 = st == 0 ? (two ? mv[2] : mv[4]) : (st == 1 ? mv[3] : mv[1]);
          const int n4 = st == 0 ? (two ? mv[3] : mv[5]) : (st == 1 ? mv[2] : mv[5]);
          const SegView V = T.view();
          bool fwd = two;
          if (!two) {
            const SegRec g = V.rec(V.locate_w(n1));
            fwd = g.step(n1, !g.rev) == n2;
          }
          const int L = T.flip(V, fwd ? n2 : n1, fwd ? n3 : n4);
          if (L < 0) {  // the table is full
            if (lane == 0) sh.fail = 1;
            break;
          }
          S.flip += L;
        }
        if (two)
          S.moves2++;
        else
          S.movesor++;
        const uint64_t t3 = global_ns();
        S.t_flip += (int64_t)(t3 - t2);
        qn2 = ls_push_warp(E, mv, two ? 4 : 6, qh2, qn2);
        if (lane == 0) {
          sh.total += sh.gain[first];
          sh.changes++;
          sh.moves_round++;
        }
        S.t_push += (int64_t)(global_ns() - t3);
      }
      if (lane == 0) {
        sh.nlog += __popc(fb);
        sh.qh = qh2;
        sh.qn = qn2;
      }
      __syncwarp();
    }
    __syncthreads();
  }
  __syncthreads();
  const int qh = sh.qh, qn = sh.qn, nl = sh.nlog;
  for (int t = tid; t < qn; t += blockDim.x) {
    int i = qh + t;
    if (i >= n) i -= n;
    E.flags[E.queue[i]] = 0;
  }
  for (int i = tid; i < nl; i += blockDim.x) E.flags[E.logb[i]] = 0;
  __syncthreads();
  return sh.fail ? -1 : sh.total;
}

}  // namespace faco
