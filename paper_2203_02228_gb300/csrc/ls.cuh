// ls.cuh -- warp-cooperative local search (Sec. 4.4, Alg 3), generic over
// the tour representation.
//
// Pop a node a from the checklist FIFO, scan its nearest-neighbour list for
// the best improving 2-opt move (successor side first, then predecessor
// side, strict '>'), flip the tour section, queue the four endpoints.  The
// scan is one warp: with k <= 16, lanes 0..15 take the successor-side moves
// of NN(a)[lane] and lanes 16..31 the predecessor-side moves; the warp
// arg-max with ties to the lowest order index is exactly the first strict
// maximum of the sequential loops.
//
// Readings shared with the oracle (decided independently there):
//   flip       reverse the forward span x..y, or the complementary span when
//              2*len > n (same cycle, opposite orientation);
//   queue      FIFO with an in-queue bit; a queued node is not queued twice;
//   verify     when the queue runs dry after a round that applied a move,
//              every node popped in that round is queued again (first-pop
//              order) and the search continues; stop after a clean round,
//              or after n applied moves (Alg 3's limit);
//   Or-opt     tried from a only when its 2-opt scan found nothing: move the
//              segment a..e (1..3 nodes following a) between the ends (u,v)
//              of a tour edge at b in NN(a) -- (b, succ b) then (pred b, b)
//              -- reversed first, then kept; u, v outside the segment and
//              {pred a, succ e}; applied as two or three edge exchanges.
//
// A Tour provides (device, lane-local unless noted): n, k; pos_of(x);
// succ(x), pred(x); adj(x, up) (succ when up, else pred, one code path for
// lanes that differ in direction); nbrs(x, pred, succ); walk(a, pred, s1,
// s2, s3) (the predecessor and three successors); coord(x); cand(x, s);
// cdist(x, s) (the cost of that candidate edge); and the warp-collective
// flip(x, y, S) (false when the representation ran out of capacity).
#pragma once

#include <climits>

#include "common.cuh"

namespace faco {

struct LsEnv {
  int n, oropt, verify;
  int32_t* queue;   // n entries, ring
  uint8_t* flags;   // n entries: bit0 queued, bit1 popped this round; zero on entry and exit
  int32_t* logb;    // n entries: nodes popped this round, first-pop order
};

struct LsStats {
  int32_t pops, moves2, movesor, verify;
  int64_t flip;
  int64_t t_eval, t_confirm, t_flip, t_push;  // device ns per phase (block search)
};

// The nodes before and after tour position t (warp-uniform t): no wrapping
// where t is not next to the route's ends.
__device__ __forceinline__ void route_walk(const int32_t* route, int n, int t, int& p, int& s1, int& s2, int& s3) {
  if (t >= 1 && t + 3 < n) {
    const int32_t* r = route + t;
    p = r[-1];
    s1 = r[1];
    s2 = r[2];
    s3 = r[3];
  } else {
    p = route[wrapn(t - 1, n)];
    s1 = route[wrapn(t + 1, n)];
    s2 = route[wrapn(t + 2, n)];
    s3 = route[wrapn(t + 3, n)];
  }
}

// Explicit tour: route[t] = node at position t, pos = inverse.  Nodes are
// node ids (with node-indexed xy/cn) or source positions (with the
// source-ordered copies); cn rows are `stride` entries apart.
struct ArrTour {
  int n, k;
  int32_t* route;
  int32_t* pos;
  const int2* xy;       // coordinates by node
  const int32_t* cn;    // candidate lists by node [n][stride]
  int stride;
  const int32_t* cd;    // their EUC_2D costs, same layout
  __device__ __forceinline__ int pos_of(int x) const { return pos[x]; }
  __device__ __forceinline__ int at_off(int p, int d) const {
    p += d;
    if (p >= n) p -= n;
    if (p < 0) p += n;
    return route[p];
  }
  __device__ __forceinline__ int succ(int x) const { return at_off(pos[x], 1); }
  __device__ __forceinline__ int succ_w(int x) const { return succ(x); }  // warp-uniform x
  __device__ __forceinline__ int pred(int x) const { return at_off(pos[x], -1); }
  __device__ __forceinline__ int adj(int x, bool up) const { return at_off(pos[x], up ? 1 : -1); }
  __device__ __forceinline__ void nbrs(int x, int& p, int& s) const {
    const int t = pos[x];
    p = at_off(t, -1);
    s = at_off(t, 1);
  }
  __device__ __forceinline__ void walk(int a, int& p, int& s1, int& s2, int& s3) const {
    route_walk(route, n, pos[a], p, s1, s2, s3);
  }
  __device__ __forceinline__ int2 coord(int x) const { return xy[x]; }
  __device__ __forceinline__ int cand(int x, int s) const { return cn[(size_t)x * stride + s]; }
  __device__ __forceinline__ int cdist(int x, int s) const { return cd[(size_t)x * stride + s]; }

  // Reverse the forward span x..y (or its complement when longer than n/2).
  __device__ __forceinline__ bool flip(int x, int y, LsStats& S) {
    const int lane = lane_id();
    int i = pos[x], j = pos[y];
    __syncwarp();  // every lane has read i and j before a position moves
    int L = j - i;
    if (L < 0) L += n;
    L += 1;
    if (2 * L > n) {
      const int i2 = (j + 1 == n) ? 0 : j + 1;
      const int j2 = (i == 0) ? n - 1 : i - 1;
      i = i2;
      j = j2;
      L = n - L;
    }
    const int half = L >> 1;
    constexpr int U = 4;
    for (int t0 = 0; t0 < half; t0 += 32 * U) {
      int ia[U], ib[U], va[U], vb[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int t = t0 + lane + 32 * u;
        ia[u] = -1;
        if (t < half) {
          ia[u] = i + t;
          if (ia[u] >= n) ia[u] -= n;
          ib[u] = j - t;
          if (ib[u] < 0) ib[u] += n;
          va[u] = route[ia[u]];
          vb[u] = route[ib[u]];
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (ia[u] >= 0) {
          route[ia[u]] = vb[u];
          route[ib[u]] = va[u];
          pos[vb[u]] = ia[u];
          pos[va[u]] = ib[u];
        }
      }
    }
    __syncwarp();
    S.flip += L;
    return true;
  }
};

// Exchange tour edges {n1,n2},{n3,n4} for {n1,n3},{n2,n4}: with n1->n2 a
// forward edge this is the Alg 3 move (n1,n2,n3,n4) -> flip n2..n3,
// otherwise the move (n2,n1,n4,n3) -> flip n1..n4.  Warp-collective.
template <class Tour>
__device__ __forceinline__ bool tour_move2(Tour& T, int n1, int n2, int n3, int n4, LsStats& S) {
  if (T.succ_w(n1) == n2) return T.flip(n2, n3, S);
  return T.flip(n1, n4, S);
}

// Both scans from a in one pass over NN(a) (one lookup of a, one of each
// neighbour b): the best 2-opt move if one gains, else (do_or) the best
// Or-opt move -- the same decision as scanning one after the other.  Returns
// the gain (0: none) and the move on every lane: mv[7] = 0 for 2-opt
// (mv[0..3]), 1 for Or-opt (mv[0..6]).
// Lane layout: with k <= 16 (TWO = false), lane = side * 16 + s (side 0: the
// edge (b, succ b), side 1: (pred b, b)); with k > 16 (TWO), lane = s and the
// two sides are two passes.  Lanes beyond k repeat entry 0 and are left out
// at the end, so that nothing diverges.  The loads that do not depend on the
// walk from a (the candidate row, b's coordinates) are issued before it; the
// move is rebuilt from the winning lane's registers.
// Bound by latency while few warps of an SM evaluate and by instruction
// issue while all do, so the costs are branch-free (euc2d_near) and run side
// by side, the choice among the moves is made of maxima and selects, both
// sides share one piece of code (swapping the ends of the edge at b only
// swaps the two orientations of an Or-opt move), no index is divided by k,
// and with TWO = false the lanes of the two sides share costs: six per lane
// instead of eight.  Of the slowest ants' time at n = 100,000 it took 2,420 us
// of 5,920 with a branch per cost, 1,375 of 3,590 branch-free, 1,046 of 3,290 in
// this form.
template <bool TWO, class Tour>
__device__ __forceinline__ int32_t eval_both(const Tour& T, int a, bool do_or, int (&mv)[8]) {
  const int n = T.n, k = T.k, lane = lane_id();
  do_or = do_or && n >= 8;
  const int s = TWO ? lane : (lane & 15);
  const bool live = s < k;
  const int sl = live ? s : 0;
  const int b = T.cand(a, sl);
  const int d_ab = T.cdist(a, sl);  // = euc2d(xa, xb), kept with the lists
  const int2 xb = T.coord(b);
  int p, s1, s2 = a, s3 = a;
  if (do_or)
    T.walk(a, p, s1, s2, s3);
  else
    T.nbrs(a, p, s1);
  const int2 xa = T.coord(a), x1 = T.coord(s1), xp = T.coord(p);
  int2 x2 = xa, x3 = xa;
  if (do_or) {
    x2 = T.coord(s2);
    x3 = T.coord(s3);
  }
  // b's tour neighbour on this lane's side (pass 0), and for k > 16 the
  // predecessor for pass 1
  int bn0, bn1 = a;
  if (TWO)
    T.nbrs(b, bn1, bn0);
  else
    bn0 = T.adj(b, lane < 16);
  const int2 xbn0 = T.coord(bn0), xbn1 = TWO ? T.coord(bn1) : xa;
  // the costs within a's tour neighbourhood are the same on every lane: one
  // lane computes the j-th, shuffles share them
  //   0 d(a,s1)  1 d(p,a)  2 d(p,s1)  3 d(s1,s2)  4 d(p,s2)  5 d(s2,s3)  6 d(p,s3)
  const int j = TWO ? lane : (lane & 15);
  int2 cu, cv;
  {
    const bool up = j == 1 || j == 2 || j == 4 || j == 6, va = j == 1, v2 = j == 3 || j == 4, v3 = j == 5 || j == 6;
    cu.x = up ? xp.x : (j == 3 ? x1.x : (j == 5 ? x2.x : xa.x));
    cu.y = up ? xp.y : (j == 3 ? x1.y : (j == 5 ? x2.y : xa.y));
    cv.x = va ? xa.x : (v2 ? x2.x : (v3 ? x3.x : x1.x));
    cv.y = va ? xa.y : (v2 ? x2.y : (v3 ? x3.y : x1.y));
  }
  // the lane's best move: a gaining 2-opt move counts kTwoOpt more than its
  // gain, so that it beats every Or-opt move; code = l * 4 + orientation * 2
  // + side (l = 0: 2-opt)
  constexpr int32_t kTwoOpt = 1 << 28;
  int32_t best = 0;
  int bcode = 0, bbn = bn0;
#pragma unroll
  for (int pass = 0; pass < (TWO ? 2 : 1); ++pass) {
    const bool hi = TWO ? pass != 0 : lane >= 16;  // side 1
    const int bn = pass == 0 ? bn0 : bn1;
    const int2 xbn = pass == 0 ? xbn0 : xbn1;
    // 0 d(b,bn)  1 d(bn,s1)  2 d(bn,a)  3 d(bn,s2), and
    //   TWO:   4 d(b,s1)  5 d(b,s2)  6 d(bn,p)  7 the j-th of a's neighbourhood
    //   else:  4 d(b,s1) on side 0, d(bn,p) on side 1
    //          5 d(b,s2) on side 0, the j-th of a's neighbourhood on side 1
    int2 u4 = xb, v4 = x1, u5 = xb, v5 = x2;
    if (!TWO) {
      u4.x = hi ? xbn.x : xb.x;
      u4.y = hi ? xbn.y : xb.y;
      v4.x = hi ? xp.x : x1.x;
      v4.y = hi ? xp.y : x1.y;
      u5.x = hi ? cu.x : xb.x;
      u5.y = hi ? cu.y : xb.y;
      v5.x = hi ? cv.x : x2.x;
      v5.y = hi ? cv.y : x2.y;
    }
    bool big = false;
    int32_t c0 = euc2d_near(xb, xbn, big), c1 = euc2d_near(xbn, x1, big), c2 = euc2d_near(xbn, xa, big),
            c3 = euc2d_near(xbn, x2, big), c4 = euc2d_near(u4, v4, big), c5 = euc2d_near(u5, v5, big), c6 = 0,
            c7 = 0;
    if (TWO) {
      c6 = euc2d_near(xbn, xp, big);
      c7 = euc2d_near(cu, cv, big);
    }
    if (__any_sync(kFull, big)) {  // an edge of 2^21 or more: the exact steps, one cost after the other
#pragma unroll 1
      for (int t = 0; t < (TWO ? 8 : 6); ++t) {
        const int2 u = t == 0 ? xb : t == 4 ? u4 : t == 5 ? u5 : t == 7 ? cu : xbn;
        const int2 v = t == 0 ? xbn : t == 1 ? x1 : t == 2 ? xa : t == 3 ? x2 : t == 4 ? v4 : t == 5 ? v5
                       : t == 6 ? xp : cv;
        const int32_t d = euc2d_m(sqdist(u, v));
        if (t == 0) c0 = d;
        if (t == 1) c1 = d;
        if (t == 2) c2 = d;
        if (t == 3) c3 = d;
        if (t == 4) c4 = d;
        if (t == 5) c5 = d;
        if (t == 6) c6 = d;
        if (t == 7) c7 = d;
      }
    }
    const int32_t nbh = TWO ? c7 : c5;
    const int nb0 = TWO ? 0 : 16;
    const int32_t c_b1 = TWO ? c4 : __shfl_sync(kFull, c4, s), c_b2 = TWO ? c5 : __shfl_sync(kFull, c5, s);
    const int32_t c_z = hi ? (TWO ? c6 : c4) : c1;  // d(bn, s1) on side 0, d(bn, p) on side 1
    const int32_t d_as = __shfl_sync(kFull, nbh, nb0), d_ap = __shfl_sync(kFull, nbh, nb0 + 1);
    // gains in 32 bits: each is a signed sum of at most six EUC_2D costs of
    // coordinates below 2^24 (each cost below 2^25)
    int32_t v = 0;
    int l = 0, o = 0;
    if (do_or) {
      const int32_t rem1 = d_ap + d_as - __shfl_sync(kFull, nbh, nb0 + 2);
      const int32_t rem2 = d_ap + __shfl_sync(kFull, nbh, nb0 + 3) - __shfl_sync(kFull, nbh, nb0 + 4);
      const int32_t rem3 = d_ap + __shfl_sync(kFull, nbh, nb0 + 5) - __shfl_sync(kFull, nbh, nb0 + 6);
      // insertion of a..e between the ends of the edge {b, bn}: one form
      // joins b to e and bn to a, the other b to a and bn to e; the reversed
      // one (orientation 0) is the first on side 0, the second on side 1
      const bool bad1 = (b == p) | (bn == p) | (bn == a) | (b == s1) | (bn == s1);
      const bool bad2 = bad1 | (b == s2) | (bn == s2);
      const bool bad3 = bad2 | (b == s3) | (bn == s3);
      const int32_t be2 = rem2 + c0 - c_b1 - c2, ba2 = rem2 + c0 - d_ab - c1;
      const int32_t be3 = rem3 + c0 - c_b2 - c2, ba3 = rem3 + c0 - d_ab - c3;
      const bool o2 = hi ? be2 > ba2 : ba2 > be2, o3 = hi ? be3 > ba3 : ba3 > be3;
      const int32_t v1 = bad1 ? 0 : rem1 + c0 - d_ab - c2;  // one node: one form only
      const int32_t v2 = bad2 ? 0 : max(be2, ba2), v3 = bad3 ? 0 : max(be3, ba3);
      v = max(max(v1, v2), max(v3, 0));
      l = v == v1 ? 1 : (v == v2 ? 2 : 3);
      o = v == v1 ? 0 : (v == v2 ? o2 : o3);
    }
    const int32_t d_out = hi ? d_ap : d_as;
    const int32_t g = d_out + c0 - d_ab - c_z;
    const bool t2 = (d_out > d_ab) & (g > 0);
    v = t2 ? g + kTwoOpt : v;
    v = live ? v : 0;
    const int code = (t2 ? 0 : l * 4 + o * 2) + (hi ? 1 : 0);
    if (pass == 0) {
      best = v;
      bcode = code;
    } else if (v > best || (v == best && (code >> 2) < (bcode >> 2))) {  // scan order: l, entry, side
      best = v;
      bcode = code;
      bbn = bn;
    }
  }
  const int32_t gm = __reduce_max_sync(kFull, best);
  mv[7] = gm < kTwoOpt;
  if (gm == 0) return 0;
  unsigned own = __ballot_sync(kFull, best == gm);
  if (own & (own - 1)) {  // equal gains: the first in scan order
    const int l = bcode >> 2, side = bcode & 1;
    const int idx = l == 0 ? side * k + s : (((l - 1) * k + s) * 2 + side) * 2 + ((bcode >> 1) & 1);
    const unsigned im = __reduce_min_sync(kFull, best == gm ? (unsigned)idx : 0xFFFFFFFFu);
    own = __ballot_sync(kFull, best == gm && (unsigned)idx == im);
  }
  const int wl = __ffs(own) - 1;
  const int bw = __shfl_sync(kFull, b, wl), bnw = __shfl_sync(kFull, bbn, wl);
  const int cw = __shfl_sync(kFull, bcode, wl);
  const int side = cw & 1;
  if (gm >= kTwoOpt) {
    mv[0] = side ? p : a;
    mv[1] = side ? a : s1;
    mv[2] = side ? bnw : bw;
    mv[3] = side ? bw : bnw;
    return gm - kTwoOpt;
  }
  const int l = cw >> 2;
  mv[0] = p; mv[1] = a; mv[2] = l == 1 ? a : (l == 2 ? s1 : s2);
  mv[3] = l == 1 ? s1 : (l == 2 ? s2 : s3); mv[4] = side ? bnw : bw; mv[5] = side ? bw : bnw;
  mv[6] = (cw >> 1) & 1;
  return gm;
}

// The 3-opt segment exchange of the initial tour (Sec. 4.3: 2-opt and
// 3-opt following Bentley; the move and its search are a reading): the
// tour edges (a,t2), (b,b'), (c,c') become (a,b'), (b,c'), (c,t2), so that,
// walking from a towards t2, a [t2..b] [b'..c] c' turns into
// a [b'..c] [t2..b] c' -- two adjacent sections swap places, neither
// reversed.  t2 is a's successor (dir 0) or predecessor (dir 1); b' runs
// over NN(a) with g1 = d(a,t2) - d(a,b') > 0 and b is the node before b' in
// the walking direction; c' runs over NN(b) with g2 = g1 + d(b,b') -
// d(b,c') > 0 and c is the node before c'; valid when, counted from a in
// the walking direction, 1 <= r(b) < r(c) <= n - 2.  gain = g2 + d(c,c') -
// d(c,t2); the first strictly largest gain in the order (dir, b', c') wins.
// The warp takes the (dir, b', c') combinations 32 at a time, lane = order
// index mod 32.  Returns the gain (0: none) and mv = {a, t2, b, b', c, c'}.
// Warp-collective; the tour's nodes and coordinates as the Tour names them.
template <class Tour>
__device__ __forceinline__ int64_t eval_or3(const Tour& T, int a, int mv[6]) {
  const int n = T.n, k = T.k, lane = lane_id();
  if (n < 8) return 0;
  int p, s1;
  T.nbrs(a, p, s1);
  const int2 xa = T.coord(a), xs = T.coord(s1), xp = T.coord(p);
  const int d_as = euc2d(xa, xs), d_ap = euc2d(xa, xp);
  const int pa = T.pos_of(a);
  const int kk = k * k, total = 2 * kk;
  int32_t best = 0;
  int bi = INT_MAX, bb = -1, bb1 = -1, bc = -1, bc1 = -1;
  for (int idx = lane; idx < total; idx += 32) {
    const int dir = idx >= kk ? 1 : 0;
    const int r = idx - dir * kk;
    const int i = r / k, j = r - i * k;
    const int2 xt2 = dir ? xp : xs;
    const int g1 = (dir ? d_ap : d_as) - T.cdist(a, i);
    if (g1 <= 0) continue;
    const int b1 = T.cand(a, i);
    const int b = T.adj(b1, dir != 0);  // dir 0: pred(b'), dir 1: succ(b')
    const int2 xb = T.coord(b), xb1 = T.coord(b1);
    const int g2 = g1 + euc2d(xb, xb1) - T.cdist(b, j);
    if (g2 <= 0) continue;
    const int c1 = T.cand(b, j);
    const int c = T.adj(c1, dir != 0);
    int rb = dir ? pa - T.pos_of(b) : T.pos_of(b) - pa;
    int rc = dir ? pa - T.pos_of(c) : T.pos_of(c) - pa;
    if (rb < 0) rb += n;
    if (rc < 0) rc += n;
    if (!(rb >= 1 && rb < rc && rc <= n - 2)) continue;
    const int2 xc = T.coord(c), xc1 = T.coord(c1);
    const int32_t g = g2 + euc2d(xc, xc1) - euc2d(xc, xt2);
    if (g > best) {  // idx grows along the lane's loop: ties keep the earlier
      best = g;
      bi = idx;
      bb = b;
      bb1 = b1;
      bc = c;
      bc1 = c1;
    }
  }
  int32_t g = best > 0 ? best : 0;
  int32_t wi = best > 0 ? bi : INT_MAX;
  warp_max_gain(g, wi);
  if (g <= 0) return 0;
  const int wl = wi & 31;
  mv[0] = a;
  mv[1] = wi >= kk ? p : s1;
  mv[2] = __shfl_sync(kFull, bb, wl);
  mv[3] = __shfl_sync(kFull, bb1, wl);
  mv[4] = __shfl_sync(kFull, bc, wl);
  mv[5] = __shfl_sync(kFull, bc1, wl);
  return g;
}

// Applies an Or-opt move {p,a,e,q,u,v,kept} as edge exchanges.
template <class Tour>
__device__ __forceinline__ bool apply_or(Tour& T, const int* mv, LsStats& S) {
  if (!tour_move2(T, mv[0], mv[1], mv[4], mv[5], S)) return false;  // {p,a},{u,v} -> {p,u},{a,v}
  if (!tour_move2(T, mv[0], mv[4], mv[3], mv[2], S)) return false;  // {p,u},{q,e} -> {p,q},{u,e}
  if (mv[6] && !tour_move2(T, mv[4], mv[2], mv[1], mv[5], S)) return false;  // {u,e},{a,v} -> {u,a},{e,v}
  return true;
}

// Queue the np (<= 32) nodes x[0..np) in order, each only if it is not
// queued yet (and not already pushed earlier in the list): lane t handles
// x[t].  Warp-collective; every lane receives the new qn.
__device__ __forceinline__ int ls_push_warp(const LsEnv& E, const int* x, int np, int qh, int qn) {
  const int lane = lane_id();
  int node = -1 - lane;  // distinct dummies for idle lanes
  if (lane < np) node = x[lane];
  const unsigned same = __match_any_sync(kFull, node);
  const bool leader = (same & ((1u << lane) - 1u)) == 0;  // first lane with this node
  uint8_t f = 0;
  if (lane < np && leader) f = E.flags[node];
  const bool push = lane < np && leader && !(f & 1);
  const unsigned bal = __ballot_sync(kFull, push);
  if (push) {
    E.flags[node] = f | 1;
    int t = qh + qn + __popc(bal & ((1u << lane) - 1u));
    if (t >= E.n) t -= E.n;
    if (t >= E.n) t -= E.n;
    E.queue[t] = node;
  }
  __syncwarp();
  return qn + __popc(bal);
}

// Runs the search from the checklist init[0..ninit) (distinct nodes).
// Returns the total gain (old length - new length), or -1 if the tour
// representation ran out of capacity (flags are left clean either way).
template <bool TWO, class Tour>
__device__ __forceinline__ int64_t ls_run(const LsEnv& E, Tour& T, const int32_t* init, int ninit,
                                          LsStats& S) {
  const int n = E.n, lane = lane_id();
  for (int i = lane; i < ninit; i += 32) {
    const int x = init[i];
    E.queue[i] = x;
    E.flags[x] = 1;
  }
  __syncwarp();
  int qh = 0, qn = ninit, nlog = 0, changes = 0, moves_round = 0;
  int64_t total = 0;
  bool ok = true;
  for (;;) {
    while (qn > 0 && changes < n) {
      const int a = E.queue[qh];
      qh = (qh + 1 == n) ? 0 : qh + 1;
      --qn;
      const uint8_t f = E.flags[a];
      __syncwarp();
      if (lane == 0) {
        E.flags[a] = (uint8_t)((f & ~1) | 2);
        if (!(f & 2)) E.logb[nlog] = a;
      }
      if (!(f & 2)) ++nlog;
      __syncwarp();
      S.pops++;
      int mv[8];
      const int32_t g = eval_both<TWO>(T, a, E.oropt != 0, mv);
      if (g > 0) {
        if (mv[7] == 0) {
          ok = T.flip(mv[1], mv[2], S);
          S.moves2++;
        } else {
          ok = apply_or(T, mv, S);
          S.movesor++;
        }
        if (!ok) break;
        qn = ls_push_warp(E, mv, mv[7] == 0 ? 4 : 6, qh, qn);
        total += g;
        ++changes;
        ++moves_round;
      }
    }
    if (!ok || changes >= n || !E.verify || moves_round == 0) break;
    // verify round: queue again every node popped in the last round
    S.verify++;
    for (int i = lane; i < nlog; i += 32) {
      const int x = E.logb[i];
      E.queue[i] = x;
      E.flags[x] = 1;
    }
    __syncwarp();
    qh = 0;
    qn = nlog;
    nlog = 0;
    moves_round = 0;
  }
  // leave the flags clean for the next search
  for (int t = lane; t < qn; t += 32) {
    int i = qh + t;
    if (i >= n) i -= n;
    E.flags[E.queue[i]] = 0;
  }
  for (int i = lane; i < nlog; i += 32) E.flags[E.logb[i]] = 0;
  __syncwarp();
  return ok ? total : -1;
}

}  // namespace faco
