// knn.cu -- candidate and backup lists (Sec. 4.1) with a uniform grid.
//
// For every node u the k + bl nearest other nodes ordered by (squared
// distance, node id): the first k form the candidate list, the next bl the
// backup list; eta = 1/d for the candidates (Sec. 2.1, d = EUC_2D cost).
// Points are bucketed into square cells (about two points per cell); a
// query takes blocks of cells around its own cell, until k + bl points are
// strictly closer than the nearest point that could lie outside the block,
// so the result is exact.
#include <climits>

#include "common.cuh"
#include "launch.h"

namespace faco {

namespace {

__device__ __forceinline__ void bbox_add(int2 p, int& mnx, int& mny, int& mxx, int& mxy, int& bad) {
  mnx = min(mnx, p.x); mny = min(mny, p.y); mxx = max(mxx, p.x); mxy = max(mxy, p.y);
  bad |= (p.x < 0 || p.y < 0 || p.x >= (1 << 24) || p.y >= (1 << 24));
}

// Warp reduction of a partial bounding box into out5 (atomics).
__device__ __forceinline__ void bbox_flush(int mnx, int mny, int mxx, int mxy, int bad, int32_t* out5) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mnx = min(mnx, __shfl_xor_sync(kFull, mnx, o));
    mny = min(mny, __shfl_xor_sync(kFull, mny, o));
    mxx = max(mxx, __shfl_xor_sync(kFull, mxx, o));
    mxy = max(mxy, __shfl_xor_sync(kFull, mxy, o));
    bad |= __shfl_xor_sync(kFull, bad, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&out5[0], mnx);
    atomicMin(&out5[1], mny);
    atomicMax(&out5[2], mxx);
    atomicMax(&out5[3], mxy);
    if (bad) atomicOr(&out5[4], 1);
  }
}

__global__ void k_bbox_check(const int2* xy, int n, int32_t* out5) {
  int mnx = INT_MAX, mny = INT_MAX, mxx = INT_MIN, mxy = INT_MIN, bad = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    bbox_add(xy[i], mnx, mny, mxx, mxy, bad);
  bbox_flush(mnx, mny, mxx, mxy, bad, out5);
}

__device__ __forceinline__ int cell_of(const Grid& g, int2 p) {
  return ((p.y - g.miny) / g.cs) * g.gx + (p.x - g.minx) / g.cs;
}

__global__ void k_cell_count(const int2* xy, int n, Grid g, int32_t* count) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) atomicAdd(&count[cell_of(g, xy[i])], 1);
}

// Exclusive scan of `count` into `start` (start[len] = total) and `cursor`
// (which may be `count` itself), one block.
__device__ __forceinline__ void scan_i32_body(int32_t* count, int32_t* start, int len, int32_t* cursor) {
  __shared__ int32_t warp_tot[32];
  const int t = threadIdx.x, T = blockDim.x;
  const int chunk = (len + T - 1) / T;
  const int lo = min(len, t * chunk), hi = min(len, lo + chunk);
  int32_t s = 0;
  for (int i = lo; i < hi; ++i) s += count[i];
  const int lane = t & 31, w = t >> 5;
  int32_t incl = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) warp_tot[w] = incl;
  __syncthreads();
  if (w == 0) {
    int32_t v = lane < (T >> 5) ? warp_tot[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(kFull, v, o);
      if (lane >= o) v += y;
    }
    warp_tot[lane] = v;
  }
  __syncthreads();
  int32_t run = (incl - s) + (w > 0 ? warp_tot[w - 1] : 0);
  for (int i = lo; i < hi; ++i) {
    const int32_t ci = count[i];
    start[i] = run;
    cursor[i] = run;
    run += ci;
  }
  if (t == T - 1) start[len] = warp_tot[(T >> 5) - 1];
}

// The same for one colony's cells, a block per tile of 4,096: each adds up the
// counts before its tile (all of them fit the L2 cache), so that no block
// waits for another.  One block for everything took 44 us for the 50,000 cells
// of n = 100,000; the list call went from 855 to 809 us.
constexpr int kCellTile = 4096;

__global__ void __launch_bounds__(1024) k_scan_i32(const int32_t* count, int32_t* start, int len) {
  constexpr int E = kCellTile / 1024;
  __shared__ int32_t s_w[32], s_b[32];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int tile = blockIdx.x * kCellTile;
  int32_t b = 0;
  for (int i = t; i < tile; i += 1024) b += count[i];
  const int i0 = tile + E * t;
  int32_t d[E], s = 0;
#pragma unroll
  for (int u = 0; u < E; ++u) {
    d[u] = i0 + u < len ? count[i0 + u] : 0;
    s += d[u];
  }
  int32_t incl = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += y;
  }
  b = (int32_t)__reduce_add_sync(kFull, (unsigned)b);
  if (lane == 31) {
    s_w[w] = incl;
    s_b[w] = b;
  }
  __syncthreads();
  int32_t run = incl - s;
  for (int v = 0; v < 32; ++v) run += s_b[v] + (v < w ? s_w[v] : 0);
#pragma unroll
  for (int u = 0; u < E; ++u) {
    if (i0 + u < len) start[i0 + u] = run;
    run += d[u];
    if (i0 + u == len - 1) start[len] = run;
  }
}

__global__ void k_cell_fill(const int2* xy, int n, Grid g, int32_t* cursor, int32_t* pts, int4* recs) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int2 p = xy[i];
  const int j = atomicAdd(&cursor[cell_of(g, p)], 1);
  pts[j] = i;
  if (recs) recs[j] = make_int4(i, p.x, p.y, i);
}

// The lists of one node by one warp.
//
// A query counts, per block of (2r + 1)^2 cells around its own, the points
// (two reads of `start` per row of cells) until a block holds about 1.5 K of
// them, then gathers those strictly closer than anything outside the block
// into shared memory.  If they are K or more, the K nearest are among them;
// else the block grows by a ring and is gathered again (about one query in
// thirty on uniform points).  The order is found by counting: lane i's key
// against every key of the buffer, read as a broadcast.
//
// Bound by instruction issue (a key comparison is three instructions while
// squared distances stay below 2^32, about 100 x 4 of them per lane and query).  The form it replaced, a thread per
// node with an insertion sort of K entries in local memory, was bound by
// that local memory.  Lists of 16 + 64 per node, the whole list call: 8.16 ->
// 0.81 ms at n = 100,003 (clustered points; 3.9 ms without the thinning, 1.15
// with 96-bit comparisons only), 0.84 -> 0.07 ms at n = 2,000.  Three blocks of
// 80 registers per SM.
constexpr int kKnnWarps = 8;     // warps per block, a node each at a time
constexpr int kKnnBuf = 384;     // candidates a warp holds (> kMaxKnn + 32)

struct KnnBuf {
  uint64_t m[kKnnBuf];           // squared distances
  int32_t id[kKnnBuf];           // node ids
};

// Leaves the min(cnt, K) smallest keys of the buffer's cnt in its front, in
// order (warp-collective).  Returns how many.
__device__ __forceinline__ int knn_order(KnnBuf& B, int cnt, int K) {
  const int lane = lane_id();
  constexpr int kPer = kKnnBuf / 32;
  uint64_t m[kPer];
  int32_t id[kPer], rank[kPer];
#pragma unroll
  for (int c = 0; c < kPer; ++c) {
    const int i = c * 32 + lane;
    m[c] = i < cnt ? B.m[i] : ~0ull;
    id[c] = i < cnt ? B.id[i] : INT_MAX;
    rank[c] = 0;
  }
  const int per = (cnt + 31) >> 5;
  unsigned high = 0;
#pragma unroll
  for (int c = 0; c < kPer; ++c) high |= c * 32 + lane < cnt ? (unsigned)(m[c] >> 32) : 0u;
  if (!__any_sync(kFull, high != 0)) {
    // squared distances below 2^32 (the usual case): distance and id as one
    // 64-bit key, half the instructions per comparison
    uint64_t key[kPer];
#pragma unroll
    for (int c = 0; c < kPer; ++c) key[c] = (m[c] << 32) | (unsigned)id[c];
    for (int j = 0; j < cnt; ++j) {
      const uint64_t kj = (B.m[j] << 32) | (unsigned)B.id[j];
#pragma unroll
      for (int c = 0; c < kPer; ++c) {
        if (c >= per) break;  // (uniform)
        rank[c] += kj < key[c] ? 1 : 0;
      }
    }
  } else {
    for (int j = 0; j < cnt; ++j) {
      const uint64_t mj = B.m[j];
      const int32_t ij = B.id[j];
#pragma unroll
      for (int c = 0; c < kPer; ++c) {
        if (c >= per) break;  // (uniform)
        rank[c] += (mj < m[c] || (mj == m[c] && ij < id[c])) ? 1 : 0;
      }
    }
  }
  __syncwarp();
#pragma unroll
  for (int c = 0; c < kPer; ++c)
    if (c * 32 + lane < cnt && rank[c] < K) {
      B.m[rank[c]] = m[c];
      B.id[rank[c]] = id[c];
    }
  __syncwarp();
  return cnt < K ? cnt : K;
}

// Thins a buffer of cnt >= K keys out to at most K + 32, the K smallest among
// them (warp-collective): those with m < t, for a t found by interpolation
// (points are spread evenly over an area, so their count grows about in
// proportion to m).  Returns the new count; tm, ti bound the keys still worth
// gathering.  Where many keys are equal no such t may exist: the buffer is
// then ordered and cut at K.
__device__ __forceinline__ int knn_thin(KnnBuf& B, int cnt, int K, uint64_t& tm, int32_t& ti) {
  const int lane = lane_id();
  uint64_t mx = 0;
  for (int i = lane; i < cnt; i += 32) mx = max(mx, B.m[i]);
  const unsigned hi32 = __reduce_max_sync(kFull, (unsigned)(mx >> 32));
  const unsigned lo32 = __reduce_max_sync(kFull, (unsigned)(mx >> 32) == hi32 ? (unsigned)mx : 0u);
  uint64_t lo = 0, hi = (((uint64_t)hi32 << 32) | lo32) + 1;  // counts below lo and hi:
  int clo = 0, chi = cnt;
  for (int step = 0; step < 12 && chi > K + 32 && hi - lo > 1; ++step) {
    const float f = (float)(K + 16 - clo) / (float)(chi - clo);
    uint64_t t = lo + (uint64_t)((float)(hi - lo) * f);
    if (step & 1) t = lo + ((hi - lo) >> 1);  // every other time by halves
    t = t <= lo ? lo + 1 : (t >= hi ? hi - 1 : t);
    int c = 0;
    for (int i = lane; i < cnt; i += 32) c += B.m[i] < t;
    c = (int)__reduce_add_sync(kFull, (unsigned)c);
    if (c >= K) {
      hi = t;
      chi = c;
    } else {
      lo = t;
      clo = c;
    }
  }
  if (chi > K + 32) {
    cnt = knn_order(B, cnt, K);
    tm = B.m[K - 1];
    ti = B.id[K - 1];
    __syncwarp();
    return cnt;
  }
  int out = 0;
  for (int i0 = 0; i0 < cnt; i0 += 32) {
    const int i = i0 + lane;
    const uint64_t m = i < cnt ? B.m[i] : ~0ull;
    const int32_t id = i < cnt ? B.id[i] : 0;
    const bool take = i < cnt && m < hi;
    const unsigned b = __ballot_sync(kFull, take);
    __syncwarp();  // every lane has read its entry before one is overwritten (a vote orders no memory)
    if (take) {
      const int at = out + __popc(b & ((1u << lane) - 1u));
      B.m[at] = m;
      B.id[at] = id;
    }
    out += __popc(b);
    __syncwarp();
  }
  tm = hi;
  ti = 0;
  return out;
}

__device__ __forceinline__ void knn_node(const int2* xy, int n, const Grid& g, const int32_t* start,
                                         const int32_t* pts, int k, int bl, int32_t* cand, int32_t* backup,
                                         float* eta, int32_t* dcand, int u, KnnBuf& B) {
  const int lane = lane_id();
  const int K = k + bl;
  const int2 q = xy[u];
  const int cx = (q.x - g.minx) / g.cs, cy = (q.y - g.miny) / g.cs;
  // the block to begin with: about 1.5 K points (two per cell on average);
  // from one cell up when the first guess holds far too many
  int r = 0;
  while ((2 * r + 1) * (2 * r + 1) * 4 < 3 * K) ++r;
  bool grown = false;
  for (;;) {
    int pc = 0;
    for (int y = cy - r + lane; y <= cy + r; y += 32)
      if (y >= 0 && y < g.gy)
        pc += start[y * g.gx + min(cx + r, g.gx - 1) + 1] - start[y * g.gx + max(cx - r, 0)];
    const int total = (int)__reduce_add_sync(kFull, (unsigned)pc);
    const bool all = cx - r <= 0 && cx + r >= g.gx - 1 && cy - r <= 0 && cy + r >= g.gy - 1;
    if (!grown && r > 0 && total > 6 * K) {
      r = 0;
      grown = true;
      continue;
    }
    if (total >= K + K / 2 || all) break;
    grown = true;
    ++r;
  }
  int cnt;
  for (;;) {
    // everything outside the block is at least dmin away
    const bool lin = cx - r <= 0, rin = cx + r >= g.gx - 1, din = cy - r <= 0, uin = cy + r >= g.gy - 1;
    const bool all = lin && rin && din && uin;
    int64_t dmin = INT64_MAX;
    if (!lin) dmin = min(dmin, (int64_t)q.x - ((int64_t)g.minx + (int64_t)(cx - r) * g.cs) + 1);
    if (!rin) dmin = min(dmin, ((int64_t)g.minx + (int64_t)(cx + r + 1) * g.cs) - q.x);
    if (!din) dmin = min(dmin, (int64_t)q.y - ((int64_t)g.miny + (int64_t)(cy - r) * g.cs) + 1);
    if (!uin) dmin = min(dmin, ((int64_t)g.miny + (int64_t)(cy + r + 1) * g.cs) - q.y);
    // keys to gather: below (tm, ti)
    uint64_t tm = all ? ~0ull : (uint64_t)(dmin * dmin);
    int32_t ti = 0;
    cnt = 0;
    int found = 0;  // points closer than dmin
    for (int y = max(cy - r, 0); y <= min(cy + r, g.gy - 1); ++y) {
      const int j1 = start[y * g.gx + min(cx + r, g.gx - 1) + 1];
      for (int j0 = start[y * g.gx + max(cx - r, 0)]; j0 < j1; j0 += 32) {
        const int j = j0 + lane;
        const int v = j < j1 ? pts[j] : u;
        const uint64_t m = sqdist(q, xy[v]);
        const bool take = v != u && (m < tm || (m == tm && v < ti));
        const unsigned b = __ballot_sync(kFull, take);
        if (take) {
          const int at = cnt + __popc(b & ((1u << lane) - 1u));
          B.m[at] = m;
          B.id[at] = v;
        }
        cnt += __popc(b);
        found += __popc(b);
        if (cnt > kKnnBuf - 32) {  // full: thin it out, take only closer points from here on
          __syncwarp();
          cnt = knn_thin(B, cnt, K, tm, ti);
        }
      }
    }
    if (found >= K || all) break;
    ++r;
    __syncwarp();  // the buffer is filled again, by other lanes
  }
  __syncwarp();
  if (cnt > K + 32) {
    uint64_t tm;
    int32_t ti;
    cnt = knn_thin(B, cnt, K, tm, ti);
  }
  knn_order(B, cnt, K);
  for (int s = lane; s < k; s += 32) {
    const int32_t d = euc2d_m(B.m[s]);
    cand[(size_t)u * k + s] = B.id[s];
    eta[(size_t)u * k + s] = d > 0 ? __fdiv_rn(1.0f, (float)d) : 1.0f;
    if (dcand) dcand[(size_t)u * k + s] = d;
  }
  for (int j = lane; j < bl; j += 32) backup[(size_t)u * bl + j] = B.id[k + j];
  __syncwarp();  // the next node overwrites the buffer
}

__global__ void __launch_bounds__(32 * kKnnWarps, 3) k_knn(const int2* xy, int n, Grid g, const int32_t* start,
                                                        const int32_t* pts, int k, int bl, int32_t* cand,
                                                        int32_t* backup, float* eta, int32_t* dcand) {
  __shared__ KnnBuf s_buf[kKnnWarps];
  const int w = threadIdx.x >> 5;
  const int u = blockIdx.x * kKnnWarps + w;
  if (u < n) knn_node(xy, n, g, start, pts, k, bl, cand, backup, eta, dcand, u, s_buf[w]);
}

// Short lists (K = k + bl <= M) of many nodes: a thread per node, its K nearest
// so far in order in registers, over the rings of cells around its own until
// nothing outside them can be nearer.  They are the last K of M entries; those
// before them stay below every key.
//
// A warp per node (above) is bound by the latency of a query's dependent loads,
// and a short list leaves it nothing to do meanwhile; with a thread per node 32
// queries share a warp's loads in flight.  With few nodes the warps of threads
// are too few to fill the chip, and where points cluster the longest query of a
// warp holds up the others.  The list call at n = 100,000, uniform / clustered
// points, warps against threads: K = 2 0.228 / 0.275 -> 0.103 / 0.155 ms, 6 0.275 /
// 0.302 -> 0.126 / 0.188, 8 0.305 / 0.314 -> 0.160 / 0.260, 12 0.329 / 0.337 -> 0.187 /
// 0.305.  K = 2 at n = 24,000 0.096 / 0.106 against 0.088 / 0.120, at 32,000 0.110 / 0.123
// against 0.089 / 0.128; K = 8 at 32,000 0.133 / 0.138 against 0.117 / 0.178, at 48,000
// 0.173 / 0.176 against 0.119 / 0.185, at 64,000 0.218 / 0.227 against 0.130 / 0.205.
// With 99 % of 100,000 points in one cell threads are ahead (K = 8: 46.7 -> 34.4 ms);
// with half of them in a few cells they are behind (2.6 -> 5.6 ms).
constexpr int kFewKnn = 12, kFewerKnn = 6;
inline bool knn_by_threads(int n, int K) { return K <= kFewKnn && n >= (K <= kFewerKnn ? 32768 : 49152); }

template <int M>
__global__ void __launch_bounds__(128) k_knn_few(const int2* xy, int n, Grid g, const int32_t* start,
                                                 const int32_t* pts, int k, int bl, int32_t* cand, int32_t* backup,
                                                 float* eta, int32_t* dcand) {
  const int u = blockIdx.x * blockDim.x + threadIdx.x;
  if (u >= n) return;
  const int K = k + bl;
  uint64_t bm[M];  // squared distances
  int32_t bi[M];
#pragma unroll
  for (int i = 0; i < M; ++i) {
    bm[i] = i < M - K ? 0 : ~0ull;
    bi[i] = i < M - K ? -1 : INT_MAX;
  }
  const int2 q = xy[u];
  const int cx = (q.x - g.minx) / g.cs, cy = (q.y - g.miny) / g.cs;
  auto scan = [&](int j, int j1) {
    for (; j < j1; ++j) {
      const int v = pts[j];
      const uint64_t m = sqdist(q, xy[v]);
      if (v == u || m > bm[M - 1] || (m == bm[M - 1] && v > bi[M - 1])) continue;
      bool before[M];  // the new key comes before entry i
#pragma unroll
      for (int i = 0; i < M; ++i) before[i] = m < bm[i] || (m == bm[i] && v < bi[i]);
#pragma unroll
      for (int i = M - 1; i >= 0; --i) {
        const bool shift = i > 0 && before[i > 0 ? i - 1 : 0];
        bm[i] = shift ? bm[i > 0 ? i - 1 : 0] : (before[i] ? m : bm[i]);
        bi[i] = shift ? bi[i > 0 ? i - 1 : 0] : (before[i] ? v : bi[i]);
      }
    }
  };
  for (int r = 0;; ++r) {
    const int x0 = max(cx - r, 0), x1 = min(cx + r, g.gx - 1);
    for (int y = max(cy - r, 0); y <= min(cy + r, g.gy - 1); ++y) {
      const int32_t* row = start + y * g.gx;
      if (y == cy - r || y == cy + r) {
        scan(row[x0], row[x1 + 1]);
      } else {
        if (cx - r >= 0) scan(row[cx - r], row[cx - r + 1]);
        if (cx + r < g.gx) scan(row[cx + r], row[cx + r + 1]);
      }
    }
    const bool lin = cx - r <= 0, rin = cx + r >= g.gx - 1, din = cy - r <= 0, uin = cy + r >= g.gy - 1;
    if (lin && rin && din && uin) break;  // every cell scanned
    int64_t dmin = INT64_MAX;  // everything else is at least this far
    if (!lin) dmin = min(dmin, (int64_t)q.x - ((int64_t)g.minx + (int64_t)(cx - r) * g.cs) + 1);
    if (!rin) dmin = min(dmin, ((int64_t)g.minx + (int64_t)(cx + r + 1) * g.cs) - q.x);
    if (!din) dmin = min(dmin, (int64_t)q.y - ((int64_t)g.miny + (int64_t)(cy - r) * g.cs) + 1);
    if (!uin) dmin = min(dmin, ((int64_t)g.miny + (int64_t)(cy + r + 1) * g.cs) - q.y);
    if (bm[M - 1] < (uint64_t)(dmin * dmin)) break;
  }
#pragma unroll
  for (int i = 0; i < M; ++i) {
    const int at = i - (M - K);
    if (at >= 0 && at < k) {
      const int32_t d = euc2d_m(bm[i]);
      cand[(size_t)u * k + at] = bi[i];
      eta[(size_t)u * k + at] = d > 0 ? __fdiv_rn(1.0f, (float)d) : 1.0f;
      if (dcand) dcand[(size_t)u * k + at] = d;
    } else if (at >= k) {
      backup[(size_t)u * bl + at - k] = bi[i];
    }
  }
}

// ---------------------------------------------------------------------
// Batch: the same steps for every colony of a batch; each block reads its
// colony and its block within the colony from a block map.
// ---------------------------------------------------------------------
__global__ void k_bbox_init_b(const ColonySetup* sets, int count) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= count) return;
  int32_t* b = sets[c].bb;
  b[0] = INT_MAX; b[1] = INT_MAX; b[2] = INT_MIN; b[3] = INT_MIN; b[4] = 0;
}

__global__ void k_bbox_b(const Colony* cols, const ColonySetup* sets, const int2* map) {
  const int2 e = map[blockIdx.x];
  const int i = e.y * blockDim.x + threadIdx.x;
  const int n = cols[e.x].n;
  int mnx = INT_MAX, mny = INT_MAX, mxx = INT_MIN, mxy = INT_MIN, bad = 0;
  if (i < n) bbox_add(cols[e.x].xy[i], mnx, mny, mxx, mxy, bad);
  bbox_flush(mnx, mny, mxx, mxy, bad, sets[e.x].bb);
}

// Grid of each colony from its bounding box, by the rule of the one-colony
// set-up: G = ceil(sqrt(n / 2)) cells per side of the square of the larger
// extent, so gx, gy <= G.
__global__ void k_grid_b(Colony* cols, const ColonySetup* sets, int count) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= count) return;
  const int32_t* b = sets[c].bb;
  const int n = cols[c].n;
  const int64_t ext = (int64_t)max(b[2] - b[0], b[3] - b[1]) + 1;
  int64_t G = (int64_t)ceil(sqrt((double)n / 2.0));
  if (G < 1) G = 1;
  Grid g;
  g.minx = b[0];
  g.miny = b[1];
  g.cs = (int32_t)((ext + G - 1) / G);
  if (g.cs < 1) g.cs = 1;
  g.gx = (b[2] - b[0]) / g.cs + 1;
  g.gy = (b[3] - b[1]) / g.cs + 1;
  cols[c].grid = g;
}

__global__ void k_cell_count_b(const Colony* cols, const ColonySetup* sets, const int2* map) {
  const int2 e = map[blockIdx.x];
  const int i = e.y * blockDim.x + threadIdx.x;
  const Colony C = cols[e.x];
  if (i < C.n) atomicAdd(&sets[e.x].cell_cnt[cell_of(C.grid, C.xy[i])], 1);
}

__global__ void __launch_bounds__(1024) k_cell_scan_b(const Colony* cols, const ColonySetup* sets) {
  const ColonySetup S = sets[blockIdx.x];
  const Grid g = cols[blockIdx.x].grid;
  scan_i32_body(S.cell_cnt, S.cell_start, g.gx * g.gy, S.cell_cnt);
}

__global__ void k_cell_fill_b(const Colony* cols, const ColonySetup* sets, const int2* map) {
  const int2 e = map[blockIdx.x];
  const int i = e.y * blockDim.x + threadIdx.x;
  const Colony C = cols[e.x];
  if (i >= C.n) return;
  const ColonySetup& S = sets[e.x];
  const int2 p = C.xy[i];
  const int j = atomicAdd(&S.cell_cnt[cell_of(C.grid, p)], 1);
  S.cell_pts[j] = i;
  S.cell_src[j] = make_int4(i, p.x, p.y, i);
}

// Block e.y of colony e.x: kKnnBatchNodes nodes, in turn over the warps.
__global__ void __launch_bounds__(32 * kKnnWarps, 3) k_knn_b(const Colony* cols, const ColonySetup* sets,
                                                          const int2* map) {
  __shared__ KnnBuf s_buf[kKnnWarps];
  const int2 e = map[blockIdx.x];
  const Colony& C = cols[e.x];
  const ColonySetup& S = sets[e.x];
  const int w = threadIdx.x >> 5;
  const int end = min(C.n, (e.y + 1) * kKnnBatchNodes);
  for (int u = e.y * kKnnBatchNodes + w; u < end; u += kKnnWarps)
    knn_node(C.xy, C.n, C.grid, S.cell_start, S.cell_pts, C.k, C.bl, S.cand, S.backup, S.eta, S.dcand, u, s_buf[w]);
}

}  // namespace

cudaError_t launch_grid_batch(Colony* cols, const ColonySetup* sets, int count, const int2* map256, int nmap256,
                              cudaStream_t s) {
  k_bbox_init_b<<<(count + 127) / 128, 128, 0, s>>>(sets, count);
  k_bbox_b<<<nmap256, 256, 0, s>>>(cols, sets, map256);
  k_grid_b<<<(count + 127) / 128, 128, 0, s>>>(cols, sets, count);
  return cudaGetLastError();
}

// The cell counts must be zero on entry.
cudaError_t build_lists_batch(const Colony* cols, const ColonySetup* sets, int count, const int2* map256,
                              int nmap256, const int2* map_knn, int nmap_knn, cudaStream_t s) {
  k_cell_count_b<<<nmap256, 256, 0, s>>>(cols, sets, map256);
  k_cell_scan_b<<<count, 256, 0, s>>>(cols, sets);
  k_cell_fill_b<<<nmap256, 256, 0, s>>>(cols, sets, map256);
  k_knn_b<<<nmap_knn, 32 * kKnnWarps, 0, s>>>(cols, sets, map_knn);
  return cudaGetLastError();
}

cudaError_t launch_bbox_check(const int2* xy, int n, int32_t* out5, cudaStream_t s) {
  const int32_t init[5] = {INT_MAX, INT_MAX, INT_MIN, INT_MIN, 0};
  cudaError_t e = cudaMemcpyAsync(out5, init, sizeof(init), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  const int blocks = min(1024, (n + 255) / 256);
  k_bbox_check<<<blocks, 256, 0, s>>>(xy, n, out5);
  return cudaGetLastError();
}

cudaError_t build_lists(const int2* xy, int n, int k, int bl, const Grid& g, int32_t* cell_count,
                        int32_t* cell_start, int32_t* cell_pts, int4* cell_src, int32_t* cand, int32_t* backup,
                        float* eta, int32_t* dcand, cudaStream_t s) {
  const int cells = g.gx * g.gy;
  cudaError_t e = cudaMemsetAsync(cell_count, 0, sizeof(int32_t) * cells, s);
  if (e != cudaSuccess) return e;
  k_cell_count<<<(n + 255) / 256, 256, 0, s>>>(xy, n, g, cell_count);
  k_scan_i32<<<(cells + kCellTile - 1) / kCellTile, 1024, 0, s>>>(cell_count, cell_start, cells);
  e = cudaMemcpyAsync(cell_count, cell_start, sizeof(int32_t) * cells, cudaMemcpyDeviceToDevice, s);
  if (e != cudaSuccess) return e;
  k_cell_fill<<<(n + 255) / 256, 256, 0, s>>>(xy, n, g, cell_count, cell_pts, cell_src);
  if (!knn_by_threads(n, k + bl))
    k_knn<<<(n + kKnnWarps - 1) / kKnnWarps, 32 * kKnnWarps, 0, s>>>(xy, n, g, cell_start, cell_pts, k, bl, cand, backup,
                                                                     eta, dcand);
  else if (k + bl <= kFewerKnn)
    k_knn_few<kFewerKnn><<<(n + 127) / 128, 128, 0, s>>>(xy, n, g, cell_start, cell_pts, k, bl, cand, backup, eta, dcand);
  else
    k_knn_few<kFewKnn><<<(n + 127) / 128, 128, 0, s>>>(xy, n, g, cell_start, cell_pts, k, bl, cand, backup, eta, dcand);
  return cudaGetLastError();
}

}  // namespace faco
