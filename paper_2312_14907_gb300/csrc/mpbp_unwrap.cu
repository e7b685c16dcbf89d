// mpbp_unwrap.cu -- the projector Pi_U of Eq. 10 on the GPU: the phases
// Phi_m = phase_scale G_m . u, wrapped (Eq. 9's W), unwrapped by
// reliability-ordered path following (Herraez et al., Appl. Opt. 2002), and
// mapped back to u with the pseudo-inverse of G.
//
// Path-following unwrappers merge pixel groups along edges taken in order of
// decreasing reliability, i.e. they integrate the wrapped phase differences
// along the maximum spanning forest of the pixel grid (edge weight = the sum
// of its pixels' reliabilities, ties broken by the edge number so that the
// order is strict and the forest unique).  Here that forest is built in
// parallel by Boruvka rounds instead of a sorted sweep:
//   - every component takes its heaviest incident edge (64-bit atomicMax of
//     (weight bits, ~edge number)); a root whose choice is shared with the
//     component on the other side keeps its place if its index is the lower;
//   - each other root hooks under the component across its edge with the
//     multiple of 2 pi that brings the phase difference across the edge into
//     [-pi, pi) (its offset relative to its new parent);
//   - pointer jumping compresses the forest, adding offsets along the way,
//     until every pixel points at its root with its offset to it.
// The rounds repeat until no root hooks; each group is then shifted so that
// its lowest-numbered pixel keeps its wrapped value.  The D phase maps form
// one graph with D disconnected parts.
//
// Two paths reach the same forest, offsets and output:
//   - maps of at most 1,280 tiles (572^2 pixels): one kernel contracts the
//     16 x 16 tiles (reliabilities and edge keys formed on the way) and lists
//     the components and edges that are left; one cluster of 8 or 16 blocks
//     per map runs the remaining rounds on those lists, which hold whatever a
//     map of such a size leaves; the caller's closing kernel applies the
//     offsets.  What bounds it is the chain of rounds (three 256^2 maps: 120 us
//     a projector call, against 237);
//   - larger maps: one cooperative launch (every block resident), bound by its
//     grid barriers (~5 us each, about 35 of them; three 256^2 maps: 226 us),
//     which are bounded in time: if one runs out, the block records
//     kErrTimeout and leaves, and the rest run out at their next barrier.
#include <cmath>
#include <climits>

#include "unwrap_launch.h"

namespace mpbp {

namespace {

constexpr float kTwoPi = 6.28318530717958647692f;
constexpr unsigned long long kBarrierNs = 100ull * 1000 * 1000;   // 0.1 s per barrier
constexpr int kUnwrapThreads = 256;

__device__ __forceinline__ float wrapf(float x) { return x - kTwoPi * floorf(x / kTwoPi + 0.5f); }

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// Sense by generation: the last block to arrive resets the count and bumps
// the generation; the others wait (bounded) for the generation to change.
// Returns false (in every thread of the block) if this block's wait ran out.
// With a.test_stall block 0 leaves without arriving, so the others' waits
// run out.
__device__ bool grid_sync(UnwrapArgs& a) {
  __shared__ int ok_s;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    volatile unsigned* genp = a.bar_gen;
    const unsigned g = *genp;
    __threadfence();
    if (a.test_stall && blockIdx.x == 0) {
      atomicOr(a.err, kErrTimeout);
      ok = 0;
    } else if (atomicAdd(a.bar_count, 1u) == gridDim.x - 1) {
      *a.bar_count = 0u;
      __threadfence();
      atomicAdd(a.bar_gen, 1u);
    } else {
      const unsigned long long t0 = global_ns();
      while (*genp == g) {
        __nanosleep(32);
        if (global_ns() - t0 > kBarrierNs) {
          atomicOr(a.err, kErrTimeout);
          ok = 0;
          break;
        }
      }
    }
    __threadfence();
    ok_s = ok;
  }
  __syncthreads();
  return ok_s != 0;
}

__device__ __forceinline__ bool in_mask(const UnwrapArgs& a, long long r) { return !a.mask || a.mask[r] != 0.0f; }

// reliability 1 / sqrt(H^2 + V^2 + D1^2 + D2^2) of a pixel from its 3 x 3
// neighbourhood P(di, dj)
template <typename Pix>
__device__ __forceinline__ float reliability_of(Pix&& P) {
  const float c = P(0, 0);
  const float h = wrapf(P(0, -1) - c) - wrapf(c - P(0, 1));
  const float vv = wrapf(P(-1, 0) - c) - wrapf(c - P(1, 0));
  const float d1 = wrapf(P(-1, -1) - c) - wrapf(c - P(1, 1));
  const float d2 = wrapf(P(-1, 1) - c) - wrapf(c - P(1, -1));
  const float dd = sqrtf(h * h + vv * vv + d1 * d1 + d2 * d2);
  return 1.0f / fmaxf(dd, 1e-30f);
}

// reliability of node v, when all eight neighbours are in the grid and the
// mask, else 0
__device__ float reliability(const UnwrapArgs& a, long long v) {
  const long long m = v / a.npix, r = v - m * a.npix;
  const int i = (int)(r / a.n2), j = (int)(r - (long long)i * a.n2);
  if (i < 1 || j < 1 || i > a.n1 - 2 || j > a.n2 - 2) return 0.0f;
  for (int di = -1; di <= 1; ++di)
    for (int dj = -1; dj <= 1; ++dj)
      if (!in_mask(a, r + (long long)di * a.n2 + dj)) return 0.0f;
  const float* w = a.wrapped + m * a.npix;
  return reliability_of([&](int di, int dj) { return w[(long long)(i + di) * a.n2 + j + dj]; });
}

// the other end of edge e = 2 v + dir (dir 0: right, 1: down), or -1
__device__ __forceinline__ long long edge_other(const UnwrapArgs& a, long long e) {
  const long long v = e >> 1;
  const long long r = v % a.npix;
  const int i = (int)(r / a.n2), j = (int)(r - (long long)i * a.n2);
  long long q;
  if (e & 1) {
    if (i + 1 >= a.n1) return -1;
    q = v + a.n2;
  } else {
    if (j + 1 >= a.n2) return -1;
    q = v + 1;
  }
  if (!in_mask(a, r) || !in_mask(a, q % a.npix)) return -1;
  return q;
}

__device__ __forceinline__ unsigned long long edge_key(float w, long long e) {
  return ((unsigned long long)__float_as_uint(w) << 32) | (unsigned long long)(0xFFFFFFFFu - (unsigned)e);
}

// Local contraction.  In every 16 x 16 tile of a map, Boruvka rounds over the
// tile in shared memory hook a component only when the heaviest edge incident
// to it -- edges that leave the tile included -- lies inside the tile.  By the
// cut property such an edge belongs to the maximum spanning forest, so the
// global rounds continue from a forest of the same tree, with about one
// component per tile left instead of one per pixel.  Writes parent and off
// (multiple of 2 pi relative to the tile-local root) of every node.
constexpr int kTile = 16;
static_assert(kTile * kTile == kUnwrapThreads, "one node per thread");

// A tile's shared state: local root and offset of every node, its node
// number, its phase, and the heaviest edge incident to each root.
struct TileState {
  int lp[kUnwrapThreads], lo[kUnwrapThreads], gid[kUnwrapThreads];
  float wv[kUnwrapThreads];
  unsigned long long bk[kUnwrapThreads];
};

// bk of every local root from the nodes' edges (0: none): kr, kd to the right
// and down, inside the tile or leaving it, kl, ku to the left and up where
// those leave the tile.  Every thread of the block; ends behind a barrier.
__device__ __forceinline__ void tile_best(TileState& s, int t, bool r_in, bool d_in, unsigned long long kr,
                                          unsigned long long kd, unsigned long long kl, unsigned long long ku) {
  s.bk[t] = 0ull;
  __syncthreads();
  const int r = s.lp[t];
  if (kr) {
    const int rq = r_in ? s.lp[t + 1] : -1;
    if (rq != r) {
      atomicMax(&s.bk[r], kr);
      if (rq >= 0) atomicMax(&s.bk[rq], kr);
    }
  }
  if (kd) {
    const int rq = d_in ? s.lp[t + kTile] : -1;
    if (rq != r) {
      atomicMax(&s.bk[r], kd);
      if (rq >= 0) atomicMax(&s.bk[rq], kd);
    }
  }
  if (kl) atomicMax(&s.bk[r], kl);
  if (ku) atomicMax(&s.bk[r], ku);
  __syncthreads();
}

// The Boruvka rounds of one tile (rows i0.., columns j0.. of a map whose nodes
// start at base); in: the thread's node exists.  Returns whether bk holds the
// heaviest edges of the final components.
__device__ bool contract_tile(TileState& s, int t, bool in, int i0, int j0, int n2, long long base,
                              unsigned long long kr, unsigned long long kd, unsigned long long kl,
                              unsigned long long ku) {
  const bool r_in = t % kTile + 1 < kTile, d_in = t / kTile + 1 < kTile;
  int *lp = s.lp, *lo = s.lo, *gid = s.gid;
  float* wv = s.wv;
  unsigned long long* bk = s.bk;
  for (int round = 0; round < 2 * kTile; ++round) {
    tile_best(s, t, r_in, d_in, kr, kd, kl, ku);
    const int r = lp[t];
    // hooks of the roots whose heaviest edge stays inside the tile
    int hook_p = -1, hook_o = 0;
    if (in && r == t && bk[t] != 0ull) {
      const long long e = 0xFFFFFFFFll - (long long)(bk[t] & 0xFFFFFFFFull);
      const long long pg = (e >> 1) - base;   // the edge's first end, within the map
      const int pi = (int)(pg / n2), pj = (int)(pg - (long long)pi * n2);
      const int qi = pi + (int)(e & 1), qj = pj + (int)(1 - (e & 1));
      if (pi >= i0 && pj >= j0 && qi < i0 + kTile && qj < j0 + kTile) {
        const int pl = (pi - i0) * kTile + (pj - j0), ql = (qi - i0) * kTile + (qj - j0);
        const bool p_in_r = lp[pl] == t;
        const int lr = p_in_r ? pl : ql, ls = p_in_r ? ql : pl;
        const int sr = lp[ls];
        if (!(bk[sr] == bk[t] && gid[t] < gid[sr])) {   // the shared edge: sr hooks under t
          const float d = (wv[lr] + kTwoPi * (float)lo[lr]) - (wv[ls] + kTwoPi * (float)lo[ls]);
          hook_p = sr;
          hook_o = -(int)floorf(d / kTwoPi + 0.5f);
        }
      }
    }
    if (!__syncthreads_or(hook_p >= 0)) return true;
    if (hook_p >= 0) {
      lp[t] = hook_p;
      lo[t] = hook_o;
    }
    __syncthreads();
    // pointer jumping to the roots (a forest of 256 nodes: at most 9 passes)
    for (int jump = 0; jump < 2 * kTile; ++jump) {
      const int p = lp[t], pp = lp[p];
      const int no = lo[t] + (pp != p ? lo[p] : 0);
      __syncthreads();
      if (pp != p) {
        lp[t] = pp;
        lo[t] = no;
      }
      if (!__syncthreads_or(pp != p)) break;
    }
  }
  return false;
}

__device__ void local_contract(const UnwrapArgs& a) {
  __shared__ TileState s;
  const int t = threadIdx.x, ti = t / kTile, tj = t % kTile;
  const int n1 = a.n1, n2 = a.n2;
  const int tpr = (n2 + kTile - 1) / kTile, tpc = (n1 + kTile - 1) / kTile;
  const int tiles_per_map = tpr * tpc;
  const int ntiles = (int)(a.nodes / a.npix) * tiles_per_map;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int m = tile / tiles_per_map, rem = tile - m * tiles_per_map;
    const int i0 = rem / tpr * kTile, j0 = rem % tpr * kTile;
    const int i = i0 + ti, j = j0 + tj;
    const bool in = i < n1 && j < n2;
    const long long base = (long long)m * a.npix;
    const long long v = in ? base + (long long)i * n2 + j : -1;
    // the node's edges (keys never change): right and down ones, inside the
    // tile or leaving it; left and up ones only where they leave it
    unsigned long long kr = 0, kd = 0, kl = 0, ku = 0;
    if (in) {
      kr = a.ekey[2 * v];
      kd = a.ekey[2 * v + 1];
      if (tj == 0 && j > 0) kl = a.ekey[2 * (v - 1)];
      if (ti == 0 && i > 0) ku = a.ekey[2 * (v - n2) + 1];
    }
    s.gid[t] = (int)v;
    s.lp[t] = t;
    s.lo[t] = 0;
    s.wv[t] = in ? a.wrapped[v] : 0.0f;
    contract_tile(s, t, in, i0, j0, n2, base, kr, kd, kl, ku);
    if (in) {
      a.parent[v] = s.gid[s.lp[t]];
      a.off[v] = s.lo[t];
    }
    __syncthreads();   // the next tile reuses the shared arrays
  }
}

// ----------------------------------------------------------------------------
// The path by tiles and maps.  Arrays of UnwrapArgs in other roles:
//   parent, off       tile-local root and offset of every node
//   parent2[root]     the component's label in its map, or -1 where no edge
//                     leaves it
//   off2[root]        what is added to off for the output
//   of component l of a map (at the map's first node + l): hook_off its root,
//   minnode its lowest node, hook_parent that node's off
//   ekey              per map, the listed edges' keys (a grid has fewer than
//                     2 npix edges)
//   best              of component l of a map, as everywhere
//   comps             per map, comp_cap places each for the components' parent
//                     and offset (two buffers), hook and hook offset
//   edge_ends         per map, the components at the ends of listed edge
//                     kMapRegEdges + k
//   lists[2 m]        components and edges listed (zero between calls)
// How many a map leaves: a listed component holds a pixel with an edge out of
// its tile, so at most 60 a tile; counted on whole 512^2 grids, 16 (smooth
// phases) to 21 (random) components and 217 (smooth), 139 (noisy), 145
// (random) edges a tile, about half as many inside a disc of half the area.
// ----------------------------------------------------------------------------

__device__ __forceinline__ unsigned long long* map_keys(const UnwrapArgs& a, int m) { return a.ekey + 2 * m * a.npix; }

// one block per tile: reliabilities, edge keys, contraction, lists
__global__ void __launch_bounds__(kUnwrapThreads) unwrap_tile_kernel(UnwrapArgs a) {
  constexpr int W = kTile + 4, R = kTile + 2;
  __shared__ TileState s;
  __shared__ float sw[W * W], srel[R * R];
  __shared__ unsigned char sin[W * W];   // in the grid and the mask
  __shared__ int lmin[kUnwrapThreads], s_n[2], s_at[2];
  const int t = threadIdx.x, ti = t / kTile, tj = t % kTile;
  const int n1 = a.n1, n2 = a.n2;
  const int tpr = (n2 + kTile - 1) / kTile, tpc = (n1 + kTile - 1) / kTile;
  const int m = blockIdx.x / (tpr * tpc), rem = blockIdx.x - m * (tpr * tpc);
  const int i0 = rem / tpr * kTile, j0 = rem % tpr * kTile;
  const long long base = (long long)m * a.npix;
  for (int k = t; k < W * W; k += kUnwrapThreads) {
    const int i = i0 - 2 + k / W, j = j0 - 2 + k % W;
    const bool ok = i >= 0 && j >= 0 && i < n1 && j < n2 && in_mask(a, (long long)i * n2 + j);
    sin[k] = ok;
    sw[k] = ok ? a.wrapped[base + (long long)i * n2 + j] : 0.0f;
  }
  if (t < 2) s_n[t] = 0;
  __syncthreads();
  for (int k = t; k < R * R; k += kUnwrapThreads) {
    const int c = (k / R + 1) * W + k % R + 1;
    bool all = true;
#pragma unroll
    for (int q = 0; q < 9; ++q) all = all && sin[c + (q / 3 - 1) * W + q % 3 - 1];
    srel[k] = all ? reliability_of([&](int di, int dj) { return sw[c + di * W + dj]; }) : 0.0f;
  }
  __syncthreads();
  const int i = i0 + ti, j = j0 + tj;
  const bool in = i < n1 && j < n2;
  const long long v = in ? base + (long long)i * n2 + j : -1;
  const int c = (ti + 2) * W + tj + 2, q = (ti + 1) * R + tj + 1;
  unsigned long long kr = 0, kd = 0, kl = 0, ku = 0;
  if (in && sin[c]) {
    if (sin[c + 1]) kr = edge_key(srel[q] + srel[q + 1], 2 * v);
    if (sin[c + W]) kd = edge_key(srel[q] + srel[q + R], 2 * v + 1);
    if (tj == 0 && sin[c - 1]) kl = edge_key(srel[q - 1] + srel[q], 2 * (v - 1));
    if (ti == 0 && sin[c - W]) ku = edge_key(srel[q - R] + srel[q], 2 * (v - n2) + 1);
  }
  s.gid[t] = (int)v;
  s.lp[t] = t;
  s.lo[t] = 0;
  // (a pixel off the mask has no edges: its phase is not read)
  s.wv[t] = sw[c];
  const bool r_in = tj + 1 < kTile, d_in = ti + 1 < kTile;
  if (!contract_tile(s, t, in, i0, j0, n2, base, kr, kd, kl, ku)) tile_best(s, t, r_in, d_in, kr, kd, kl, ku);
  // lists: the components that an edge leaves, and those edges, each by the
  // tile of its first end
  lmin[t] = kUnwrapThreads;
  __syncthreads();
  const int root = s.lp[t];
  if (in) atomicMin(&lmin[root], t);   // t grows with the node number
  const bool listed = in && root == t && s.bk[t] != 0ull;
  const bool er = kr && !(r_in && s.lp[t + 1] == root), ed = kd && !(d_in && s.lp[t + kTile] == root);
  const int lc = listed ? atomicAdd(&s_n[0], 1) : 0;
  const int le = er || ed ? atomicAdd(&s_n[1], (int)er + (int)ed) : 0;
  __syncthreads();
  if (t < 2) s_at[t] = s_n[t] ? atomicAdd(&a.lists[2 * m + t], s_n[t]) : 0;
  __syncthreads();
  if (in) {
    a.parent[v] = s.gid[root];
    a.off[v] = s.lo[t];
    if (root == t) {
      const int lm = lmin[t];
      if (listed) {
        const int l = s_at[0] + lc;
        a.parent2[v] = l;
        a.hook_off[base + l] = (int)v;
        a.minnode[base + l] = s.gid[lm];
        a.hook_parent[base + l] = s.lo[lm];
      } else {
        a.parent2[v] = -1;
        a.off2[v] = -s.lo[lm];
      }
    }
    const long long k = s_at[1] + le;
    unsigned long long* const ek = map_keys(a, m);
    if (er && k < 2 * a.npix) ek[k] = kr;   // (always, from counts that start at 0)
    if (ed && k + er < 2 * a.npix) ek[k + er] = kd;
  }
}

// A map's cluster: threads a block, edges a thread keeps in registers (the
// smallest cluster's are the ones that need no place in edge_ends).
constexpr int kMapThreads = 1024;
constexpr int kMapEdges = 8;
constexpr int kMapRegEdges = 8 * kMapThreads * kMapEdges;

// (warp-wide instructions: the lanes come out of strided loops of their own)
__device__ __forceinline__ void cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// One cluster per map: the remaining rounds on the listed components and
// edges, in L2, with the cluster's hardware barrier (about 1 us a phase with
// the reads around it, against 5 us for the grid's; one block instead of
// eight, its state in shared memory, took longer than the whole grid: it is
// bound by its SM's issue and by one lane a clock for its scattered reads).
// A thread takes every all-th listed edge: the first kMapEdges in registers,
// the rest in L2, where each round leaves those between two components at the
// front of the thread's own places.
__global__ void __launch_bounds__(kMapThreads) unwrap_map_kernel(UnwrapArgs a, int blocks) {
  const int m = blockIdx.x / blocks;
  const int t = (blockIdx.x % blocks) * kMapThreads + threadIdx.x;   // within the cluster
  const int all = blocks * kMapThreads;
  const long long base = (long long)m * a.npix;
  const int cap = (int)a.comp_cap;
  const int nc = min(a.lists[2 * m], cap);   // (never above, from counts that start at 0)
  const int ne = (int)min((long long)a.lists[2 * m + 1], 2 * a.npix);
  unsigned long long* const ek = map_keys(a, m);
  int* const pool = a.comps + 6ll * m * cap;
  int* const par[2] = {pool, pool + cap};
  int* const off[2] = {pool + 2 * cap, pool + 3 * cap};
  int* const hp = pool + 4 * cap;
  int* const ho = pool + 5 * cap;
  int2* const el = a.edge_ends + (long long)m * a.spill_cap - kMapRegEdges;   // by edge number
  unsigned long long* const best = a.best + base;
  int* const flags = a.map_flags + 3 * m;   // rotating: the next slot is cleared two uses after its last read
  int use = 0, cur = 0;
  auto label = [&](long long v) { return a.parent2[a.parent[v]]; };
  auto ends = [&](unsigned long long key, long long& p, long long& q) {
    const long long e = 0xFFFFFFFFll - (long long)(key & 0xFFFFFFFFull);
    p = e >> 1;
    q = p + ((e & 1) ? a.n2 : 1);
  };
  for (int l = t; l < nc; l += all) {
    par[0][l] = l;
    off[0][l] = 0;
    best[l] = 0ull;
  }
  if (t < 3) flags[t] = 0;
  unsigned long long key[kMapEdges];   // 0: none, or inside a component
  int la[kMapEdges], lb[kMapEdges];
#pragma unroll
  for (int i = 0; i < kMapEdges; ++i) {
    const int k = t + i * all;
    key[i] = k < ne ? ek[k] : 0ull;
    la[i] = lb[i] = 0;
    if (key[i]) {
      long long p, q;
      ends(key[i], p, q);
      la[i] = label(p);
      lb[i] = label(q);
    }
  }
  int spill = 0;   // the thread's edges kMapEdges, kMapEdges + 1, ... at place t + i all
  for (int k = t + kMapEdges * all; k < ne; k += all, ++spill) {
    long long p, q;
    ends(ek[k], p, q);
    el[k] = make_int2(label(p), label(q));
  }
  cluster_sync();
  for (int round = 0; round < a.max_rounds; ++round) {
    // heaviest incident edge of every component
#pragma unroll
    for (int i = 0; i < kMapEdges; ++i) {
      if (!key[i]) continue;
      la[i] = __ldcg(par[cur] + la[i]);   // the components the ends are in by now
      lb[i] = __ldcg(par[cur] + lb[i]);
      if (la[i] == lb[i]) {
        key[i] = 0ull;
        continue;
      }
      if (key[i] > __ldcg(best + la[i])) atomicMax(best + la[i], key[i]);
      if (key[i] > __ldcg(best + lb[i])) atomicMax(best + lb[i], key[i]);
    }
    int kept = t + kMapEdges * all;
    for (int k = kept, end = kept + spill * all; k < end; k += all) {
      const unsigned long long kk = ek[k];
      const int2 e = el[k];
      const int ca = __ldcg(par[cur] + e.x), cb = __ldcg(par[cur] + e.y);
      if (ca == cb) continue;
      if (kk > __ldcg(best + ca)) atomicMax(best + ca, kk);
      if (kk > __ldcg(best + cb)) atomicMax(best + cb, kk);
      ek[kept] = kk;
      el[kept] = make_int2(ca, cb);
      kept += all;
    }
    spill = (kept - t) / all - kMapEdges;
    cluster_sync();
    const int fs = use % 3;
    for (int l = t; l < nc; l += all) {
      const unsigned long long b = __ldcg(best + l);
      int h = -1;
      if (b != 0ull) {   // a root: nothing else has one
        long long p, q;
        ends(b, p, q);
        const int lp = label(p), lq = label(q);
        const bool p_in = __ldcg(par[cur] + lp) == l;
        const int s = __ldcg(par[cur] + (p_in ? lq : lp));
        if (!(__ldcg(best + s) == b && a.hook_off[base + l] < a.hook_off[base + s])) {   // else s hooks under l
          const float dp = a.wrapped[p] + kTwoPi * (float)(a.off[p] + __ldcg(off[cur] + lp));
          const float dq = a.wrapped[q] + kTwoPi * (float)(a.off[q] + __ldcg(off[cur] + lq));
          const float d = p_in ? dp - dq : dq - dp;
          h = s;
          ho[l] = -(int)floorf(d / kTwoPi + 0.5f);
          flags[fs] = 1;
        }
      }
      hp[l] = h;
    }
    if (t == 0) flags[(use + 1) % 3] = 0;
    cluster_sync();
    const bool any = __ldcg(flags + fs) != 0;
    ++use;
    if (!any) break;
    // pointer jumping, four hops a pass, until every component is under a
    // root; the first pass applies the hooks and clears best (the cap only
    // guards against a forest that is not one)
    for (int jump = 0; jump < 32; ++jump) {
      const int fj = use % 3;
      auto up = [&](int x, int& o) {
        if (jump == 0) {
          const int h = __ldcg(hp + x);
          if (h >= 0) {
            o = __ldcg(ho + x);
            return h;
          }
        }
        o = __ldcg(off[cur] + x);
        return __ldcg(par[cur] + x);
      };
      for (int l = t; l < nc; l += all) {
        int o = 0, sum = 0, x = l;
#pragma unroll
        for (int hop = 0; hop < 4; ++hop) {
          const int y = up(x, o);
          sum += o;   // a root's is 0
          if (y == x) break;
          x = y;
        }
        par[cur ^ 1][l] = x;
        off[cur ^ 1][l] = sum;
        if (up(x, o) != x) flags[fj] = 1;
        if (jump == 0) best[l] = 0ull;
      }
      if (t == 0) flags[(use + 1) % 3] = 0;
      cluster_sync();
      const bool more = __ldcg(flags + fj) != 0;
      ++use;
      cur ^= 1;
      if (!more) break;
    }
  }
  // each group's lowest-numbered node keeps its wrapped value
  for (int l = t; l < nc; l += all) hp[l] = INT_MAX;
  cluster_sync();
  for (int l = t; l < nc; l += all) atomicMin(hp + __ldcg(par[cur] + l), a.minnode[base + l]);
  cluster_sync();
  for (int l = t; l < nc; l += all) {
    const int r = __ldcg(par[cur] + l);
    if (a.minnode[base + l] == __ldcg(hp + r)) ho[r] = a.hook_parent[base + l] + __ldcg(off[cur] + l);
  }
  cluster_sync();
  for (int l = t; l < nc; l += all)
    a.off2[a.hook_off[base + l]] = __ldcg(off[cur] + l) - __ldcg(ho + __ldcg(par[cur] + l));
}

// the unwrapped phase of node v after the tile and map kernels
__device__ __forceinline__ float unwrapped_at(const UnwrapArgs& a, long long v) {
  return a.wrapped[v] + kTwoPi * (float)(a.off[v] + a.off2[a.parent[v]]);
}

__global__ void unwrap_close_kernel(UnwrapArgs a, int maps) {
  if (blockIdx.x == 0 && threadIdx.x < 2 * maps) a.lists[threadIdx.x] = 0;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < a.nodes;
       v += (long long)gridDim.x * blockDim.x)
    a.out[v] = unwrapped_at(a, v);
}

// The cooperative path.
__global__ void __launch_bounds__(kUnwrapThreads) unwrap_kernel(UnwrapArgs a) {
  const long long n = a.nodes;
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long stride = (long long)gridDim.x * blockDim.x;
  int* par[2] = {a.parent, a.parent2};
  int* off[2] = {a.off, a.off2};
  int cur = 0;   // which buffer holds the forest

  for (long long v = tid; v < n; v += stride) {
    a.rel[v] = reliability(a, v);
    a.best[v] = 0ull;
    a.minnode[v] = INT_MAX;   // read only by the closing phase
  }
  if (!grid_sync(a)) return;
  // edge keys (0: no edge), computed once
  for (long long e = tid; e < 2 * n; e += stride) {
    const long long q = edge_other(a, e);
    a.ekey[e] = q < 0 ? 0ull : edge_key(a.rel[e >> 1] + a.rel[q], e);
  }
  if (!grid_sync(a)) return;
  local_contract(a);   // writes parent and off of every node
  if (!grid_sync(a)) return;

  int flag_it = 0;   // flags rotate over 3 slots (see next_flag)
  auto next_flag = [&]() {
    // the slot of the next use is cleared now; it was last read two uses ago
    if (blockIdx.x == 0 && threadIdx.x == 0) a.flags[(flag_it + 1) % 3] = 0;
  };

  for (int round = 0; round < a.max_rounds; ++round) {
    int* P = par[cur];
    int* O = off[cur];
    // heaviest incident edge of every component (best[] is all zero here)
    for (long long e = tid; e < 2 * n; e += stride) {
      const unsigned long long key = a.ekey[e];
      if (!key) continue;
      const long long p = e >> 1, q = p + ((e & 1) ? a.n2 : 1);
      const int rp = P[p], rq = P[q];
      if (rp == rq) continue;
      atomicMax(&a.best[rp], key);
      atomicMax(&a.best[rq], key);
    }
    if (!grid_sync(a)) return;
    // hooks, decided from a consistent snapshot
    const int fs = flag_it % 3;
    for (long long r = tid; r < n; r += stride) {
      a.hook_parent[r] = -1;
      if (P[r] != (int)r || a.best[r] == 0ull) continue;
      const long long e = 0xFFFFFFFFll - (long long)(a.best[r] & 0xFFFFFFFFull);
      const long long p = e >> 1, q = p + ((e & 1) ? a.n2 : 1);
      const bool p_in_r = P[p] == (int)r;
      const long long pr = p_in_r ? p : q, ps = p_in_r ? q : p;
      const int s = P[ps];
      if (a.best[s] == a.best[r] && r < s) continue;   // the shared edge: s hooks under r
      const float d = (a.wrapped[pr] + kTwoPi * (float)O[pr]) - (a.wrapped[ps] + kTwoPi * (float)O[ps]);
      a.hook_parent[r] = s;
      a.hook_off[r] = -(int)floorf(d / kTwoPi + 0.5f);
      a.flags[fs] = 1;
    }
    next_flag();
    if (!grid_sync(a)) return;
    const bool any = *(volatile int*)&a.flags[fs] != 0;
    ++flag_it;
    if (!any) break;
    // pointer jumping until every node points at its root, four hops a pass
    // (the depth shrinks fourfold per pass; an acyclic forest of n nodes
    // needs at most log4(n) + 1 passes, the cap only guards against a forest
    // that is not), stopping after the pass that leaves every node under a
    // root.  The first pass reads the forest with the Boruvka round's hooks
    // applied (a hooked root's parent and offset from hook_parent/hook_off)
    // and clears best[]: every decision that read it is behind the barrier.
    for (int jump = 0;; ++jump) {
      if (jump > 64) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(a.err, kErrTimeout);
        break;
      }
      const bool first = jump == 0;
      const int* Pi = par[cur];
      const int* Oi = off[cur];
      int* Po = par[cur ^ 1];
      int* Oo = off[cur ^ 1];
      auto up = [&](int x, int& o) {   // parent of x, o = x's offset to it
        if (first) {
          const int h = a.hook_parent[x];
          if (h >= 0) {
            o = a.hook_off[x];
            return h;
          }
        }
        o = Oi[x];
        return Pi[x];
      };
      const int fj = flag_it % 3;
      for (long long v = tid; v < n; v += stride) {
        int o1, o2, o3, o4;
        const int p1 = up((int)v, o1);
        const int p2 = up(p1, o2);
        const int p3 = up(p2, o3);
        const int p4 = up(p3, o4);
        int ov = o1;
        if (p2 != p1) ov += o2;
        if (p3 != p2) ov += o3;
        if (p4 != p3) ov += o4;
        Po[v] = p4;
        Oo[v] = ov;
        // another pass only if the new parent is not a root (a root stays one)
        int o5;
        if (up(p4, o5) != p4) a.flags[fj] = 1;
        if (first) a.best[v] = 0ull;
      }
      next_flag();
      if (!grid_sync(a)) return;
      const bool changed = *(volatile int*)&a.flags[fj] != 0;
      ++flag_it;
      cur ^= 1;
      if (!changed) break;
    }
  }

  // each group's lowest-numbered node keeps its wrapped value
  int* P = par[cur];
  int* O = off[cur];
  for (long long v = tid; v < n; v += stride) atomicMin(&a.minnode[P[v]], (int)v);
  if (!grid_sync(a)) return;
  for (long long v = tid; v < n; v += stride) {
    const int mn = a.minnode[P[v]];
    a.out[v] = a.wrapped[v] + kTwoPi * (float)(O[v] - O[mn]);
  }
}

// Phi_m = phase_scale G_m . u, wrapped
__global__ void project_phase_kernel(ProjectArgs a) {
  const long long n = a.npix * a.D;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int m = (int)(i / a.npix);
    const long long r = i - (long long)m * a.npix;
    float ph = 0.0f;
    for (int c = 0; c < a.C; ++c) ph = fmaf(a.g_scaled[m * kMaxComp + c], a.u[c * a.npix + r], ph);
    a.phi[i] = ph;
    a.wrapped[i] = wrapf(ph);
  }
}

// u += (Phi' - Phi) pinv^T / phase_scale inside the mask; tiles: Phi' from the
// tile and map kernels' offsets
__global__ void project_correct_kernel(ProjectArgs a, UnwrapArgs uw, int tiles) {
  if (tiles && blockIdx.x == 0 && threadIdx.x < 2 * a.D) uw.lists[threadIdx.x] = 0;
  for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < a.npix;
       r += (long long)gridDim.x * blockDim.x) {
    if (a.mask && a.mask[r] == 0.0f) continue;
    for (int c = 0; c < a.C; ++c) {
      float s = 0.0f;
      for (int m = 0; m < a.D; ++m) {
        const long long i = m * a.npix + r;
        s = fmaf(a.pinv_scaled[c * kMaxPeaks + m], (tiles ? unwrapped_at(uw, i) : a.unwrapped[i]) - a.phi[i], s);
      }
      a.u[c * a.npix + r] += s;
    }
  }
}

}  // namespace

bool unwrap_prepare(int num_sms, int* grid) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, unwrap_kernel, kUnwrapThreads, 0) != cudaSuccess ||
      per_sm < 1)
    return false;
  *grid = num_sms * (per_sm < 2 ? per_sm : 2);   // 2 per SM: measured fastest (fewer barrier arrivals)
  return true;
}

// The map kernel's launch: `maps` clusters of `blocks` blocks.
static cudaLaunchConfig_t map_config(int maps, int blocks, cudaLaunchAttribute* at, cudaStream_t s) {
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = (unsigned)blocks;
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3((unsigned)(maps * blocks));
  c.blockDim = dim3(kMapThreads);
  c.stream = s;
  c.attrs = at;
  c.numAttrs = 1;
  return c;
}

int unwrap_map_blocks() {
  cudaLaunchAttribute at;
  int n = 0;
  const cudaLaunchConfig_t c = map_config(1, 16, &at, nullptr);
  if (cudaFuncSetAttribute(unwrap_map_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
      cudaOccupancyMaxActiveClusters(&n, unwrap_map_kernel, &c) == cudaSuccess && n > 0)
    return 16;
  cudaGetLastError();
  return 8;
}

static long long map_tiles(int n1, int n2) {
  return (long long)((n1 + kTile - 1) / kTile) * ((n2 + kTile - 1) / kTile);
}

// Places for the components a map can list: each holds a pixel of its own on
// its tile's rim, 4 (kTile - 1) of them.
long long unwrap_comp_cap(int n1, int n2) {
  const long long n = map_tiles(n1, n2) * 4 * (kTile - 1), npix = (long long)n1 * n2;
  return n < npix ? n : npix;
}

// Places for the listed edges that the smallest cluster's registers do not
// hold (a grid has fewer than 2 npix edges).
long long unwrap_spill_cap(int n1, int n2) {
  const long long n = 2ll * n1 * n2 - kMapRegEdges;
  return n > 0 ? n : 0;
}

// The cluster's size.  A larger one has more reads in flight, a smaller one
// cheaper barriers and room for more maps at a time (256 tiles, noisy phases on
// the whole grid: three maps 107 us a call with sixteen blocks, 117 with eight,
// but 16 maps 345 against 276; 399 and 625 tiles, three maps, smooth: 103 and
// 129 us with sixteen, 123 and 170 with eight).
static int map_blocks(const UnwrapArgs& a) { return a.max_blocks < 16 || map_tiles(a.n1, a.n2) <= 300 ? 8 : 16; }

// Against the cooperative path, three maps, noisy phases, on the whole grid and
// in a disc of half its area: 128^2 86 and 76 us a call (132 and 109), 256^2 117
// and 101 (254 and 216), 512^2 304 and 182 (894 and 630), 560^2 284 and 176
// (1,101 and 679); 16 maps of 512^2 836 and 536 (3,603 and 3,254).  Smooth,
// random and constant phases likewise: none of these is slower.  Larger maps,
// not measured, stay with the cooperative path.
constexpr long long kTilesPerBlock = 80;

bool unwrap_by_tiles(const UnwrapArgs& a) {
  return !a.test_stall && map_tiles(a.n1, a.n2) <= a.max_blocks * kTilesPerBlock;
}

cudaError_t unwrap_tiles_launch(const UnwrapArgs& a, cudaStream_t s) {
  const int maps = (int)(a.nodes / a.npix);
  unwrap_tile_kernel<<<(unsigned)(map_tiles(a.n1, a.n2) * maps), kUnwrapThreads, 0, s>>>(a);
  cudaLaunchAttribute at;
  const int blocks = map_blocks(a);
  const cudaLaunchConfig_t c = map_config(maps, blocks, &at, s);
  const cudaError_t e = cudaGetLastError();
  return e != cudaSuccess ? e : cudaLaunchKernelEx(&c, unwrap_map_kernel, a, blocks);
}

cudaError_t unwrap_close_launch(const UnwrapArgs& a, int num_sms, cudaStream_t s) {
  const long long b = (a.nodes + 255) / 256;
  unwrap_close_kernel<<<(int)(b < num_sms * 8 ? b : num_sms * 8), 256, 0, s>>>(a, (int)(a.nodes / a.npix));
  return cudaGetLastError();
}

cudaError_t unwrap_launch(const UnwrapArgs& a, int grid, cudaStream_t s) {
  void* args[] = {const_cast<UnwrapArgs*>(&a)};
  return cudaLaunchCooperativeKernel((const void*)unwrap_kernel, dim3(grid), dim3(kUnwrapThreads), args, 0, s);
}

cudaError_t project_phase_launch(const ProjectArgs& a, int num_sms, cudaStream_t s) {
  const long long n = a.npix * a.D;
  const long long b = (n + 255) / 256;
  project_phase_kernel<<<(int)(b < num_sms * 8 ? b : num_sms * 8), 256, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t project_correct_launch(const ProjectArgs& a, const UnwrapArgs& uw, bool tiles, int num_sms,
                                   cudaStream_t s) {
  const long long b = (a.npix + 255) / 256;
  project_correct_kernel<<<(int)(b < num_sms * 8 ? b : num_sms * 8), 256, 0, s>>>(a, uw, tiles ? 1 : 0);
  return cudaGetLastError();
}

}  // namespace mpbp
