// One block per graph: a whole minimum spanning forest in one block.
//
// A batch of graphs with at most 2^16 vertices each needs no passes over the
// union of the graphs: a graph's vertex labels (16 bits each) and its
// components' minima (32-bit keys) fit one SM's shared memory, where a random
// access costs a few cycles.  In the union passes every label or best[] gather
// takes a line of the L1 pipeline (one per cycle and SM), which held them at 2
// to 3 times their streaming time.  Here the two passes over a graph's edges
// stream from memory and gather from shared memory, and everything between
// them runs behind block barriers.
//
// The method is Filter-Borůvka with one partition level (Alg. 2): the light
// edges of the graph (weight up to a sampled pivot, about 1.5 n of them) are
// written to a list and contracted by Borůvka rounds; the second pass keeps
// the heavy edges between different components, and rounds on those finish.
// Keys are w << pb | position in the list being contracted; the lists keep the
// order of the edge ids, so keys order edges by (w, id).  They take 32 bits
// where the graph's weights allow (w <= 255 and up to 2^22 edges), else 64.
//
// GB300, 4096 graphs of 2^8 to 2^16 vertices (337 M edges): 12.1 ms as a union,
// 5.1 to 5.7 ms here (runs of the same code differ by that much), of which 0.14
// ms for the ids.  What bounds it is latency between
// barriers with one or two graphs per SM: half of the issue slots and half of
// L1's throughput are used (ncu, 224 KB blocks).  An edge's record is one
// 16-byte store and a live edge 8 bytes (three arrays: 5.63 ms); separate warps'
// lists instead of block-wide ones behind a scan: 5.63 against 5.95 ms.
#include <algorithm>
#include <cstdint>

#include "device.cuh"
#include "internal.h"

namespace mstgpu {

namespace {

// An entry of the component array: a key (or INF: no edge), then link | other
// component once it has hooked, or root | new id.
template <class K>
struct Entry {
  static constexpr int bits = 8 * sizeof(K);
  static constexpr K INF = ((K)1 << (bits - 1)) - 1;
  static constexpr K LINK = (K)1 << (bits - 1);
  static constexpr K ROOT = (K)3 << (bits - 2);
  static constexpr K LONE = ROOT | 0x10000u;  // a root without edges, before its id
};
constexpr uint32_t DEAD_TOP = 65535;      // components without edges left take ids from here downwards
constexpr uint32_t WIDE_PB = 30;          // position bits of a 64-bit key: the tags above a 32-bit weight stay clear
constexpr uint32_t JSTEPS = 8;            // links followed per jump pass

template <int T>
struct Shared {
  uint32_t warp[2][T / 32];
  uint32_t dead;
  uint32_t cnt;
  u64 wsum;
  uint32_t graph;
};

// What a block works on: one graph and its part of the scratch arrays.  Warp w
// takes the w-th part of the graph's edges and keeps the edges it lists in the
// matching part of the arrays (positions base.. of the warp), so the passes
// need no block barrier and positions still follow the edge ids.
struct Work {
  uint32_t n, m;
  uint64_t off;          // position of the graph's first edge
  uint4 *ent;            // a listed edge by position: ends (16 bits each), edge id, weight
  uint2 *live;           // the warps' live edges: ends, key (64-bit keys: position)
  u64 *gbest;            // [n] minima that do not fit shared memory
  // this warp's edges, as positions from the graph's first edge rounded down to
  // a multiple of four (that is skip edges earlier)
  uint32_t skip, wlo, whi;
  uint32_t base;         // this warp's first position in the lists
};

// Block-wide exclusive scan (one value per thread) behind a single barrier:
// every warp adds up the warps' sums for itself.  The sums alternate between
// two buffers, so a buffer is rewritten one barrier after its last reads.
template <int T>
__device__ __forceinline__ uint32_t scan(Shared<T> &sh, uint32_t &flip, uint32_t x, uint32_t &total) {
  constexpr int W = T / 32;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  flip ^= 1u;
  uint32_t incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) sh.warp[flip][wid] = incl;
  __syncthreads();
  const uint32_t mine = lane < W ? sh.warp[flip][lane] : 0u;
  uint32_t sums = mine;
#pragma unroll
  for (int o = 1; o < W; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, sums, o);
    if (lane >= o) sums += y;
  }
  total = __shfl_sync(0xffffffffu, sums, W - 1);
  return __shfl_sync(0xffffffffu, sums - mine, wid) + incl - x;
}

// Four consecutive entries from position j (a multiple of 4); positions outside
// [lo, hi) give 0.  lim: entries of the array from here on.
__device__ __forceinline__ void load4(const uint32_t *p, uint32_t j, uint32_t lo, uint32_t hi, uint32_t lim, bool vec,
                                      uint32_t (&x)[4]) {
  if (vec && j + 4 <= lim && j < hi) {
    const uint4 t = __ldcs(reinterpret_cast<const uint4 *>(p + j));
    x[0] = t.x, x[1] = t.y, x[2] = t.z, x[3] = t.w;
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = (j + k >= lo && j + k < hi) ? __ldcs(p + j + k) : 0u;
  }
}

// The smallest x with more than `rank` of the threads' values <= x.
template <int T>
__device__ __forceinline__ uint32_t quantile(uint32_t v, int rank) {
  uint32_t x = 0;
  for (uint32_t b = 0x80000000u; b; b >>= 1)  // the largest x with count(v < x) <= rank
    if (__syncthreads_count(v < (x | b)) <= rank) x |= b;
  return x;
}

// One pass over the warp's edges.  HEAVY 0: the light edges (w <= pw) become
// the list; 1: the heavy ones between different components.  Either relaxes
// best[] in shared memory (indexed by component; in pass 0 by vertex) if asked
// to.  Returns the length of the warp's list.
template <class K, bool HEAVY>
__device__ __forceinline__ uint32_t stream_pass(const BlockArgs &a, const Work &g, uint32_t pw, uint32_t pb,
                                                uint32_t wlim, const uint16_t *lab, K *best, bool relax,
                                                uint32_t &bad) {
  const uint64_t first = g.off - g.skip;
  const uint32_t *ps = a.src + first, *pd = a.dst + first, *pw4 = a.w + first;
  const uint32_t lim = (uint32_t)min(a.m_total - first, (uint64_t)0xffffffffu);
  const uint32_t lo = max(g.skip, g.wlo), hi = g.whi;
  const bool vec = ((((uintptr_t)ps | (uintptr_t)pd | (uintptr_t)pw4) & 15u) == 0);
  const int lane = threadIdx.x & 31;
  uint32_t len = 0;
  uint32_t j = g.wlo + 4 * lane;
  uint32_t nu[4], nv[4], nw[4];
  load4(ps, j, lo, hi, lim, vec, nu);
  load4(pd, j, lo, hi, lim, vec, nv);
  load4(pw4, j, lo, hi, lim, vec, nw);
  for (uint32_t tb = g.wlo; tb < hi; tb += 128, j += 128) {
    uint32_t u[4], v[4], w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) u[k] = nu[k], v[k] = nv[k], w[k] = nw[k];
    if (tb + 128 < hi) {  // the next tile's loads run under this tile's work
      load4(ps, j + 128, lo, hi, lim, vec, nu);
      load4(pd, j + 128, lo, hi, lim, vec, nv);
      load4(pw4, j + 128, lo, hi, lim, vec, nw);
    }
    uint32_t keep = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const bool in = j + k >= lo && j + k < hi;
      bool ok = in;
      if (!HEAVY && in) {
        if (u[k] >= g.n || v[k] >= g.n) {
          bad |= 1u;
          ok = false;
        }
        if (sizeof(K) == 4 && w[k] >= wlim) bad |= 2u;
      }
      ok = ok && (HEAVY ? w[k] > pw : (w[k] <= pw && u[k] != v[k]));
      if (HEAVY) ok = ok && lab[u[k]] != lab[v[k]];
      keep |= (ok ? 1u : 0u) << k;
    }
    const uint32_t c = (uint32_t)__popc(keep);
    uint32_t incl = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += y;
    }
    uint32_t p = g.base + len + incl - c;
    len += __shfl_sync(0xffffffffu, incl, 31);
    // few lanes keep more than one edge: as many steps as the busiest one has
    for (; keep; keep &= keep - 1, ++p) {
      const uint32_t k = (uint32_t)__ffs(keep) - 1;
      const uint32_t x = k & 2 ? (k & 1 ? u[3] : u[2]) : (k & 1 ? u[1] : u[0]);
      const uint32_t y = k & 2 ? (k & 1 ? v[3] : v[2]) : (k & 1 ? v[1] : v[0]);
      const uint32_t z = k & 2 ? (k & 1 ? w[3] : w[2]) : (k & 1 ? w[1] : w[0]);
      g.ent[p] = make_uint4(x | (y << 16), j + k - g.skip, z, 0);
      if (relax) {
        const K key = ((K)z << pb) | p;
        const uint32_t c0 = HEAVY ? lab[x] : x, c1 = HEAVY ? lab[y] : y;
        if (key < best[c0]) atomicMin(best + c0, key);
        if (key < best[c1]) atomicMin(best + c1, key);
      }
    }
  }
  __syncwarp();
  return len;
}

// Ends and key of the warp's live edge i (first: the list as the pass left it).
template <class K>
__device__ __forceinline__ uint32_t live_edge(const Work &g, uint32_t i, uint32_t pb, bool first, K &key) {
  if (first) {
    const uint4 e = g.ent[g.base + i];
    key = ((K)e.z << pb) | (g.base + i);
    return e.x;
  }
  const uint2 e = g.live[g.base + i];
  key = sizeof(K) == 4 ? (K)e.y : ((K)g.ent[e.y].z << pb) | e.y;
  return e.x;
}

// The minima of the live edges over components [lo, hi) into best[0..hi-lo).
template <int T, class K>
__device__ __forceinline__ void relax_range(const Work &g, uint32_t len, uint32_t pb, bool first, bool identity,
                                            const uint16_t *lab, uint32_t lo, uint32_t hi, K *best) {
  for (uint32_t i = threadIdx.x; i < hi - lo; i += T) best[i] = Entry<K>::INF;
  __syncthreads();
  for (uint32_t i = threadIdx.x & 31; i < len; i += 32) {
    K key;
    const uint32_t x = live_edge<K>(g, i, pb, first, key);
    const uint32_t c0 = identity ? (x & 0xffffu) : lab[x & 0xffffu], c1 = identity ? (x >> 16) : lab[x >> 16];
    if (c0 >= lo && c0 < hi && key < best[c0 - lo]) atomicMin(best + (c0 - lo), key);
    if (c1 >= lo && c1 < hi && key < best[c1 - lo]) atomicMin(best + (c1 - lo), key);
  }
  __syncthreads();
}

// Hooking, new ids and pointer jumping over the components' minima B[0..k):
// afterwards an entry holds ROOT | its component's new id.  Returns the number
// of live components.  Four components per thread at a time: their dependent
// loads overlap (one at a time, hooking alone took 47 us of a graph with 2^15
// vertices).
template <int T, class K>
__device__ __forceinline__ uint32_t contract(const BlockArgs &a, const Work &g, Shared<T> &sh, uint32_t &flip, K *B,
                                             uint32_t k, uint32_t pb, bool identity, const uint16_t *lab, u64 &wacc,
                                             uint32_t &chosen) {
  constexpr int Q = 4;
  const uint32_t pmask = (1u << pb) - 1u;
  // hooking, in place: an entry is a key until its component has linked
  volatile K *vb = B;
  for (uint32_t b = threadIdx.x; b < k; b += Q * T) {
    K key[Q], ob[Q];
    uint2 e[Q];  // ends and edge id
    uint32_t other[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const uint32_t c = b + q * T;
      key[q] = c < k ? vb[c] : (K)Entry<K>::INF;
      e[q] = make_uint2(0, 0);
      if (key[q] != Entry<K>::INF) {
        const uint4 t = g.ent[(uint32_t)key[q] & pmask];
        e[q] = make_uint2(t.x, t.y);
      }
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const uint32_t x = e[q].x & 0xffffu, y = e[q].x >> 16;
      other[q] = (identity ? x ^ y : (uint32_t)lab[x] ^ (uint32_t)lab[y]) ^ (b + q * T);
      ob[q] = key[q] != Entry<K>::INF ? vb[other[q]] : 0;
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const uint32_t c = b + q * T;
      if (c >= k) continue;
      if (key[q] == Entry<K>::INF) {
        vb[c] = Entry<K>::LONE;  // no edge left
      } else if (c < other[q] && (ob[q] == key[q] || ob[q] == (Entry<K>::LINK | c))) {
        // both chose this edge: the other's key is this one, or it already
        // linked here (then its minimum joins the two, and so is the same edge)
        vb[c] = Entry<K>::ROOT;
      } else {
        vb[c] = Entry<K>::LINK | other[q];
        const uint64_t bit = g.off + e[q].y;
        atomicOr(a.bits + (bit >> 5), 1u << (bit & 31));
        wacc += key[q] >> pb;
        ++chosen;
      }
    }
  }
  __syncthreads();
  // new ids: roots with edges 0.., the others from the dead end
  const uint32_t per = (k + T - 1) / T | 1u;  // odd: no bank conflicts between threads
  const uint32_t c0 = threadIdx.x * per, c1 = min(k, c0 + per);
  uint32_t live = 0, dead = 0;
#pragma unroll 4
  for (uint32_t c = c0; c < c1; ++c) {
    const K x = B[c];
    live += x == Entry<K>::ROOT ? 1u : 0u;
    dead += x == Entry<K>::LONE ? 1u : 0u;
  }
  uint32_t total, dead_total;
  uint32_t id = scan<T>(sh, flip, live, total);
  uint32_t dd = sh.dead + scan<T>(sh, flip, dead, dead_total);
#pragma unroll 4
  for (uint32_t c = c0; c < c1; ++c) {
    const K x = B[c];
    if (x == Entry<K>::ROOT)
      B[c] = Entry<K>::ROOT | id++;
    else if (x == Entry<K>::LONE)
      B[c] = Entry<K>::ROOT | (DEAD_TOP - dd++);
  }
  __syncthreads();
  if (threadIdx.x == 0) sh.dead += dead_total;  // (read again after later barriers)
  // pointer jumping: every pass reaches (JSTEPS + 1) times as far
  for (int pass = 0; pass < 32; ++pass) {
    bool left = false;
    for (uint32_t b = threadIdx.x; b < k; b += Q * T) {
      K x[Q];
      uint32_t pend = 0;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        x[q] = b + q * T < k ? vb[b + q * T] : (K)Entry<K>::ROOT;
        pend |= (x[q] < Entry<K>::ROOT ? 1u : 0u) << q;
      }
      const uint32_t moved = pend;
      for (uint32_t s = 0; pend && s < JSTEPS; ++s) {
#pragma unroll
        for (int q = 0; q < Q; ++q)
          if (pend >> q & 1) {
            x[q] = vb[(uint32_t)x[q] & 0xffffu];
            if (x[q] >= Entry<K>::ROOT) pend &= ~(1u << q);
          }
      }
#pragma unroll
      for (int q = 0; q < Q; ++q)
        if (moved >> q & 1) vb[b + q * T] = x[q];
      left |= pend != 0;
    }
    if (!__syncthreads_or((int)left)) break;
  }
  return total;
}

// Drops the edges inside components from the warp's list, in place (first:
// from the list as the pass left it); relaxes the others into best[] in shared
// memory if asked to.  Returns the list's new length.
template <class K>
__device__ __forceinline__ uint32_t drop_inner(const Work &g, uint32_t len, uint32_t pb, bool first,
                                               const uint16_t *lab, K *best, bool relax) {
  const int lane = threadIdx.x & 31;
  const uint32_t below = (1u << lane) - 1u;
  uint32_t kept = 0;
  for (uint32_t t0 = 0; t0 < len; t0 += 128) {
    uint32_t x[4];
    K key[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t i = t0 + q * 32 + lane;
      x[q] = 0, key[q] = 0;
      if (i < len) x[q] = live_edge<K>(g, i, pb, first, key[q]);
    }
    __syncwarp();  // every lane has read its edges: survivors overwrite them
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t c0 = lab[x[q] & 0xffffu], c1 = lab[x[q] >> 16];
      const bool ok = t0 + q * 32 + lane < len && c0 != c1;
      const uint32_t b = __ballot_sync(0xffffffffu, ok);
      if (ok) {
        g.live[g.base + kept + __popc(b & below)] =
            make_uint2(x[q], sizeof(K) == 4 ? (uint32_t)key[q] : (uint32_t)key[q] & ((1u << pb) - 1u));
        if (relax) {
          if (key[q] < best[c0]) atomicMin(best + c0, key[q]);
          if (key[q] < best[c1]) atomicMin(best + c1, key[q]);
        }
      }
      kept += __popc(b);
    }
    __syncwarp();
  }
  return kept;
}

// Borůvka rounds on the warps' lists (`len` edges in this one's) over
// components 0..k-1 (identity: the vertices themselves, lab not set yet).
// relaxed: shared memory holds their minima (at `buf` with identity, behind lab
// otherwise).  Afterwards lab holds each vertex's component, `k` live ones and
// sh.dead others from DEAD_TOP downwards.
template <int T, class K>
__device__ __forceinline__ void rounds(const BlockArgs &a, const Work &g, Shared<T> &sh, uint32_t &flip, uint32_t len,
                                       uint32_t &k, uint32_t pb, bool identity, bool relaxed, unsigned char *buf,
                                       u64 &wacc, uint32_t &chosen) {
  uint16_t *lab = reinterpret_cast<uint16_t *>(buf);
  K *behind = reinterpret_cast<K *>(buf + ((2u * g.n + 15u) & ~15u));
  K *const gb = reinterpret_cast<K *>(g.gbest);
  const uint32_t cap_id = a.smem / sizeof(K), cap_lab = (a.smem - ((2u * g.n + 15u) & ~15u)) / sizeof(K);
  // (the components halve in every round: the bound is never met)
  for (uint32_t round = 0; round < 40; ++round) {
    const int any = __syncthreads_or((int)(len > 0));
    if (!any && !identity) break;
    K *B = identity ? reinterpret_cast<K *>(buf) : behind;
    const uint32_t cap = identity ? cap_id : cap_lab;
    const bool spilled = !relaxed && k > cap;
    if (spilled) {  // ranges of components in turn, collected in global memory
      for (uint32_t lo = 0; lo < k; lo += cap) {
        const uint32_t hi = min(k, lo + cap);
        relax_range<T, K>(g, len, pb, round == 0, identity, lab, lo, hi, B);
        for (uint32_t i = threadIdx.x; i < hi - lo; i += T) gb[lo + i] = B[i];
        __syncthreads();
      }
    } else if (!relaxed) {
      relax_range<T, K>(g, len, pb, round == 0, identity, lab, 0, k, B);
    }
    const uint32_t live = spilled ? contract<T, K>(a, g, sh, flip, gb, k, pb, identity, lab, wacc, chosen)
                                  : contract<T, K>(a, g, sh, flip, B, k, pb, identity, lab, wacc, chosen);
    // labels
    if (identity && !spilled) {  // in place: label v overwrites the entry of vertex v / 2, read before
      for (uint32_t v0 = 0; v0 < g.n; v0 += 4 * T) {
        uint32_t x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint32_t v = v0 + q * T + threadIdx.x;
          x[q] = v < g.n ? (uint32_t)B[v] : 0u;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint32_t v = v0 + q * T + threadIdx.x;
          if (v < g.n) lab[v] = (uint16_t)x[q];
        }
      }
    } else {
#pragma unroll 4
      for (uint32_t v = threadIdx.x; v < g.n; v += T) {
        const uint32_t l = identity ? v : lab[v];
        if (l < k) lab[v] = (uint16_t)(spilled ? gb[l] : B[l]);
      }
    }
    k = live;
    identity = false;
    __syncthreads();
    // drop the edges inside components and relax the rest for the next round
    relaxed = k <= cap_lab;
    if (relaxed)
      for (uint32_t i = threadIdx.x; i < k; i += T) behind[i] = Entry<K>::INF;
    __syncthreads();
    len = drop_inner<K>(g, len, pb, round == 0, lab, behind, relaxed);
  }
}

// The forest of one graph with keys of type K: bits of its edges set, sh.cnt
// and sh.wsum their number and weight.  False (nothing set) when a weight does
// not fit the keys.
template <int T, class K>
__device__ __forceinline__ bool solve_keys(const BlockArgs &a, const Work &g, Shared<T> &sh, unsigned char *buf,
                                           uint32_t pb, uint32_t wlim, uint32_t pw, bool split) {
  uint32_t flip = 0;
  const uint32_t lab_bytes = (2u * g.n + 15u) & ~15u;
  K *best = reinterpret_cast<K *>(buf);
  const bool fits = g.n <= a.smem / sizeof(K);
  if (fits)
    for (uint32_t i = threadIdx.x; i < g.n; i += T) best[i] = Entry<K>::INF;
  if (threadIdx.x == 0) {
    sh.dead = 0;
    sh.cnt = 0;
    sh.wsum = 0;
  }
  __syncthreads();
  uint32_t bad = 0;
  uint32_t len = stream_pass<K, false>(a, g, pw, pb, wlim, nullptr, best, fits, bad);
  if (bad & 1u) atomicOr(a.err, ERR_VERTEX);
  if (__syncthreads_or((int)(bad & 1u))) return true;
  if (__syncthreads_or((int)bad)) return false;
  u64 wacc = 0;
  uint32_t chosen = 0, k = g.n;
  rounds<T, K>(a, g, sh, flip, len, k, pb, true, fits, buf, wacc, chosen);
  if (split) {
    // all components again: live ones 0..k-1, then the others
    uint16_t *lab = reinterpret_cast<uint16_t *>(buf);
    const uint32_t kl = k;
    for (uint32_t v = threadIdx.x; v < g.n; v += T) {
      const uint32_t l = lab[v];
      if (l >= kl) lab[v] = (uint16_t)(kl + (DEAD_TOP - l));
    }
    k += sh.dead;
    __syncthreads();
    if (threadIdx.x == 0) sh.dead = 0;
    K *hb = reinterpret_cast<K *>(buf + lab_bytes);
    const bool hfits = k <= (a.smem - lab_bytes) / sizeof(K);
    if (hfits)
      for (uint32_t i = threadIdx.x; i < k; i += T) hb[i] = Entry<K>::INF;
    __syncthreads();
    len = stream_pass<K, true>(a, g, pw, pb, wlim, lab, hb, hfits, bad);
    __syncthreads();
    rounds<T, K>(a, g, sh, flip, len, k, pb, false, hfits, buf, wacc, chosen);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    wacc += __shfl_xor_sync(0xffffffffu, wacc, o);
    chosen += __shfl_xor_sync(0xffffffffu, chosen, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (chosen) atomicAdd(&sh.cnt, chosen);
    if (wacc) atomicAdd(&sh.wsum, wacc);
  }
  __syncthreads();
  return true;
}

// The forest of one graph (n, m > 0).
template <int T>
__device__ __forceinline__ void solve_graph(const BlockArgs &a, Work g, Shared<T> &sh, unsigned char *buf) {
  constexpr uint32_t W = T / 32;
  g.skip = (uint32_t)g.off & 3u;
  const uint32_t end = g.m + g.skip, part = (end + W * 128 - 1) / (W * 128) * 128;
  g.wlo = min(end, (threadIdx.x >> 5) * part);
  g.whi = min(end, g.wlo + part);
  g.base = g.wlo > g.skip ? g.wlo - g.skip : 0u;
  const uint32_t pb = block_pos_bits(g.m), wlim = block_weight_limit(g.m);
  // the pivot: about 1.5 n light edges, from one sampled weight per thread
  const uint64_t j = g.off + __umul64hi(splitmix64_at(0x5eedULL + g.off, threadIdx.x), (u64)g.m);
  const uint32_t sw = __ldg(a.w + j);
  const bool wide = __syncthreads_or(sw >= wlim);
  uint32_t pw = 0xffffffffu;
  const bool split = g.m > 3 * g.n && g.m > 2048;
  if (split) pw = quantile<T>(sw, (int)((u64)T * 3 * g.n / (2 * (u64)g.m)));
  if (!wide && solve_keys<T, uint32_t>(a, g, sh, buf, pb, wlim, pw, split)) return;
  solve_keys<T, u64>(a, g, sh, buf, WIDE_PB, wlim, pw, split);
}

// Graphs order[first .. first + num) one after another, each by the block that
// takes it from the queue.
template <int T, int MINB>
__global__ void __launch_bounds__(T, MINB) block_batch_kernel(const __grid_constant__ BlockArgs a) {
  extern __shared__ __align__(16) unsigned char buf[];
  __shared__ Shared<T> sh;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) sh.graph = atomicAdd(a.queue, 1u);
    __syncthreads();
    const uint32_t i = sh.graph;
    if (i >= a.num) return;
    const uint32_t gi = a.order[a.first + i];
    const uint64_t off = a.edge_off[gi], v0 = a.vert_off[gi];
    const Work g{a.gn[gi], (uint32_t)(a.edge_off[gi + 1] - off), off, a.ent + off, a.live + off,
                 a.gbest + v0, 0, 0, 0, 0};
    if (g.m > 0 && g.n > 0) {
      solve_graph<T>(a, g, sh, buf);
    } else if (threadIdx.x == 0) {
      if (g.m > 0) atomicOr(a.err, ERR_VERTEX);
      sh.cnt = 0;
      sh.wsum = 0;
    }
    if (threadIdx.x == 0) {
      a.totals[gi] = sh.wsum;
      a.sizes[gi] = sh.cnt;
      a.solved[gi] = 1;
    }
  }
}

// A single graph (edges 0..m-1): zeroes its bitmap, solves it and writes the
// ascending ids, their number and their weight.
template <int T>
__global__ void __launch_bounds__(T, 1) block_single_kernel(const __grid_constant__ BlockArgs a, uint32_t n, uint32_t m,
                                                            uint32_t *out_ids, uint32_t *out_count) {
  extern __shared__ __align__(16) unsigned char buf[];
  __shared__ Shared<T> sh;
  const uint32_t words = (m + 31) / 32;
  for (uint32_t i = threadIdx.x; i < words; i += T) a.bits[i] = 0;
  if (threadIdx.x == 0) *a.err = 0;
  __syncthreads();
  const Work g{n, m, 0, a.ent, a.live, a.gbest, 0, 0, 0, 0};
  solve_graph<T>(a, g, sh, buf);
  __threadfence_block();
  __syncthreads();
  uint32_t flip = 0, base = 0;
  for (uint32_t i0 = 0; i0 < words; i0 += T) {
    uint32_t word = i0 + threadIdx.x < words ? __ldcg(a.bits + i0 + threadIdx.x) : 0u;
    uint32_t total;
    uint32_t p = base + scan<T>(sh, flip, (uint32_t)__popc(word), total);
    for (; word; word &= word - 1) out_ids[p++] = (i0 + threadIdx.x) * 32 + (uint32_t)__ffs(word) - 1;
    base += total;
  }
  if (threadIdx.x == 0) {
    *out_count = sh.cnt;
    *a.totals = sh.wsum;
  }
  publish_state(a.rb);
}

constexpr size_t BIG_SMEM = BLOCK_BIG_N * 4, MID_SMEM = BLOCK_MID_N * 4, SMALL_SMEM = BLOCK_SMALL_N * 4;

template <int T, int MINB>
int resident_blocks(size_t smem) {
  int dev = 0, sms = 0, b = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (cudaFuncSetAttribute(block_batch_kernel<T, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, block_batch_kernel<T, MINB>, T, smem) != cudaSuccess)
    b = 0;
  cudaGetLastError();
  return sms * b;
}

constexpr int SINGLE_T = 1024;

// False when the launch was refused (nothing runs; the error is the caller's to act on, not left pending).
template <class... Args>
bool launch(void (*kernel)(Args...), unsigned grid, int threads, size_t smem, cudaStream_t s, Args... args) {
  void *p[] = {&args...};
  if (cudaLaunchKernel((const void *)kernel, dim3(grid), dim3((unsigned)threads), p, smem, s) == cudaSuccess)
    return true;
  cudaGetLastError();
  return false;
}

}  // namespace

bool launch_block_single(const BlockArgs &args, uint32_t n, uint32_t m, uint32_t *out_ids, uint32_t *out_count,
                         cudaStream_t s) {
  static PerDevice set_of;
  const int set = set_of.get(current_device(), []() -> int {
    const bool ok = cudaFuncSetAttribute(block_single_kernel<SINGLE_T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)BIG_SMEM) == cudaSuccess;
    cudaGetLastError();
    return ok;
  });
  if (!set) return false;
  BlockArgs a = args;
  // room for the vertices' minima in either key size and for labels with minima behind them
  a.smem = (uint32_t)std::min<size_t>(BIG_SMEM, std::max<size_t>((size_t)n * 10 + 64, 16384));
  return launch<BlockArgs>(block_single_kernel<SINGLE_T>, 1, SINGLE_T, a.smem, s, a, n, m, out_ids, out_count);
}

bool launch_block_batch(const BlockArgs &args, int kind, cudaStream_t s) {
  if (args.num == 0) return true;
  static PerDevice blocks_of[3];
  constexpr size_t smem[3] = {BIG_SMEM, MID_SMEM, SMALL_SMEM};
  const int blocks = blocks_of[kind].get(current_device(), [&] {
    return kind == 0 ? resident_blocks<1024, 1>(smem[0])
                     : kind == 1 ? resident_blocks<512, 2>(smem[1]) : resident_blocks<256, 4>(smem[2]);
  });
  if (blocks <= 0) return false;
  BlockArgs a = args;
  a.smem = (uint32_t)smem[kind];
  const unsigned grid = std::min<unsigned>(a.num, (unsigned)blocks);
  if (kind == 0) return launch<BlockArgs>(block_batch_kernel<1024, 1>, grid, 1024, smem[0], s, a);
  if (kind == 1) return launch<BlockArgs>(block_batch_kernel<512, 2>, grid, 512, smem[1], s, a);
  return launch<BlockArgs>(block_batch_kernel<256, 4>, grid, 256, smem[2], s, a);
}

}  // namespace mstgpu
