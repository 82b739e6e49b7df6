// The Borůvka rounds of one call in a single persistent kernel.
//
// Every round (Section 2.3) is a few short passes over lists that shrink
// quickly, so a round loop driven by the host, or by a CUDA graph's
// conditional node, mostly waits between launches: on GB300 a graph iteration
// of two rounds cost about 25 us before its first kernel, and a call about
// 50 us more to enter the loop, against 5-30 us of work in a late round.  Here
// all blocks of one cooperative launch stay resident and pass from phase to
// phase through a grid barrier (about 1.5 us); once a list fits one block, the
// other blocks leave and the last rounds run behind block barriers.
//
// Components are renumbered densely in every round: the roots that hooking
// leaves get the ids 0..k-1 of the next round, so that later rounds read and
// write compact, coalesced vertex arrays (no list of active vertices), and a
// few components' minima fit a shared-memory table.
#include <algorithm>
#include <cstdint>

#include "device.cuh"
#include "internal.h"

namespace mstgpu {

namespace {

constexpr int RB = 512;            // threads per block; two blocks per SM (64 registers)
constexpr int RI = 4;              // edges per thread at a time of a long list
constexpr int RT = RB * RI;        // edges per tile of a long list
constexpr int RW = RB / 32;
constexpr int GROUP = 4;           // warps that claim output places together
constexpr int HI = 16;             // vertices per thread and tile of a long hooking pass
constexpr uint32_t ROOT = 0x80000000u;  // link entry: a root with its next-round id, or a resolved vertex
constexpr uint32_t FIN = 0xffffffffu;   // link entry: component without edges left
constexpr uint32_t RSTEPS = 32;         // parent steps per jump pass
constexpr uint32_t RPASSES = 256;       // jump passes per round (each multiplies the reach)
// Components up to which a round's minima are first collected in shared memory
// per block.  With few components and many edges every block would send its
// minima to the same few words: a GNM round (n=2^16, m=2^20) with 300
// components left took 46 us, most of it those atomics queueing; 12 us with
// the table.
constexpr uint32_t STAB = 4096;
// Components up to which a round keeps only the lightest edge between each two
// (pair_phase): their pairs and the byte labels fill the shared memory that a
// block has anyway.
constexpr uint32_t PAIR_COMPS = 124, PAIRS = PAIR_COMPS * (PAIR_COMPS - 1) / 2;
constexpr uint32_t NO_PAIRS = 0xffffffffu;
// Labels of up to LABS components are then read from shared memory.  A gather
// answered by L1 costs a cycle per line, so up to 32 per warp, however few
// lines the table has; in shared memory about four.
constexpr uint32_t LABS = 4096;
// A call's last rounds run in one block from this size on.
constexpr uint64_t SOLO_EDGES = 4096, SOLO_VERTS = 4096;
constexpr uint32_t BAR_SPINS = 1u << 24;  // polls of the grid barrier before giving up, by default

struct Smem {
  uint32_t out[4][RT];  // a hooking tile's vertices; the relabel's claims
  u64 tab[STAB];        // per-block minima of a round with few components
};
static_assert(PAIRS * sizeof(u64) + LABS <= sizeof(Smem), "pairs and labels fit");

// All blocks of the launch are resident (cooperative launch), so a wait for
// the others ends; it is bounded all the same.  A block that gives up has
// arrived at that barrier but arrives at no later one, so the others, whose
// phases only read what was complete at the last barrier they passed, give up
// at the next.  Whatever of parent[] is unfinished then stays so: the passes
// queued behind the launch look at the error first (ERR_ROUNDS).
// FIXED: the limit is BAR_SPINS.  A limit read at run time changes the long
// phases' registers (RMAT n=2^22 m=2^26, plain: 2719 -> 2737 us; RGG2D n=2^22
// 903 -> 910), so it has an instance of its own.
template <bool FIXED>
struct GridSync {
  uint32_t nb, bid;  // blocks that take part, this block's number
  uint32_t *bar, *err;
  uint32_t limit;    // polls
  uint32_t target;
  bool solo;
  // False when the wait ran out (the error is latched; the kernel ends).
  __device__ __forceinline__ bool sync() {
    if (solo) {
      __syncthreads();
      return true;
    }
    int bad = 0;
    __syncthreads();
    if (threadIdx.x == 0) {
      target += nb;
      __threadfence();
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
      uint32_t spins = 0;
      for (;;) {
        uint32_t v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
        if ((int32_t)(v - target) >= 0) break;
        if (++spins >= (FIXED ? BAR_SPINS : limit)) {
          atomicOr(err, ERR_BARRIER);
          bad = 1;
          break;
        }
      }
      __threadfence();
    }
    return !__syncthreads_or(bad);
  }
};

__device__ __forceinline__ bool aligned16_list(const EdgeList &l) {
  return ((((uintptr_t)l.u | (uintptr_t)l.v | (uintptr_t)l.w | (uintptr_t)l.id) & 15u) == 0);
}

// best[x] = min(best[x], key): the current value first (it only falls, so a
// stale copy costs an extra atomic at most).
__device__ __forceinline__ void relax(u64 *best, uint32_t x, u64 key, u64 cur) {
  if (key < cur) atomicMin(best + x, key);
}

// minEdges over the call's first list: vertex check, best[] of both ends, and
// the ends by id where the hook will look them up and nothing recorded them.
__device__ __forceinline__ void min_edges_phase(const RoundsArgs &a, KeyLayout kl, uint64_t m, uint32_t nb, uint32_t bid) {
  const bool vec = aligned16_list(a.in);
  const bool record = a.record_first && !kl.packed;
  for (uint64_t tb = (uint64_t)bid * RT; tb < m; tb += (uint64_t)nb * RT) {
    const uint64_t j0 = tb + 4 * threadIdx.x;
    uint32_t eu[RI], ev[RI], ew[RI], ei[RI];
    if (vec && tb + RT <= m) {
      const uint4 x = __ldg(reinterpret_cast<const uint4 *>(a.in.u + j0));
      const uint4 y = __ldg(reinterpret_cast<const uint4 *>(a.in.v + j0));
      const uint4 z = __ldg(reinterpret_cast<const uint4 *>(a.in.w + j0));
      eu[0] = x.x, eu[1] = x.y, eu[2] = x.z, eu[3] = x.w;
      ev[0] = y.x, ev[1] = y.y, ev[2] = y.z, ev[3] = y.w;
      ew[0] = z.x, ew[1] = z.y, ew[2] = z.z, ew[3] = z.w;
      if (a.in.id) {
        const uint4 t = __ldg(reinterpret_cast<const uint4 *>(a.in.id + j0));
        ei[0] = t.x, ei[1] = t.y, ei[2] = t.z, ei[3] = t.w;
      } else {
#pragma unroll
        for (int k = 0; k < RI; ++k) ei[k] = (uint32_t)(j0 + k);
      }
    } else {
#pragma unroll
      for (int k = 0; k < RI; ++k) {
        const uint64_t j = j0 + k;
        const bool in = j < m;
        eu[k] = in ? a.in.u[j] : 0u;
        ev[k] = in ? a.in.v[j] : 0u;
        ew[k] = in ? a.in.w[j] : 0u;
        ei[k] = in ? (a.in.id ? a.in.id[j] : (uint32_t)j) : 0u;
      }
    }
    u64 cu[RI], cv[RI];
    uint32_t ok = 0;
#pragma unroll
    for (int k = 0; k < RI; ++k) {
      bool v = eu[k] != ev[k] && j0 + k < m;
      if (a.validate && j0 + k < m && (eu[k] >= a.n || ev[k] >= a.n)) {
        atomicOr(a.err, ERR_VERTEX);
        v = false;
      }
      ok |= (v ? 1u : 0u) << k;
      cu[k] = v ? __ldca(a.best + eu[k]) : 0ULL;
      cv[k] = v ? __ldca(a.best + ev[k]) : 0ULL;
    }
#pragma unroll
    for (int k = 0; k < RI; ++k) {
      relax(a.best, eu[k], relax_key(kl, ew[k], ei[k], ev[k]), cu[k]);
      relax(a.best, ev[k], relax_key(kl, ew[k], ei[k], eu[k]), cv[k]);
      if (record && (ok >> k & 1)) {
        a.cur_u[ei[k]] = eu[k];
        a.cur_v[ei[k]] = ev[k];
      }
    }
  }
}

// Hooking over the round's vertices 0..nc-1 (round 0: all vertices of the
// call): a vertex with a minimum edge links to the edge's other end; of a
// 2-cycle the smaller id stays root and takes the next free id of the next
// round.  `link` gets the other end, or ROOT | next id; a component without
// edges gets FIN (in round 0 its entry, a plain representative, is kept).
// A tile of 512 * I vertices is first reduced to those with an edge, so that
// the dependent gathers behind them run with full warps however sparse the
// call is (a light list of RMAT n=2^24 touches 6% of the vertices).  Vertices
// and the roots' new ids keep their order inside a tile: neighbouring ids of a
// geometric graph stay neighbours in every round (ids out of order there made
// the RGG2D n=2^22 first relabel 263 us instead of 213).
template <int I>
__device__ __forceinline__ void hook_phase(const RoundsArgs &a, const KeyLayout &kl, int r, uint64_t nc, uint64_t off,
                                           bool rec, uint32_t nb, uint32_t bid, Smem &sm, uint32_t *s_warp,
                                           uint32_t *s_base) {
  static_assert(I * RB <= 4 * RT, "a tile's vertices fit the output stage");
  uint32_t *link = r == 0 ? a.parent : a.link + off;
  const uint32_t *rep = a.rep + off;
  uint32_t *rep_next = a.rep + (r == 0 ? 0 : off + nc);
  const uint32_t *eu = rec ? a.cur_u : a.src, *ev = rec ? a.cur_v : a.dst;
  uint32_t *s_c = &sm.out[0][0];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t below = (1u << lane) - 1u;
  u64 wacc = 0;
  constexpr uint64_t T = (uint64_t)RB * I;
  constexpr int C = I >= 4 ? 4 : I;  // vertices with an edge in flight per thread
  const int wshift = kl.packed ? kl.idbits + kl.vbits : 32;
  for (uint64_t tb = (uint64_t)bid * T; tb < nc; tb += (uint64_t)nb * T) {
    // warp w reduces the tile's vertices [w * 32 I, (w + 1) * 32 I)
    const uint64_t c0 = tb + (uint64_t)wid * (32 * I) + lane;
    uint32_t act = 0, cnt = 0;
#pragma unroll
    for (int q = 0; q < I; ++q) act |= (c0 + 32 * q < nc && a.best[c0 + 32 * q] != KEY_INF ? 1u : 0u) << q;
#pragma unroll
    for (int q = 0; q < I; ++q) cnt += __popc(__ballot_sync(0xffffffffu, act >> q & 1));
    uint32_t total;
    uint32_t p = block_exclusive_scan<RB>(lane == 0 ? cnt : 0u, total, s_warp);
    p = __shfl_sync(0xffffffffu, p, 0);
    if (r == 0 && threadIdx.x == 0 && total) s_base[1] = (uint32_t)atomicAdd(&a.st->ca, (u64)total);
#pragma unroll
    for (int q = 0; q < I; ++q) {
      const uint32_t b = __ballot_sync(0xffffffffu, act >> q & 1);
      if (act >> q & 1)
        s_c[p + __popc(b & below)] = (uint32_t)(c0 + 32 * q);
      else if (r > 0 && c0 + 32 * q < nc)
        link[c0 + 32 * q] = FIN;
      p += __popc(b);
    }
    __syncthreads();
    // warp w hooks the entries [w * per, (w + 1) * per) of the reduced tile
    const uint32_t per = ((total + RW - 1) / RW + 31u) & ~31u;  // at most 32 I
    const uint32_t lo = wid * per + lane, hi = min(total, (wid + 1) * per);
    uint32_t roots = 0;
#pragma unroll
    for (int q = 0; q < I / C; ++q) {
      if ((uint32_t)q * (32 * C) >= per) break;
      uint32_t c[C], oth[C];
      u64 kk[C];
#pragma unroll
      for (int k = 0; k < C; ++k) {
        const uint32_t i = lo + (q * C + k) * 32;
        c[k] = i < hi ? s_c[i] : 0u;
        kk[k] = i < hi ? a.best[c[k]] : KEY_INF;
        if (r == 0 && i < hi) a.act[s_base[1] + i] = c[k];
      }
#pragma unroll
      for (int k = 0; k < C; ++k) {
        oth[k] = 0;
        if (kk[k] == KEY_INF) continue;
        if (kl.packed) {
          oth[k] = (uint32_t)(kk[k] & ((1ULL << kl.vbits) - 1));
        } else {
          const uint32_t e = (uint32_t)kk[k];
          oth[k] = __ldca(eu + e) ^ __ldca(ev + e) ^ c[k];
        }
      }
      u64 ob[C];
#pragma unroll
      for (int k = 0; k < C; ++k) ob[k] = kk[k] != KEY_INF ? a.best[oth[k]] : 0ULL;
#pragma unroll
      for (int k = 0; k < C; ++k) {
        if (kk[k] == KEY_INF) continue;
        if (same_edge(kl, ob[k], kk[k]) && c[k] < oth[k]) {
          roots |= 1u << (q * C + k);
        } else {
          link[c[k]] = oth[k];
          const uint32_t e = key_edge_id(kl, kk[k]);
          atomicOr(a.chosen_bits + (e >> 5), 1u << (e & 31));
          wacc += kk[k] >> wshift;
        }
      }
    }
    cnt = 0;
#pragma unroll
    for (int b = 0; b < I; ++b) cnt += __popc(__ballot_sync(0xffffffffu, roots >> b & 1));
    uint32_t did = block_exclusive_scan<RB>(lane == 0 ? cnt : 0u, total, s_warp);
    if (threadIdx.x == 0 && total) s_base[0] = (uint32_t)atomicAdd(&a.st->cv[r], (u64)total);
    __syncthreads();
    did = s_base[0] + __shfl_sync(0xffffffffu, did, 0);
#pragma unroll
    for (int b = 0; b < I; ++b) {
      const uint32_t m = __ballot_sync(0xffffffffu, roots >> b & 1);
      if (roots >> b & 1) {
        const uint32_t c = s_c[lo + b * 32], d = did + __popc(m & below);
        link[c] = ROOT | d;
        if (a.want_parent) rep_next[d] = r == 0 ? c : rep[c];
      }
      did += __popc(m);
    }
    __syncthreads();  // s_c, s_warp and s_base are reused by the next tile
  }
  wsum_add(a.wsum, wacc);
}

// The same for a short pass (rounds of few components, small calls): a lane per
// vertex, and no block barriers; the GROUP warps of a group claim their roots'
// ids, and in round 0 places in `act`, together.  A chain of L2 round trips
// between two grid barriers: 3.1 to 5.2 us a pass in GNM n=2^16 m=2^20, 21 with
// 541,226 components.  Against the tiles of the long pass, whole solves: that GNM
// 208 -> 204 us, RGG3D n=2^21 596 -> 586, grid 2048 x 2048 582 -> 572.  Sparse
// first rounds need the tiles (RMAT n=2^24: about 95 us, a lane per vertex four
// to five times that).
__device__ __forceinline__ void hook_short(const RoundsArgs &a, const KeyLayout &kl, int r, uint64_t nc, uint64_t off,
                                           bool rec, uint32_t nb, uint32_t bid, Smem &sm) {
  uint32_t *link = r == 0 ? a.parent : a.link + off;
  const uint32_t *rep = a.rep + off;
  uint32_t *rep_next = a.rep + (r == 0 ? 0 : off + nc);
  const uint32_t *eu = rec ? a.cur_u : a.src, *ev = rec ? a.cur_v : a.dst;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t *s_tot = reinterpret_cast<uint32_t *>(sm.tab), *s_pos = s_tot + RW;  // per warp, two per group
  const uint32_t below = (1u << lane) - 1u;
  u64 wacc = 0;
  for (uint64_t tile = (uint64_t)bid * RW + wid; tile / GROUP * GROUP * 32 < nc; tile += (uint64_t)nb * RW) {
    const uint64_t c64 = tile * 32 + lane;
    const uint32_t c = (uint32_t)c64;
    const u64 k = c64 < nc ? a.best[c] : KEY_INF;
    const bool act = k != KEY_INF;
    bool root = false;
    if (act) {
      const uint32_t e = key_edge_id(kl, k);
      const uint32_t oth = kl.packed ? (uint32_t)(k & ((1ULL << kl.vbits) - 1)) : __ldca(eu + e) ^ __ldca(ev + e) ^ c;
      root = same_edge(kl, a.best[oth], k) && c < oth;
      if (!root) {
        link[c] = oth;
        atomicOr(a.chosen_bits + (e >> 5), 1u << (e & 31));
        wacc += k >> (kl.packed ? kl.idbits + kl.vbits : 32);
      }
    } else if (r > 0 && c64 < nc) {
      link[c] = FIN;
    }
    const uint32_t rm = __ballot_sync(0xffffffffu, root), am = __ballot_sync(0xffffffffu, act);
    if (lane == 0) s_tot[wid] = __popc(rm) | (r == 0 ? __popc(am) << 16 : 0);
    asm volatile("bar.sync %0, %1;" ::"r"(1 + wid / GROUP), "n"(32 * GROUP) : "memory");
    uint32_t sum = 0, mine = 0;
#pragma unroll
    for (int q = 0; q < GROUP; ++q) {
      const uint32_t t = s_tot[wid / GROUP * GROUP + q];
      mine += q < wid % GROUP ? t : 0u;
      sum += t;
    }
    if (wid % GROUP == 0 && lane < 2) {
      const uint32_t n = lane ? sum >> 16 : sum & 0xffffu;
      s_pos[wid / GROUP * 2 + lane] = n ? (uint32_t)atomicAdd(lane ? &a.st->ca : &a.st->cv[r], (u64)n) : 0u;
    }
    asm volatile("bar.sync %0, %1;" ::"r"(1 + wid / GROUP), "n"(32 * GROUP) : "memory");
    if (root) {
      const uint32_t d = s_pos[wid / GROUP * 2] + (mine & 0xffffu) + __popc(rm & below);
      link[c] = ROOT | d;
      if (a.want_parent) rep_next[d] = r == 0 ? c : rep[c];
    }
    if (r == 0 && act) a.act[s_pos[wid / GROUP * 2 + 1] + (mine >> 16) + __popc(am & below)] = c;
  }
  wsum_add(a.wsum, wacc);
}

// Pointer jumping (Section 4.2): every vertex that is not a root follows the
// links to its root and takes the root's next-round id; best[] goes back to
// INF.  Other threads' progress may be read on the way (an entry is either a
// vertex nearer the root or the final id).  At most RSTEPS steps per pass: a pass
// multiplies every vertex's reach by at least RSTEPS + 1, so long chains want
// several short passes, and the trees of other graphs are less deep.  `flag` is
// raised once per warp at most, and not where it is up already: raised by every
// thread, its atomics queued at one word for most of a pass.  Plain solve of 16
// paths of 2^16 vertices with ascending weights, joined end to end: 388 us with
// 256 steps and a flag per thread, 319 with 256 steps, 226 with 64, 192 with 32.
__device__ __forceinline__ void jump_phase(const RoundsArgs &a, int r, uint64_t cnt, uint64_t off, bool reset,
                                        uint32_t *flag, uint32_t nb, uint32_t bid) {
  uint32_t *link = r == 0 ? a.parent : a.link + off;
  const uint64_t stride = (uint64_t)nb * RB;
  bool left = false;
  for (uint64_t i0 = (uint64_t)bid * RB + threadIdx.x; i0 < cnt; i0 += 4 * stride) {
    uint32_t c[4], q[4], pend = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint64_t i = i0 + k * stride;
      const bool in = i < cnt;
      c[k] = in ? (r == 0 ? __ldca(a.act + i) : (uint32_t)i) : 0u;
      q[k] = in ? __ldca(link + c[k]) : ROOT;
      if (reset && in) a.best[c[k]] = KEY_INF;
      pend |= (q[k] & ROOT ? 0u : 1u) << k;
    }
    const uint32_t moved = pend;
    for (uint32_t s = 0; pend && s < RSTEPS; ++s) {
      uint32_t t[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) t[k] = (pend >> k & 1) ? __ldca(link + q[k]) : 0u;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (pend >> k & 1) {
          q[k] = t[k];
          if (t[k] & ROOT) pend &= ~(1u << k);
        }
    }
    left |= pend != 0;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (moved >> k & 1) __stcg(link + c[k], q[k]);
  }
  if (__any_sync(0xffffffffu, left) && (threadIdx.x & 31) == 0 && !__ldcg(flag)) atomicOr(flag, 1u);
}

// Relabel, self-loop removal and compaction of the round's list, with the next
// round's minEdges on the survivors (Section 4.3).  A warp takes 32 * I edges at
// a time; the GROUP warps of a group claim their survivors' places with one
// atomic, and write them from registers (a store's lanes are dense).  `tab`:
// collect the minima in shared memory first.  Bound by the label and best[]
// gathers, four per edge, which warps that wait for no more than their group
// keep coming.  Its first two passes take 1040 and 673 us in RMAT n=2^22 m=2^26
// (254 and 383 G gathers/s), 207 and 128 in RGG2D n=2^22, 33 and 16 in GNM n=2^16
// m=2^20.  Whole solves, with whole blocks passing from load to gather to a staged
// store behind barriers: that RMAT 3.23 ms (now 2.88), that RGG2D 997 us (936),
// that GNM 233 (229).  A claim per warp queues at the counter and scatters
// neighbours over the next list (the RMAT's first two passes a seventh longer);
// groups of eight wait longer (a twentieth).
template <int I>
__device__ __forceinline__ void relabel_phase(const RoundsArgs &a, KeyLayout kl, int r, uint64_t m, uint64_t off,
                                               bool tab, uint32_t nb, uint32_t bid, Smem &sm) {
  const uint32_t *link = r == 0 ? a.parent : a.link + off;
  const EdgeOut out = a.list[(a.first_slot + r) & 1], prev = a.list[(a.first_slot + r + 1) & 1];
  const EdgeList in = r == 0 ? a.in : EdgeList{prev.u, prev.v, prev.w, prev.id};
  u64 *counter = &a.st->ce[r];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t below = (1u << lane) - 1u;
  uint32_t *s_tot = &sm.out[0][0], *s_pos = s_tot + RW;  // per warp, per group
  for (uint64_t tile = (uint64_t)bid * RW + wid; tile / GROUP * GROUP * (32 * I) < m; tile += (uint64_t)nb * RW) {
    const uint64_t j0 = tile * (32 * I) + lane;
    uint32_t eu[I], ev[I], ew[I], ei[I];
#pragma unroll
    for (int k = 0; k < I; ++k) {
      const uint64_t j = j0 + 32 * k;
      const bool ok = j < m;
      eu[k] = ok ? __ldcg(in.u + j) : 0u;
      ev[k] = ok ? __ldcg(in.v + j) : eu[k];
      ew[k] = ok ? __ldcg(in.w + j) : 0u;
      ei[k] = ok && in.id ? __ldcg(in.id + j) : (uint32_t)j;
    }
#pragma unroll
    for (int k = 0; k < I; ++k) {
      const bool self = eu[k] == ev[k];
      eu[k] = self ? 0u : __ldca(link + eu[k]) & ~ROOT;
      ev[k] = self ? 0u : __ldca(link + ev[k]) & ~ROOT;
    }
    uint32_t keep[I], total = 0;
#pragma unroll
    for (int k = 0; k < I; ++k) {
      keep[k] = __ballot_sync(0xffffffffu, eu[k] != ev[k]);
      total += __popc(keep[k]);
    }
    if (lane == 0) s_tot[wid] = total;
    asm volatile("bar.sync %0, %1;" ::"r"(1 + wid / GROUP), "n"(32 * GROUP) : "memory");
    uint32_t sum = 0, mine = 0;
#pragma unroll
    for (int q = 0; q < GROUP; ++q) {
      const uint32_t t = s_tot[wid / GROUP * GROUP + q];
      mine += q < wid % GROUP ? t : 0u;
      sum += t;
    }
    if (wid % GROUP == 0 && lane == 0) s_pos[wid / GROUP] = sum ? (uint32_t)atomicAdd(counter, (u64)sum) : 0u;
    u64 cx[I], cy[I];
#pragma unroll
    for (int k = 0; k < I; ++k) {
      const bool has = eu[k] != ev[k];
      cx[k] = !has ? 0ULL : tab ? sm.tab[eu[k]] : __ldca(a.best + eu[k]);
      cy[k] = !has ? 0ULL : tab ? sm.tab[ev[k]] : __ldca(a.best + ev[k]);
    }
    asm volatile("bar.sync %0, %1;" ::"r"(1 + wid / GROUP), "n"(32 * GROUP) : "memory");
    uint32_t p = s_pos[wid / GROUP] + mine;
#pragma unroll
    for (int k = 0; k < I; ++k) {
      const uint32_t o = p + __popc(keep[k] & below);
      p += __popc(keep[k]);
      if (eu[k] == ev[k]) continue;
      out.u[o] = eu[k];
      out.v[o] = ev[k];
      out.w[o] = ew[k];
      out.id[o] = ei[k];
      const u64 kx = relax_key(kl, ew[k], ei[k], ev[k]), ky = relax_key(kl, ew[k], ei[k], eu[k]);
      if (tab) {
        if (kx < cx[k]) atomicMin(&sm.tab[eu[k]], kx);
        if (ky < cy[k]) atomicMin(&sm.tab[ev[k]], ky);
      } else {
        relax(a.best, eu[k], kx, cx[k]);
        relax(a.best, ev[k], ky, cy[k]);
      }
      if (!kl.packed) {
        a.cur_u[ei[k]] = eu[k];
        a.cur_v[ei[k]] = ev[k];
      }
    }
  }
}

// Clears the pairs' table.  It lies where the round's survivors would have gone
// (room for all of the round's edges, at least 4 np entries of 4 bytes).
__device__ __noinline__ void pair_clear(uint32_t *table_mem, uint32_t np, uint32_t nb, uint32_t bid) {
  for (uint32_t i = bid * RB + threadIdx.x; i < np; i += nb * RB) reinterpret_cast<u64 *>(table_mem)[i] = KEY_INF;
}

// Relabel of a round that leaves few components (at most PAIR_COMPS): of the
// edges between two components only the lightest can be in the forest, so the
// list shrinks to one entry per pair at once, and block 0 finishes the call
// on them.  Every block collects its pairs' minima in shared memory and then
// sends them to the table; nothing is staged or written per edge, and an edge's
// id is read only where its weight is not above the pair's minimum.  Bound by
// reading 12 bytes per edge: RMAT n=2^22 m=2^26, which keeps 64 million edges
// until its last rounds, passes over them in 241 us (3.2 TB/s; the shared-memory
// lookups are the rest); relabel, minEdges and three more rounds in its place made
// the solve 4.1 ms instead of 3.4.  The pair functions
// are calls, with their arguments by value: inlined, their registers cost the
// long phases spills (RGG2D's first relabel 200 -> 223 us).
template <int I>
__device__ __noinline__ void pair_phase(EdgeList in, const uint32_t *link, uint64_t m, uint32_t nc, uint32_t np,
                                        uint32_t *table_mem, uint32_t nb, uint32_t bid) {
  extern __shared__ __align__(128) unsigned char smem_dyn[];
  u64 *pt = reinterpret_cast<u64 *>(smem_dyn), *table = reinterpret_cast<u64 *>(table_mem);
  const bool lab = nc <= LABS;
  uint8_t *s_lab = reinterpret_cast<uint8_t *>(pt + PAIRS);
  for (uint32_t i = threadIdx.x; i < np; i += RB) pt[i] = KEY_INF;
  if (lab)
    for (uint32_t i = threadIdx.x; i < nc; i += RB) s_lab[i] = (uint8_t)__ldca(link + i);
  __syncthreads();
  constexpr uint64_t T = (uint64_t)RB * I;
  const uint64_t nfull = I == RI && aligned16_list(in) ? m / T : 0;
  uint32_t fu[I], fv[I], fw[I];  // the next tile
  const auto fetch = [&](uint64_t tile) {
    const uint64_t j0 = tile * T + (uint64_t)I * threadIdx.x;
    if constexpr (I == RI) {
      if (tile < nfull) {
        const uint4 x = __ldcg(reinterpret_cast<const uint4 *>(in.u + j0));
        const uint4 y = __ldcg(reinterpret_cast<const uint4 *>(in.v + j0));
        const uint4 z = __ldcg(reinterpret_cast<const uint4 *>(in.w + j0));
        fu[0] = x.x, fu[1] = x.y, fu[2] = x.z, fu[3] = x.w;
        fv[0] = y.x, fv[1] = y.y, fv[2] = y.z, fv[3] = y.w;
        fw[0] = z.x, fw[1] = z.y, fw[2] = z.z, fw[3] = z.w;
        return;
      }
    }
#pragma unroll
    for (int k = 0; k < I; ++k) {
      const bool ok = j0 + k < m;
      fu[k] = ok ? __ldca(in.u + j0 + k) : 0u;
      fv[k] = ok ? __ldca(in.v + j0 + k) : fu[k];
      fw[k] = ok ? __ldca(in.w + j0 + k) : 0u;
    }
  };
  fetch(bid);
  for (uint64_t tile = bid; tile * T < m; tile += nb) {
    const uint64_t j0 = tile * T + (uint64_t)I * threadIdx.x;
    uint32_t pi[I], ew[I];  // pair (PAIRS: both ends in one component) and weight
#pragma unroll
    for (int k = 0; k < I; ++k) {
      // the ends of an edge that is not there are equal
      const uint32_t x = lab ? s_lab[fu[k]] : __ldca(link + fu[k]) & ~ROOT;
      const uint32_t y = lab ? s_lab[fv[k]] : __ldca(link + fv[k]) & ~ROOT;
      const uint32_t hi = max(x, y);
      pi[k] = x == y ? PAIRS : hi * (hi - 1) / 2 + min(x, y);
      ew[k] = fw[k];
    }
    fetch(tile + nb);
#pragma unroll
    for (int k = 0; k < I; ++k) {
      if (pi[k] == PAIRS) continue;
      const u64 cur = pt[pi[k]];
      if (ew[k] > (uint32_t)(cur >> 32)) continue;
      const u64 key = (u64)ew[k] << 32 | (in.id ? __ldca(in.id + j0 + k) : (uint32_t)(j0 + k));
      if (key < cur) atomicMin(pt + pi[k], key);
    }
  }
  __syncthreads();
  // each block begins at another pair, so that they do not queue at the same ones
  const uint32_t first = (uint32_t)((uint64_t)np * bid / nb);
  for (uint32_t t = threadIdx.x; t < np; t += RB) {
    const uint32_t i = t + first < np ? t + first : t + first - np;
    const u64 k = pt[i];
    if (k != KEY_INF) relax(table, i, k, __ldca(table + i));
  }
}

// The call's last rounds over the table of pairs, in one block's shared memory:
// a warp looks through a component's row, and everything else is one thread per
// component: 17 us for all of them in GNM n=2^16 m=2^20 (108 components left); with
// the pairs written as a list, and rounds over that, the solve took 229 us instead
// of 204.
// rep: representatives of the nn components, replaced by those of their final
// ones; or nullptr.
__device__ __noinline__ void pair_rounds(const uint32_t *table_mem, uint32_t nn, uint32_t *chosen_bits, u64 *wsum,
                                         uint32_t *rep) {
  extern __shared__ __align__(128) unsigned char smem_dyn[];
  u64 *pt = reinterpret_cast<u64 *>(smem_dyn), *s_cmin = pt + PAIRS, *s_rmin = s_cmin + PAIR_COMPS;
  uint32_t *s_lab = reinterpret_cast<uint32_t *>(s_rmin + PAIR_COMPS), *s_far = s_lab + PAIR_COMPS,
           *s_part = s_far + PAIR_COMPS, *s_next = s_part + PAIR_COMPS;
  static_assert((PAIRS + 2 * PAIR_COMPS) * sizeof(u64) + 4 * PAIR_COMPS * sizeof(uint32_t) <= sizeof(Smem), "fits");
  const uint32_t t = threadIdx.x, lane = t & 31, wid = t >> 5, np = nn * (nn - 1) / 2;
  const bool comp = t < nn;
  for (uint32_t i = t; i < np; i += RB) pt[i] = __ldcg(reinterpret_cast<const u64 *>(table_mem) + i);
  if (comp) s_lab[t] = t;
  u64 wacc = 0;
  for (uint32_t round = 0; round < nn; ++round) {  // every round but the last merges
    if (comp) s_cmin[t] = KEY_INF;
    __syncthreads();
    for (uint32_t c = wid; c < nn; c += RW) {
      const uint32_t lc = s_lab[c];
      u64 k = KEY_INF;
      uint32_t far = 0;
      for (uint32_t d = lane; d < nn; d += 32) {
        if (s_lab[d] == lc) continue;
        const uint32_t h = max(c, d);
        const u64 q = pt[h * (h - 1) / 2 + min(c, d)];
        if (q < k) k = q, far = d;
      }
#pragma unroll
      for (int x = 16; x > 0; x >>= 1) {
        const u64 q = __shfl_xor_sync(0xffffffffu, k, x);
        const uint32_t d = __shfl_xor_sync(0xffffffffu, far, x);
        if (q < k) k = q, far = d;
      }
      if (lane == 0) {
        s_rmin[c] = k;
        s_far[c] = far;
        if (k != KEY_INF) atomicMin(s_cmin + lc, k);
      }
    }
    __syncthreads();
    // (an edge has one end in a component, so one row holds its minimum)
    if (comp && s_rmin[t] != KEY_INF && s_rmin[t] == s_cmin[s_lab[t]]) s_part[s_lab[t]] = s_lab[s_far[t]];
    __syncthreads();
    bool merges = false;
    if (comp && s_lab[t] == t) {
      const u64 k = s_cmin[t];
      merges = k != KEY_INF;
      const uint32_t y = merges ? s_part[t] : t;
      const bool root = !merges || (s_cmin[y] == k && t < y);
      s_next[t] = root ? t : y;
      if (!root) {
        atomicOr(chosen_bits + ((uint32_t)k >> 5), 1u << (k & 31));
        wacc += k >> 32;
      }
    }
    if (!__syncthreads_or(merges)) break;
    if (comp) {
      uint32_t q = s_next[s_lab[t]];
      for (uint32_t s = 0; s < nn && s_next[q] != q; ++s) q = s_next[q];
      s_lab[t] = q;
    }
  }
  wsum_add(wsum, wacc);
  if (rep) {
    __syncthreads();
    const uint32_t v = comp ? rep[s_lab[t]] : 0u;
    __syncthreads();
    if (comp) rep[t] = v;
  }
}

// The call's vertices (act) back to representatives in the caller's numbering:
// parent[v] = the representative of v's final component.
__device__ __forceinline__ void compose_phase(const RoundsArgs &a, const uint64_t *s_off, int levels) {
  const uint64_t cnt = a.st->ca;
  for (uint64_t i = (uint64_t)blockIdx.x * RB + threadIdx.x; i < cnt; i += (uint64_t)gridDim.x * RB) {
    const uint32_t v = __ldca(a.act + i);
    uint32_t d = a.parent[v] & ~ROOT;
    int l = 1;
    for (; l < levels; ++l) {
      const uint32_t q = __ldca(a.link + s_off[l] + d);
      if (q == FIN) break;
      d = q & ~ROOT;
    }
    a.parent[v] = __ldca(a.rep + s_off[l] + d);
  }
}

template <bool FIXED>
__global__ void __launch_bounds__(RB, 2) rounds_kernel(const __grid_constant__ RoundsArgs a) {
  extern __shared__ __align__(128) unsigned char smem_dyn[];
  Smem &sm = *reinterpret_cast<Smem *>(smem_dyn);
  __shared__ uint32_t s_warp[RW + 1], s_base[2];
  // the round's edges, vertices, next round's vertices, vertices to jump, and each round's part of link and rep
  __shared__ uint64_t s_m, s_nc, s_nn, s_cnt, s_off[ROUNDS_MAX + 2];
  __shared__ uint32_t s_np;  // pairs of the next round's components, if the round ends by pairs
  GridSync<FIXED> g{gridDim.x, blockIdx.x, &a.st->bar, a.err, a.spin_limit, 0, gridDim.x == 1};

  const uint64_t m0 = a.m_dev ? min((uint64_t)*a.m_dev, a.m) : a.m;
  const KeyLayout kl = resolve_layout(a.kl, a.max_w);
  if (!a.best_ready) {
    min_edges_phase(a, kl, m0, g.nb, g.bid);
    if (!g.sync()) return;
  }
  // an error set before the barrier, or by another block that gave up at it: one answer per block
  if (__syncthreads_or((int)(*(volatile uint32_t *)a.err & (ERR_VERTEX | ERR_OVERFLOW | ERR_ROUNDS)))) return;

  const bool rec0 = a.ends_rec || a.record_first;
  if (threadIdx.x == 0) {
    s_m = m0;
    s_off[0] = 0;
    s_off[1] = 0;
    s_nc = a.n;
  }
  __syncthreads();
  int r = 0;
  uint32_t pass = 0;
  bool ok = true, alone = false;
  for (; s_m > 0 && s_nc > 0; ++r) {
    if (r >= (int)a.max_rounds) {
      if (threadIdx.x == 0) atomicOr(a.err, ERR_JUMP);
      break;
    }
    if (s_nc >= (uint64_t)4 * RB * g.nb)
      hook_phase<HI>(a, kl, r, s_nc, s_off[r], r > 0 || rec0, g.nb, g.bid, sm, s_warp, s_base);
    else
      hook_short(a, kl, r, s_nc, s_off[r], r > 0 || rec0, g.nb, g.bid, sm);
    if (!(ok = g.sync())) break;
    if (threadIdx.x == 0) {  // components left with a root, vertices to jump
      s_nn = __ldca(&a.st->cv[r]);
      s_cnt = r == 0 ? __ldca(&a.st->ca) : s_nc;
      if (r > 0) s_off[r + 1] = s_off[r] + s_nc;
      // pairs where they are few beside the edges
      const uint32_t np = s_nn <= PAIR_COMPS ? (uint32_t)(s_nn * (s_nn - 1) / 2) : 0u;
      s_np = s_nn <= PAIR_COMPS && s_m > SOLO_EDGES && s_m >= (uint64_t)4 * np ? np : NO_PAIRS;
    }
    __syncthreads();
    // no vertex had an edge; or all are in one component, so no edge between
    // components is left (a star of 2^20 vertices and 2^23 edges read its edges
    // once more for nothing: 574 -> 532 us)
    if (s_nn == 0 || (s_nn == 1 && !a.want_parent)) {
      ++r;
      break;
    }
    for (uint32_t tries = 0;; ++tries, ++pass) {
      uint32_t *flag = &a.st->jflag[pass & 3];
      if (g.bid == 0 && threadIdx.x == 0) a.st->jflag[(pass + 2) & 3] = 0;
      jump_phase(a, r, s_cnt, s_off[r], tries == 0, flag, g.nb, g.bid);
      if (tries == 0 && s_np != NO_PAIRS) pair_clear(a.list[(a.first_slot + r) & 1].u, s_np, g.nb, g.bid);
      if (!(ok = g.sync()) || !__ldca(flag)) break;
      if (tries >= RPASSES) {
        if (threadIdx.x == 0) atomicOr(a.err, ERR_JUMP);
        ok = false;
        break;
      }
    }
    ++pass;
    if (!ok) break;
    if (s_nn == 1) {
      ++r;
      break;
    }
    if (s_np != NO_PAIRS) {
      const EdgeOut out = a.list[(a.first_slot + r) & 1], prev = a.list[(a.first_slot + r + 1) & 1];
      const EdgeList in = r == 0 ? a.in : EdgeList{prev.u, prev.v, prev.w, prev.id};
      const uint32_t *link = r == 0 ? a.parent : a.link + s_off[r];
      if (s_m >= (uint64_t)RT * g.nb)
        pair_phase<RI>(in, link, s_m, (uint32_t)s_nc, s_np, out.u, g.nb, g.bid);
      else
        pair_phase<1>(in, link, s_m, (uint32_t)s_nc, s_np, out.u, g.nb, g.bid);
      if (!(ok = g.sync())) break;
      alone = alone || !g.solo;
      if (blockIdx.x != 0) break;
      ++r;
      pair_rounds(out.u, (uint32_t)s_nn, a.chosen_bits, a.wsum, a.want_parent ? a.rep + s_off[r] : nullptr);
      break;
    }
    const bool tab = s_nn <= STAB;
    if (tab) {
      for (uint32_t i = threadIdx.x; i < (uint32_t)s_nn; i += RB) sm.tab[i] = KEY_INF;
      __syncthreads();
    }
    if (s_m >= (uint64_t)RT * g.nb)
      relabel_phase<RI>(a, kl, r, s_m, s_off[r], tab, g.nb, g.bid, sm);
    else
      relabel_phase<1>(a, kl, r, s_m, s_off[r], tab, g.nb, g.bid, sm);
    if (tab) {  // one atomic per component and block at most
      __syncthreads();
      for (uint32_t i = threadIdx.x; i < (uint32_t)s_nn; i += RB) {
        const u64 k = sm.tab[i];
        if (k != KEY_INF) relax(a.best, i, k, __ldca(a.best + i));
      }
    }
    if (!(ok = g.sync())) break;
    if (threadIdx.x == 0) {
      s_m = __ldca(&a.st->ce[r]);
      s_nc = s_nn;
    }
    __syncthreads();
    if (!g.solo && s_m > 0 && s_m <= SOLO_EDGES && s_nc <= SOLO_VERTS) {  // block 0 finishes alone
      alone = true;
      if (blockIdx.x != 0) break;
      g.solo = true;
      g.nb = 1;
    }
  }
  if (!ok || !a.want_parent) return;
  __syncthreads();
  if (alone) {  // the other blocks come back for the last pass and learn the rounds they missed
    if (blockIdx.x == 0) {
      for (int i = threadIdx.x; i <= r; i += RB) a.st->off[i] = s_off[i];
      if (threadIdx.x == 0) a.st->levels = (uint32_t)r;
    }
    g.solo = false;
    g.nb = gridDim.x;
    if (!g.sync()) return;
    if (blockIdx.x != 0) {
      r = (int)__ldcg(&a.st->levels);
      for (int i = threadIdx.x; i <= r; i += RB) s_off[i] = __ldcg(&a.st->off[i]);
    }
    __syncthreads();
  }
  compose_phase(a, s_off, r);
}

template <bool FIXED>
bool launch(const RoundsArgs &a, uint64_t max_edges, bool clear, int sms, cudaStream_t s) {
  static PerDevice per_sm_of;  // resident blocks per SM (0: not available)
  const int per_sm = per_sm_of.get(current_device(), []() -> int {
    int b = 0;
    if (cudaFuncSetAttribute(rounds_kernel<FIXED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem)) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, rounds_kernel<FIXED>, RB, sizeof(Smem)) != cudaSuccess)
      b = 0;
    cudaGetLastError();
    return b < 2 ? b : 2;
  });
  if (per_sm <= 0 || a.n >= ROOT) return false;
  if (clear && cudaMemsetAsync(a.st, 0, sizeof(RoundsState), s) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  // as many blocks as the first round's tiles can use; a graph that fits one
  // block's last rounds from the start needs no grid barrier at all
  const uint64_t want = std::max(max_edges, (uint64_t)a.n) / RB + 1;
  unsigned grid = (unsigned)std::min<uint64_t>(want, (uint64_t)sms * per_sm);
  if (max_edges <= SOLO_EDGES && a.n <= SOLO_VERTS) grid = 1;
  RoundsArgs arg = a;
  void *args[] = {&arg};
  if (cudaLaunchCooperativeKernel((const void *)rounds_kernel<FIXED>, dim3(grid), dim3(RB), args, sizeof(Smem), s) ==
      cudaSuccess)
    return true;
  cudaGetLastError();
  return false;
}

}  // namespace

bool launch_rounds(const RoundsArgs &a, uint64_t max_edges, bool clear, int sms, cudaStream_t s) {
  return a.spin_limit == BAR_SPINS ? launch<true>(a, max_edges, clear, sms, s)
                                   : launch<false>(a, max_edges, clear, sms, s);
}

}  // namespace mstgpu
