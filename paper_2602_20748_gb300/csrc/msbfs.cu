// Product-graph breadth-first search for many start vertices at once.
//
// What is computed (Section 2.2, automata-based approach): for every start
// vertex s, the product vertices (v, q) of G x DFA reachable from (s, q0),
// with a visited set per start vertex so that each is expanded once; (s, v)
// is a result when some reached (v, q) has q accepting (Definition 1).  The
// search runs level by level until the frontier is empty, with no hop limit
// (the paper's Section 3 shows hop-limited depth-first search losing
// answers).
//
// How (design of this engine, not the paper's hop-limited DFS / segment
// pooling): start vertices are packed as bit lanes, K = 64 * NW of them per
// lane group, G groups per launch.  For every (state, vertex, group) there is
// one K-bit word in each of three arrays: VIS (visited) and two frontier
// words used in ping-pong, laid out [state][vertex][group][word] so that the
// G words of one (state, vertex) are contiguous (G * 8 * NW bytes, 512 for
// 16 groups of 256 lanes).  A level is expanded either
//   * top-down ("push"): the sparse list of (group, state, vertex) frontier
//     entries is scanned, the out-edges on the labels of the state's
//     transitions are spread evenly over the lanes of a warp, and the new
//     lanes are OR-ed into the next frontier word with atomics; long rows are
//     cut into chunks shared by all warps (spill_chunk gives their length);
//   * bottom-up ("pull"): a warp takes 32 vertices and all groups at once: for
//     each in-edge on an incoming transition from a state that is present in
//     the frontier, it gathers the neighbour's G frontier words (one
//     coalesced 512-byte read) and ORs them into the vertex's; the gathers of
//     a warp's vertices are listed first and read several at a time
//     (pull_staged; pull_lanes with an automaton per lane); rows with at least
//     heavy_row in-edges are cut (at graph load) into chunks shared by all
//     warps; or
//   * top-down by block 0 alone when the frontier has few entries and edges
//     (SOLO_SLOTS, SOLO_EDGES): no grid barrier between such levels,
// chosen per level from the byte cost of each given the DFA states present
// in the frontier.  New lanes land in the next frontier word; a commit phase
// folds them into VIS and clears the old frontier.  The whole search is one
// persistent cooperative launch; levels are separated by a grid barrier whose
// waits are bounded by a time limit (on expiry the kernel records
// RPQ_ERR_TIMEOUT and returns).
#include <algorithm>

#include "device_common.cuh"
#include "grid_barrier.cuh"
#include "push_split.cuh"
#include "rpq_internal.h"

namespace rpq {

constexpr int BFS_THREADS = 256;

template <int NW>
struct Word {
  u64 w[NW];
};

template <int NW>
__device__ __forceinline__ Word<NW> load_cg(const u64 *p) {
  Word<NW> x;
  if constexpr (NW % 2 == 0) {
#pragma unroll
    for (int i = 0; i < NW; i += 2) {
      ulonglong2 a = __ldcg(reinterpret_cast<const ulonglong2 *>(p + i));
      x.w[i] = a.x;
      x.w[i + 1] = a.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < NW; i++) x.w[i] = __ldcg(p + i);
  }
  return x;
}

// PER consecutive words at p (16-byte aligned when PER is even), or all ones
// when !on.
template <int PER>
__device__ __forceinline__ void load_vis(const u64 *p, bool on, u64 (&v)[PER]) {
  if constexpr (PER % 2 == 0) {
#pragma unroll
    for (int k = 0; k < PER; k += 2) {
      const ulonglong2 a = on ? __ldcg(reinterpret_cast<const ulonglong2 *>(p + k)) : make_ulonglong2(~0ull, ~0ull);
      v[k] = a.x;
      v[k + 1] = a.y;
    }
  } else {
#pragma unroll
    for (int k = 0; k < PER; k++) v[k] = on ? __ldcg(p + k) : ~0ull;
  }
}

template <int NW>
__device__ __forceinline__ void store_w(u64 *p, const Word<NW> &x) {
  if constexpr (NW % 2 == 0) {
#pragma unroll
    for (int i = 0; i < NW; i += 2) *reinterpret_cast<ulonglong2 *>(p + i) = make_ulonglong2(x.w[i], x.w[i + 1]);
  } else {
#pragma unroll
    for (int i = 0; i < NW; i++) p[i] = x.w[i];
  }
}

template <int NW>
__device__ __forceinline__ bool any_bits(const Word<NW> &x) {
  u64 a = 0;
#pragma unroll
  for (int i = 0; i < NW; i++) a |= x.w[i];
  return a != 0;
}

template <int NW>
__device__ __forceinline__ u32 popc_w(const Word<NW> &x) {
  u32 c = 0;
#pragma unroll
  for (int i = 0; i < NW; i++) c += __popcll(x.w[i]);
  return c;
}

// First u64 of the word of (group g, state q, vertex v).
template <int NW>
__device__ __forceinline__ u64 widx(const BfsParams &p, u32 g, u32 q, u32 v) {
  return (((u64)q * p.n + v) * p.G + g) * NW;
}

// Automaton modes of a launch: one automaton for every lane (of one lane
// group, or of several), one per lane group (multi), or one per lane (lane
// mode; AM_LANES where its bottom-up levels are pull_lanes).
constexpr int AM_ONE = 0, AM_GROUP = 1, AM_LANE = 2, AM_MANY = 3, AM_LANES = 4;
constexpr bool per_lane(int am) { return am == AM_LANE || am == AM_LANES; }

// Automaton of group g: its own in multi mode, else the launch's (the union
// in lane mode).
template <int AM>
__device__ __forceinline__ const QueryDesc &gdesc(const BfsParams &p, u32 g) {
  if constexpr (AM == AM_GROUP)
    return p.qg[g];
  else
    return p.q;
}

// Out-degree of v summed over the labels leaving DFA state q; *rows (if
// given) gets the number of those labels present in the graph.
__device__ __forceinline__ u32 degsum(const BfsParams &p, const QueryDesc &qd, u32 q, u32 v, u32 *rows = nullptr) {
  u32 s = 0, r = 0;
  const u32 n1 = p.n + 1;
  for (u32 t = qd.out_begin[q]; t < qd.out_begin[q + 1]; t++) {
    u32 l = qd.out_label[t];
    if (l >= p.L) continue;
    const u32 *off = p.out_off + (u64)l * n1 + v;
    s += __ldg(off + 1) - __ldg(off);
    r++;
  }
  if (rows) *rows = r;
  return s;
}

// Lane mode: the rows a top-down step over (q, v) reads -- the out-degree of
// v summed over the union's transitions leaving q (returned; their number in
// *rows) -- and, for the lanes set in m (group g's words), each lane's own
// product-edge count: deg_l(v) for every label l its automaton leaves q on,
// added into W.
template <int NW>
__device__ __forceinline__ u32 la_degsum(const BfsParams &p, u32 q, u32 v, u32 g, const Word<NW> &m, u64 &W,
                                         u32 *rows) {
  // per (state, label) group: its transitions' lanes are disjoint, so the
  // lanes of m taking any of them are popc(m & OR of their masks); the
  // degree sum and row count still count every transition
  u32 s = 0, r = 0;
  const u32 n1 = p.n + 1;
  const u64 gw = (u64)p.G * NW;
  for (u32 gi = p.la_grp_begin[q]; gi < p.la_grp_begin[q + 1]; gi++) {
    const u32 e = p.la_grp[gi];
    const u32 l = e & 0xFFFFu, c = e >> 16;
    if (l >= p.L) continue;
    const u32 *off = p.out_off + (u64)l * n1 + v;
    const u32 d = __ldg(off + 1) - __ldg(off);
    const u64 *mk = p.la_gmask + gi * gw + (u64)g * NW;
    u32 lanes = 0;
#pragma unroll
    for (int k = 0; k < NW; k++) lanes += __popcll(m.w[k] & __ldg(mk + k));
    W += (u64)lanes * d;
    s += c * d;
    r += c;
  }
  *rows = r;
  return s;
}

// List entries are (group * Q + state) << 32 | vertex; this bit marks one that
// the bottom-up phase that produced it has committed.
constexpr u64 ENTRY_DONE = 1ull << 63;

// A warp's current run of reserved list slots [pos, end) (warp-uniform) and
// how many it reserves at a time in this phase (0: exactly what it appends).
struct Appender {
  u64 pos = 0, end = 0;
  u32 seg = 0;
};

// Warp-aggregated append of `entry` for the lanes with `take` set.  All 32
// lanes must call it.  With segments, the warp fills its reserved slots and
// reserves seg more with one atomic add when they run out, so the list
// counter sees one atomic per segment instead of one per append; slots left
// over are read (and skipped) by the next level and the commit.
__device__ __forceinline__ void warp_append(const BfsParams &p, Appender &a, bool take, u64 entry,
                                            unsigned long long *count, u64 *list) {
  const u32 b = __ballot_sync(FULL_MASK, take);
  if (!b) return;
  const u32 k = __popc(b), r = __popc(b & lanemask_lt());
  u64 at;
  if (a.seg == 0) {
    u64 base = 0;
    if (lane_id() == __ffs(b) - 1) base = atomicAdd(count, (unsigned long long)k);
    base = __shfl_sync(FULL_MASK, base, __ffs(b) - 1);
    at = base + r;
  } else {
    const u64 room = a.end - a.pos;
    u64 nb = 0;
    if (k > room) {
      if (lane_id() == 0) nb = atomicAdd(count, (unsigned long long)a.seg);
      nb = __shfl_sync(FULL_MASK, nb, 0);
    }
    at = r < room ? a.pos + r : nb + (r - room);
    if (k > room) {
      a.pos = nb + (k - room);
      a.end = nb + a.seg;
    } else {
      a.pos += k;
    }
  }
  if (take) {
    if (at < p.list_cap)
      list[at] = entry;
    else
      atomicCAS(&p.ctl->err, 0u, ERR_LIST_OVERFLOW);
  }
}

// End of a phase: the warp's reserved slots not used hold NO_ENTRY.
__device__ __forceinline__ void append_close(const BfsParams &p, Appender &a, u64 *list) {
  for (u64 i = a.pos + lane_id(); i < a.end; i += 32)
    if (i < p.list_cap) list[i] = NO_ENTRY;
  a.pos = a.end = 0;
}

// Adds v (the same in every lane) to one of the warp's statistics.
__device__ __forceinline__ void stat_add(u64 *stat, int i, u64 v) {
  if (lane_id() == 0) stat[i] += v;
}

template <int NW, int AM>
__device__ void seed_phase(const BfsParams &p, u64 *stat) {
  const u32 K = 64 * NW;
  const u64 total = (u64)p.G * K;
  const u64 stride = (u64)gridDim.x * blockDim.x;
  u64 W = 0, N = 0, mf = 0, gx = 0, gn = 0;
  Appender app;
  for (u64 base = (u64)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); base < total; base += stride) {
    u64 i = base + lane_id();
    bool take = false;
    u64 entry = 0;
    if (i < total) {
      u32 s = p.lanesrc[i];
      if (s != NO_SOURCE) {
        u32 g = (u32)(i / K), lane = (u32)(i % K);
        u64 wi = widx<NW>(p, g, 0, s);  // start state 0
        // lanes may repeat a start vertex, so seeds share words: atomics, and
        // one list entry per (group, vertex)
        const u64 bit = 1ull << (lane % 64);
        atomicOr((unsigned long long *)(p.vis + wi + lane / 64), bit);
        const u64 oldf = atomicOr((unsigned long long *)(p.fr0 + wi + lane / 64), bit);
        if constexpr (NW == 1)
          take = oldf == 0;
        else
          take = atomicMax(p.claim + ((u64)s * p.G + g), p.stamp_base + 1) < p.stamp_base + 1;
        entry = ((u64)g * p.Q << 32) | s;
        if (take && p.fbits) atomicOr(p.fbits + (s >> 5), 1u << (s & 31));  // state 0, bitmap 0
        u32 rows = 0, d;
        if constexpr (per_lane(AM)) {
          Word<NW> me;
#pragma unroll
          for (int k = 0; k < NW; k++) me.w[k] = (lane / 64 == (u32)k) ? bit : 0ull;
          d = la_degsum<NW>(p, 0, s, g, me, W, &rows);
        } else {
          d = degsum(p, gdesc<AM>(p, g), 0, s, &rows);
          W += d;
        }
        N += 1;
        if (take) {
          mf += d;
          gx += rows;
          gn += 1;
        }
      }
    }
    warp_append(p, app, take, entry, &p.ctl->n_list[0], p.list0);
  }
  append_close(p, app, p.list0);
  W = warp_sum(W);
  N = warp_sum(N);
  mf = warp_sum(mf);
  gx = warp_sum(gx);
  gn = warp_sum(gn);
  if (lane_id() == 0) {
    stat[ST_W] += W;
    stat[ST_N] += N;
    if (gx) atomicAdd(&p.ctl->stats[ST_GROUP_X], gx);
    if (mf) atomicAdd(&p.ctl->mf[0], mf);
    if (gn) atomicAdd(&p.ctl->n_true[0], gn);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&p.ctl->smask[0], 1u);
}

// Target of a top-down row: state and group, packed as in the rows' shared
// records (relax runs once per edge and would pay a division to unpack a list
// entry's group * Q + state).
__device__ __forceinline__ u32 pack_target(u32 q2, u32 g) { return q2 << 16 | g; }
__device__ __forceinline__ u64 target_entry(const BfsParams &p, u32 tg, u32 w) {
  return (u64)((tg & 0xFFFFu) * p.Q + (tg >> 16)) << 32 | w;
}

// One top-down relaxation of an edge to (target tg, w) with source lanes fm:
// the lanes not yet visited there are OR-ed into the next frontier word;
// returns whether this thread must list the target in the next frontier.
template <int NW>
__device__ __forceinline__ bool relax(const BfsParams &p, u64 *FB, u32 tg, u32 w, const u64 *fm, u32 stamp) {
  const u32 g = tg & 0xFFFFu, q2 = tg >> 16;
  const u64 wi = widx<NW>(p, g, q2, w);
  Word<NW> vis = load_cg<NW>(p.vis + wi);
  Word<NW> m;
#pragma unroll
  for (int i = 0; i < NW; i++) m.w[i] = fm[i] & ~vis.w[i];
  if (!any_bits(m)) return false;
  if constexpr (NW == 1) {
    u64 old = atomicOr((unsigned long long *)(FB + wi), m.w[0]);
    return old == 0;
  } else {
#pragma unroll
    for (int i = 0; i < NW; i++)
      if (m.w[i]) atomicOr((unsigned long long *)(FB + wi + i), m.w[i]);
    u32 old = atomicMax(p.claim + (((u64)q2 * p.n + w) * p.G + g), stamp);
    return old < stamp;
  }
}

// Top-down expansion of the entries of the current list.  A warp takes `grab`
// entries at a time and spreads the edges of their rows evenly over its lanes
// (prefix sum of row lengths, owner found by binary search); rows longer than
// `chunk` are queued in chunks for the spill sub-phase.  n_warps: the warps
// that share the level, those of the grid or of block 0 alone.  The entries'
// frontier words and the rows' targets are kept in the warp's shared scratch:
// an edge reads its owner's with three loads instead of ten shuffles, and the
// words do not sit in registers through the edge loop.
template <int NW, int AM>
__device__ void push_level(const BfsParams &p, int lp, u32 cur, u32 nxt, u64 n_cur, u64 mf, u64 n_warps, u32 chunk,
                           u32 seg, u32 stamp, u64 *scratch, u64 *stat) {
  // scratch: [32][NW] words of the entries, in lane mode [32][NW] of them
  // masked by the row's transition, [32] (first edge - prefix, target)
  u64 *s_fm = scratch + lane_id() * NW;
  u64 *s_words = per_lane(AM) ? scratch + 32 * NW : scratch;
  uint2 *s_row = reinterpret_cast<uint2 *>(s_words + 32 * NW);
  const u64 *list = lp ? p.list1 : p.list0;
  u64 *nlist = lp ? p.list0 : p.list1;
  const u64 *F = lp ? p.fr1 : p.fr0;
  u64 *FB = lp ? p.fr0 : p.fr1;
  const u32 Q = p.Q, n1 = p.n + 1;
  const u32 lane = lane_id();
  u64 edges = 0, rows = 0, entries = 0;
  Appender app;
  app.seg = seg;
  const u32 grab = push_grab(n_cur, mf, n_warps);
  for (u64 it = grid_warp() * grab; it < n_cur; it = next_item(&p.ctl->cursor[cur], n_warps, grab)) {
    u64 idx = it + lane;
    u64 e = lane < grab && idx < n_cur ? __ldcg(&list[idx]) : NO_ENTRY;
    bool valid = e != NO_ENTRY;
    if (!__any_sync(FULL_MASK, valid)) continue;
    if (!valid) e = 0;
    u32 gq = (u32)((e & ~ENTRY_DONE) >> 32), v = (u32)e;
    u32 g = gq / Q, q = gq - g * Q;
    __syncwarp();  // the previous entries' edges are done
    if (valid) store_w<NW>(s_fm, load_cg<NW>(F + widx<NW>(p, g, q, v)));
    entries += valid;
    const QueryDesc &qd = gdesc<AM>(p, valid ? g : 0);
    u32 t_beg, nt;
    if constexpr (per_lane(AM)) {
      t_beg = valid ? p.la_out_begin[q] : 0;
      nt = valid ? p.la_out_begin[q + 1] - t_beg : 0;
    } else {
      t_beg = valid ? qd.out_begin[q] : 0;
      nt = valid ? qd.out_begin[q + 1] - t_beg : 0;
    }
    u32 max_nt = __reduce_max_sync(FULL_MASK, nt);
    for (u32 j = 0; j < max_nt; j++) {
      u32 rbeg = 0, rlen = 0, tg = 0;
      if (per_lane(AM) && j) __syncwarp();  // the previous transition's edges are done
      if (j < nt) {
        u32 t = t_beg + j;
        u32 l, to;
        bool any = true;
        if constexpr (per_lane(AM)) {
          // the entry's lanes that take this transition
          const u32 e = p.la_trans[t];
          l = e & 0xFFFFu;
          to = e >> 16;
          const u64 *mk = p.la_mask + (u64)t * ((u64)p.G * NW) + (u64)g * NW;
          Word<NW> fmt;
#pragma unroll
          for (int k = 0; k < NW; k++) fmt.w[k] = s_fm[k] & __ldg(mk + k);
          any = any_bits(fmt);
          store_w<NW>(s_words + lane * NW, fmt);
        } else {
          l = qd.out_label[t];
          to = qd.out_to[t];
        }
        tg = pack_target(to, g);
        if (l < p.L && any) {
          const u32 *off = p.out_off + (u64)l * n1 + v;
          rbeg = __ldg(off);
          rlen = __ldg(off + 1) - rbeg;
          rows++;
        }
      }
      // long rows, one at a time: the warp writes a row's chunk records together
      const u32 longs = __ballot_sync(FULL_MASK, p.spill && rlen > chunk);
      if (longs) __syncwarp();
      for (u32 big = longs; big; big &= big - 1) {
        const u32 o = __ffs(big) - 1;
        const u32 o_beg = __shfl_sync(FULL_MASK, rbeg, o), o_len = __shfl_sync(FULL_MASK, rlen, o);
        const u32 o_tg = __shfl_sync(FULL_MASK, tg, o);
        u64 at = 0;
        u32 fit = 0;
        if (lane == 0) fit = spill_reserve(&p.ctl->spill_count[cur], (o_len + chunk - 1) / chunk, p.spill_cap, &at);
        at = __shfl_sync(FULL_MASK, at, 0);
        fit = __shfl_sync(FULL_MASK, fit, 0);
        for (u32 c = lane; c < fit; c += 32) {
          u64 *rec = p.spill + (at + c) * (2 + NW);
          rec[0] = ((u64)o_tg << 32) | (o_beg + c * chunk);
          rec[1] = min(chunk, o_len - c * chunk);
#pragma unroll
          for (int t = 0; t < NW; t++) rec[2 + t] = s_words[o * NW + t];
        }
        // the chunks that did not fit stay with this warp
        if (lane == o) {
          const u32 moved = min(rlen, fit * chunk);
          rbeg += moved;
          rlen -= moved;
        }
      }
      // exclusive prefix of row lengths across the warp
      u32 pre = rlen;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        u32 t = __shfl_up_sync(FULL_MASK, pre, o);
        if (lane >= (u32)o) pre += t;
      }
      u32 total = __shfl_sync(FULL_MASK, pre, 31);
      pre -= rlen;
      edges += (lane == 0) ? total : 0;
      if (total == 0) continue;
      if (!per_lane(AM)) __syncwarp();  // the previous transition's edges are done
      s_row[lane] = make_uint2(rbeg - pre, tg);
      __syncwarp();
      for (u32 k0 = 0; k0 < total; k0 += 32) {
        u32 k = k0 + lane;
        // owner: the largest lane o with pre[o] <= k
        u32 o = 0;
#pragma unroll
        for (u32 step = 16; step > 0; step >>= 1) {
          u32 pv = __shfl_sync(FULL_MASK, pre, o + step);
          if (pv <= k) o += step;
        }
        const uint2 row = s_row[o];
        bool take = false;
        u32 w = 0;
        if (k < total) {
          w = __ldg(p.out_col + (u32)(row.x + k));
          take = relax<NW>(p, FB, row.y, w, s_words + o * NW, stamp);
        }
        warp_append(p, app, take, target_entry(p, row.y, w), &p.ctl->n_list[nxt], nlist);
      }
    }
  }
  append_close(p, app, nlist);
  edges = warp_sum(edges);
  rows = warp_sum(rows);
  entries = warp_sum(entries);
  stat_add(stat, ST_GROUP_EDGES, edges);
  stat_add(stat, ST_GROUP_ROWS, rows);
  // per relaxation a column id and the target's visited word (the spilled
  // share is counted by the spill phase); per row its two offsets; per entry
  // the list entry and its frontier word
  stat_add(stat, ST_ALG_BYTES, edges * (4 + 8 * NW) + rows * 8 + entries * (8 + 8 * NW));
}

// The queued chunks of long rows: a warp per chunk, taken dynamically.
template <int NW>
__device__ void spill_phase(const BfsParams &p, int lp, u32 cur, u32 nxt, u32 seg, u32 stamp, u64 *stat) {
  u64 *nlist = lp ? p.list0 : p.list1;
  u64 *FB = lp ? p.fr0 : p.fr1;
  const u32 lane = lane_id();
  const u64 count = min(*(volatile unsigned long long *)&p.ctl->spill_count[cur], (unsigned long long)p.spill_cap);
  u64 edges = 0;
  Appender app;
  app.seg = seg;
  for (u64 it = grid_warp(); it < count; it = next_item(&p.ctl->spill_cursor[cur], grid_warps(), 1)) {
    const u64 *rec = p.spill + it * (2 + NW);
    const u64 h = __ldcg(rec);
    const u32 tg = (u32)(h >> 32), b = (u32)h;
    const u32 len = (u32)__ldcg(rec + 1);
    Word<NW> fm;
#pragma unroll
    for (int t = 0; t < NW; t++) fm.w[t] = __ldcg(rec + 2 + t);
    edges += (lane == 0) ? len : 0;
    for (u32 k0 = 0; k0 < len; k0 += 32) {
      u32 k = k0 + lane;
      bool take = false;
      u32 w = 0;
      if (k < len) {
        w = __ldg(p.out_col + b + k);
        take = relax<NW>(p, FB, tg, w, fm.w, stamp);
      }
      warp_append(p, app, take, target_entry(p, tg, w), &p.ctl->n_list[nxt], nlist);
    }
  }
  append_close(p, app, nlist);
  edges = warp_sum(edges);
  stat_add(stat, ST_GROUP_EDGES, edges);
  stat_add(stat, ST_ALG_BYTES, edges * (4 + 8 * NW));
}

// Bottom-up work for target (q2, w) over in-edges [beg, end) of one
// transition group with active source states `from`: every lane ORs the
// gathered frontier words of its PER words into acc.  With EARLY (few enough
// lanes that a vertex can run out of unvisited ones) a lane stops gathering
// once acc covers all its lanes not yet visited, and the sub-warp (lanes
// sg_mask) leaves the row when all its lanes have.  Returns the in-edges
// examined.
template <int NW, int PER, bool EARLY, bool LANE>
__device__ __forceinline__ u32 gather_row(const BfsParams &p, const u64 *F, const u32 *bits, u32 from, u32 beg,
                                          u32 end, u32 lane_off, bool lane_on, u32 sg_mask,
                                          const u64 (&vis)[PER], u64 (&acc)[PER], u32 &gathers,
                                          const unsigned short *tin) {
  const u32 n = p.n;
  const u64 wpv = (u64)p.G * NW;
  // lane mode: the gathered words of source state s are masked with the lanes
  // that take this group's transition from s (tin[s]); else all lanes
  auto lane_mask = [&](u32 st, u64 (&mk)[PER]) {
    if constexpr (LANE) {
      const u64 *mp = p.la_mask + (u64)tin[st] * wpv + lane_off;
#pragma unroll
      for (int k = 0; k < PER; k++) mk[k] = __ldg(mp + k);
    } else {
#pragma unroll
      for (int k = 0; k < PER; k++) mk[k] = ~0ull;
    }
  };
  auto done = [&]() {
    bool d = true;
#pragma unroll
    for (int k = 0; k < PER; k++) d &= (acc[k] | vis[k]) == ~0ull;
    return d;
  };
  // a lane with no source state on this row (another group's label in a
  // multi launch) has nothing to gather here
  bool fin = !lane_on || from == 0 || (EARLY && done());
  if (EARLY && (__ballot_sync(sg_mask, !fin) & sg_mask) == 0) return 0;
  u32 i = beg;
  // four in-edges per step keep four gathers in flight
  for (; i + 4 <= end; i += 4) {
    u32 v0 = __ldg(p.in_col + i), v1 = __ldg(p.in_col + i + 1), v2 = __ldg(p.in_col + i + 2),
        v3 = __ldg(p.in_col + i + 3);
    if (!fin) {
      for (u32 fb = from; fb; fb &= fb - 1) {
        u64 mk[PER];
        lane_mask(__ffs(fb) - 1, mk);
        const u64 qb = (u64)(__ffs(fb) - 1) * n;
        // with a frontier bitmap, neighbours outside the frontier are skipped
        bool h0 = true, h1 = true, h2 = true, h3 = true;
        if (bits) {
          h0 = (__ldcg(bits + ((qb + v0) >> 5)) >> ((qb + v0) & 31)) & 1u;
          h1 = (__ldcg(bits + ((qb + v1) >> 5)) >> ((qb + v1) & 31)) & 1u;
          h2 = (__ldcg(bits + ((qb + v2) >> 5)) >> ((qb + v2) & 31)) & 1u;
          h3 = (__ldcg(bits + ((qb + v3) >> 5)) >> ((qb + v3) & 31)) & 1u;
        }
        gathers += (u32)h0 + (u32)h1 + (u32)h2 + (u32)h3;
        const u64 *f0 = F + (qb + v0) * wpv + lane_off, *f1 = F + (qb + v1) * wpv + lane_off;
        const u64 *f2 = F + (qb + v2) * wpv + lane_off, *f3 = F + (qb + v3) * wpv + lane_off;
        if constexpr (PER == 2) {
          const ulonglong2 z = make_ulonglong2(0, 0);
          ulonglong2 a0 = h0 ? __ldcg(reinterpret_cast<const ulonglong2 *>(f0)) : z;
          ulonglong2 a1 = h1 ? __ldcg(reinterpret_cast<const ulonglong2 *>(f1)) : z;
          ulonglong2 a2 = h2 ? __ldcg(reinterpret_cast<const ulonglong2 *>(f2)) : z;
          ulonglong2 a3 = h3 ? __ldcg(reinterpret_cast<const ulonglong2 *>(f3)) : z;
          acc[0] |= (a0.x | a1.x | a2.x | a3.x) & mk[0];
          acc[1] |= (a0.y | a1.y | a2.y | a3.y) & mk[1];
        } else {
          acc[0] |= ((h0 ? __ldcg(f0) : 0ull) | (h1 ? __ldcg(f1) : 0ull) | (h2 ? __ldcg(f2) : 0ull) |
                     (h3 ? __ldcg(f3) : 0ull)) &
                    mk[0];
        }
      }
      if (EARLY) fin = done();
    }
    if (EARLY && (__ballot_sync(sg_mask, !fin) & sg_mask) == 0) return i + 4 - beg;
  }
  for (; i < end; i++) {
    u32 v = __ldg(p.in_col + i);
    if (fin) continue;
    for (u32 fb = from; fb; fb &= fb - 1) {
      const u64 bi = (u64)(__ffs(fb) - 1) * n + v;
      if (bits && !((__ldcg(bits + (bi >> 5)) >> (bi & 31)) & 1u)) continue;
      gathers++;
      u64 mk[PER];
      lane_mask(__ffs(fb) - 1, mk);
      const u64 *f = F + bi * wpv + lane_off;
#pragma unroll
      for (int k = 0; k < PER; k++) acc[k] |= __ldcg(f + k) & mk[k];
    }
  }
  return end - beg;
}

// Bottom-up target (q2, w), all groups: new lanes = acc & ~VIS go to the next
// frontier word, and one lane per group appends the list entry.  When chunks
// of long in-rows of the same vertex may also produce (q2, w) in this level
// (shared), the word is or-ed atomically and the entry is claimed (the first
// producer appends); otherwise this sub-warp is the only producer, the word
// was zero, and no atomic result has to be waited for.
template <int NW, int PER>
__device__ __forceinline__ void pull_finish(const BfsParams &p, Appender &app, u64 *FB, u64 *nlist, u32 nxt, u32 q2,
                                            u32 w, u32 stamp, u32 lane, bool lane_on, u32 my_g, bool shared,
                                            const u64 (&vis)[PER], const u64 (&acc)[PER]) {
  const u64 base = ((u64)q2 * p.n + w) * p.G * NW + (u64)lane * PER;
  bool take = false;
  bool nz = false;
  u64 nw[PER];
#pragma unroll
  for (int k = 0; k < PER; k++) {
    nw[k] = lane_on ? (acc[k] & ~vis[k]) : 0;
    nz |= nw[k] != 0;
  }
  if constexpr (NW == 1) {
    if (nz) {
      if (shared) {
        take = atomicOr((unsigned long long *)(FB + base), nw[0]) == 0;
      } else {
        FB[base] = nw[0];
        take = true;
      }
    }
  } else {
#pragma unroll
    for (int k = 0; k < PER; k++)
      if (nw[k]) {
        if (shared)
          atomicOr((unsigned long long *)(FB + base + k), nw[k]);
        else
          FB[base + k] = nw[k];
      }
    // NW / PER lanes hold one group's word
    bool gnz = nz;
#pragma unroll
    for (int o = 1; o < NW / PER; o <<= 1) gnz |= __shfl_xor_sync(FULL_MASK, gnz, o);
    if (gnz && lane_on && (lane % (NW / PER)) == 0)
      take = !shared || atomicMax(p.claim + (((u64)q2 * p.n + w) * p.G + my_g), stamp) < stamp;
  }
  warp_append(p, app, take, ((u64)(my_g * p.Q + q2) << 32) | w, &p.ctl->n_list[nxt], nlist);
}

// What a block's warps committed in a level, in shared memory: added to the
// control block once per block and level.  One atomic per warp and counter
// queued up to 4,864 x 5 of them on two lines: 4-5 us of every commit.
struct CommitSums {
  unsigned long long mf, gx, n_true;
  unsigned int smask;
};

// By one thread, when the block's warps have committed.  gx is kept to the end.
__device__ __forceinline__ void publish_sums(BfsCtl *c, CommitSums &s, u32 nxt) {
  if (s.n_true == 0) return;
  if (s.mf) atomicAdd(&c->mf[nxt], s.mf);
  atomicAdd(&c->n_true[nxt], s.n_true);
  atomicOr(&c->smask[nxt], s.smask);
  s.mf = s.n_true = 0;
  s.smask = 0;
}

// ---------------------------------------------------------------------------
// Bottom-up expansion of several lane groups under one automaton (G > 1, 256
// lanes each), the form of large source lists on graphs with rows of very
// different lengths (where all rows are long pull_level is faster, see
// set_chunks).
//
// What bounds it: gathers of G * 32 bytes from random rows of the frontier
// array.  Walking one vertex's in-row after another, the row offsets, the
// column ids and the gathers of every row were three dependent round trips,
// with at most four gathers in flight and one in a row's tail.  Here the
// gathers of 32 consecutive vertices are listed first, by all lanes together
// (coalesced offsets and column ids, one round trip each for the whole list),
// in shared memory; a vertex is then one round trip of up to six gathers (six
// and eight differ by 1%, four and eight by 2%).
// With a frontier bitmap only neighbours in the frontier are listed, and only
// vertices with such a neighbour read their visited words.
//
// A vertex produced by one sub-warp alone (no chunks of long rows, no second
// piece of the list) is also committed by it: it has the visited words in
// registers, and the vertex's degrees, counted once per vertex by the lane
// that lists it, serve all its groups; its entries carry ENTRY_DONE, and the
// commit phase passes over them.
// ---------------------------------------------------------------------------
constexpr u32 STAGE = 256;           // gathers listed at a time per warp
constexpr u64 STAGE_ROW = (1ull << 58) - 1;  // low bits: state * n + vertex; above: the owning vertex's lane


// The k-th set bit of m (0-based).
__device__ __forceinline__ u32 nth_bit(u32 m, u32 k) {
  for (; k; k--) m &= m - 1;
  return __ffs(m) - 1;
}

// ORs the listed rows lst[first], lst[first + step], ... below cnt into acc,
// DEEP gathers in flight.  Lanes that are off must pass cnt = 0.
template <int DEEP>
__device__ __forceinline__ void gather_list(const u64 *F, u64 wpv, u32 lane_off, const u64 *lst, u32 first, u32 step,
                                            u32 cnt, u64 (&acc)[2]) {
  for (u32 k = first; k < cnt; k += DEEP * step) {
    ulonglong2 a[DEEP];
#pragma unroll
    for (int t = 0; t < DEEP; t++) {
      const u32 j = k + t * step;
      a[t] = make_ulonglong2(0, 0);
      if (j < cnt)
        a[t] = __ldcg(reinterpret_cast<const ulonglong2 *>(F + (lst[j] & STAGE_ROW) * wpv + lane_off));
    }
#pragma unroll
    for (int t = 0; t < DEEP; t++) {
      acc[0] |= a[t].x;
      acc[1] |= a[t].y;
    }
  }
}

template <int NW>
__device__ void pull_staged(const BfsParams &p, int lp, u32 cur, u32 nxt, u32 active, u32 stamp, const u32 *bits,
                            u64 *scratch, CommitSums &sums, u64 *stat) {
  static_assert(NW == 4, "two words per lane, two lanes per group");
  const u64 *F = lp ? p.fr1 : p.fr0;
  u64 *FB = lp ? p.fr0 : p.fr1;
  u64 *nlist = lp ? p.list0 : p.list1;
  const u32 n = p.n, Q = p.Q, n1 = p.n + 1;
  const u32 lane = lane_id();
  const u32 lanes_used = p.G * 2;
  u32 SW = 1;
  while (SW < lanes_used) SW <<= 1;
  const u32 VPW = 32 / SW;  // vertices a warp works on at once
  const u32 sg = lane / SW, li = lane % SW;
  const bool lane_on = li < lanes_used;
  const u32 lane_off = li * 2, my_g = li / 2;
  const u64 wpv = (u64)p.G * NW;
  u64 *lst = scratch;  // [STAGE]
  // the listed vertices: lane | shared << 5 | rows << 6, first gather, gathers,
  // out-degree
  __shared__ uint4 s_vertex[BFS_THREADS / 32][32];
  uint4 *vertex = s_vertex[threadIdx.x >> 5];
  const bool chunked = p.hchunk != nullptr;
  const u64 gword = 8ull * NW * p.G;  // bytes of the G words of one (state, vertex)
  u64 W = 0, mf = 0;
  u32 N = 0, gv = 0, gx = 0, states = 0;
  Appender app;
  app.seg = (u64)n * Q * p.G >= grid_warps() * 2 * APPEND_SEG ? p.append_seg : min(p.append_seg, 32u);

  // Long in-rows first (the light rows' shorter items then fill the phase's
  // end): their precomputed chunks, a warp per (target state, transition
  // group, chunk), the sub-warps sharing the list.
  if (chunked) {
    for (u64 it = grid_warp();; it = next_item(&p.ctl->heavy_cursor[cur], grid_warps(), 1)) {
      u64 acc_base = 0, ci = 0;
      u32 q2 = 0, from = 0;
      bool found = false;
      for (u32 q = 0; q < Q && !found; q++)
        for (u32 j = p.q.in_begin[q]; j < p.q.in_begin[q + 1]; j++) {
          const u32 l = p.q.in_label[j];
          if (!(p.q.in_from[j] & active) || l >= p.L) continue;
          const u64 cnt = p.hchunk_end[l] - p.hchunk_beg[l];
          if (it < acc_base + cnt) {
            found = true;
            q2 = q;
            from = p.q.in_from[j] & active;
            ci = p.hchunk_beg[l] + (it - acc_base);
            break;
          }
          acc_base += cnt;
        }
      if (!found) break;
      const u32 *rec = p.hchunk + 3 * ci;
      const u32 w = __ldg(rec), beg = __ldg(rec + 1), len = __ldg(rec + 2) - beg;
      u64 vis[2], acc[2] = {0, 0};
      load_vis<2>(p.vis + ((u64)q2 * n + w) * wpv + lane_off, lane_on, vis);
      if (__all_sync(FULL_MASK, (vis[0] & vis[1]) == ~0ull)) continue;
      for (u32 fb = from; fb; fb &= fb - 1) {
        const u64 qb = (u64)(__ffs(fb) - 1) * n;
        for (u32 e0 = 0; e0 < len; e0 += STAGE) {
          u32 cnt = 0;
          __syncwarp();  // the previous list is consumed
          for (u32 k = e0; k < min(len, e0 + STAGE); k += 32) {
            u64 row = 0;
            bool in = k + lane < len;
            if (in) {
              row = qb + __ldg(p.in_col + beg + k + lane);
              if (bits) in = (__ldcg(bits + (row >> 5)) >> (row & 31)) & 1u;
            }
            const u32 b = __ballot_sync(FULL_MASK, in);
            if (in) lst[cnt + __popc(b & lanemask_lt())] = row;
            cnt += __popc(b);
          }
          __syncwarp();
          gather_list<6>(F, wpv, lane_off, lst, sg, VPW, lane_on ? cnt : 0, acc);
          stat_add(stat, ST_ALG_BYTES, cnt * gword);
        }
      }
      for (u32 o = SW; o < 32; o <<= 1) {
        acc[0] |= __shfl_xor_sync(FULL_MASK, acc[0], o);
        acc[1] |= __shfl_xor_sync(FULL_MASK, acc[1], o);
      }
      stat_add(stat, ST_PULL_EDGES, len);
      stat_add(stat, ST_PULL_VERTICES, 1);
      stat_add(stat, ST_ALG_BYTES, gword + len * (bits ? 8 : 4));
      pull_finish<NW, 2>(p, app, FB, nlist, nxt, q2, w, stamp, li, lane_on && sg == 0, my_g, true, vis, acc);
    }
  }

  u32 cv = 32;  // vertices a warp takes at a time (see pull_level)
  while (cv > VPW && n < 2 * grid_warps() * cv) cv >>= 1;
  for (u64 c0 = grid_warp() * cv; c0 < n;) {
    const u32 v = (u32)(c0 + lane);
    const bool mine = lane < cv && c0 + lane < n;
    for (u32 q2 = 0; q2 < Q; q2++) {
      const u32 gb = p.q.in_begin[q2], ge = p.q.in_begin[q2 + 1];
      // this lane's vertex: its light in-rows on active transitions (gathers
      // to list), and whether chunks of a long one produce it too
      u32 tot = 0, lens = 0;
      bool shared = false;
      if (mine)
        for (u32 j = gb; j < ge; j++) {
          const u32 from = p.q.in_from[j] & active, l = p.q.in_label[j];
          if (!from || l >= p.L) continue;
          const u32 *off = p.in_off + (u64)l * n1 + v;
          const u32 len = __ldg(off + 1) - __ldg(off);
          if (len >= p.heavy_row && chunked)
            shared = true;
          else
            lens += len, tot += len * __popc(from);
        }
      u32 pre = tot;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const u32 t = __shfl_up_sync(FULL_MASK, pre, o);
        if (lane >= (u32)o) pre += t;
      }
      const u32 T = __shfl_sync(FULL_MASK, pre, 31);
      if (T == 0) continue;
      pre -= tot;
      lens = __reduce_add_sync(FULL_MASK, lens);
      stat_add(stat, ST_PULL_EDGES, lens);
      stat_add(stat, ST_ALG_BYTES, lens * (bits ? 8 : 4));
      shared |= tot && pre / STAGE != (pre + tot - 1) / STAGE;  // listed in two pieces
      // the vertex's out-degree over the labels leaving q2, for its commit
      u32 rows = 0, deg = 0;
      if (tot && !shared) deg = degsum(p, p.q, q2, v, &rows);
      for (u32 p0 = 0; p0 < T; p0 += STAGE) {
        const u32 pend = min(T, p0 + STAGE);
        u32 listed = 0;
        __syncwarp();  // the previous list is consumed
        for (u32 k0 = p0; k0 < pend; k0 += 32) {
          const u32 k = k0 + lane;
          // owner: the largest lane o with pre[o] <= k
          u32 o = 0;
#pragma unroll
          for (u32 step = 16; step > 0; step >>= 1) {
            const u32 pv = __shfl_sync(FULL_MASK, pre, o + step);
            if (pv <= k) o += step;
          }
          u32 r = k - __shfl_sync(FULL_MASK, pre, o);
          bool in = k < pend;
          u64 row = 0;
          if (in) {
            // the r-th gather of vertex c0 + o: its groups in order, every
            // in-edge once per active source state
            u32 col = 0, st = 0;
            for (u32 j = gb; j < ge; j++) {
              const u32 from = p.q.in_from[j] & active, l = p.q.in_label[j];
              if (!from || l >= p.L) continue;
              const u32 *off = p.in_off + (u64)l * n1 + (u32)(c0 + o);
              const u32 beg = __ldg(off), len = __ldg(off + 1) - beg;
              if (len >= p.heavy_row && chunked) continue;
              const u32 np = __popc(from);
              if (r < len * np) {
                col = beg + (np == 1 ? r : r / np);
                st = nth_bit(from, np == 1 ? 0 : r % np);
                break;
              }
              r -= len * np;
            }
            row = (u64)st * n + __ldg(p.in_col + col);
            if (bits) in = (__ldcg(bits + (row >> 5)) >> (row & 31)) & 1u;
          }
          const u32 b = __ballot_sync(FULL_MASK, in);
          if (in) lst[listed + __popc(b & lanemask_lt())] = row | (u64)o << 58;
          listed += __popc(b);
        }
        __syncwarp();
        // this lane's vertex's part of the list: [first, first + cnt)
        u32 first, cnt;
        if (bits) {
          u32 lo = 0, hi = listed;
          while (lo < hi) {
            const u32 mid = (lo + hi) >> 1;
            if ((u32)(lst[mid] >> 58) < lane)
              lo = mid + 1;
            else
              hi = mid;
          }
          first = lo;
          const u32 up = __shfl_down_sync(FULL_MASK, lo, 1);
          cnt = (lane == 31 ? listed : up) - lo;
        } else {
          const u32 s = max(pre, p0), e = min(pre + tot, pend);
          first = s - p0;
          cnt = e > s ? e - s : 0;
        }
        const u32 M = __ballot_sync(FULL_MASK, cnt != 0);
        const u32 nz = __popc(M);
        if (cnt) vertex[__popc(M & lanemask_lt())] = make_uint4(lane | (u32)shared << 5 | rows << 6, first, cnt, deg);
        __syncwarp();
        stat_add(stat, ST_PULL_VERTICES, nz);
        stat_add(stat, ST_ALG_BYTES, (listed + nz) * gword);
        for (u32 r0 = 0; r0 < nz; r0 += VPW) {
          const bool work = r0 + sg < nz;
          const uint4 x = vertex[work ? r0 + sg : 0];
          const bool osh = (x.x >> 5) & 1u;
          const bool on = work && lane_on;
          const u32 w = (u32)c0 + (x.x & 31u);
          const u64 base = ((u64)q2 * n + w) * wpv + lane_off;
          u64 vis[2], acc[2] = {0, 0};
          load_vis<2>(p.vis + base, on, vis);
          gather_list<6>(F, wpv, lane_off, lst + x.y, 0, 1, on ? x.z : 0, acc);
          const u64 n0 = acc[0] & ~vis[0], n1w = acc[1] & ~vis[1];  // zero for lanes that are off
          const bool nz_l = (n0 | n1w) != 0;
          if (!__any_sync(FULL_MASK, nz_l)) continue;
          if (nz_l) {
            if (osh) {
              if (n0) atomicOr((unsigned long long *)(FB + base), n0);
              if (n1w) atomicOr((unsigned long long *)(FB + base + 1), n1w);
            } else {
              *reinterpret_cast<ulonglong2 *>(FB + base) = make_ulonglong2(n0, n1w);
              *reinterpret_cast<ulonglong2 *>(p.vis + base) = make_ulonglong2(vis[0] | n0, vis[1] | n1w);
              const u32 c = __popcll(n0) + __popcll(n1w);
              N += c;
              W += (u64)c * x.w;
            }
          }
          // one lane per group lists the entry
          bool take = __shfl_xor_sync(FULL_MASK, nz_l, 1) | nz_l;
          take = take && on && (li & 1) == 0;
          if (take && osh) take = atomicMax(p.claim + (((u64)q2 * n + w) * p.G + my_g), stamp) < stamp;
          if (take && !osh) {
            mf += x.w;
            gx += x.x >> 6;
            gv += 1;
            states |= 1u << q2;
          }
          warp_append(p, app, take, ((u64)(my_g * Q + q2) << 32) | w | (osh ? 0ull : ENTRY_DONE),
                      &p.ctl->n_list[nxt], nlist);
        }
      }
    }
    if (p.pull_dynamic)
      c0 = next_item(&p.ctl->cursor[cur], grid_warps(), cv);
    else
      c0 += grid_warps() * cv;
  }
  append_close(p, app, nlist);
  W = warp_sum(W);
  mf = warp_sum(mf);
  const u64 s_gv = warp_sum((u64)gv), s_gx = warp_sum((u64)gx);
  states = __reduce_or_sync(FULL_MASK, states);
  stat_add(stat, ST_W, W);
  stat_add(stat, ST_N, warp_sum((u64)N));
  // counted above: per in-edge a column id (and a bitmap word), per gather a
  // frontier row, per vertex its visited words; here per entry committed its
  // list entry, its new frontier word and its visited word written
  stat_add(stat, ST_ALG_BYTES, s_gv * (8 + 16 * NW));
  if (lane == 0 && s_gv) {
    atomicAdd(&sums.mf, mf);
    atomicAdd(&sums.gx, s_gx);
    atomicAdd(&sums.n_true, s_gv);
    atomicOr(&sums.smask, states);
  }
}

// ---------------------------------------------------------------------------
// Bottom-up expansion in lane mode, by source state, for launches whose lanes
// fill a warp's row (G * 2 > 16 lanes of two words) and whose union automaton
// has at most LANE_SRC_Q states.
//
// Target q2's new lanes at vertex w are the OR over the union's transitions
// t = (s, l, q2) and the in-edges (v, w) of label l of F[s][v] & mask(t).  A
// row F[s][v] serves every target of (s, l): it is gathered once and masked
// into the targets' accumulators (shared memory, one 16-byte word per lane and
// target).  What bounds it: the gathers, about one per in-edge and source
// state.  A vertex's rows are short and spread over its labels, so walking
// them one by one kept one or two gathers in flight, each behind its row's
// offsets and column ids.  Here the gathers of 16 in-edges at a time are
// listed by all lanes together, without the rows a frontier bitmap shows
// empty, and read eight at once whatever rows and labels they belong to; a
// row's gathers of one state are ORed before they are masked, and a vertex's
// visited words are read together when its list ends.  A batch of 4,096
// queries on R-MAT 2^22 (3,704 lanes, 8 states, 189 transitions): its three
// dense levels 90 / 105 / 103 -> 51 / 58 / 56 ms.  Masking every gather by
// itself (one apply per in-edge and state) took 82 / 101 / 99 ms: the masks
// and accumulators pass the load/store unit once per target of each.  Three
// blocks per SM (80 registers) beat four (314 against 327 ms of traversal).
// ---------------------------------------------------------------------------
constexpr u32 LANE_EDGES = 16;                          // in-edges listed at a time
constexpr u32 LANE_LIST = LANE_EDGES * LANE_SRC_Q;      // their gathers
constexpr u64 LANE_ROW = (1ull << 44) - 1;              // state * n + vertex; above: label * 8 + state, owner lane

struct LaneTables {  // of a level, in shared memory
  u32 grp[RPQ_MAX_LABELS * LANE_SRC_Q];  // [label][state]: first transition | targets << 16 (0: none, or state not active)
  unsigned char act[RPQ_MAX_LABELS];     // [label]: active states with a transition on it
};

template <int NW>
__device__ void pull_lanes(const BfsParams &p, int lp, u32 cur, u32 nxt, u32 active, u32 stamp, const u32 *bits,
                           u64 *scratch, LaneTables &tab, u64 *stat) {
  static_assert(NW == 4, "two words per lane");
  const u64 *F = lp ? p.fr1 : p.fr0;
  u64 *FB = lp ? p.fr0 : p.fr1;
  u64 *nlist = lp ? p.list0 : p.list1;
  const u32 n = p.n, Q = p.Q, L = p.L, n1 = p.n + 1;
  const u32 lane = lane_id();
  const bool lane_on = lane < p.G * 2;
  const u32 lane_off = lane * 2;
  const u64 wpv = (u64)p.G * NW, gword = 8ull * NW * p.G;
  ulonglong2 *sacc = reinterpret_cast<ulonglong2 *>(scratch) + lane;  // target q2's words at sacc[32 * q2]
  u64 *lst = scratch + LANE_SRC_Q * 2 * 32;                           // [LANE_LIST]
  const bool chunked = p.hchunk != nullptr;
  u32 *nbits = p.fbits ? p.fbits + (lp ? 0 : p.fbits_words) : nullptr;  // the next frontier's bitmap
  Appender app;
  app.seg = (u64)n * Q * p.G >= grid_warps() * 2 * APPEND_SEG ? p.append_seg : min(p.append_seg, 32u);

  for (u32 i = threadIdx.x; i < L * LANE_SRC_Q; i += blockDim.x) {
    const u32 l = i / LANE_SRC_Q, s = i % LANE_SRC_Q;
    tab.grp[i] = s < Q && ((active >> s) & 1u) ? p.la_sl[s * L + l] : 0u;
  }
  __syncthreads();
  u64 lset = 0;  // labels with an active transition
  u32 sts_all = 0;  // states with one
  for (u32 l = 0; l < L; l++) {
    u32 a = 0;
    for (u32 s = 0; s < Q; s++) a |= (tab.grp[l * LANE_SRC_Q + s] >> 16 ? 1u : 0u) << s;
    if (a) lset |= 1ull << l;
    sts_all |= a;
    if (threadIdx.x == 0) tab.act[l] = (unsigned char)a;
  }
  __syncthreads();

  u32 tmask = 0;  // targets with an accumulator
  // row (words r) of a gather from (label, state) tag into its targets
  auto apply = [&](u32 tag, const ulonglong2 r) {
    const u32 e = tab.grp[tag];
    u64 at = (u64)(e & 0xFFFFu) * wpv + lane_off;
    for (u32 tm = e >> 16; tm; tm &= tm - 1, at += wpv) {
      const u32 to = __ffs(tm) - 1;
      ulonglong2 m = make_ulonglong2(0, 0);
      if (lane_on) m = __ldg(reinterpret_cast<const ulonglong2 *>(p.la_mask + at));
      m.x &= r.x;
      m.y &= r.y;
      if ((tmask >> to) & 1u) {
        const ulonglong2 a = sacc[32 * to];
        m.x |= a.x;
        m.y |= a.y;
      }
      sacc[32 * to] = m;
      tmask |= 1u << to;
    }
  };
  // the accumulated vertex: lanes not yet visited go to the next frontier
  auto flush = [&](u32 w, bool shared) {
    ulonglong2 v[LANE_SRC_Q];
#pragma unroll
    for (u32 q2 = 0; q2 < LANE_SRC_Q; q2++) {
      v[q2] = make_ulonglong2(~0ull, ~0ull);
      if (lane_on && ((tmask >> q2) & 1u))
        v[q2] = __ldcg(reinterpret_cast<const ulonglong2 *>(p.vis + ((u64)q2 * n + w) * wpv + lane_off));
    }
    u32 found = 0;
#pragma unroll
    for (u32 q2 = 0; q2 < LANE_SRC_Q; q2++)
      if ((tmask >> q2) & 1u) {
        ulonglong2 a = sacc[32 * q2];
        a.x &= ~v[q2].x;
        a.y &= ~v[q2].y;
        sacc[32 * q2] = a;
        if (a.x | a.y) found |= 1u << q2;
      }
    stat_add(stat, ST_PULL_VERTICES, __popc(tmask));
    stat_add(stat, ST_ALG_BYTES, __popc(tmask) * gword);
    u32 any = __reduce_or_sync(FULL_MASK, found);
    for (; any; any &= any - 1) {
      const u32 q2 = __ffs(any) - 1;
      const bool nz = (found >> q2) & 1u;
      if (lane == 0 && nbits) {
        const u64 bi = (u64)q2 * n + w;
        atomicOr(nbits + (bi >> 5), 1u << (bi & 31));
      }
      const u64 base = ((u64)q2 * n + w) * wpv + lane_off;
      if (nz) {
        const ulonglong2 a = sacc[32 * q2];
        if (shared) {
          if (a.x) atomicOr((unsigned long long *)(FB + base), a.x);
          if (a.y) atomicOr((unsigned long long *)(FB + base + 1), a.y);
        } else {
          *reinterpret_cast<ulonglong2 *>(FB + base) = a;
        }
      }
      bool take = __shfl_xor_sync(FULL_MASK, nz, 1) | nz;
      take = take && (lane & 1) == 0;
      if (take && shared)
        take = atomicMax(p.claim + (((u64)q2 * n + w) * p.G + lane / 2), stamp) < stamp;
      warp_append(p, app, take, ((u64)(lane / 2 * Q + q2) << 32) | w, &p.ctl->n_list[nxt], nlist);
    }
    tmask = 0;
  };

  // Long in-rows first, an item per (label, chunk): the chunk's rows of each
  // active source state are ORed together and masked once.
  if (chunked) {
    for (u64 it = grid_warp();; it = next_item(&p.ctl->heavy_cursor[cur], grid_warps(), 1)) {
      u64 acc_base = 0, ci = 0;
      u32 l = 0;
      bool found = false;
      for (u64 lb = lset; lb && !found; lb &= lb - 1) {
        l = __ffsll((long long)lb) - 1;
        const u64 cnt = p.hchunk_end[l] - p.hchunk_beg[l];
        found = it < acc_base + cnt;
        if (found) ci = p.hchunk_beg[l] + (it - acc_base);
        acc_base += cnt;
      }
      if (!found) break;
      const u32 *rec = p.hchunk + 3 * ci;
      const u32 w = __ldg(rec), beg = __ldg(rec + 1), len = __ldg(rec + 2) - beg;
      for (u32 sm = tab.act[l]; sm; sm &= sm - 1) {
        const u32 st = __ffs(sm) - 1;
        u64 g[2] = {0, 0};
        for (u32 e0 = 0; e0 < len; e0 += LANE_LIST) {
          u32 cnt = 0;
          __syncwarp();  // the previous list is consumed
          for (u32 k = e0; k < min(len, e0 + LANE_LIST); k += 32) {
            u64 row = 0;
            bool in = k + lane < len;
            if (in) {
              row = (u64)st * n + __ldg(p.in_col + beg + k + lane);
              if (bits) in = (__ldcg(bits + (row >> 5)) >> (row & 31)) & 1u;
            }
            const u32 b = __ballot_sync(FULL_MASK, in);
            if (in) lst[cnt + __popc(b & lanemask_lt())] = row;
            cnt += __popc(b);
          }
          __syncwarp();
          gather_list<8>(F, wpv, lane_off, lst, 0, 1, lane_on ? cnt : 0, g);
          stat_add(stat, ST_ALG_BYTES, cnt * gword);
        }
        if (__any_sync(FULL_MASK, (g[0] | g[1]) != 0)) apply(l * LANE_SRC_Q + st, make_ulonglong2(g[0], g[1]));
      }
      stat_add(stat, ST_PULL_EDGES, len);
      stat_add(stat, ST_ALG_BYTES, len * 4);
      if (tmask) flush(w, true);
    }
  }

  u32 cv = 32;  // vertices a warp takes at a time (see pull_level)
  while (cv > 1 && n < 2 * grid_warps() * cv) cv >>= 1;
  for (u64 c0 = grid_warp() * cv; c0 < n;) {
    // this lane's vertex: its light in-edges on active labels, and whether
    // chunks of a long row produce it too
    u32 tot = 0;
    bool sh = false;
    if (lane < cv && c0 + lane < n)
      for (u64 lb = lset; lb; lb &= lb - 1) {
        const u32 *off = p.in_off + (u64)(__ffsll((long long)lb) - 1) * n1 + c0 + lane;
        const u32 len = __ldg(off + 1) - __ldg(off);
        if (len >= p.heavy_row && chunked)
          sh = true;
        else
          tot += len;
      }
    const u32 shared = __ballot_sync(FULL_MASK, sh);
    u32 pre = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u32 t = __shfl_up_sync(FULL_MASK, pre, o);
      if (lane >= (u32)o) pre += t;
    }
    const u32 T = __shfl_sync(FULL_MASK, pre, 31);
    pre -= tot;
    stat_add(stat, ST_PULL_EDGES, T);
    stat_add(stat, ST_ALG_BYTES, T * 4ull);
    u32 own = 32;  // lane of the vertex being accumulated (32: none)
    for (u32 p0 = 0; p0 < T; p0 += LANE_EDGES) {
      // in-edges p0 + lane: owner, label, the states to gather it from
      const u32 k = p0 + lane;
      u32 o = 0;
#pragma unroll
      for (u32 step = 16; step > 0; step >>= 1) {
        const u32 pv = __shfl_sync(FULL_MASK, pre, o + step);
        if (pv <= k) o += step;
      }
      u32 r = k - __shfl_sync(FULL_MASK, pre, o);
      u32 l = 0, u = 0, sm = 0;
      if (lane < LANE_EDGES && k < T) {
        for (u64 lb = lset; lb; lb &= lb - 1) {
          l = __ffsll((long long)lb) - 1;
          const u32 *off = p.in_off + (u64)l * n1 + c0 + o;
          const u32 beg = __ldg(off), len = __ldg(off + 1) - beg;
          if (len >= p.heavy_row && chunked) continue;
          if (r < len) {
            u = __ldg(p.in_col + beg + r);
            sm = tab.act[l];
            break;
          }
          r -= len;
        }
        if (bits) {
          u32 bw[LANE_SRC_Q];
#pragma unroll
          for (u32 st = 0; st < LANE_SRC_Q; st++) {
            const u64 row = (u64)st * n + u;
            bw[st] = (sm >> st) & 1u ? __ldcg(bits + (row >> 5)) >> (row & 31) : 0u;
          }
          sm = 0;
#pragma unroll
          for (u32 st = 0; st < LANE_SRC_Q; st++) sm |= (bw[st] & 1u) << st;
        }
      }
      u32 at = __popc(sm);
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const u32 t = __shfl_up_sync(FULL_MASK, at, d);
        if (lane >= (u32)d) at += t;
      }
      const u32 listed = __shfl_sync(FULL_MASK, at, 31);
      at -= __popc(sm);
      // a row's gathers are listed state by state, so that a state's rows are
      // ORed before they are masked: behind those of the row's smaller states
      // and of its earlier in-edges
      const u32 same = __match_any_sync(FULL_MASK, lane < LANE_EDGES && k < T ? o << 6 | l : 1u << 31 | lane);
      at = __shfl_sync(FULL_MASK, at, __ffs(same) - 1);
      __syncwarp();  // the previous list is consumed
      auto entry = [&](u32 st) {
        return ((u64)st * n + u) | (u64)(l * LANE_SRC_Q + st) << 44 | (u64)o << 58;
      };
      if (bits) {
        for (u32 sts = sts_all; sts; sts &= sts - 1) {
          const u32 st = __ffs(sts) - 1;
          const u32 has = __ballot_sync(FULL_MASK, (sm >> st) & 1u) & same;
          if ((sm >> st) & 1u) lst[at + __popc(has & lanemask_lt())] = entry(st);
          at += __popc(has);
        }
      } else {  // every in-edge of the row has the same states
        at += __popc(same & lanemask_lt());
        for (u32 m = sm; m; m &= m - 1, at += __popc(same)) lst[at] = entry(__ffs(m) - 1);
      }
      __syncwarp();
      stat_add(stat, ST_ALG_BYTES, listed * gword);
      for (u32 i = 0; i < listed;) {
        const u32 o2 = (u32)(lst[i] >> 58);
        if (o2 != own) {
          if (tmask) flush((u32)c0 + own, (shared >> own) & 1u);
          own = o2;
        }
        // the run of this vertex in the list: [i, j)
        u32 j = i, hi = listed;
        while (j < hi) {
          const u32 mid = (j + hi) >> 1;
          if ((u32)(lst[mid] >> 58) == o2)
            j = mid + 1;
          else
            hi = mid;
        }
        constexpr u32 DEEP = 8;
        ulonglong2 g = make_ulonglong2(0, 0);
        for (; i < j; i += DEEP) {
          ulonglong2 a[DEEP];
#pragma unroll
          for (u32 t = 0; t < DEEP; t++) {
            a[t] = make_ulonglong2(0, 0);
            if (lane_on && i + t < j)
              a[t] = __ldcg(reinterpret_cast<const ulonglong2 *>(F + (lst[i + t] & LANE_ROW) * wpv + lane_off));
          }
#pragma unroll
          for (u32 t = 0; t < DEEP; t++)
            if (i + t < j) {
              g.x |= a[t].x;
              g.y |= a[t].y;
              const u32 tag = (u32)(lst[i + t] >> 44);
              if (i + t + 1 < j && (u32)(lst[i + t + 1] >> 44) == tag) continue;
              if (__any_sync(FULL_MASK, (g.x | g.y) != 0)) apply(tag & (RPQ_MAX_LABELS * LANE_SRC_Q - 1), g);
              g = make_ulonglong2(0, 0);
            }
        }
        i = j;
      }
    }
    if (tmask) flush((u32)c0 + own, (shared >> own) & 1u);
    if (p.pull_dynamic)
      c0 = next_item(&p.ctl->cursor[cur], grid_warps(), cv);
    else
      c0 += grid_warps() * cv;
  }
  append_close(p, app, nlist);
}

// Bottom-up expansion.  Light rows: one vertex per sub-warp of SW lanes (the
// smallest power of two holding the vertex's G * NW words at PER words per
// lane), all groups at once, so a warp covers 32 / SW vertices (32 for a
// single start vertex).  Long rows: their precomputed chunks, a warp per
// chunk taken dynamically over the (target state, transition group) pairs
// whose source states are active; the sub-warps split the chunk's edges and
// OR their gathers together.
template <int NW, int AM>
__device__ void pull_level(const BfsParams &p, int lp, u32 cur, u32 nxt, u32 active, u32 stamp, const u32 *bits,
                           u64 *scratch, u64 *stat) {
  constexpr int PER = (NW >= 2) ? 2 : 1;
  const u64 *F = lp ? p.fr1 : p.fr0;
  u64 *FB = lp ? p.fr0 : p.fr1;
  u64 *nlist = lp ? p.list0 : p.list1;
  const u32 n = p.n, Q = p.Q, n1 = p.n + 1;
  const u32 lane = lane_id();
  const u32 lanes_used = p.G * NW / PER;
  u32 SW = 1;
  while (SW < lanes_used) SW <<= 1;
  const u32 VPW = 32 / SW;  // vertices per warp
  const u32 sg = lane / SW, li = lane % SW;
  const u32 sg_mask = SW == 32 ? FULL_MASK : (((1u << SW) - 1u) << (sg * SW));
  const bool lane_on = li < lanes_used;
  const u32 lane_off = li * PER;
  const u32 my_g = lane_on ? lane_off / NW : 0;
  const u64 wpv = (u64)p.G * NW;
  const u64 warp = grid_warp(), n_warps = grid_warps();
  // vertices a warp takes at a time: 32, fewer (but no fewer than it works on
  // at once) on graphs too small to give every warp two such chunks
  u32 cv = 32;
  while (cv > VPW && n < 2 * n_warps * cv) cv >>= 1;
  const bool chunked = p.hchunk != nullptr;
  const u64 gword = 8ull * NW * p.G;  // bytes of the G words of one (state, vertex)
  u64 edges = 0, words = 0, bytes = 0;
  Appender app;
  // small graphs: shorter segments, so that unused slots do not outnumber the entries
  app.seg = (u64)n * Q * p.G >= n_warps * 2 * APPEND_SEG ? p.append_seg : min(p.append_seg, 32u);
  // lane mode by source state: this warp's per-target accumulators
  u64 *lane_acc = scratch;

  // A warp takes cv consecutive vertices at a time: lane i first finds, with
  // coalesced reads of the in-row offsets, the target states into which
  // vertex c0 + i has a light in-row on an active transition; only those
  // (vertex, state) pairs are then visited, VPW vertices at a time (their
  // offsets are in L1 by then).  With pull_dynamic the chunks are taken from
  // a cursor (the level's list cursor, unused by bottom-up levels), so a
  // warp whose chunks had little work takes more of them; else chunk k goes
  // to warp k mod warps.
  for (u64 c0 = warp * cv; c0 < n;) {
    // hmask: states with a long in-row (its chunks also produce); with a
    // sparse frontier (bits), lane i also tests up to PRESCAN in-edges of
    // its own vertex against the frontier bitmap, so that a state none of
    // whose in-neighbours is in the frontier is dropped here, 32 vertices at
    // a time; tmask: states whose light rows are longer than that and showed
    // no hit yet -- the sub-warp tests the rest of them below
    constexpr u32 PRESCAN = 16;
    u32 qmask = 0, hmask = 0, tmask = 0;
    if (lane < cv && c0 + lane < n) {
      const u32 v = (u32)(c0 + lane);
      for (u32 q2 = 0; q2 < Q; q2++)
        for (u32 j = p.q.in_begin[q2]; j < p.q.in_begin[q2 + 1]; j++) {
          const u32 l = p.q.in_label[j];
          const u32 from = p.q.in_from[j] & active;
          if (!from || l >= p.L) continue;
          const u32 *off = p.in_off + (u64)l * n1 + v;
          const u32 beg = __ldg(off), len = __ldg(off + 1) - beg;
          if (len >= p.heavy_row && chunked) {
            hmask |= 1u << q2;
            continue;
          }
          if (len == 0 || (((qmask & ~tmask) >> q2) & 1u)) continue;  // a hit is known already
          if (!bits) {
            qmask |= 1u << q2;
            continue;
          }
          bool hit = false;
          const u32 scan = min(len, PRESCAN);
          for (u32 i = 0; i < scan && !hit; i += 4) {
            u32 u[4];
#pragma unroll
            for (int t = 0; t < 4; t++) u[t] = i + t < scan ? __ldg(p.in_col + beg + i + t) : NO_SOURCE;
            for (u32 fb = from; fb; fb &= fb - 1) {
              const u64 qb = (u64)(__ffs(fb) - 1) * n;
#pragma unroll
              for (int t = 0; t < 4; t++)
                if (u[t] != NO_SOURCE) hit |= (__ldcg(bits + ((qb + u[t]) >> 5)) >> ((qb + u[t]) & 31)) & 1u;
            }
          }
          bytes += (u64)scan * (4 + 4 * __popc(from));
          if (hit) {
            qmask |= 1u << q2;
            tmask &= ~(1u << q2);
          } else if (len > PRESCAN) {
            qmask |= 1u << q2;
            tmask |= 1u << q2;
          }
        }
    }
    const u32 M = __ballot_sync(FULL_MASK, qmask != 0);
    for (u32 s0 = 0; s0 < 32 && (M >> s0); s0 += VPW) {
      if (VPW < 32 && ((M >> s0) & ((1u << VPW) - 1u)) == 0) continue;
      const u32 s = s0 + sg;
      const u32 vq = __shfl_sync(FULL_MASK, qmask, s);
      const u32 vh = __shfl_sync(FULL_MASK, hmask, s);
      const u32 vt = __shfl_sync(FULL_MASK, tmask, s);
      const bool wv = vq != 0;
      const u32 w = wv ? (u32)(c0 + s) : 0;
    if constexpr (AM == AM_LANE) {
      if (p.lane_by_source && Q <= LANE_SRC_Q) {
        // Lane mode by source state.  Target q2's new lanes are the OR over
        // its union transitions t = (s, l, q2) and the in-edges (v, w) of
        // label l of F[s][v] & mask(t); since the mask does not depend on v,
        // that is the OR over t of mask(t) & (OR over v of F[s][v]).  So the
        // frontier words of each (label, source state) are gathered once and
        // ORed over the in-edges, then masked into every target taking a
        // transition from them (accumulated per lane in shared memory); the
        // per-target order gathers each (s, v) once per target instead.
        u64 *sacc = lane_acc;  // [q2][k][lane]
        u32 wmask = 0;  // targets with lanes to find (uniform within the sub-warp)
        for (u32 q2 = 0; q2 < Q; q2++) {
          const bool any = wv && ((vq >> q2) & 1u);
          u64 vis[PER];
          load_vis<PER>(p.vis + ((u64)q2 * n + w) * wpv + lane_off, lane_on && any, vis);
          bool full = true;
#pragma unroll
          for (int k = 0; k < PER; k++) {
            full &= vis[k] == ~0ull;
            sacc[(q2 * PER + k) * 32 + lane] = 0;
          }
          const u32 fb = __ballot_sync(FULL_MASK, full);
          if (any && (fb & sg_mask) != sg_mask) wmask |= 1u << q2;
        }
        u64 lset = 0;  // labels of the work targets' active transitions
        for (u32 q2 = 0; q2 < Q; q2++)
          if ((wmask >> q2) & 1u)
            for (u32 j = p.q.in_begin[q2]; j < p.q.in_begin[q2 + 1]; j++)
              if ((p.q.in_from[j] & active) && p.q.in_label[j] < p.L) lset |= 1ull << p.q.in_label[j];
        for (; lset; lset &= lset - 1) {
          const u32 l = __ffsll((long long)lset) - 1;
          const u32 *off = p.in_off + (u64)l * n1 + w;
          const u32 beg = __ldg(off), end = __ldg(off + 1);
          if (beg == end || (end - beg >= p.heavy_row && chunked)) continue;
          u32 S = 0;  // source states of those transitions on label l
          for (u32 q2 = 0; q2 < Q; q2++)
            if ((wmask >> q2) & 1u)
              for (u32 j = p.q.in_begin[q2]; j < p.q.in_begin[q2 + 1]; j++)
                if (p.q.in_label[j] == l) S |= p.q.in_from[j] & active;
          for (; S; S &= S - 1) {
            const u32 st = __ffs(S) - 1;
            u64 g[PER], none[PER];
#pragma unroll
            for (int k = 0; k < PER; k++) g[k] = none[k] = 0;
            u32 gat = 0;
            const u32 ex = gather_row<NW, PER, false, false>(p, F, bits, 1u << st, beg, end, lane_off, lane_on,
                                                             sg_mask, none, g, gat, nullptr);
            edges += (li == 0) ? ex : 0;
            bytes += (li == 0) ? 8 + (u64)ex * (4 + (bits ? 4 : 0)) + (u64)gat * gword : 0;
            bool nz = false;
#pragma unroll
            for (int k = 0; k < PER; k++) nz |= g[k] != 0;
            if (!nz) continue;
            for (u32 q2 = 0; q2 < Q; q2++) {
              if (!((wmask >> q2) & 1u)) continue;
              for (u32 j = p.q.in_begin[q2]; j < p.q.in_begin[q2 + 1]; j++) {
                if (p.q.in_label[j] != l || !((p.q.in_from[j] >> st) & 1u)) continue;
                const u64 *mk = p.la_mask + (u64)p.la_in_t[(u64)j * Q + st] * wpv + lane_off;
#pragma unroll
                for (int k = 0; k < PER; k++) sacc[(q2 * PER + k) * 32 + lane] |= g[k] & __ldg(mk + k);
              }
            }
          }
        }
        for (u32 q2 = 0; q2 < Q; q2++) {
          const bool work = ((wmask >> q2) & 1u) != 0;
          if (!__any_sync(FULL_MASK, work)) continue;
          u64 vis[PER], acc[PER];
          load_vis<PER>(p.vis + ((u64)q2 * n + w) * wpv + lane_off, lane_on && work, vis);
#pragma unroll
          for (int k = 0; k < PER; k++) acc[k] = sacc[(q2 * PER + k) * 32 + lane];
          words += (li == 0 && work);
          bytes += (li == 0 && work) ? gword : 0;
          pull_finish<NW, PER>(p, app, FB, nlist, nxt, q2, w, stamp, li, lane_on && work, my_g,
                               ((vh >> q2) & 1u) != 0, vis, acc);
        }
        continue;
      }
    }
    for (u32 q2 = 0; q2 < Q; q2++) {
      const u32 gb = p.q.in_begin[q2], ge = p.q.in_begin[q2 + 1];
      bool any = wv && ((vq >> q2) & 1u);
      if (bits && __any_sync(FULL_MASK, any && ((vt >> q2) & 1u))) {
        // sparse frontier, rows the pre-scan left undecided: a vertex none of
        // whose in-neighbours is in the frontier is skipped before its
        // visited words are read (the sub-warp's lanes test the in-edges in
        // turn: a column id and a bitmap word each)
        bool hit = false;
        if (!((vt >> q2) & 1u)) any = false, hit = wv && ((vq >> q2) & 1u);
        for (u32 j = gb; j < ge && !hit && any; j++) {
          const u32 l = p.q.in_label[j];
          const u32 from = p.q.in_from[j] & active;
          if (!from || l >= p.L) continue;
          const u32 *off = p.in_off + (u64)l * n1 + w;
          const u32 beg = __ldg(off), end = __ldg(off + 1);
          if (end - beg >= p.heavy_row && chunked) continue;
          for (u32 i = beg + li; i < end && !hit; i += SW) {
            const u32 u = __ldg(p.in_col + i);
            bytes += 4 + 4 * __popc(from);
            for (u32 fb = from; fb && !hit; fb &= fb - 1) {
              const u64 bi = (u64)(__ffs(fb) - 1) * n + u;
              hit = (__ldcg(bits + (bi >> 5)) >> (bi & 31)) & 1u;
            }
          }
        }
        any = (__ballot_sync(FULL_MASK, hit) & sg_mask) != 0;
      }
      const u64 base = ((u64)q2 * n + w) * wpv + lane_off;
      u64 vis[PER];
      load_vis<PER>(p.vis + base, lane_on && any, vis);
      u64 acc[PER];
#pragma unroll
      for (int k = 0; k < PER; k++) acc[k] = 0;
      // the in-rows' gathers into acc
      auto gather_all = [&]() {
        for (u32 j = gb; j < ge; j++) {
          const u32 l = p.q.in_label[j];
          const u32 from = p.q.in_from[j] & active;
          if (!from || l >= p.L) continue;
          const u32 *off = p.in_off + (u64)l * n1 + w;
          const u32 beg = __ldg(off), end = __ldg(off + 1);
          if (end - beg >= p.heavy_row && chunked) continue;
          // in multi mode each lane gathers through its own group's transitions
          u32 lfrom = from;
          if constexpr (AM == AM_GROUP) lfrom = lane_on ? p.from_tab[((u64)my_g * Q + q2) * p.L + l] & active : 0u;
          u32 gat = 0;
          const u32 ex = gather_row<NW, PER, true, AM == AM_LANE>(p, F, bits, lfrom, beg, end, lane_off, lane_on,
                                                                   sg_mask, vis, acc, gat,
                                                                   p.la_in_t + (u64)j * Q);
          edges += (li == 0) ? ex : 0;
          // column ids, frontier-bit words when tested, gathered frontier words
          bytes += (li == 0) ? 8 + (u64)ex * (4 + (bits ? 4 * __popc(from) : 0)) + (u64)gat * gword : 0;
        }
        words += (li == 0);
        bytes += (li == 0) ? gword : 0;
      };
      // whether every lane of the sub-warp's vertex is visited; a warp-wide
      // ballot, so every lane of the warp must call it
      auto all_visited = [&]() {
        bool full = true;
#pragma unroll
        for (int k = 0; k < PER; k++) full &= vis[k] == ~0ull;
        return (__ballot_sync(FULL_MASK, full) & sg_mask) == sg_mask;
      };
      // the gathers stop early on the visited words: read them first
      const bool allv = all_visited();
      const bool work = any && !allv;
      if (!__any_sync(FULL_MASK, work)) continue;
      if (work) gather_all();
      pull_finish<NW, PER>(p, app, FB, nlist, nxt, q2, w, stamp, li, lane_on && work, my_g, ((vh >> q2) & 1u) != 0,
                           vis, acc);
    }
    }
    if (p.pull_dynamic)
      c0 = next_item(&p.ctl->cursor[cur], n_warps, cv);
    else
      c0 += n_warps * cv;
  }

  bool chunks_done = !chunked;
  if constexpr (AM == AM_LANE) {
    if (chunked && p.lane_by_source && Q <= LANE_SRC_Q) {
      // Long in-rows by source state: an item is a chunk of a label's long
      // in-rows; its frontier words are gathered once per active source
      // state with a transition on that label and masked into every target
      // taking one (the light rows' scheme, see above).
      u64 lact = 0;  // labels with an active transition
      for (u32 j = 0; j < p.q.in_begin[Q]; j++)
        if ((p.q.in_from[j] & active) && p.q.in_label[j] < p.L) lact |= 1ull << p.q.in_label[j];
      for (u64 it = warp;; it = next_item(&p.ctl->heavy_cursor[cur], n_warps, 1)) {
        u64 acc_base = 0, ci = 0;
        u32 ls = 0;
        bool found = false;
        for (u64 lb = lact; lb; lb &= lb - 1) {
          const u32 l = __ffsll((long long)lb) - 1;
          const u64 cnt = p.hchunk_end[l] - p.hchunk_beg[l];
          if (it < acc_base + cnt) {
            found = true;
            ls = l;
            ci = p.hchunk_beg[l] + (it - acc_base);
            break;
          }
          acc_base += cnt;
        }
        if (!found) break;
        const u32 *rec = p.hchunk + 3 * ci;
        const u32 w = __ldg(rec), beg = __ldg(rec + 1), end = __ldg(rec + 2);
        // targets with a transition on ls from an active state and lanes not
        // yet visited (the whole warp works on vertex w)
        u32 wmask = 0;
        for (u32 q2 = 0; q2 < Q; q2++) {
          bool has = false;
          for (u32 j = p.q.in_begin[q2]; j < p.q.in_begin[q2 + 1]; j++)
            has |= p.q.in_label[j] == ls && (p.q.in_from[j] & active) != 0;
          u64 vis[PER];
          load_vis<PER>(p.vis + ((u64)q2 * n + w) * wpv + lane_off, lane_on && has, vis);
          bool full = true;
#pragma unroll
          for (int k = 0; k < PER; k++) {
            full &= vis[k] == ~0ull;
            lane_acc[(q2 * PER + k) * 32 + lane] = 0;
          }
          const u32 fbal = __ballot_sync(FULL_MASK, full);  // every lane, before the test
          if (has && fbal != FULL_MASK) wmask |= 1u << q2;
        }
        if (!wmask) continue;
        u32 S = 0;
        for (u32 q2 = 0; q2 < Q; q2++)
          if ((wmask >> q2) & 1u)
            for (u32 j = p.q.in_begin[q2]; j < p.q.in_begin[q2 + 1]; j++)
              if (p.q.in_label[j] == ls) S |= p.q.in_from[j] & active;
        // the sub-warps take consecutive slices of the chunk's edges
        const u32 len = end - beg, per = (len + VPW - 1) / VPW;
        const u32 sb = beg + min(len, sg * per), se = beg + min(len, (sg + 1) * per);
        u64 ex_tot = 0, gat_tot = 0;
        for (; S; S &= S - 1) {
          const u32 st = __ffs(S) - 1;
          u64 g[PER], none[PER];
#pragma unroll
          for (int k = 0; k < PER; k++) g[k] = none[k] = 0;
          u32 gat = 0;
          ex_tot += gather_row<NW, PER, false, false>(p, F, bits, 1u << st, sb, se, lane_off, lane_on, sg_mask,
                                                      none, g, gat, nullptr);
          gat_tot += gat;
          for (u32 o = SW; o < 32; o <<= 1) {
#pragma unroll
            for (int k = 0; k < PER; k++) g[k] |= __shfl_xor_sync(FULL_MASK, g[k], o);
          }
          for (u32 q2 = 0; q2 < Q; q2++) {
            if (!((wmask >> q2) & 1u)) continue;
            for (u32 j = p.q.in_begin[q2]; j < p.q.in_begin[q2 + 1]; j++) {
              if (p.q.in_label[j] != ls || !((p.q.in_from[j] >> st) & 1u)) continue;
              const u64 *mk = p.la_mask + (u64)p.la_in_t[(u64)j * Q + st] * wpv + lane_off;
#pragma unroll
              for (int k = 0; k < PER; k++) lane_acc[(q2 * PER + k) * 32 + lane] |= g[k] & __ldg(mk + k);
            }
          }
        }
        const u64 ex_all = warp_sum((u64)(li == 0 ? ex_tot : 0));
        const u64 gat_all = warp_sum((u64)(li == 0 ? gat_tot : 0));
        edges += (lane == 0) ? ex_all : 0;
        bytes += (lane == 0) ? 12 + ex_all * (4 + (bits ? 4 : 0)) + gat_all * gword : 0;
        for (u32 q2 = 0; q2 < Q; q2++) {
          if (!((wmask >> q2) & 1u)) continue;  // uniform across the warp
          u64 vis[PER], acc[PER];
          load_vis<PER>(p.vis + ((u64)q2 * n + w) * wpv + lane_off, lane_on, vis);
#pragma unroll
          for (int k = 0; k < PER; k++) acc[k] = lane_acc[(q2 * PER + k) * 32 + lane];
          words += (lane == 0);
          bytes += (lane == 0) ? gword : 0;
          pull_finish<NW, PER>(p, app, FB, nlist, nxt, q2, w, stamp, li, lane_on && sg == 0, my_g, true, vis, acc);
        }
      }
      chunks_done = true;
    }
  }
  if (!chunks_done) {
    for (u64 it = warp;; it = next_item(&p.ctl->heavy_cursor[cur], n_warps, 1)) {
      // map the item number to (target state, transition group, chunk)
      u64 acc_base = 0, ci = 0;
      u32 q2s = 0, from = 0, ls = 0, js = 0;
      bool found = false;
      for (u32 q2 = 0; q2 < Q && !found; q2++)
        for (u32 j = p.q.in_begin[q2]; j < p.q.in_begin[q2 + 1]; j++) {
          const u32 l = p.q.in_label[j];
          if (!(p.q.in_from[j] & active) || l >= p.L) continue;
          const u64 cnt = p.hchunk_end[l] - p.hchunk_beg[l];
          if (it < acc_base + cnt) {
            found = true;
            q2s = q2;
            ls = l;
            js = j;
            from = p.q.in_from[j] & active;
            ci = p.hchunk_beg[l] + (it - acc_base);
            break;
          }
          acc_base += cnt;
        }
      if (!found) break;
      const u32 *rec = p.hchunk + 3 * ci;
      const u32 w = __ldg(rec), beg = __ldg(rec + 1), end = __ldg(rec + 2);
      const u64 base = ((u64)q2s * n + w) * wpv + lane_off;
      u64 vis[PER];
      load_vis<PER>(p.vis + base, lane_on, vis);
      bool full = true;
#pragma unroll
      for (int k = 0; k < PER; k++) full &= vis[k] == ~0ull;
      if (__all_sync(FULL_MASK, full)) continue;
      u64 acc[PER];
#pragma unroll
      for (int k = 0; k < PER; k++) acc[k] = 0;
      // the sub-warps take consecutive slices of the chunk's edges
      const u32 len = end - beg, per = (len + VPW - 1) / VPW;
      const u32 sb = beg + min(len, sg * per), se = beg + min(len, (sg + 1) * per);
      u32 lfrom = from;
      if constexpr (AM == AM_GROUP) lfrom = lane_on ? p.from_tab[((u64)my_g * Q + q2s) * p.L + ls] & active : 0u;
      u32 gat = 0;
      const u32 ex = gather_row<NW, PER, true, AM == AM_LANE>(p, F, bits, lfrom, sb, se, lane_off, lane_on, sg_mask,
                                                               vis, acc, gat, p.la_in_t + (u64)js * Q);
      for (u32 o = SW; o < 32; o <<= 1) {
#pragma unroll
        for (int k = 0; k < PER; k++) acc[k] |= __shfl_xor_sync(FULL_MASK, acc[k], o);
      }
      const u64 ex_all = warp_sum((u64)(li == 0 ? ex : 0));
      const u64 gat_all = warp_sum((u64)(li == 0 ? gat : 0));
      edges += (lane == 0) ? ex_all : 0;
      bytes += (lane == 0) ? 12 + gword + ex_all * (4 + (bits ? 4 * __popc(from) : 0)) + gat_all * gword : 0;
      words += (lane == 0);
      pull_finish<NW, PER>(p, app, FB, nlist, nxt, q2s, w, stamp, li, lane_on && sg == 0, my_g, true, vis, acc);
    }
  }
  append_close(p, app, nlist);
  stat_add(stat, ST_PULL_EDGES, warp_sum(edges));
  stat_add(stat, ST_PULL_VERTICES, warp_sum(words));
  stat_add(stat, ST_ALG_BYTES, warp_sum(bytes));
}

// Commit of a level: fold the new frontier words into VIS, count work, note
// the DFA states present in the new frontier, clear the old frontier words.
// set_bits: the next frontier may be sparse enough for bottom-up levels to
// test its bitmap, so its bits are set (pull_lanes has set its own);
// clear_bits: this level's bits were set and are cleared, entry by entry (1)
// or all words (2).
template <int NW, int AM>
__device__ void commit_phase(const BfsParams &p, int lp, u32 nxt, u64 n_cur, u64 n_warps, bool set_bits,
                             int clear_bits, CommitSums &sums, u64 *stat) {
  const u64 *list = lp ? p.list1 : p.list0;
  const u64 *nlist = lp ? p.list0 : p.list1;
  u64 *F = lp ? p.fr1 : p.fr0;
  const u64 *FB = lp ? p.fr0 : p.fr1;
  const u32 Q = p.Q;
  const u64 n_next = *(volatile unsigned long long *)&p.ctl->n_list[nxt];
  const u64 stride = n_warps * 32;
  const u64 tid = (u64)blockIdx.x * blockDim.x + threadIdx.x;
  u64 W = 0, N = 0, mf = 0, gv = 0, gx = 0;
  u32 states = 0;
  for (u64 j = tid; j < n_next; j += stride) {
    u64 e = __ldcg(&nlist[j]);
    if (e == NO_ENTRY) continue;
    u32 gq = (u32)((e & ~ENTRY_DONE) >> 32), w = (u32)e;
    u32 g = gq / Q, q = gq - g * Q;
    if (set_bits) {
      const u64 bi = (u64)q * p.n + w;
      atomicOr(p.fbits + (lp ? 0 : p.fbits_words) + (bi >> 5), 1u << (bi & 31));
    }
    if (e & ENTRY_DONE) continue;
    u64 wi = widx<NW>(p, g, q, w);
    Word<NW> m = load_cg<NW>(FB + wi);
    Word<NW> v = load_cg<NW>(p.vis + wi);
#pragma unroll
    for (int t = 0; t < NW; t++) v.w[t] |= m.w[t];
    store_w<NW>(p.vis + wi, v);
    u32 c = popc_w(m);
    u32 rows = 0, d;
    if constexpr (per_lane(AM)) {
      d = la_degsum<NW>(p, q, w, g, m, W, &rows);
    } else {
      d = degsum(p, gdesc<AM>(p, g), q, w, &rows);
      W += (u64)c * d;
    }
    N += c;
    mf += d;
    gx += rows;
    gv += 1;
    states |= 1u << q;
  }
  Word<NW> zero;
#pragma unroll
  for (int t = 0; t < NW; t++) zero.w[t] = 0;
  for (u64 j = tid; j < n_cur; j += stride) {
    u64 e = __ldcg(&list[j]);
    if (e == NO_ENTRY) continue;
    u32 gq = (u32)((e & ~ENTRY_DONE) >> 32);
    u32 g = gq / Q;
    store_w<NW>(F + widx<NW>(p, g, gq - g * Q, (u32)e), zero);
    if (clear_bits == 1) {
      // the retired frontier's bitmap: every set bit belongs to one of these entries
      const u64 bi = (u64)(gq - g * Q) * p.n + (u32)e;
      p.fbits[(lp ? p.fbits_words : 0) + (bi >> 5)] = 0u;
    }
  }
  if (clear_bits == 2)  // a dense frontier's: all of it
    for (u64 j = tid; j < ((u64)p.n * Q + 31) / 32; j += stride) p.fbits[(lp ? p.fbits_words : 0) + j] = 0u;
  if (tid == 0) stat[ST_ALG_BYTES] += n_cur * (8 + 8 * NW);
  W = warp_sum(W);
  N = warp_sum(N);
  mf = warp_sum(mf);
  gv = warp_sum(gv);
  gx = warp_sum(gx);
  states = __reduce_or_sync(FULL_MASK, states);
  // per new entry: the entry, its new frontier word, its visited word read and
  // written; per old entry: the entry and its frontier word cleared
  if (lane_id() == 0) stat[ST_ALG_BYTES] += gv * (8 + 24 * NW);
  if (lane_id() == 0) {
    stat[ST_W] += W;
    stat[ST_N] += N;
    if (gv) {
      atomicAdd(&sums.mf, mf);
      atomicAdd(&sums.gx, gx);
      atomicAdd(&sums.n_true, gv);
      atomicOr(&sums.smask, states);
    }
  }
}

// Bytes a bottom-up level moves when the frontier holds the states `active`:
// per target state with an active incoming transition, its visited words;
// per such transition group, the row offsets and per in-edge a column id
// and the gathered frontier words.  An estimate in single precision: every
// thread evaluates it at the start of every level, and in double precision it
// took most of the 8 us between the end of one level's commit and the start of
// the next (2 us now, the barrier).
template <int NW>
__device__ float pull_bytes(const BfsParams &p, u32 active) {
  float b = 0;
  const float wv = 8.0f * NW * p.G, nf = (float)p.n;
  for (u32 q2 = 0; q2 < p.Q; q2++) {
    bool any = false;
    for (u32 j = p.q.in_begin[q2]; j < p.q.in_begin[q2 + 1]; j++) {
      const u32 f = p.q.in_from[j] & active, l = p.q.in_label[j];
      if (!f || l >= p.L) continue;
      any = true;
      b += 8.0f * nf + (float)p.label_edges[l] * (4.0f + wv * __popc(f));
    }
    if (any) b += wv * nf;
  }
  return b;
}

// Levels of at most SOLO_SLOTS list slots and SOLO_EDGES out-edges are run by
// block 0 alone, with __syncthreads between the phases: a level is then the
// latency of its loads and atomics (7-8 us for a handful of entries), where
// the grid pays two more barriers and the wake-up of 4,864 warps (17-19 us).
// Above 512 edges the block's eight warps take longer than that.  The other
// blocks wait at a grid barrier, for at most SOLO_RUN levels at a time, so
// that no wait comes near the time limit.
constexpr u64 SOLO_SLOTS = 512, SOLO_EDGES = 512;
constexpr u32 SOLO_RUN = 64;

template <int NW, int AM, int BLOCKS = AM == AM_LANES ? 3 : 4>
__global__ void __launch_bounds__(BFS_THREADS, BLOCKS) msbfs_kernel(const __grid_constant__ BfsParams p) {
  // per-warp statistics (lane 0 adds to them once per phase), summed into the
  // control block at the end; in registers they were spilled by every phase
  __shared__ u64 s_stat[BFS_THREADS / 32][ST_COUNT];
  u64 *stat = s_stat[threadIdx.x >> 5];
  if (lane_id() < ST_COUNT) stat[lane_id()] = 0;
  __syncwarp();
  BfsCtl *c = p.ctl;
  unsigned epoch = 0;  // grid barriers passed
  __shared__ CommitSums sums;
  // per-warp scratch of the expansion phases: a push keeps its entries' words
  // and rows there, lane mode its accumulators, pull_staged its lists
  constexpr int SCRATCH = AM == AM_LANES  ? LANE_SRC_Q * 2 * 32 + LANE_LIST
                          : AM == AM_LANE ? LANE_SRC_Q * 2 * 32
                          : AM == AM_MANY ? STAGE
                                          : 32 * NW + 32;
  __shared__ __align__(16) u64 s_scratch[BFS_THREADS / 32][SCRATCH];
  u64 *scratch = s_scratch[threadIdx.x >> 5];
  if (threadIdx.x == 0) sums = CommitSums{};  // seen by the block after the seeds' barrier
  const bool tracer = blockIdx.x == 0 && threadIdx.x == 0;

  seed_phase<NW, AM>(p, stat);
  if (!grid_sync(c, p.nblocks, epoch, p.time_limit_ns)) return;

  // Bottom-up levels by pull_lanes cost less than the estimate's bytes with a
  // bitmap: the batch above goes top-down in its second level at a factor above
  // 0.4 (60 ms, not 22).
  constexpr float LANES_PULL = 0.4f;
  constexpr bool lanes_staged = AM == AM_LANES;
  bool have_bits = p.fbits != nullptr;  // this level's frontier has a bitmap (the seeds set theirs)
  u32 level = 0, run = 0;  // run: levels left of block 0's run, 0 outside one
  for (;; level++) {
    const u32 cur = level % 3, nxt = (level + 1) % 3, old = (level + 2) % 3;
    const int lp = level & 1;
    const u64 n_cur = *(volatile unsigned long long *)&c->n_list[cur];
    if (n_cur == 0) break;
    const u64 mf = *(volatile unsigned long long *)&c->mf[cur];
    const u32 active = *(volatile unsigned *)&c->smask[cur];
    const u64 n_true = *(volatile unsigned long long *)&c->n_true[cur];
    const bool solo = n_cur <= SOLO_SLOTS && mf <= SOLO_EDGES && p.force != 2;
    if (solo && run == 0) {
      // every block has read this level's counters before block 0 goes on
      if (!grid_sync(c, p.nblocks, epoch, p.time_limit_ns)) return;
      if (blockIdx.x != 0) {
        if (!grid_sync(c, p.nblocks, epoch, p.time_limit_ns)) return;
        level = *(volatile unsigned *)&c->next_level - 1;
        // a top-down level of block 0 built this frontier
        have_bits = p.fbits && *(volatile unsigned long long *)&c->n_list[(level + 1) % 3] * 4 < (u64)p.n * p.Q;
        continue;
      }
      run = SOLO_RUN;
    }
    const float push_cost = (float)mf * (4.0f + 8.0f * NW) + (float)n_true * (16.0f + 8.0f * NW);
    float pull_cost = pull_bytes<NW>(p, active);
    // pull_lanes tests the frontier's bitmap up to a seventh of the words: the
    // rows it shows empty outweigh the test then (second and third level of the
    // batch above 31 -> 22 and 50 -> 48 ms, its dense levels 57 -> 61)
    const bool lanes_bits = lanes_staged && have_bits && n_cur * 7 < (u64)p.n * __popc(active) * p.G;
    if (lanes_bits) pull_cost *= LANES_PULL;
    const bool push = solo || p.force == 1 || (p.force != 2 && p.alpha * push_cost < pull_cost);
    if (tracer) {
      // counters of the level after next start at zero
      c->n_list[old] = 0;
      c->cursor[old] = 0;
      c->mf[old] = 0;
      c->n_true[old] = 0;
      c->spill_count[old] = 0;
      c->spill_cursor[old] = 0;
      c->heavy_cursor[old] = 0;
      c->smask[old] = 0;
      if (level < (u32)TRACE_LEVELS) {
        c->trace_t[level] = globaltimer_ns();
        c->trace_n[level] = (u32)min(n_cur, (u64)~0u);
        c->trace_mode[level] = push ? 1 : 2;
        c->trace_mf[level] = mf;
      }
      stat[ST_GROUP_W] += mf;
      stat[ST_GROUP_VERTICES] += n_true;
      if (push)
        stat[ST_PUSH_LEVELS] += 1;
      else
        stat[ST_PULL_LEVELS] += 1;
    }
    const u32 stamp = p.stamp_base + level + 2;  // the seeds used stamp_base + 1
    const u64 n_warps = (run ? 1ull : (u64)p.nblocks) * (BFS_THREADS / 32);
    if (mf == 0) {
      // no out-edges: the next frontier is empty, only this one is cleared
    } else if (push) {
      const u32 seg = mf < PUSH_EXACT ? 0u : p.append_seg;
      push_level<NW, AM>(p, lp, cur, nxt, n_cur, mf, n_warps, run ? ~0u : spill_chunk(mf, n_warps, p.spill_cap), seg,
                         stamp, scratch, stat);
      if (run) {
        __syncthreads();
      } else {
        if (!grid_sync(c, p.nblocks, epoch, p.time_limit_ns)) return;
        if (*(volatile unsigned long long *)&c->spill_count[cur] != 0) {
          spill_phase<NW>(p, lp, cur, nxt, seg, stamp, stat);
          if (!grid_sync(c, p.nblocks, epoch, p.time_limit_ns)) return;
        }
      }
    } else {
      // a sparse frontier: test the frontier bitmap before each gather
      // (implies n_cur * 4 < n * Q, so the commit that built this frontier set
      // its bits)
      const bool sparse = lanes_staged ? lanes_bits : p.fbits && n_cur * 4 < (u64)p.n * __popc(active);
      const u32 *bits = sparse ? p.fbits + (lp ? p.fbits_words : 0) : nullptr;
      // pull_level's early exit pays where few lanes are live: one lane
      // group, the per-group automata of a multi launch (typically one start
      // vertex each), or per-lane automata (lanes of short queries go quiet
      // early)
      if constexpr (AM == AM_MANY) {
        pull_staged<NW>(p, lp, cur, nxt, active, stamp, bits, scratch, sums, stat);
      } else if constexpr (AM == AM_LANES) {
        __shared__ LaneTables tab;
        pull_lanes<NW>(p, lp, cur, nxt, active, stamp, bits, scratch, tab, stat);
      } else {
        pull_level<NW, AM>(p, lp, cur, nxt, active, stamp, bits, scratch, stat);
      }
      if (!grid_sync(c, p.nblocks, epoch, p.time_limit_ns)) return;
    }
    {
      // bitmaps only where a bottom-up level may test them: a frontier with
      // fewer than n * Q / 4 entries (the seeds always set theirs)
      const u64 n_next = *(volatile unsigned long long *)&c->n_list[nxt];
      const u64 sparse_cap = (u64)p.n * p.Q;
      const bool pulled_lanes = lanes_staged && mf != 0 && !push;
      const bool set_bits = p.fbits && n_next * 4 < sparse_cap && !pulled_lanes;
      const int clear_bits = !have_bits ? 0 : level == 0 || n_cur * 4 < sparse_cap ? 1 : 2;
      have_bits = p.fbits && (n_next * 4 < sparse_cap || pulled_lanes);
      if (tracer && level < (u32)TRACE_LEVELS) c->trace_c[level] = (u32)globaltimer_ns();
      commit_phase<NW, AM>(p, lp, nxt, n_cur, n_warps, set_bits, clear_bits, sums, stat);
      if (run) {
        __syncthreads();
        if (threadIdx.x == 0) publish_sums(c, sums, nxt);
        __syncthreads();
        const u64 mf_next = *(volatile unsigned long long *)&c->mf[nxt];
        if (--run == 0 || n_next == 0 || n_next > SOLO_SLOTS || mf_next > SOLO_EDGES) {
          run = 0;
          if (tracer) c->next_level = level + 1;
          if (!grid_sync(c, p.nblocks, epoch, p.time_limit_ns)) return;
        }
        continue;
      }
    }
    if (!grid_sync(c, p.nblocks, epoch, p.time_limit_ns, [&] { publish_sums(c, sums, nxt); })) return;
  }
  if (threadIdx.x == 0 && sums.gx) atomicAdd(&c->stats[ST_GROUP_X], sums.gx);
  __syncwarp();
  if (lane_id() < ST_COUNT && stat[lane_id()]) atomicAdd(&c->stats[lane_id()], stat[lane_id()]);
  if (tracer) {
    c->levels = level;
    c->trace_t[level < (u32)TRACE_LEVELS ? level : TRACE_LEVELS] = globaltimer_ns();
  }
}

// VIS words start as the mask of empty lanes of their group, so empty lanes
// look visited everywhere (this also lets bottom-up levels stop early).
template <int NW>
__global__ void vis_init_kernel(u64 *__restrict__ vis, u64 total, u32 G, const u64 *__restrict__ empty) {
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (u64)gridDim.x * blockDim.x) {
    u32 g = (u32)((i / NW) % G);
    vis[i] = empty[(u64)g * NW + (i % NW)];
  }
}

cudaError_t launch_vis_init(const BfsParams &p, const unsigned long long *empty, cudaStream_t st) {
  u64 total = (u64)p.Q * p.n * p.G;
  u64 blocks = (total + 255) / 256;
  if (blocks > 152ull * 32) blocks = 152ull * 32;
  if (blocks == 0) blocks = 1;
  vis_init_kernel<1><<<(unsigned)blocks, 256, 0, st>>>(p.vis, total, p.G, empty);
  return cudaGetLastError();
}

// Start of a launch whose lanes are filled from the first on: VIS words as
// above (lane i is empty from `live` on), the control block and the emission's
// accumulators zeroed, and up to 64 start vertices written from the kernel's
// own parameters.  One launch for what took five calls, and with one
// allocation and one read-back where there were three and two, a lookup on a
// 1,000-vertex graph takes 98 us for 112, and one on 2^20 vertices 536 for 553.
// More than 64 start vertices are copied from the host as before.
struct StartLanes {
  u32 id[64];
};
template <int NW>
__global__ void start_kernel(const BfsParams p, u64 total, u32 live, u64 *__restrict__ small, u32 *__restrict__ lanesrc,
                             const __grid_constant__ StartLanes lanes) {
  const u64 tid = (u64)blockIdx.x * blockDim.x + threadIdx.x, step = (u64)gridDim.x * blockDim.x;
  if (lanesrc && tid < 64) lanesrc[tid] = lanes.id[tid];
  if (tid < 4) small[tid] = 0;
  static_assert(sizeof(BfsCtl) % 4 == 0, "cleared by words");
  for (u64 i = tid; i < sizeof(BfsCtl) / 4; i += step) reinterpret_cast<u32 *>(p.ctl)[i] = 0;
  const u32 row = p.G * NW;
  for (u64 i = tid; i < total; i += step) {
    const u32 first = (u32)(i % row) * 64;  // first lane of the word
    p.vis[i] = first + 64 <= live ? 0ull : first >= live ? ~0ull : ~0ull << (live - first);
  }
}

cudaError_t launch_start(int nw, const BfsParams &p, uint32_t live, unsigned long long *small, uint32_t *lanesrc,
                         const uint32_t *ids, cudaStream_t st) {
  const u64 total = (u64)p.Q * p.n * p.G * nw;
  const u64 blocks = std::min<u64>(std::max<u64>((total + 255) / 256, 16), 152ull * 32);
  StartLanes lanes;
  for (uint32_t i = 0; i < 64; i++) lanes.id[i] = ids && i < live ? ids[i] : NO_SOURCE;
  if (nw == 1)
    start_kernel<1><<<(unsigned)blocks, 256, 0, st>>>(p, total, live, small, ids ? lanesrc : nullptr, lanes);
  else
    start_kernel<4><<<(unsigned)blocks, 256, 0, st>>>(p, total, live, small, ids ? lanesrc : nullptr, lanes);
  return cudaGetLastError();
}

// Lane mode: VIS words start as empty_q[(q * G + g) * NW + k], the lanes that
// are empty or whose automaton has no state q (so they look visited there).
template <int NW>
__global__ void vis_init_lane_kernel(u64 *__restrict__ vis, u64 total, u64 per_state, u32 G,
                                     const u64 *__restrict__ empty_q) {
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (u64)gridDim.x * blockDim.x) {
    const u64 q = i / per_state;
    const u32 gk = (u32)(i % ((u64)G * NW));
    vis[i] = empty_q[q * G * NW + gk];
  }
}

cudaError_t launch_vis_init_lane(int nw, const BfsParams &p, const unsigned long long *empty_q, cudaStream_t st) {
  const u64 per_state = (u64)p.n * p.G * nw;
  const u64 total = per_state * p.Q;
  u64 blocks = (total + 255) / 256;
  if (blocks > 152ull * 32) blocks = 152ull * 32;
  if (blocks == 0) blocks = 1;
  if (nw == 1)
    vis_init_lane_kernel<1><<<(unsigned)blocks, 256, 0, st>>>(p.vis, total, per_state, p.G, empty_q);
  else
    vis_init_lane_kernel<4><<<(unsigned)blocks, 256, 0, st>>>(p.vis, total, per_state, p.G, empty_q);
  return cudaGetLastError();
}

// flag[i] = 1 when start vertex srcs[i] has an edge on a label of label_mask
// in the traversal's forward direction (off = the forward offsets).
__global__ void source_filter_kernel(const u32 *__restrict__ off, u32 n, u32 L, unsigned long long label_mask,
                                     const u32 *__restrict__ srcs, u64 count, unsigned char *__restrict__ flag) {
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (u64)gridDim.x * blockDim.x) {
    const u32 s = srcs[i];
    unsigned char f = 0;
    for (unsigned long long m = label_mask; m && !f; m &= m - 1) {
      const u32 l = __ffsll(m) - 1;
      if (l >= L) break;
      const u32 *o = off + (u64)l * (n + 1) + s;
      f = __ldg(o + 1) > __ldg(o);
    }
    flag[i] = f;
  }
}

cudaError_t launch_source_filter(const uint32_t *off, uint32_t n, uint32_t L, unsigned long long label_mask,
                                 const uint32_t *srcs, unsigned long long count, unsigned char *flag,
                                 cudaStream_t st) {
  if (count == 0) return cudaSuccess;
  u64 blocks = (count + 255) / 256;
  if (blocks > 152ull * 16) blocks = 152ull * 16;
  source_filter_kernel<<<(unsigned)blocks, 256, 0, st>>>(off, n, L, label_mask, srcs, count, flag);
  return cudaGetLastError();
}

cudaError_t launch_msbfs(int nw, const BfsParams &p, int blocks, int threads, cudaStream_t st) {
  void *args[] = {(void *)&p};
  void *kernel = nw == 1   ? (void *)msbfs_kernel<1, AM_ONE>
                 : p.G == 1 || p.walk_rows ? (void *)msbfs_kernel<4, AM_ONE>
                                           : (void *)msbfs_kernel<4, AM_MANY>;
  return cudaLaunchCooperativeKernel(kernel, blocks, threads, args, 0, st);
}

int msbfs_max_blocks(int nw, int threads, int *blocks_per_sm, int *sms) {
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
  if (nw == 1)
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, msbfs_kernel<1, AM_ONE>, threads, 0) ==
                   cudaSuccess
               ? 0
               : -1;
  // launch_msbfs takes either kernel: the grid has to fit both
  int many = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, msbfs_kernel<4, AM_ONE>, threads, 0) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&many, msbfs_kernel<4, AM_MANY>, threads, 0) != cudaSuccess)
    return -1;
  *blocks_per_sm = std::min(*blocks_per_sm, many);
  return 0;
}

cudaError_t preload_static_msbfs_kernels() {
  cudaFuncAttributes a;
  cudaError_t e = cudaFuncGetAttributes(&a, msbfs_kernel<1, AM_ONE>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, start_kernel<1>);
  return e;
}

cudaError_t launch_msbfs_multi(const BfsParams &p, int blocks, int threads, cudaStream_t st) {
  void *args[] = {(void *)&p};
  return cudaLaunchCooperativeKernel((void *)msbfs_kernel<1, AM_GROUP>, blocks, threads, args, 0, st);
}

static void *lane_kernel(int nw, LaneKernel k) {
  if (k == LaneKernel::staged) return (void *)msbfs_kernel<4, AM_LANES>;
  if (k == LaneKernel::few) return nw == 1 ? (void *)msbfs_kernel<1, AM_LANE, 3> : (void *)msbfs_kernel<4, AM_LANE, 3>;
  return nw == 1 ? (void *)msbfs_kernel<1, AM_LANE> : (void *)msbfs_kernel<4, AM_LANE>;
}

cudaError_t launch_msbfs_lane(int nw, LaneKernel k, const BfsParams &p, int blocks, int threads, cudaStream_t st) {
  void *args[] = {(void *)&p};
  return cudaLaunchCooperativeKernel(lane_kernel(nw, k), blocks, threads, args, 0, st);
}

int msbfs_lane_max_blocks(int nw, LaneKernel k, int threads, int *blocks_per_sm) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, lane_kernel(nw, k), threads, 0) == cudaSuccess
             ? 0
             : -1;
}

int msbfs_multi_max_blocks(int threads, int *blocks_per_sm) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, msbfs_kernel<1, AM_GROUP>, threads, 0) ==
                 cudaSuccess
             ? 0
             : -1;
}

}  // namespace rpq
