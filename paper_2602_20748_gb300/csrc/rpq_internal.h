// Internal declarations shared by the host API and the CUDA kernels of the
// RPQ engine.  Not part of the public ABI (see include/rpq.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/rpq.h"

namespace rpq {

// ---------------------------------------------------------------------------
// Compiled query: the minimal DFA in the forms the kernels use.
// ---------------------------------------------------------------------------
struct QueryDesc {
  uint32_t n_states;    // 0 means the empty language
  uint32_t final_mask;  // bit q: state q accepts
  uint32_t n_labels;    // largest label id used + 1
  uint32_t n_trans;
  // Top-down form: transitions leaving state q are [out_begin[q], out_begin[q+1]).
  uint16_t out_begin[RPQ_MAX_STATES + 1];
  uint8_t out_label[RPQ_MAX_TRANSITIONS];
  uint8_t out_to[RPQ_MAX_TRANSITIONS];
  // Bottom-up form: for target state q, groups [in_begin[q], in_begin[q+1]) of
  // (label, bitmask of source states that reach q on that label).
  uint16_t in_begin[RPQ_MAX_STATES + 1];
  uint8_t in_label[RPQ_MAX_TRANSITIONS];
  uint32_t in_from[RPQ_MAX_TRANSITIONS];
};

// Host-side compiled query.
struct HostQuery {
  QueryDesc d;
  std::vector<int32_t> next;  // n_states * n_labels, -1 = none
  // Minimal DFA of the reversed language, for evaluation from the target end
  // over in-edges (absent when it would exceed RPQ_MAX_STATES).
  bool has_rev = false;
  QueryDesc rev;
  std::vector<int32_t> rev_next;
};

// Parses and compiles; returns RPQ_OK or an error code with *msg set.
int compile_regex(const char *regex, const char *const *names, uint32_t n_names, HostQuery *out, std::string *msg);
// The minimal DFA of L(alpha) followed by one edge of label x (x above every
// label alpha uses).
int dfa_then_label(const HostQuery &alpha, uint32_t x, HostQuery *out, std::string *msg);

// ---------------------------------------------------------------------------
// Device-resident graph: one CSR per edge label over the full id space, for
// out-edges (sorted by label, src, dst) and in-edges (label, dst, src).
// off[l * (n + 1) + v] is the first edge of row v of label l.
// ---------------------------------------------------------------------------
// In-edge rows with at least HEAVY_ROW edges are cut into chunks of HCHUNK
// edges at graph load; bottom-up levels share the chunks among all warps
// instead of scanning such a row with one warp.  At 32 edges the warps' shares
// come out evener than at 128, though such a vertex's words are then or-ed
// atomically: 1,500 reverse targets on R-MAT 2^18 1.78 -> 1.52 ms,
// configuration 2 20.2 -> 19.0 (24: 19.3, 48: 19.2, 64: 19.4, 256: 20.5).
// Where most rows are that long they may stay whole (see set_chunks).
// Launches of few start vertices leave a row at the first frontier vertices
// they meet, so for them only rows of LONG_ROW edges are chunked (one lookup
// on R-MAT 2^20: 0.55 ms, 0.60 with chunks from 32); the lists keep the two
// classes of rows apart.
constexpr uint32_t HEAVY_ROW = 32;
constexpr uint32_t LONG_ROW = 128;
constexpr uint32_t FEW_STARTS = 32;  // fewer start vertices than this chunk LONG_ROW rows only
constexpr uint32_t HCHUNK = 256;

// Chunks (vertex, first edge, end edge) of one direction's rows with at least
// HEAVY_ROW edges, grouped by label and class: label l's chunks of rows of
// LONG_ROW edges and more are [off[2 l], off[2 l + 1]), those of shorter rows
// follow up to off[2 l + 2] (host copy of the 2 L + 1 offsets).  One list, so that
// a launch finds a record with one base and one offset (a list per class made
// configuration 2 1.2% slower); where the budget needs the room of the shorter
// rows' chunks it is built again without them.
struct ChunkLists {
  uint32_t *rec = nullptr;
  std::vector<uint32_t> off;
  std::vector<uint32_t> light;  // per label, the edges in rows below HEAVY_ROW
  uint32_t shorter = 0;         // chunks of the shorter rows in the list
  std::vector<uint32_t> shorter_rows;  // per label, the rows of the second class (listed or not)
};

struct DevGraph {
  uint32_t n = 0;
  uint32_t L = 0;
  uint64_t m = 0;
  uint32_t *out_off = nullptr;
  uint32_t *out_col = nullptr;
  uint32_t *in_off = nullptr;
  uint32_t *in_col = nullptr;
  uint8_t *vlabel = nullptr;
  ChunkLists chunks_in, chunks_out;
  std::vector<uint8_t> vlabel_host;   // vertex labels (host copy), empty if none
  std::vector<uint64_t> label_edges;  // edges per label (host copy)
};

// ---------------------------------------------------------------------------
// Traversal control block (device memory, one per launch).
// ---------------------------------------------------------------------------
enum StatIdx {
  ST_W = 0,          // product-edge relaxations (per start vertex)
  ST_N,              // product vertices visited (per start vertex)
  ST_PUSH_LEVELS,
  ST_PULL_LEVELS,
  ST_GROUP_EDGES,    // edges read by top-down levels
  ST_GROUP_ROWS,     // adjacency rows opened by top-down levels
  ST_GROUP_VERTICES, // lane-group product vertices discovered
  ST_PULL_EDGES,     // in-edges read by bottom-up levels
  ST_PULL_VERTICES,  // (vertex, state) words examined bottom-up
  ST_ALG_BYTES,      // algorithmic bytes of the traversal (see the kernel)
  ST_GROUP_W,        // W_g: out-degree over the state's labels, summed over lane-group product vertices
  ST_GROUP_X,        // X_g: (label) adjacency rows of lane-group product vertices
  ST_COUNT
};

constexpr int TRACE_LEVELS = 64;
constexpr unsigned long long NO_ENTRY = ~0ull;      // a reserved list slot left empty
constexpr unsigned int ERR_LIST_OVERFLOW = 1000u;   // BfsCtl::err: an append ran past list_cap
constexpr unsigned int APPEND_SEG = 128;             // list slots a warp reserves at a time, at most
// Launches of several words per vertex reserve half as many (configuration 2
// 1% faster); with one word a warp appends up to 32 entries at once (one lookup
// on R-MAT 2^20: 550 us, 600 with 64).
inline unsigned int append_seg(int nw) { return nw == 1 ? APPEND_SEG : APPEND_SEG / 2; }

// The words that all blocks poll or add to, and that every level reads, have a
// 128-byte line each (a trace entry written into the line of the barrier's flag
// or of a counter cost the small calls 2-3%).  The size counts: what
// run_rpq_static takes and the serving slots that fit a budget depend on it.
struct BfsCtl {
  // grid barrier (grid_barrier.cuh): blocks that have arrived, over all
  // barriers; the last barrier completed << 1 | error
  unsigned int bar_count;
  unsigned int pad0[31];
  unsigned int bar_flag;
  unsigned int err;
  unsigned int err_where;
  unsigned int pad1[29];
  unsigned long long n_list[3];
  unsigned long long pad2[13];
  unsigned long long cursor[3];
  unsigned long long pad3[13];
  unsigned long long mf[3];  // frontier out-edges
  unsigned long long pad4[13];
  unsigned long long n_true[3];        // frontier entries without the lists' unused slots
  unsigned long long spill_count[3];   // top-down row chunks queued this level
  unsigned long long spill_cursor[3];
  unsigned long long heavy_cursor[3];  // bottom-up row chunks taken
  unsigned long long pad5[4];
  unsigned int smask[3];    // DFA states present in each frontier
  unsigned int next_level;  // first level after a run of one-block levels
  unsigned long long levels;
  unsigned long long stats[ST_COUNT];
  unsigned long long pad6[12];
  // per-level trace (first TRACE_LEVELS levels): start time (ns), frontier
  // out-edges and entries (at most 2^32 - 1), start time of the commit phase (its
  // low half), direction (1 top-down, 2 bottom-up)
  unsigned long long trace_t[TRACE_LEVELS + 1];
  unsigned long long trace_mf[TRACE_LEVELS];
  unsigned int trace_n[TRACE_LEVELS];
  unsigned int trace_c[TRACE_LEVELS];
  unsigned char trace_mode[TRACE_LEVELS];
};
static_assert(sizeof(BfsCtl) == 2592, "see above");

// A top-down row longer than the level's chunk length (at most SPILL_EDGES
// edges, see spill_chunk) is cut into chunks that all warps share in a
// sub-phase of the level.
constexpr unsigned int SPILL_EDGES = 1024;
constexpr unsigned int SPILL_EDGES_MIN = 64;
constexpr unsigned long long SPILL_CAP = 1ull << 18;  // chunks per level

struct BfsParams {
  // graph
  const uint32_t *out_off;
  const uint32_t *out_col;
  const uint32_t *in_off;
  const uint32_t *in_col;
  const uint32_t *hchunk;               // chunks of long in_off rows (nullptr: the list could not be built again)
  uint32_t hchunk_beg[RPQ_MAX_LABELS];  // per label, the chunks of rows of
  uint32_t hchunk_end[RPQ_MAX_LABELS];  // at least heavy_row edges
  uint32_t heavy_row;
  bool walk_rows;  // several lane groups: bottom-up levels walk each row (see set_chunks)
  unsigned long long label_edges[RPQ_MAX_LABELS];
  uint32_t n;
  uint32_t L;             // edge labels of the graph
  // lane groups
  uint32_t G;             // groups in this launch
  uint32_t Q;             // DFA states
  const uint32_t *lanesrc;  // [G * 64 * NW], 0xFFFFFFFF = empty lane
  // workspace
  unsigned long long *vis;     // [Q][n][G][NW]: groups innermost
  unsigned long long *fr0;     // frontier ping
  unsigned long long *fr1;     // frontier pong
  unsigned int *claim;         // [Q][n][G] level stamps (NW > 1)
  unsigned long long *spill;   // SPILL_CAP chunk records (nullptr: no spilling)
  unsigned long long spill_cap;  // records usable per level (<= SPILL_CAP)
  unsigned long long *list0;   // entries ((g*Q+q) << 32 | v)
  unsigned long long *list1;
  // Optional frontier bitmaps (nullptr: none), two of fbits_words words: bit
  // q*n + v of bitmap (level & 1) is set when some group holds (q, v) in the
  // level's frontier; bottom-up levels over a sparse frontier test it before
  // gathering a neighbour's frontier words.  Zero between searches.
  unsigned int *fbits;
  unsigned long long fbits_words;
  // List appends: a warp reserves append_seg slots at a time (0: one atomic
  // add per warp-aggregated append); unused reserved slots hold NO_ENTRY.
  unsigned int append_seg;
  unsigned long long list_cap;  // entries per list (overflow sets ERR_LIST_OVERFLOW)
  // Per-group automata (multi mode; nullptr otherwise): group g runs qg[g].
  // q is then the union of the groups' automata over states 0 .. Q-1: it
  // drives the bottom-up iteration and the cost estimates, while qg[g] drives
  // group g's top-down steps and work counters and from_tab[(g * Q + q2) * L
  // + l] is the set of group g's states that reach q2 on label l.
  const QueryDesc *qg;
  const unsigned int *from_tab;
  // Per-lane automata (lane mode; nullptr otherwise): every lane runs its own
  // minimal DFA (states 0 .. Q_i - 1, start state 0).  q then holds the union
  // of the lanes' automata in its bottom-up form (in_begin / in_label /
  // in_from over states 0 .. Q - 1): it drives bottom-up iteration and the
  // cost estimates.  The union's transitions (state, label, target) are listed
  // per source state: transition t of state s is la_trans[t] for
  // la_out_begin[s] <= t < la_out_begin[s + 1], the label in the low 16 bits
  // and the target above; la_mask[t * G * NW + g * NW + k] holds the lanes of
  // word k of group g that take it.  la_in_t[j * Q + s] is the transition
  // from state s of bottom-up group j (the group's label into its target).
  const unsigned short *la_out_begin;
  const unsigned int *la_trans;
  const unsigned long long *la_mask;
  const unsigned short *la_in_t;
  // the union's transitions grouped by (state, label): groups la_grp_begin[q]
  // .. la_grp_begin[q + 1] of state q, la_grp[i] = label | (transitions << 16),
  // la_gmask[i * G * NW ..] the OR of the group's lane masks (a lane's own DFA
  // takes at most one transition per (state, label), so the masks are disjoint)
  const unsigned short *la_grp_begin;
  const unsigned int *la_grp;
  const unsigned long long *la_gmask;
  // la_sl[s * L + l] (unions of at most 8 states): first transition of (state
  // s, label l) | the set of its targets << 16; its transitions are
  // consecutive, targets ascending
  const unsigned int *la_sl;
  BfsCtl *ctl;
  unsigned int stamp_base;     // claim stamps continue across launches
  unsigned int nblocks;
  unsigned int pull_dynamic;   // bottom-up levels take vertex chunks from a cursor (else round-robin)
  unsigned int lane_by_source; // lane mode: light bottom-up rows gathered once per (label, source state)
  int force;                   // 0 auto, 1 push only, 2 pull only
  float alpha;                 // push if alpha * push_cost < pull_cost
  unsigned long long time_limit_ns;
  QueryDesc q;
};

// The labels that a launch's automaton takes and the graph has.
inline uint64_t label_set(const BfsParams &p) {
  uint64_t set = 0;
  for (uint32_t j = 0; j < p.q.in_begin[p.q.n_states]; j++)
    if (p.q.in_label[j] < p.L) set |= 1ull << p.q.in_label[j];
  return set;
}
// The chunks of a launch of `starts` start vertices, and how launches of several
// lane groups read the other rows bottom-up.
//
// Where rows of 32 to 127 edges are the ordinary ones, more than one vertex in
// eight over the launch's labels, they stay whole: an item per row costs more
// than the row, and there is nothing to even out.  500,000 vertices of degree 40,
// a* from 64 start vertices: 1,825 us with their chunks, 512 without.  In R-MAT
// graphs of degree 16 to 100 at most one vertex in eleven has such a row, and the
// chunks make the calls 1.05 to 1.4 times as fast.
//
// There, and where the rows below 32 edges are long on average, levels walk a
// vertex's rows (pull_level) instead of listing the gathers of 32 vertices
// (pull_staged): the list costs more than it hides, the more so the fewer words a
// gather reads.  300 start vertices (two groups) on 500,000 of degree 40 / 20:
// 2,068 / 1,636 us listed, 1,313 / 1,274 walked; 4,096 on degree 20: 7.40 and
// 7.23 ms, degree 10: 6.8 and 7.4.  R-MAT 2^20 of degree 64, 300: 3.14 ms listed,
// 3.94 walked; its rows below 32 edges have 4 on average.
//
// Both need vertices enough for every warp to work on several at a time: of
// degree 100, 300 start vertices take 244 us on 16,000 vertices by chunks and
// lists, 290 by whole rows (32,000: 300 and 309; 64,000: 461 and 441), of degree
// 25 per label 296 listed and 352 walked on 32,000 (128,000: 534 and 437).
// Launches of one group have rows enough on any graph; the staged lane levels
// list rows anyhow (3,000 lanes on 128,000 vertices of degree 50 per label: 54 ms
// by chunks, 68 without).
constexpr uint32_t WHOLE_MIN = 1u << 15, WALK_MIN = 1u << 17;
inline void set_chunks(BfsParams &p, const ChunkLists &c, uint64_t starts, bool lanes_staged = false) {
  const uint64_t labels = label_set(p);
  uint64_t rows = 0, light = 0, vertices = 0;  // over the labels
  for (uint32_t l = 0; l < p.L; l++)
    if ((labels >> l) & 1u) {
      rows += c.shorter_rows[l];
      light += c.light[l];
      vertices += p.n;
    }
  const bool whole = rows * 8 > vertices && (p.G == 1 || p.n >= WHOLE_MIN) && !lanes_staged;
  p.walk_rows = whole || !c.rec || (p.n >= WALK_MIN && light > vertices * (p.G <= 4 ? 8 : 16));
  const bool shorter = c.shorter > 0 && starts >= FEW_STARTS && !whole;
  p.hchunk = c.rec;
  p.heavy_row = shorter ? HEAVY_ROW : LONG_ROW;
  for (uint32_t l = 0; l < p.L; l++) {
    p.hchunk_beg[l] = c.off[2 * l];
    p.hchunk_end[l] = c.off[2 * l + (shorter ? 2 : 1)];
  }
}

// Lane-mode bottom-up levels gather by source state for unions of at most
// LANE_SRC_Q states (larger ones per target state), and by the staged form,
// pull_lanes, in launches whose lanes fill a warp's row.  It needs 80 registers,
// so its kernel runs three blocks per SM; the plain form is a kernel of its own,
// at four: 1,797 lanes on R-MAT 2^24 (0.55 of the SMs), its three dense levels
// 636 / 777 / 767 ms, 853 / 1,049 / 1,038 at three.  Launches whose grid fits
// three blocks per SM anyway take a third build, the plain levels at 80 registers
// (200 lanes on 30,000 vertices of degree 40: 2.05 ms, 2.30 at 64).
enum class LaneKernel { plain, few, staged };
constexpr uint32_t LANE_SRC_Q = 8;
inline bool lanes_staged(int nw, uint32_t G, uint32_t Q, bool by_source) {
  return nw == 4 && by_source && Q <= LANE_SRC_Q && G * nw / 2 > 16;
}

// Launchers (return cudaError_t of the launch).
cudaError_t launch_vis_init(const BfsParams &p, const unsigned long long *empty, cudaStream_t st);
// Before a launch_msbfs of `live` start vertices, in lanes 0 .. live - 1: VIS,
// the control block and small[0 .. 4) set up; with ids (at most 64), lanesrc
// [0 .. 64) too.
cudaError_t launch_start(int nw, const BfsParams &p, uint32_t live, unsigned long long *small, uint32_t *lanesrc,
                         const uint32_t *ids, cudaStream_t st);
cudaError_t launch_msbfs(int nw, const BfsParams &p, int blocks, int threads, cudaStream_t st);
// Per-group automata (p.qg set): one lane word per group (NW = 1).
cudaError_t launch_msbfs_multi(const BfsParams &p, int blocks, int threads, cudaStream_t st);
int msbfs_multi_max_blocks(int threads, int *blocks_per_sm);
// Per-lane automata (p.la_* set), NW = 1 or 4.  VIS starts as empty_q[(q * G +
// g) * NW + k]: the lanes that are empty or whose automaton has no state q.
cudaError_t launch_msbfs_lane(int nw, LaneKernel k, const BfsParams &p, int blocks, int threads, cudaStream_t st);
int msbfs_lane_max_blocks(int nw, LaneKernel k, int threads, int *blocks_per_sm);
cudaError_t launch_vis_init_lane(int nw, const BfsParams &p, const unsigned long long *empty_q, cudaStream_t st);
// flag[i] = whether srcs[i] has an edge (offsets `off`, per label) on a label of label_mask.
cudaError_t launch_source_filter(const uint32_t *off, uint32_t n, uint32_t L, unsigned long long label_mask,
                                 const uint32_t *srcs, unsigned long long count, unsigned char *flag,
                                 cudaStream_t st);
// Edges per label that a launch's automaton takes, on average.
inline uint64_t label_edges(const BfsParams &p) {
  uint64_t m = 0, n_labels = 0;
  for (uint64_t set = label_set(p), l = 0; l < p.L; l++)
    if ((set >> l) & 1u) {
      m += p.label_edges[l];
      n_labels++;
    }
  return n_labels ? m / n_labels : 0;
}
// Blocks of a traversal launch over n vertices with `edges` edges per label:
// enough that a bottom-up level gives every sub-warp (the lanes it uses per
// vertex, two words each, rounded up to a power of two) a vertex, or GRID_EDGES
// edges where vertices have more, at most max_blocks.  Beyond that, blocks only
// make the barriers of a small graph's levels dearer (by the labels' sum instead
// of their average 600 lanes on 8,000 vertices of degree 100 took 3.35 ms for
// 2.95); sized by vertices alone, 64 start vertices on 1,000 vertices with 2.5 *
// 10^6 edges ran on four blocks, 3,390 us for (a|b)+.c where the full grid takes
// 299 and this rule 199.  Of a* there 4 edges are up to 13% faster and up to 5%
// slower, 64 lose 40% with 2 * 10^5 edges.
constexpr uint32_t GRID_EDGES = 16;
inline int bfs_grid(int max_blocks, int nw, uint32_t G, uint32_t n, uint64_t edges) {
  const uint32_t lanes = nw == 1 ? G : G * nw / 2;
  uint64_t sw = 1;
  while (sw < lanes) sw <<= 1;
  const uint64_t units = n > edges / GRID_EDGES ? n : edges / GRID_EDGES;
  const uint64_t want = (units * sw + 255) / 256;
  return want < (uint64_t)max_blocks ? (int)want : max_blocks;
}
int msbfs_max_blocks(int nw, int threads, int *blocks_per_sm, int *sms);

struct EmitParams {
  const unsigned long long *vis;
  uint32_t n;
  uint32_t G;
  uint32_t Q;
  uint32_t final_mask;
  const uint32_t *lanesrc;
  uint32_t tiles;                // 32-vertex tiles per segment (emit_tiles)
  uint32_t segs;                 // segments per group
  uint32_t *cnt;                 // [G * K][segs]
  const unsigned long long *off; // exclusive offsets of cnt (write pass)
  uint32_t *dst;                 // output destinations (write pass)
  unsigned long long *digest;    // [2]: sum, xor
  const uint32_t *final_g;       // per-group accepting masks (multi mode), else nullptr
  // per-lane accepting lanes (lane mode), else nullptr: word [q * G * NW + g
  // * NW + k] holds the lanes of word k of group g whose automaton accepts in
  // state q (final_mask is then the union of the lanes' accepting states)
  const unsigned long long *final_lane;
  // write pass: lanes whose rows also go out as bitsets over the vertices.
  // lane_slot[lane] = the lane's bitset index (bitset at bits + slot *
  // bwords, bwords a multiple of 4), NO_SOURCE for none; nullptr: no
  // bitsets.  With keep_lists = 0 such lanes write no destinations (their
  // counts must have been zeroed before the offsets were scanned).
  const uint32_t *lane_slot;
  unsigned long long *bits;
  uint64_t bwords;
  uint32_t keep_lists;
};
constexpr int EMIT_TILES = 128;  // 32-vertex tiles per segment at most
constexpr int EMIT_TILES_MIN = 8;
constexpr int EMIT_SEG = 32 * EMIT_TILES;
// Tiles per segment for a launch of G groups over n vertices, a block per
// segment and group: as long as possible (a row's first and last 32 words in
// a segment are stored word by word), but short enough for two blocks (12 of
// the two-warp blocks of nw = 1) per residency slot of the write pass.  With
// 4,096-vertex segments 300 sources on 65,537 vertices ran on 34 blocks, one
// source on R-MAT 2^20 on 256 blocks of two warps.
inline uint32_t emit_tiles(int nw, uint32_t G, uint32_t n) {
  const uint64_t want = nw == 1 ? 152ull * 12 : 152ull * 6;
  uint32_t t = EMIT_TILES;
  while (t > EMIT_TILES_MIN && ((uint64_t)n + 32 * t - 1) / (32 * t) * G < want) t >>= 1;
  return t;
}
inline uint32_t emit_segs(uint32_t tiles, uint32_t n) { return (uint32_t)(((uint64_t)n + 32 * tiles - 1) / (32 * tiles)); }
cudaError_t launch_emit(int nw, bool write, bool digest, const EmitParams &p, cudaStream_t st);
// Digest (sum, xor of splitmix64(src << 32 | dst)) of a materialized chunk's
// rows, added into digest[0..1].
// live: the lanes that may have rows (the first ones).
cudaError_t launch_row_digest(const uint32_t *lanesrc, const unsigned long long *lane_off, uint32_t live,
                              const uint32_t *dst, unsigned long long *digest, cudaStream_t st);
// Per-lane row count and digest (lane_stats[3 * lane + {0, 1, 2}] = rows,
// digest sum, digest xor over the lane's (source, y) rows); lane_stats zeroed
// by the caller.
cudaError_t launch_emit_lane_stats(int nw, const EmitParams &p, unsigned long long *lane_stats, cudaStream_t st);

// Write pass into interleaved (src, dst) rows of a caller's buffer (NW = 1).
cudaError_t launch_emit_pairs(const EmitParams &p, uint32_t *out, cudaStream_t st);

// Load (under the runtime's lazy module loading) the kernels the entry point
// that allocates nothing launches, so that their first use allocates nothing.
cudaError_t preload_static_msbfs_kernels();
cudaError_t preload_static_emit_kernels();
cudaError_t preload_scan_kernels();

// cnt[lane][*] = 0 for every lane with lane_slot[lane] != NO_SOURCE.
cudaError_t launch_zero_lane_counts(uint32_t *cnt, uint32_t segs, uint32_t n_lanes, const uint32_t *lane_slot,
                                    cudaStream_t st);
// lane_off[i] = off[i * segs] for the first `live` lanes, *total from there to
// lane_off[n_lanes] (lanes without a start vertex are the last ones); with
// lanesrc_out, also copies the lanes' start vertices there.
cudaError_t launch_gather_lane_off(const unsigned long long *off, uint32_t segs, uint32_t n_lanes, uint32_t live,
                                   const unsigned long long *total, unsigned long long *lane_off,
                                   const uint32_t *lanesrc, uint32_t *lanesrc_out, cudaStream_t st);

// Pair expansion for fetch: out[2k], out[2k+1] = (src, dst) of row first + k.
cudaError_t launch_expand_pairs(const uint32_t *lanesrc, const unsigned long long *lane_off, uint32_t n_lanes,
                                const uint32_t *dst, unsigned long long first, unsigned long long count,
                                uint32_t *out, cudaStream_t st);

// Device-wide exclusive scans.  `tmp` must hold scan_tmp_words(n) words.
size_t scan_tmp_words(size_t n);
cudaError_t exclusive_scan_u32_to_u64(const uint32_t *in, unsigned long long *out, size_t n,
                                      unsigned long long *total, unsigned long long *tmp, cudaStream_t st);
cudaError_t exclusive_scan_u64(const unsigned long long *in, unsigned long long *out, size_t n,
                               unsigned long long *total, unsigned long long *tmp, cudaStream_t st);

// Start-in-the-middle plan: (src, dst, label) triples of the out-CSR (triple
// e = out_col index e), and of a materialized chunk's rows with label x from
// position base.
cudaError_t launch_csr_triples(const uint32_t *off, const uint32_t *col, uint32_t n, uint32_t L, uint32_t *src,
                               uint32_t *dst, uint16_t *lab, cudaStream_t st);
cudaError_t launch_chunk_triples(const uint32_t *lanesrc, const unsigned long long *lane_off, uint32_t n_lanes,
                                 const uint32_t *cdst, unsigned long long base, uint16_t x, uint32_t *src,
                                 uint32_t *dst, uint16_t *lab, cudaStream_t st);

// Graph construction.  Returns RPQ_OK or an error code with *msg set.
int build_graph(DevGraph *g, uint32_t n, uint32_t L, uint64_t m, const uint32_t *d_src, const uint32_t *d_dst,
                const uint16_t *d_lab, cudaStream_t st, std::string *msg);
void free_graph_arrays(DevGraph *g, cudaStream_t st);  // all but vlabel
// Builds the list of the CSR `off` again without the shorter rows (see
// ChunkLists); the other streams that read the old one are done.
cudaError_t drop_shorter_chunks(const uint32_t *off, uint32_t n, uint32_t L, ChunkLists *c, cudaStream_t st);
int graph_key_bits(uint32_t n, uint32_t L);

// Stable LSD radix sort of 64-bit keys over bits [lo_bit, hi_bit); the result
// is in *a afterwards (the two buffers are swapped as needed).
cudaError_t sort_keys_u64(unsigned long long **a, unsigned long long **b, size_t m, int lo_bit, int hi_bit,
                          cudaStream_t st);
// Distinct keys of a sorted array, in order; *d_count (device) gets their number.
cudaError_t unique_keys_u64(const unsigned long long *sorted, size_t m, unsigned long long *out,
                            unsigned long long *d_count, cudaStream_t st);

}  // namespace rpq
