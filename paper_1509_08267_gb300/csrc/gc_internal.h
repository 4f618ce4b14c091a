// Internal declarations shared by the library's translation units (kernels, C ABI, server).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "gc.h"

namespace gc {

// Adjacency entries a warp loads per step of a work item (kStep / 32 per lane, issued together).
#ifndef GC_STEP
#define GC_STEP 128
#endif
constexpr int kStep = GC_STEP;

// Accumulator slot of a vertex of degree > T1 (its row is split into warp work items):
//   [0, kAccWords)  round window: colors 0..511 of the neighbours read this round
//   kAccFlag        conflict flag of this round
//   kAccDone        work items of this round finished (when the last item finishes the vertex)
//   kAccSurv        compact mode: list entries whose neighbour was not final when read this round
//   kAccNewLen      compact mode: entries written to the other list region this round
// Compact mode only, kept for the whole run (the slot belongs to the vertex):
//   [kAccFin, kAccFin+kAccWords)  colors 0..511 of neighbours found final
//   kAccSrc         where the vertex's list of possibly-changing neighbours is: 0 its CSR row,
//                   1 region A, 2 region B of its space in the list pool
//   kAccLen         entries in that list
//   kAccOffLo/Hi    offset of region A in the list pool (region B follows it, each deg entries)
//   kAccDeg         the vertex's degree
// The round part (words [0, 20)) is zero whenever a round starts: only vertices with several work
// items use it, and whoever finishes such a vertex clears it.
constexpr int kAccWords = 16;
constexpr int kAccFlag = 16;
constexpr int kAccDone = 17;
constexpr int kAccSurv = 18;
constexpr int kAccNewLen = 19;
constexpr int kAccFin = 32;
constexpr int kAccSrc = 48;
constexpr int kAccLen = 49;
constexpr int kAccOffLo = 51;
constexpr int kAccOffHi = 52;
constexpr int kAccDeg = 53;
constexpr int kAccStride = 64;  // 256 B per slot
// Ordered mode: vertices of degree <= min(T1, kOrdSmall) are one thread's work; larger rows are
// split into work items of min(CH, kOrdChunk) entries; a vertex of several items merges them in an
// accumulator slot of kOrdSlotWords words (window 0..15, done counter kAccDone).
constexpr int kOrdSmall = 8;
constexpr int kOrdMid = 32;  // degree <= kOrdMid (and > the small bound): an 8-lane group each
// Priority of the recoloring pass (gc_recolor): key(v) = (-min(c(v), 2^20 - 1), h(v), v) for the
// given coloring c, the color classes in decreasing color order.
constexpr int32_t kPriorityRecolor = 3;
constexpr int kOrdChunk = 128;
constexpr int kOrdSingleChunk = 64;  // default work-item size of the ordered mode on a single graph
constexpr int kOrdSlotWords = 32;
constexpr int kOrdPad = 32, kOrdSet = 4 * kOrdPad;  // words from one counter, or counter set, to the next

// One row of a batch's offset tables: graph g's vertices [v0, v1) of n, entries [e0, e1) of nnz.  Every
// row is checked against the totals by itself: a table that rises and falls again has rows that look
// right next to each other and lie outside the arrays.
inline __host__ __device__ bool batch_row_ok(int32_t g, int64_t v0, int64_t v1, int64_t e0, int64_t e1, int64_t n,
                                             int64_t nnz) {
    return 0 <= v0 && v0 <= v1 && v1 <= n && 0 <= e0 && e0 <= e1 && e1 <= nnz && (g != 0 || (v0 == 0 && e0 == 0));
}

// Priority digests of the value keys (largest first, smallest last): 24 bits in the order of the 31
// priority bits (kKeyCap - value over 11 hash bits), of which a vertex state keeps the top 8 or 16.  The
// keys are cut into bins -- one per value below 128, eight per power of two above, the larger value
// first -- and each bin gets the part of the range that its vertices' degrees are of all of them, so that
// a worklist row meets every digest equally often; inside its bin a key lies by what is left of the value
// and by the hash.  (A fixed logarithmic code of the value gave the vertices of one degree one digest: on
// a mesh every neighbour tied, 85% of the row sweeps had to be resolved by the full keys and round 1 could
// not stop early.  Largest first, a whole call: 160^3 stencil 9.96 ms with it, 2.34 now; 3,000^2 grid 5.27 and
// 1.08; 600 cliques of 150 in a batch 23.4 and 4.7; R-MAT n = 5,000 3.1 and 0.41.)
constexpr uint32_t kKeyCap = (1u << 20) - 1u;
constexpr int kDigestExact = 128;
constexpr int kDigestBins = kDigestExact + 8 * 13;
struct DigestBin {
    uint32_t base, width;  // in 2^-24 of the range
};
inline __host__ __device__ int value_lead(uint32_t value) {  // position of the leading one
#ifdef __CUDA_ARCH__
    return 31 - __clz(static_cast<int>(value));
#else
    return 31 - __builtin_clz(value);
#endif
}
inline __host__ __device__ int digest_bin(uint32_t value) {
    if (value < static_cast<uint32_t>(kDigestExact)) return static_cast<int>(value);
    const int lead = value_lead(value);  // 7..19
    return kDigestExact + 8 * (lead - 7) + static_cast<int>(value >> (lead - 3) & 7u);
}
// A bin's part of the range: `before` of `total` lie in the bins of larger values, `count` in the bin.
inline __host__ __device__ DigestBin digest_range(uint64_t before, uint64_t count, uint64_t total) {
    if (total == 0) return DigestBin{0u, 0u};
    return DigestBin{static_cast<uint32_t>((before << 24) / total), static_cast<uint32_t>((count << 24) / total)};
}
inline __host__ __device__ uint32_t key_digest24(const DigestBin *bins, uint32_t p31) {
    const uint32_t value = kKeyCap - (p31 >> 11), h = p31 & 2047u;
    const DigestBin b = bins[digest_bin(value)];
    uint32_t inside = h;  // place in the bin, in 2^-11 of it
    if (value >= static_cast<uint32_t>(kDigestExact)) {
        const int s = value_lead(value) - 3;  // bits of the value below the bin's
        const uint32_t rest = ~value & ((1u << s) - 1u);
        inside = s <= 11 ? rest << (11 - s) | h >> s : rest >> (s - 11);
    }
    const uint32_t x = b.base + static_cast<uint32_t>(static_cast<uint64_t>(b.width) * inside >> 11);
    return x < (1u << 24) ? x : (1u << 24) - 1u;
}

// Worklist counters: three sets used round-robin (read / append / clear), kCnt words each.
constexpr int kCnt = 4;
//   kCntSmall   vertices of degree <= T1
//   kCntItems   larger vertices (their accumulator slots, in non-compact mode, are numbered by it)
//   kCntChunks  work items
//   kCntMulti   deterministic mode: larger vertices with more than one work item
constexpr int kCntSmall = 0, kCntItems = 1, kCntChunks = 2, kCntMulti = 3;

// Bytes per work item in the work-item buffers (deterministic items are 48 bytes, in-place 16).
constexpr size_t kItemBytes = 48;

// Grid barrier of the persistent round kernels: arrivals so far in the current launch (launch_rounds
// zeroes it before every launch).
struct alignas(128) GridBar {
    unsigned count;
    unsigned pad[31];
};

// Everything the setup, round and count kernels need.  A single graph uses plain CSR addressing;
// with BATCH the vertices of graph g are the global ids [g_vbase[g], g_vbase[g] + g_n[g]), its own
// local rowptr (g_n[g] + 1 entries) starts at rowptr[g_rbase[g]] and its local neighbour ids start at
// colidx[g_ebase[g]] (g_m[g] entries).  gc_color_batch and the server both fill this table.
struct RoundParams {
    int32_t n;    // total vertices (single graph: n)
    int32_t G;    // graphs in the table
    int64_t nnz;  // single graph: adjacency entries
    const int32_t *rowptr;
    const int32_t *colidx;
    const int64_t *g_vbase;  // [G]
    const int32_t *g_n;      // [G]
    const int64_t *g_ebase;  // [G]
    const int64_t *g_rbase;  // [G]
    const int64_t *g_m;      // [G]
    int32_t *vg;             // [n] graph id per vertex (batch)
    uint64_t seed;
    const uint64_t *g_seed;  // [G] per-graph priority seeds (the server); nullptr: `seed` for every graph

    // In-place and ordered modes: vertex state words, low 32 bits = color (int32, -1 = uncolored), high
    // 32 bits = FINAL and the vertex's priority bits, so one gather gives a neighbour's color and
    // priority.  (Partition mode: colors now, and as the round began.)
    uint64_t *col0;
    uint64_t *col1;
    // Deterministic mode (set_det_state): 16 bits per vertex and buffer -- color (saturated at 127) << 9
    // | priority digest (8 bits: the hash's top bits, or key_digest24's) << 1 | FINAL -- which is all that nearly every adjacency
    // entry needs of its neighbour, so the gathered array is a quarter of the state words' size, and
    // one subtraction tells a neighbour of equal color and smaller digest.  Entry n stands for no
    // neighbour (color 127, digest 255).  The exact color of a saturated one is in cx0 / cx1 (written
    // only then); prio holds the 31 priority bits, read when colors and digests are equal.
    uint16_t *s16a;  // read in odd rounds, written in even ones (like cx0)
    uint16_t *s16b;  // written in odd rounds (like cx1)
    int32_t *cx0, *cx1;
    uint32_t *prio;
    const uint8_t *g_done;  // [G] graphs the set-up skips (colored by small_batch_kernel), or nullptr
    int64_t ci_len;  // entries of colidx that may be read (16-byte loads stay inside them)
    int32_t *small0, *small1;  // thread-per-vertex worklists (two parities)
    int4 *chunk0, *chunk1;     // warp work items, kItemBytes each (two parities)
    int4 *ord0, *ord1;         // ordered mode: the ready vertices, n entries (two parities): small ones from
                               // the front, medium-degree ones from the back
    unsigned ord_items;        // ordered mode: entries chunk0 / chunk1 hold
    unsigned *ord_cnt;         // [3][kOrdSet] its counter sets, a counter per 128 bytes: every releasing warp adds
                               // to them, and atomics on one line queue
    int32_t *items;            // setup scratch: larger vertices found by the binning pass
    unsigned *tmp;             // [2] setup scratch counters: larger vertices, their work items
    unsigned *cnt;             // [3][kCnt] worklist counters
    unsigned *acc;             // [slots][kAccStride]
    int32_t *lists;                   // compact mode: list pool (two regions of deg entries per larger vertex)
    unsigned long long *list_total;   // compact mode: setup adds 2 * deg of every larger vertex
    unsigned long long *list_alloc;   // compact mode: expand's allocation counter in the list pool
    int32_t slot_per_vertex;          // compact mode, 1: vertex V's slot is V and its list regions start
                                      // at 2 x its first entry (no allocation; the server's layout)
    int32_t sort_shift;               // log2 of the vertex block of the thread-worklist sort (sort_shift(n))
    unsigned *deg_hist;               // [2 * sort_bins(n)] optional: setup counts thread-per-vertex rows per
                                      // (vertex block, degree) bin, zeroed by the caller; list positions per
                                      // bin follow
    GridBar *bar;
    int32_t *err;              // [4] status, vertex, entry, extra
    int32_t *passes;           // [2] first round not executed by the last launch, last round executed
    int32_t *graph_last;       // [G] last round whose worklist held a vertex of graph g
    unsigned long long *stats; // [4 * stats_cap + 1] per round |W_r|, sum of degrees, end time (ns),
                               // adjacency entries read; last entry: start time of the launch (optional)
    int32_t stats_cap;
    int32_t pass_begin;        // first round this launch runs (the worklist of that round is current)
    int32_t pass_end;          // rounds >= pass_end are not run by this launch
    int32_t cap_is_error;      // reaching pass_end with work left is GC_ERR_NO_CONVERGENCE
    int64_t spin_ns;
    int32_t T1;  // largest degree handled by one thread
    int32_t CH;  // adjacency entries per warp work item
    int32_t priority;  // GC_PRIORITY_* or kPriorityRecolor: what the 31 priority bits of a state word hold
    const int32_t *prio_rank;  // smallest last: the peel levels; recoloring: the given coloring (int32[n])
    int32_t spread;  // in-place mode: phase 1 takes the thread worklist in a spread order (set when no
                     // vertex is past T1: the degree-sorted order then balances nothing)
    // Deterministic mode from C_1 = 0: the colors of round r are at most r - 1 (a loser's First Fit
    // color exceeds the largest color around it by at most one).  A sweep that knows its vertex loses
    // and has seen every color 0..r-1 around it knows the vertex's next color (r) and stops early.
    int32_t early_exit;
    // Hand-over to the core phase (deterministic compact mode).  core_max > 0: the round kernel stops
    // at the top of the first round whose worklist has at most core_max vertices whose lists hold at
    // most core_emax entries, and sets *core_go; the core kernels (gc_core.cu) finish the coloring.
    int32_t core_max;
    int64_t core_emax;
    unsigned long long *ecnt;  // [3] entries in the lists of each counter set's worklist (core_max > 0)
    int32_t *core_go;          // set to 1 by the round kernel when it hands over
};

// Places the deterministic mode's vertex state in two buffers: the exact colors of both parities in
// the first (8 n bytes), the priority bits and both 16-bit arrays in the second (8 n + kDetPad bytes).
constexpr size_t kDetPad = 64;
inline void set_det_state(RoundParams &P, void *buf0, void *buf1, size_t n) {
    P.cx0 = static_cast<int32_t *>(buf0);
    P.cx1 = P.cx0 + n;
    P.prio = static_cast<uint32_t *>(buf1);
    P.s16a = reinterpret_cast<uint16_t *>(P.prio + n);
    P.s16b = P.s16a + n + 1;
}

// Core phase (gc_core.cu).  Once the worklist is small, its vertices get local ids 0..m-1 (the core)
// and their rows are rebuilt as lists of the local ids of neighbours still on the worklist, the
// neighbour's key order in the top bit (kCoreSmaller: smaller key than the row's vertex); the colors
// of neighbours already final go into the vertex's window of final colors.  Each round every block
// keeps the colors of all m core vertices in shared memory (8 bits each, saturated at 255, the exact
// value in cex; and a FINAL bit each), so a row's neighbour colors come from shared memory instead
// of L2.  Rows are cut once into pieces of at most kCorePiece entries, which every round's list of
// active pieces hands out to the warps.
constexpr uint32_t kCoreSmaller = 0x80000000u;
constexpr int64_t kCoreEntries = int64_t{1} << 27;  // list entries the core phase takes at most
constexpr int kCoreCnt = 8;  // counter words per set
#ifndef GC_CORE_PIECE
#define GC_CORE_PIECE 2048
#endif
constexpr int kCorePiece = GC_CORE_PIECE;
// Per core vertex, kCoreRecWords words: [0, 16) the window of neighbour colors 0..511 and kCoreFlag
// (some smaller-key neighbour has the vertex's color), which the row build leaves for the core's first
// round, [kAccFin, kAccFin + 16) the window of final neighbours' colors, then the row's offset in the
// pool, degree, global id, row length, graph, the hand-over list's length and the vertex's range of
// pieces.
constexpr int kCoreRecWords = 64;
constexpr int kCoreFlag = 16;
constexpr int kCoreOffLo = 48, kCoreOffHi = 49, kCoreDeg = 50, kCoreGid = 51, kCoreFill = 52, kCoreG = 53;
constexpr int kCoreListLen = 56, kCorePcBeg = 57, kCorePcEnd = 58;
constexpr int kCoreTail = 59;  // the vertex's tail id (tail phase)
// Tail phase (gc_tail.cu).  Once the core's worklist has at most tail_max vertices, one thread-block
// cluster of tail_nc blocks runs the remaining rounds: the worklist vertices get tail ids 0..k-1 in
// key order, every block keeps all k colors in shared memory and owns the rows (bitmaps over the
// tail ids) of the vertices t with t % tail_nc equal to its rank, and new colors are stored into
// every block's copy through distributed shared memory.  kTailOwned rows per block.  Default
// threshold kTailDefault: a cluster has a tenth of the GPU's SMs, so the tail pays off only once a
// round's work is small (on R-MAT scale 22: 0.3 ms saved at 256-512 vertices, less at 768, a loss
// from 1,024).
constexpr int kTailOwned = 256;
constexpr int kTailDefault = 384;
struct CoreParams {
    int32_t max_v;        // vertex capacity M (shared memory holds M 8-bit colors and M FINAL bits; a
                          // multiple of 16)
    int64_t max_e;        // list entries the core may hold (the pool's size)
    int64_t max_pieces;   // piece capacity: max_e / kCorePiece + M
    unsigned *rec;        // [M][kCoreRecWords]
    int32_t *cex;         // [2][M] exact colors, double-buffered like col0 / col1
    uint8_t *c8;          // [2][M] colors saturated at 255, double-buffered like cex
    unsigned *fbits;      // [M / 32 + 1] FINAL bit of every core vertex (zero at hand-over)
    int4 *pieces;         // [max_pieces] {local vertex, pool offset, entries, flags}
    int32_t *active;      // each round's worklist: [2][M] pieces of the one-piece vertices, [2][M] {first piece,
                          // pieces} of the others
    uint2 *log;           // [2][M] {local vertex, 8-bit color | FINAL << 8} of the vertices a round finished
    int32_t *pool;        // [max_e] the rows
    unsigned long long *bump;  // pool allocation counter
    unsigned *cnt;        // [3][kCoreCnt] per-round counters: vertices finished (log entries), losers, one-piece
                          // vertices, grabs, vertices of several pieces
    unsigned *m;          // [4]: larger vertices numbered by the index kernel, m, pieces
    int32_t tail_max;     // tail phase once the worklist has at most this many vertices (0: never)
    int32_t tail_nc;      // blocks of the tail's cluster (tail_max <= kTailOwned * tail_nc)
    unsigned *tail;       // [4]: 1 when the core handed over to the tail, the tail's first round, the round
                          // the core left for the host's sake (0: it did not)
    const int *leave;     // a host word that asks the rounds to stop when it is not 0, or nullptr
};

// Small graphs (gc_small.cu).  A batch's graphs of at most kSmallBatchVertices vertices and
// kSmallBatchEntries entries are colored by one block each; a single graph of at most
// kSmallOneVertices vertices whose rows average at most kSmallOneRow entries by one block (up to
// kSmallBlockVertices vertices and kSmallBlockEntries entries) or one cluster (kSmallOneEntries).
constexpr int32_t kSmallBatchVertices = 4096;
constexpr int64_t kSmallBatchEntries = int64_t{1} << 18;
constexpr int32_t kSmallOneVertices = 16384, kSmallBlockVertices = 2048;
constexpr int64_t kSmallOneEntries = int64_t{1} << 19, kSmallBlockEntries = int64_t{1} << 15;
constexpr int64_t kSmallOneRow = 64;
struct SmallBatch {
    int32_t *queue;            // [G] the small graphs, largest first
    unsigned *queued, *taken;  // their number; how many blocks have taken
    unsigned long long *left;  // vertices of the other graphs
    uint8_t *g_done;           // [G] 1: small
};
struct SmallOne {
    uint32_t *exchange;   // [2][cap] a cluster's new states
    unsigned *cnt;        // [3] a cluster's losers per round
    int32_t *out;         // [n] the colors (written only if nothing is wrong)
    int32_t *result;      // [9] {0: done, 1: too large, -1: error in [5..8]; entries, last round, colors, largest}
    int32_t cap;          // vertices the shared arrays hold (a multiple of 4)
    int64_t max_entries;  // larger graphs are left alone
};
// The cluster a single graph runs as (16 or 8 blocks, 0: none).
int small_one_blocks();
cudaError_t launch_small_one(const RoundParams &P, const SmallOne &A, int blocks, cudaStream_t s);
// After launch_batch_tables: picks the small graphs and colors them (nnz: the batch's entries; *grid: the
// blocks launched, of 256 threads).
cudaError_t launch_small_batch(const RoundParams &P, const SmallBatch &B, int64_t nnz, cudaStream_t s, int *grid);

// Launch wrappers (gc_kernels.cu).  All return the launch's cudaError_t.
// gc_color_batch: graph table from the offset tables, graph id per vertex, graph_last = 1 (0 if empty).
cudaError_t launch_batch_tables(const RoundParams &P, const int64_t *vtx_off, const int64_t *edge_off,
                                int64_t *g_vbase, int32_t *g_n, int64_t *g_ebase, int64_t *g_rbase, int64_t *g_m,
                                cudaStream_t s);
// Binning of vertices [v_begin, v_end) into the worklist of round P.pass_begin.  g_fixed >= 0: all
// of them belong to graph g_fixed (vg is written, and graph_last[g_fixed] is raised to pass_begin
// if any of them has a neighbour); otherwise vg must be filled already.
cudaError_t launch_setup(const RoundParams &P, int mode, bool batch, int32_t v_begin, int32_t v_end,
                         int32_t g_fixed, cudaStream_t s);
// With P.deg_hist: writes the thread-per-vertex entries of [v_begin, v_end) (counted by setup) to
// the current small list in increasing order of degree.  Without it, setup appended them already.
cudaError_t launch_sort_small(const RoundParams &P, bool batch, int32_t v_begin, int32_t v_end, cudaStream_t s);
// The thread-worklist sort's vertex-block size (log2) for n vertices, and its bins for vertex ids
// below v_end (P.deg_hist holds twice as many words).
int32_t sort_shift(int64_t n);
int32_t sort_bins(int32_t v_end, int32_t shift);
// Turns the n_items larger vertices found by setup into work items of round P.pass_begin
// (n_items < 0: the count setup left in P.tmp[0] on the device).
// compact: every larger vertex gets a persistent slot and list-pool space (deterministic mode).
cudaError_t launch_expand(const RoundParams &P, int mode, bool batch, bool compact, int32_t n_items,
                          cudaStream_t s);
// After the deterministic launch_setup with a value key: the vertices' priority digests.  cnt:
// [kDigestBins] zeroed counters.
cudaError_t launch_digests(const RoundParams &P, unsigned long long *cnt, cudaStream_t s);
// compact (deterministic mode only): larger vertices sweep packed lists of the neighbours that can
// still change instead of their whole rows.
// Round-kernel variants: kRoundWide is compiled for 3 resident blocks per SM (80 registers a thread),
// for graphs whose adjacency entries are mostly in larger vertices; kRoundNarrow for 4 (64); kRoundSmall
// (deterministic mode, no larger vertex) has no work-item code.
enum RoundVariant { kRoundNarrow = 0, kRoundWide = 1, kRoundSmall = 2 };
cudaError_t launch_rounds(const RoundParams &P, int mode, bool batch, bool compact, int grid, int block,
                          cudaStream_t s, RoundVariant v = kRoundNarrow);
cudaError_t round_kernel_occupancy(int mode, bool batch, bool compact, int block, int *blocks_per_sm,
                                   RoundVariant v = kRoundNarrow);
// Distinct colors and largest color per graph over vertices [v_begin, v_end) (graphs g_begin..g_end-1).
// `colors_sel` != NULL: deterministic mode's state, the buffer that round *colors_sel wrote (s16b / cx1
// when it is odd, else s16a / cx0); NULL: the state words col0.  `out` != NULL receives the colors of
// [v_begin, v_end) (out[0] is vertex v_begin) unless err[0] != 0.
cudaError_t launch_count_colors(const RoundParams &P, bool batch, const int32_t *colors_sel, int32_t v_begin,
                                int32_t v_end, int32_t g_begin, int32_t g_end, unsigned *bitmap, int32_t *gmax,
                                int32_t *gcount, int32_t *out, cudaStream_t s);
// Ordered mode (GC_MODE_ORDERED): after the in-place launch_setup (every vertex with neighbours
// uncolored) with P.T1 <= kOrdSmall and P.CH <= kOrdChunk, with the counter sets and P.acc's slots
// zeroed, counts each vertex's smaller-key neighbours into its word W[n], lists the first ready
// vertices (P.ord0 / ord1 hold n entries each, chunk0 / chunk1 P.ord_items work items) and runs the
// cooperative round kernel on `grid` blocks.
cudaError_t ordered_kernel_occupancy(bool batch, int block, int *blocks_per_sm);
// Smallest-last levels (single graph): launch_peel_init sets the words W to deg(v), level[v] = 0, the two
// threshold words kw[2] and adds the work items the lists may need (vertices past kOrdMid, P.CH
// entries each) to *items; launch_peel (counter sets zeroed, P.T1 <= kOrdSmall, P.CH <= kOrdChunk,
// lists as the ordered mode's; rlist0 / rlist1 int32[n] scratch with two counters rcnt) writes
// level[v] >= 1, the number of levels to passes[0] and the degeneracy to passes[1].
cudaError_t launch_peel_init(const RoundParams &P, unsigned long long *W, int32_t *level, unsigned *kw, unsigned *items,
                             cudaStream_t s);
cudaError_t peel_kernel_occupancy(int block, int *blocks_per_sm);
cudaError_t launch_peel(const RoundParams &P, unsigned long long *W, int32_t *level, unsigned *kw, int32_t *rlist0,
                        int32_t *rlist1, unsigned *rcnt, int grid, int block, cudaStream_t s);
cudaError_t launch_ordered(const RoundParams &P, bool batch, unsigned long long *W, int grid, int block, cudaStream_t s);
// Partition mode (GC_MODE_PARTITION, single graph): set-up (rows checked, colors -1, W_1 = V) and
// the cooperative round kernel with p blocks of consecutive ids.
cudaError_t launch_partition_init(const RoundParams &P, cudaStream_t s);
cudaError_t partition_kernel_occupancy(int block, int *blocks_per_sm);
cudaError_t launch_partition_rounds(const RoundParams &P, int32_t p, int grid, int block, cudaStream_t s);
cudaError_t launch_validate(int32_t n, const int32_t *rowptr, const int32_t *colidx, int flags, int32_t *err,
                            cudaStream_t s);
// gc_det_round: one fused deterministic round over the worklist vertices work[0, nwork).
cudaError_t launch_det_round_block(int32_t n, const int32_t *rowptr, const int32_t *colidx, uint64_t seed,
                                  const int32_t *cur, const int32_t *work, int32_t nwork, int32_t *next, int32_t *lost,
                                  int32_t *err, cudaStream_t s);
// Core phase (after launch_rounds handed over, *P.core_go = 1; every kernel returns at once when
// it did not): local ids and rows, the round kernel, and the final colors written back to both buffers
// of the vertex state.  core_max_vertices: the largest M the shared memory of one block per SM allows.
int32_t core_max_vertices();
cudaError_t launch_core(const RoundParams &P, const CoreParams &Q, bool batch, cudaStream_t s);
// After a core that left (Q.tail[2] = P.pass_begin): the core vertices' colors back into both state
// buffers and the unfinished ones onto the worklist of that round, the larger ones for launch_expand.  The
// worklist counters and P.tmp must be zero.
cudaError_t launch_core_return(const RoundParams &P, const CoreParams &Q, cudaStream_t s);
// Tail phase: the largest cluster (16 or 8 blocks) the tail kernel can run as, 0 if none; the launch
// (every block returns at once unless the core handed over).
int32_t tail_cluster_size();
cudaError_t launch_tail(const RoundParams &P, const CoreParams &Q, bool batch, cudaStream_t s);

}  // namespace gc

namespace gc {
int set_last_error(int code, const char *fmt, ...);
}
