// Small graphs of the deterministic mode (sm_103a): a whole coloring by one block, or by one
// thread-block cluster, with the vertex states in shared memory.
//
// The rule is Algorithm 1's (Section 3.1) as in gc_kernels.cu: in round r a worklist vertex v loses
// iff a neighbour of equal color in C_r has a smaller key, and a loser's next color is the least color
// absent from C_r over its neighbours.  A graph of a few thousand vertices needs a dozen rounds of
// microseconds of work; on the whole GPU each round is a grid barrier and a chain of L2 round trips, and
// the call is a dozen launches.  Here a round is a block (or cluster) barrier, a neighbour's state is a
// shared-memory word, and set-up, rounds and color count are one launch:
//
//   small_batch_kernel   the small graphs of a batch, one block of 256 threads each, largest first from
//                        a queue; their colors go into the batch's vertex state, marked FINAL, and the
//                        regular kernels skip their vertices
//   small_one_kernel     a single graph on one block of 1,024 threads, or on a cluster whose blocks own
//                        equal ranges of vertices; every block keeps all states, the owners' new ones
//                        pass through global memory (L2) between two cluster barriers
//
// What bounds them: latency -- the row and entry loads of a round (L1 and L2 hits), its barriers, and for
// the batch the L1 lookups of 32 rows in 32 places.  ER n = 1,000, degree 8 (9 rounds): 30 us of kernel,
// 290 -> 64 us a call from Python; n = 10,000, degree 16 (12 rounds) on 16 blocks: 73 us, 407 -> 123;
// 4,096 graphs of 100..4,000 vertices: 5.1 -> 2.43 ms (without the degree sort 5.8; a shared atomic
// per entry of a long row instead of register masks: 4.1).  A single graph past kSmallOneVertices or
// denser than kSmallOneRow entries a row is left to the core phase, whose 152 blocks then win.
//
// State word: color << 17 | 16-bit key digest << 1.  A neighbour's word minus (own color << 17) is below
// twice the own digest exactly for an equal color and a smaller digest; equal digests (hash key: one pair in
// 65,536; value keys: hardly more than the pairs whose 31 priority bits are equal) compare the full keys.
#include <algorithm>

#include "gc_device.cuh"

namespace gc {
namespace {

constexpr int kSmallRow = 128;  // longest row one thread sweeps; longer ones take a warp
constexpr int kWinWords = 32;  // a warp's color window: 1,024 colors at a time
constexpr uint32_t kNobody32 = 0xfffffffeu;  // state of the entry past the last vertex's (index cap)

struct SmallGraph {
    const int32_t *rp;  // local row offsets
    int64_t e0;         // first entry in colidx
    int64_t m;
    int32_t n, vbase, g;
    uint64_t seed;
    int64_t ci_len;  // entries of colidx that may be read
};

struct SmallShared {
    unsigned count[2][2];  // [parity][small, large] worklist vertices of this block
    int bad;               // a malformed row or entry was found
    int stop;              // ... as of the last barrier: leave
    unsigned colors;
    int32_t top;
    unsigned at[kSmallRow + 1];  // set-up: vertices per degree, then their list positions
};

// bins: the value keys' table, nullptr for the hash key.
__device__ __forceinline__ uint32_t small_digest(const DigestBin *bins, uint32_t p31) {
    return bins ? key_digest24(bins, p31) >> 8 : p31 >> 15;
}

// The full keys of two vertices of graph g: is u's smaller?
__device__ __noinline__ bool small_key_less(const RoundParams &P, const SmallGraph &g, int32_t u, int32_t v) {
    uint32_t p[2];
    const int32_t x[2] = {u, v};
    for (int k = 0; k < 2; ++k) {
        const uint64_t h = vertex_hash(g.seed, static_cast<uint32_t>(x[k]));
        const int32_t d = __ldg(g.rp + x[k] + 1) - __ldg(g.rp + x[k]);
        constexpr int32_t kCap = static_cast<int32_t>(kKeyCap);
        p[k] = P.priority == GC_PRIORITY_HASH
                   ? static_cast<uint32_t>(h >> 33)
                   : static_cast<uint32_t>(kCap - min(d, kCap)) << 11 | static_cast<uint32_t>(h >> 53);
    }
    return key_less(p[0], p[1], static_cast<uint32_t>(u), static_cast<uint32_t>(v), g.seed);
}

__device__ __forceinline__ void small_bad(const RoundParams &P, SmallShared &S, const SmallGraph &g, int32_t v, int64_t j) {
    set_error(P.err, GC_ERR_INVALID_GRAPH, g.vbase + v, j);
    S.bad = 1;
}

// Equal digests (a vertex that is its own neighbour always gets here before it can win) or malformed
// entries: did v lose, by the full keys (one thread; rare).
__device__ __noinline__ bool small_exact(const RoundParams &P, const SmallGraph &g, SmallShared &S, const uint32_t *cur,
                                         int32_t v) {
    const int32_t b = __ldg(g.rp + v), e = __ldg(g.rp + v + 1);
    for (int32_t j = b; j < e; ++j) {
        const int32_t u = load_entry(P.colidx + g.e0 + j);
        if (static_cast<uint32_t>(u) >= static_cast<uint32_t>(g.n) || u == v) {
            small_bad(P, S, g, v, j);
            continue;
        }
        if (cur[u] >> 17 == cur[v] >> 17 && small_key_less(P, g, u, v)) return true;
    }
    return false;
}

// The same by a warp (longer rows).
__device__ __noinline__ bool small_exact_warp(const RoundParams &P, const SmallGraph &g, SmallShared &S,
                                              const uint32_t *cur, int32_t v, int lane) {
    const int32_t b = __ldg(g.rp + v), e = __ldg(g.rp + v + 1);
    bool lose = false;
    for (int32_t j = b + lane; j < e; j += 32) {
        const int32_t u = load_entry(P.colidx + g.e0 + j);
        if (static_cast<uint32_t>(u) >= static_cast<uint32_t>(g.n) || u == v)
            small_bad(P, S, g, v, j);
        else if (cur[u] >> 17 == cur[v] >> 17)
            lose |= small_key_less(P, g, u, v);
    }
    return __any_sync(kFull, lose);
}

// A row's degree, or -1 for a malformed one.
__device__ __forceinline__ int32_t small_degree(const SmallGraph &g, int32_t v, int64_t &b) {
    b = __ldg(g.rp + v);
    const int64_t e = __ldg(g.rp + v + 1);
    const bool ok = b >= 0 && b <= e && e <= g.m && (v != 0 || b == 0) && (v != g.n - 1 || e == g.m);
    return ok ? static_cast<int32_t>(e - b) : -1;
}

// The value keys' digests of one graph (block-wide; both arrays kDigestBins long).
__device__ void small_digests(const SmallGraph &g, DigestBin *bins, unsigned *cnt) {
    for (int t = static_cast<int>(threadIdx.x); t < kDigestBins; t += static_cast<int>(blockDim.x)) cnt[t] = 0u;
    __syncthreads();
    for (int32_t v = static_cast<int32_t>(threadIdx.x); v < g.n; v += static_cast<int32_t>(blockDim.x)) {
        int64_t b;
        const int32_t d = small_degree(g, v, b);
        if (d > 0) atomicAdd(&cnt[digest_bin(min(static_cast<uint32_t>(d), kKeyCap))], static_cast<unsigned>(d));
    }
    __syncthreads();
    if (threadIdx.x < 32) digest_table(cnt, bins, static_cast<int>(threadIdx.x));
}

// Set-up of one graph by the calling block: rows checked (every block of a cluster checks all of them
// and comes to the same end), the states of all vertices, and the block's worklist: the vertices of
// [lo, hi) with neighbours, rows up to kSmallRow at the list's front by increasing degree (a counting
// sort: the 32 rows a warp sweeps side by side then have similar lengths), longer ones at its back.
// bins: room for the value keys' table and counts (key_room), or nullptr.  Ends with a block barrier.
__device__ void small_setup(const RoundParams &P, const SmallGraph &g, SmallShared &S, uint32_t *st, uint16_t *list,
                            int32_t cap, int32_t lo, int32_t hi, uint32_t *st2, DigestBin *bins) {
    const int lane = threadIdx.x & 31;
    if (bins) small_digests(g, bins, reinterpret_cast<unsigned *>(bins + kDigestBins));
    for (int t = static_cast<int>(threadIdx.x); t <= kSmallRow; t += static_cast<int>(blockDim.x)) S.at[t] = 0u;
    __syncthreads();
#pragma unroll 4
    for (int32_t v = static_cast<int32_t>(threadIdx.x); v < g.n; v += static_cast<int32_t>(blockDim.x)) {
        int64_t b;
        int32_t d = small_degree(g, v, b);
        if (d < 0) {
            small_bad(P, S, g, v, b);
            d = 0;
        }
        const uint64_t h = vertex_hash(g.seed, static_cast<uint32_t>(v));
        constexpr int32_t kCap = static_cast<int32_t>(kKeyCap);
        const uint32_t p31 = bins ? static_cast<uint32_t>(kCap - min(d, kCap)) << 11 | static_cast<uint32_t>(h >> 53)
                                  : static_cast<uint32_t>(h >> 33);
        const uint32_t w = small_digest(bins, p31) << 1;
        st[v] = w;
        if (st2) st2[v] = w;
        if (v >= lo && v < hi && d > 0 && d <= kSmallRow) atomicAdd(&S.at[d], 1u);
    }
    __syncthreads();
    if (S.bad) return;  // (every thread: nothing sets it before the next barrier)
    if (threadIdx.x < 32) {
        // list positions of the degrees 1..kSmallRow
        unsigned c[kSmallRow / 32], sum = 0;
#pragma unroll
        for (int k = 0; k < kSmallRow / 32; ++k) {
            c[k] = S.at[1 + lane * (kSmallRow / 32) + k];
            sum += c[k];
        }
        unsigned incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        unsigned run = incl - sum;
#pragma unroll
        for (int k = 0; k < kSmallRow / 32; ++k) {
            S.at[1 + lane * (kSmallRow / 32) + k] = run;
            run += c[k];
        }
        if (lane == 31) S.count[1][0] = incl;
    }
    __syncthreads();
#pragma unroll 4
    for (int32_t v = lo + static_cast<int32_t>(threadIdx.x); v < hi; v += static_cast<int32_t>(blockDim.x)) {
        const int32_t d = __ldg(g.rp + v + 1) - __ldg(g.rp + v);
        if (d <= 0) continue;
        if (d <= kSmallRow)
            list[atomicAdd(&S.at[d], 1u)] = static_cast<uint16_t>(v);
        else
            list[static_cast<unsigned>(cap) - 1u - atomicAdd(&S.count[1][1], 1u)] = static_cast<uint16_t>(v);
    }
    __syncthreads();
}

// Entries [4 h, 4 h + 4) of the eight from p (the row is slots [lo, hi) from there; `left` entries of the
// array may be read from p).
__device__ __forceinline__ void small_load(const int32_t *p, bool vec, int64_t left, int32_t lo, int32_t hi,
                                           int32_t (&u)[8]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (vec && left >= 4 * h + 4 && hi > 4 * h) {
            const int4 x = __ldg(reinterpret_cast<const int4 *>(p + 4 * h));
            u[4 * h] = x.x;
            u[4 * h + 1] = x.y;
            u[4 * h + 2] = x.z;
            u[4 * h + 3] = x.w;
        } else {
#pragma unroll
            for (int q = 4 * h; q < 4 * h + 4; ++q) u[q] = q >= lo && q < hi ? __ldg(p + q) : 0;
        }
    }
}

// One vertex of a row up to kSmallRow entries (one thread): its next color, or -1 if it did not lose.
// Eight entries a step from the aligned group of four that holds the row's first (a batch's graphs start
// anywhere in colidx), the next step's loaded before this one's states are looked up.  W: words of the
// color window (colors of round `pass` are below `pass`; 128 when all of a four-word window are there,
// the most a row of 128 can need).  Slots outside the row and malformed entries read the state of entry
// `nobody`, which has no color of a window and no smaller digest; their number tells of malformed ones.
template <int W>
__device__ __forceinline__ int32_t small_row(const RoundParams &P, const SmallGraph &g, SmallShared &S,
                                             const uint32_t *cur, int32_t nobody, int32_t v, int32_t b, int32_t e) {
    const uint32_t own = cur[v], cvs = own & 0xfffe0000u, dig2 = own & 0x1fffeu;
    const bool vec = (reinterpret_cast<uintptr_t>(P.colidx) & 15u) == 0;
    const int64_t j0 = g.e0 + b;
    int32_t lo = static_cast<int32_t>(j0 & 3), hi = lo + (e - b);
    const int32_t *p = P.colidx + (j0 - lo);
    int64_t left = g.ci_len - (j0 - lo);
    uint32_t least = ~0u, m[W];
#pragma unroll
    for (int w = 0; w < W; ++w) m[w] = 0u;
    int none = -lo;  // slots that named no vertex, less those outside the row
    int32_t u[8], un[8];
    small_load(p, vec, left, lo, hi, u);
#pragma unroll
    for (int q = 0; q < 3; ++q)
        if (q < lo) u[q] = -1;
    for (;;) {
        if (hi < 8) {
#pragma unroll
            for (int q = 1; q < 8; ++q)
                if (q >= hi) u[q] = -1;
            none -= 8 - hi;
        }
        const bool more = hi > 8;
        if (more) small_load(p + 8, vec, left - 8, 0, hi - 8, un);
        uint32_t x[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const bool ok = static_cast<uint32_t>(u[q]) < static_cast<uint32_t>(g.n);
            if (!ok) ++none;
            x[q] = cur[ok ? u[q] : nobody];
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            least = min(least, x[q] - cvs);
#pragma unroll
            for (int k = 0; k < W; ++k) m[k] |= bit_or_none((x[q] >> 17) - 32u * k);
        }
        if (!more) break;
        p += 8;
        left -= 8;
        hi -= 8;
#pragma unroll
        for (int q = 0; q < 8; ++q) u[q] = un[q];
    }
    bool lose = least < dig2;
    if (least >> 1 == dig2 >> 1 || none != 0) lose = small_exact(P, g, S, cur, v);
    return lose ? first_free_words<W>(m) : -1;
}

// The same for a longer row (one warp): four entries per lane and step, the next step's loaded first;
// colors 0..63 in registers, the others up to 1,023 in the warp's shared window (shared atomics of 32
// lanes on a few words queue), further ones in more sweeps.
__device__ __forceinline__ int32_t small_long_row(const RoundParams &P, const SmallGraph &g, SmallShared &S,
                                                  const uint32_t *cur, int32_t nobody, int32_t v, unsigned *win,
                                                  int lane) {
    const uint32_t own = cur[v], cvs = own & 0xfffe0000u, dig2 = own & 0x1fffeu;
    const int32_t b = __ldg(g.rp + v), e = __ldg(g.rp + v + 1);
    const int32_t *ci = P.colidx + g.e0;
    for (int32_t base = 0;; base += 32 * kWinWords) {
        win[lane] = 0u;
        __syncwarp();
        uint32_t least = ~0u, m0 = 0, m1 = 0;
        int none = 0;  // malformed entries
        int32_t u[4], un[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int32_t j = b + 32 * q + lane;
            u[q] = j < e ? __ldg(ci + j) : -1;
            none -= j < e ? 0 : 1;
        }
        for (int32_t j0 = b;; j0 += 128) {
            const bool more = j0 + 128 < e;
            if (more) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int32_t j = j0 + 128 + 32 * q + lane;
                    un[q] = j < e ? __ldg(ci + j) : -1;
                    none -= j < e ? 0 : 1;
                }
            }
            uint32_t x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const bool ok = static_cast<uint32_t>(u[q]) < static_cast<uint32_t>(g.n);
                if (!ok) ++none;
                x[q] = cur[ok ? u[q] : nobody];
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                least = min(least, x[q] - cvs);
                const uint32_t c = (x[q] >> 17) - static_cast<uint32_t>(base);
                m0 |= bit_or_none(c);
                m1 |= bit_or_none(c - 32u);
                if (c >= 64u && c < 32u * kWinWords) atomicOr(&win[c >> 5], 1u << (c & 31u));
            }
            if (!more) break;
#pragma unroll
            for (int q = 0; q < 4; ++q) u[q] = un[q];
        }
        m0 = __reduce_or_sync(kFull, m0);
        m1 = __reduce_or_sync(kFull, m1);
        if (base == 0) {
            least = __reduce_min_sync(kFull, least);
            bool lose = least < dig2;
            if (least >> 1 == dig2 >> 1 || __any_sync(kFull, none != 0)) lose = small_exact_warp(P, g, S, cur, v, lane);
            if (!lose) return -1;
        }
        __syncwarp();
        const unsigned word = lane == 0 ? m0 : lane == 1 ? m1 : win[lane];
        const unsigned open = __ballot_sync(kFull, word != ~0u);
        if (open) {
            const int l = __ffs(static_cast<int>(open)) - 1;
            return base + 32 * l + __ffs(static_cast<int>(~__shfl_sync(kFull, word, l))) - 1;
        }
        __syncwarp();
    }
}

// Round `pass` over the block's worklist of its parity: next states into `nxt`, the losers into the
// other parity's list.
__device__ void small_round(const RoundParams &P, const SmallGraph &g, SmallShared &S, const uint32_t *cur,
                            uint32_t *nxt, const uint16_t *list, uint16_t *next, int32_t cap, int pass, unsigned *win) {
    const int par = pass & 1;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, nwarps = static_cast<int>(blockDim.x >> 5);
    const unsigned ns = S.count[par][0], nl = S.count[par][1];
    unsigned *cn = S.count[par ^ 1];
    // long rows first, a warp each
    for (unsigned i = static_cast<unsigned>(wib); i < nl; i += static_cast<unsigned>(nwarps)) {
        const int32_t v = list[static_cast<unsigned>(cap) - 1u - i];
        const int32_t nc = small_long_row(P, g, S, cur, cap, v, win, lane);
        if (lane == 0) {
            const uint32_t own = cur[v];
            nxt[v] = nc >= 0 ? static_cast<uint32_t>(nc) << 17 | (own & 0x1fffeu) : own;
            if (nc >= 0) next[static_cast<unsigned>(cap) - 1u - atomicAdd(cn + 1, 1u)] = static_cast<uint16_t>(v);
        }
        __syncwarp();
    }
    for (unsigned base = static_cast<unsigned>(wib) * 32u; base < ns; base += blockDim.x) {
        const unsigned i = base + static_cast<unsigned>(lane);
        int32_t v = 0, nc = -1;
        if (i < ns) {
            v = list[i];
            const int32_t b = __ldg(g.rp + v), e = __ldg(g.rp + v + 1);
            nc = pass <= 32   ? small_row<1>(P, g, S, cur, cap, v, b, e)
                 : pass <= 64 ? small_row<2>(P, g, S, cur, cap, v, b, e)
                              : small_row<4>(P, g, S, cur, cap, v, b, e);
            const uint32_t own = cur[v];
            nxt[v] = nc >= 0 ? static_cast<uint32_t>(nc) << 17 | (own & 0x1fffeu) : own;
        }
        const unsigned m = __ballot_sync(kFull, nc >= 0);
        if (m == 0u) continue;
        unsigned at = 0;
        if (lane == 0) at = atomicAdd(cn, static_cast<unsigned>(__popc(m)));
        at = __shfl_sync(kFull, at, 0) + __popc(m & lanemask_lt());
        if (nc >= 0) next[at] = static_cast<uint16_t>(v);
    }
}

// ------------------------------------------------------------------------------------------
// the small graphs of a batch

constexpr int kBatchThreads = 256;
constexpr int kBatchBlocks = 3;  // per SM: 4 (64 registers) spill and leave little L1 for the rows, 2 idle

// Dynamic shared memory: states [2][cap + 4], lists [2][cap], windows, a value key's table and counts.
constexpr size_t key_room(bool value_key) { return value_key ? (sizeof(DigestBin) + 4) * kDigestBins : 0; }
template <int THREADS>
constexpr size_t small_smem(int32_t cap, bool value_key) {
    return 12 * static_cast<size_t>(cap) + 32 + 4 * kWinWords * (THREADS / 32) + key_room(value_key);
}

__global__ void __launch_bounds__(kBatchThreads, kBatchBlocks) small_batch_kernel(const __grid_constant__ RoundParams P,
                                                                   const __grid_constant__ SmallBatch B) {
    extern __shared__ __align__(16) unsigned char s_small[];
    __shared__ SmallShared S;
    __shared__ unsigned s_q;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int32_t cap = kSmallBatchVertices;
    uint32_t *st[2] = {reinterpret_cast<uint32_t *>(s_small), reinterpret_cast<uint32_t *>(s_small) + cap + 4};
    uint16_t *list[2] = {reinterpret_cast<uint16_t *>(st[1] + cap + 4),
                         reinterpret_cast<uint16_t *>(st[1] + cap + 4) + cap};
    unsigned *win = reinterpret_cast<unsigned *>(list[1] + cap) + kWinWords * wib;
    DigestBin *bins = P.priority == GC_PRIORITY_HASH
                          ? nullptr
                          : reinterpret_cast<DigestBin *>(reinterpret_cast<unsigned *>(list[1] + cap) +
                                                          kWinWords * (kBatchThreads / 32));
    const unsigned count = __ldcg(B.queued);
    if (threadIdx.x < 2) st[threadIdx.x][cap] = kNobody32;
    for (;;) {
        __syncthreads();  // the previous graph is done with
        if (threadIdx.x == 0) {
            s_q = atomicAdd(B.taken, 1u);
            S.count[0][0] = S.count[0][1] = S.count[1][0] = S.count[1][1] = 0u;
            S.bad = 0;
        }
        __syncthreads();
        if (s_q >= count) return;
        SmallGraph g;
        g.g = __ldcg(B.queue + s_q);
        g.n = __ldg(P.g_n + g.g);
        g.vbase = static_cast<int32_t>(__ldg(P.g_vbase + g.g));
        g.e0 = __ldg(P.g_ebase + g.g);
        g.m = __ldg(P.g_m + g.g);
        g.rp = P.rowptr + __ldg(P.g_rbase + g.g);
        g.seed = P.g_seed ? __ldg(P.g_seed + g.g) : P.seed;
        g.ci_len = P.ci_len;
        small_setup(P, g, S, st[1], list[1], cap, 0, g.n, st[0], bins);
        if (threadIdx.x == 0) S.stop = S.bad;
        __syncthreads();
        int pass = 1;
        for (;; ++pass) {
            // round `pass` reads parity pass & 1
            const int par = pass & 1;
            const unsigned left = S.count[par][0] + S.count[par][1];
            if (left == 0u || S.stop) break;
            if (pass >= P.pass_end) {
                if (P.cap_is_error && threadIdx.x == 0) set_error(P.err, GC_ERR_NO_CONVERGENCE, pass, 0);
                break;
            }
            small_round(P, g, S, st[par], st[par ^ 1], list[par], list[par ^ 1], cap, pass, win);
            __syncthreads();
            if (threadIdx.x == 0) {
                S.count[par][0] = S.count[par][1] = 0u;
                S.stop = S.bad;
            }
            __syncthreads();
        }
        // FINAL in both buffers of the batch's state; the color count and, if no error was posted, the copy
        // to the caller's array read them
        const uint32_t *fin = st[pass & 1];
        for (int32_t v = static_cast<int32_t>(threadIdx.x); v < g.n; v += static_cast<int32_t>(blockDim.x)) {
            const int32_t c = static_cast<int32_t>(fin[v] >> 17);
            det_store(DetState{P.s16a, P.cx0}, g.vbase + v, c, 0u, true);
            det_store(DetState{P.s16b, P.cx1}, g.vbase + v, c, 0u, true);
        }
        if (threadIdx.x == 0) P.graph_last[g.g] = max(1, pass - 1);
    }
}

// Which graphs of a batch are small: at most kSmallBatchVertices vertices and kSmallBatchEntries
// entries, and no more than four times an SM's share of the batch's entries (a block takes about a
// nanosecond per entry and round; a batch with little else to do is better spread over the GPU).  When
// they hold less than half of the entries none is taken: the last of them then runs about as long as
// the regular rounds take for all of them (256 mixed graphs: 12.9 ms with the small ones apart, 11.7
// without).  One block: a counting sort by the entries' bit length, largest first, into the queue;
// g_done marks them for the regular kernels, and the vertices left for those are counted.
constexpr int kQueueThreads = 1024;
__global__ void __launch_bounds__(kQueueThreads) small_queue_kernel(RoundParams P, SmallBatch B, int64_t share) {
    __shared__ unsigned s_n[64], s_at[64];
    __shared__ unsigned long long s_left, s_small, s_all;
    if (P.err[0] != 0) {  // the tables are wrong: the call ends with that error, nothing is colored
        if (threadIdx.x == 0) {
            *B.queued = *B.taken = 0u;
            *B.left = 0ull;
        }
        return;
    }
    if (threadIdx.x < 64) s_n[threadIdx.x] = 0u;
    if (threadIdx.x == 0) s_left = s_small = s_all = 0ull;
    __syncthreads();
    auto bucket = [&](int32_t g) -> int {  // -1: not small
        const int32_t n = P.g_n[g];
        const int64_t m = P.g_m[g];
        if (n <= 0 || n > kSmallBatchVertices || m < 0 || m > kSmallBatchEntries || m > share) return -1;
        return 63 - __clzll(static_cast<long long>(m + 1));
    };
    unsigned long long left = 0, small = 0, all = 0;
    for (int32_t g = static_cast<int32_t>(threadIdx.x); g < P.G; g += kQueueThreads) {
        const unsigned long long m = static_cast<unsigned long long>(max(P.g_m[g], int64_t{0}));
        all += m;
        if (bucket(g) >= 0) small += m;
    }
    if (all) atomicAdd(&s_all, all);
    if (small) atomicAdd(&s_small, small);
    __syncthreads();
    const bool use = 2ull * s_small >= s_all;
    for (int32_t g = static_cast<int32_t>(threadIdx.x); g < P.G; g += kQueueThreads) {
        const int b = use ? bucket(g) : -1;
        B.g_done[g] = b >= 0 ? 1 : 0;
        if (b >= 0)
            atomicAdd(&s_n[b], 1u);
        else
            left += static_cast<unsigned long long>(P.g_n[g]);
    }
    if (left) atomicAdd(&s_left, left);
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned at = 0;
        for (int b = 63; b >= 0; --b) {
            s_at[b] = at;
            at += s_n[b];
        }
        *B.queued = at;
        *B.taken = 0u;
        *B.left = s_left;
    }
    __syncthreads();
    for (int32_t g = static_cast<int32_t>(threadIdx.x); g < P.G; g += kQueueThreads) {
        const int b = use ? bucket(g) : -1;
        if (b >= 0) B.queue[atomicAdd(&s_at[b], 1u)] = g;
    }
}

// ------------------------------------------------------------------------------------------
// a single graph

constexpr int kOneThreads = 1024;

__device__ __forceinline__ unsigned small_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned small_blocks() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// Cluster barrier: release the block's writes, acquire everyone else's.
__device__ __forceinline__ void small_cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The whole call for one graph: every exit is taken by all blocks of the cluster at once (they decide
// on the row offsets alone, which all of them check, and on the shared loser and error counts).
// Result: {status (0: done, 1: too large for this kernel, else an error in P.err), entries, rounds,
// colors}, then the error's words.
template <bool CLUSTER>
__global__ void __launch_bounds__(kOneThreads, 1) small_one_kernel(const __grid_constant__ RoundParams P,
                                                                   const __grid_constant__ SmallOne A) {
    extern __shared__ __align__(16) unsigned char s_small[];
    __shared__ SmallShared S;
    const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned rank = CLUSTER ? small_rank() : 0u, ncl = CLUSTER ? small_blocks() : 1u;
    const int32_t cap = A.cap;
    uint32_t *st[2] = {reinterpret_cast<uint32_t *>(s_small), reinterpret_cast<uint32_t *>(s_small) + cap + 4};
    uint16_t *list[2] = {reinterpret_cast<uint16_t *>(st[1] + cap + 4),
                         reinterpret_cast<uint16_t *>(st[1] + cap + 4) + cap};
    unsigned *win = reinterpret_cast<unsigned *>(list[1] + cap) + kWinWords * wib;
    DigestBin *bins = P.priority == GC_PRIORITY_HASH
                          ? nullptr
                          : reinterpret_cast<DigestBin *>(reinterpret_cast<unsigned *>(list[1] + cap) +
                                                          kWinWords * (kOneThreads / 32));
    SmallGraph g;
    g.g = 0;
    g.n = P.n;
    g.vbase = 0;
    g.e0 = 0;
    g.rp = P.rowptr;
    g.seed = P.seed;
    g.m = __ldg(P.rowptr + P.n);
    g.ci_len = g.m;
    if (threadIdx.x < 2) st[threadIdx.x][cap] = kNobody32;
    const bool lead = rank == 0 && threadIdx.x == 0;
    if (g.m < 0 || g.m > A.max_entries) {
        if (lead) {
            A.result[1] = static_cast<int32_t>(g.m);
            A.result[0] = 1;
        }
        return;
    }
    if (threadIdx.x == 0) {
        S.count[0][0] = S.count[0][1] = S.count[1][0] = S.count[1][1] = 0u;
        S.bad = 0;
        S.colors = 0u;
        S.top = -1;
    }
    if (lead) {
        for (int k = 0; k < 3; ++k) atomicExch(A.cnt + k, 0u);
        atomicExch(P.err, 0);
    }
    const int32_t lo = static_cast<int32_t>(static_cast<int64_t>(g.n) * rank / ncl);
    const int32_t hi = static_cast<int32_t>(static_cast<int64_t>(g.n) * (rank + 1) / ncl);
    if (CLUSTER)
        small_cluster_sync();
    else
        __syncthreads();
    small_setup(P, g, S, st[1], list[1], cap, lo, hi, CLUSTER ? nullptr : st[0], bins);
    if (threadIdx.x == 0) S.stop = S.bad;
    if (CLUSTER) {
        // the exchange buffers start with the block's own vertices' states; before the barrier, because
        // round 1 writes them from whichever thread has the vertex on its list
        for (int32_t v = lo + static_cast<int32_t>(threadIdx.x); v < hi; v += kOneThreads) {
            const uint32_t w = st[1][v];
            __stcg(A.exchange + v, w);
            __stcg(A.exchange + cap + v, w);
        }
    }
    __syncthreads();
    // this block's worklist; the cluster's size is known once the first round has run, and a round over
    // an empty list changes nothing
    unsigned left = 1u;
    int pass = 1;
    bool bad = false;
    for (;; ++pass) {
        const int par = pass & 1;
        if (!CLUSTER) left = S.count[par][0] + S.count[par][1];
        bad = !CLUSTER && S.stop != 0;
        if (left == 0u || bad) break;
        if (pass >= P.pass_end) {
            if (P.cap_is_error && lead) set_error(P.err, GC_ERR_NO_CONVERGENCE, pass, 0);
            bad = true;
            break;
        }
        // a cluster keeps C_pass in st[1] and writes C_{pass+1} to the exchange buffer of its parity
        uint32_t *cur = CLUSTER ? st[1] : st[par];
        uint32_t *nxt = CLUSTER ? A.exchange + static_cast<size_t>(par ^ 1) * cap : st[par ^ 1];
        small_round(P, g, S, cur, nxt, list[par], list[par ^ 1], cap, pass, win);
        __syncthreads();
        if (CLUSTER) {
            // the cluster's losers (a malformed entry counts as 2^24: it ends the rounds everywhere)
            if (threadIdx.x == 0) {
                const unsigned mine = S.count[par ^ 1][0] + S.count[par ^ 1][1] + (S.bad ? 1u << 24 : 0u);
                if (mine) atomicAdd(A.cnt + (pass + 1) % 3, mine);
                if (rank == 0) A.cnt[(pass + 2) % 3] = 0u;
                S.count[par][0] = S.count[par][1] = 0u;
            }
            small_cluster_sync();
            // the count and the new states in one round trip
            const uint4 *src = reinterpret_cast<const uint4 *>(nxt);
            constexpr int kLoads = kSmallOneVertices / 4 / kOneThreads;
            uint4 x[kLoads];
#pragma unroll
            for (int k = 0; k < kLoads; ++k) {
                const int32_t i = static_cast<int32_t>(threadIdx.x) + k * kOneThreads;
                if (i < (g.n + 3) >> 2) x[k] = __ldcg(src + i);
            }
            left = __ldcg(A.cnt + (pass + 1) % 3);
            bad = left >= 1u << 24;
            if (bad) break;
#pragma unroll
            for (int k = 0; k < kLoads; ++k) {
                const int32_t i = static_cast<int32_t>(threadIdx.x) + k * kOneThreads;
                if (i < (g.n + 3) >> 2) reinterpret_cast<uint4 *>(st[1])[i] = x[k];
            }
        } else if (threadIdx.x == 0) {
            S.count[par][0] = S.count[par][1] = 0u;
            S.stop = S.bad;
        }
        __syncthreads();
    }
    // colors, their number, the result
    const uint32_t *fin = CLUSTER ? st[1] : st[pass & 1];
    if (!bad) {
        for (int32_t v = lo + static_cast<int32_t>(threadIdx.x); v < hi; v += kOneThreads)
            A.out[v] = static_cast<int32_t>(fin[v] >> 17);
    }
    if (rank != 0) return;
    if (!bad) {
        unsigned *bits = reinterpret_cast<unsigned *>(list[0]);  // n bits
        for (int32_t i = static_cast<int32_t>(threadIdx.x); i < (g.n + 31) >> 5; i += kOneThreads) bits[i] = 0u;
        __syncthreads();
        int32_t top = -1;
        for (int32_t v = static_cast<int32_t>(threadIdx.x); v < g.n; v += kOneThreads) {
            const uint32_t c = fin[v] >> 17;
            if (!(bits[c >> 5] >> (c & 31u) & 1u)) atomicOr(&bits[c >> 5], 1u << (c & 31u));
            top = max(top, static_cast<int32_t>(c));
        }
        __syncthreads();
        unsigned k = 0;
        for (int32_t i = static_cast<int32_t>(threadIdx.x); i < (g.n + 31) >> 5; i += kOneThreads) k += __popc(bits[i]);
        k = __reduce_add_sync(kFull, k);
        top = __reduce_max_sync(kFull, top);
        if (lane == 0) {
            if (k) atomicAdd(&S.colors, k);
            atomicMax(&S.top, top);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        A.result[1] = static_cast<int32_t>(g.m);
        A.result[2] = pass - 1;
        A.result[3] = static_cast<int32_t>(S.colors);
        A.result[4] = S.top;
        for (int k = 0; k < 4; ++k) A.result[5 + k] = __ldcg(P.err + k);
        A.result[0] = bad ? -1 : 0;
    }
}

template <bool CLUSTER>
cudaError_t one_config(int32_t cap, bool value_key, int blocks, cudaLaunchConfig_t &cfg, cudaLaunchAttribute *at) {
    const void *fn = reinterpret_cast<const void *>(&small_one_kernel<CLUSTER>);
    const size_t smem = small_smem<kOneThreads>(cap, value_key);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e == cudaSuccess && blocks > 8) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3(static_cast<unsigned>(blocks));
    cfg.blockDim = dim3(kOneThreads);
    cfg.dynamicSmemBytes = smem;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = static_cast<unsigned>(blocks);
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = CLUSTER ? 1 : 0;
    return e;
}

}  // namespace

int small_one_blocks() {
    for (int blocks : {16, 8}) {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute at[1];
        int n = 0;
        if (one_config<true>(kSmallOneVertices, true, blocks, cfg, at) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&n, small_one_kernel<true>, &cfg) == cudaSuccess && n >= 1)
            return blocks;
        cudaGetLastError();
    }
    return 0;
}

cudaError_t launch_small_one(const RoundParams &P, const SmallOne &A, int blocks, cudaStream_t s) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    const bool value_key = P.priority != GC_PRIORITY_HASH;
    cudaError_t e = blocks > 1 ? one_config<true>(A.cap, value_key, blocks, cfg, at)
                               : one_config<false>(A.cap, value_key, 1, cfg, at);
    if (e != cudaSuccess) return e;
    cfg.stream = s;
    return blocks > 1 ? cudaLaunchKernelEx(&cfg, small_one_kernel<true>, P, A)
                      : cudaLaunchKernelEx(&cfg, small_one_kernel<false>, P, A);
}

cudaError_t launch_small_batch(const RoundParams &P, const SmallBatch &B, int64_t nnz, cudaStream_t s, int *grid) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    small_queue_kernel<<<1, kQueueThreads, 0, s>>>(P, B, std::max<int64_t>(int64_t{1} << 14, 4 * nnz / sms));
    const size_t smem = small_smem<kBatchThreads>(kSmallBatchVertices, P.priority != GC_PRIORITY_HASH);
    e = cudaFuncSetAttribute(small_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, small_batch_kernel, kBatchThreads, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    *grid = std::min(P.G, sms * per_sm);
    small_batch_kernel<<<*grid, kBatchThreads, smem, s>>>(P, B);
    return cudaGetLastError();
}

}  // namespace gc
