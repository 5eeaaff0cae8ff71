// Kernel 2 (Sec. 2.3): level-synchronous, direction-optimising BFS.
//
// One persistent cooperative kernel runs the whole search; levels are
// separated by a software grid barrier (bounded waits), which is the level
// synchronisation of Sec. 2.3.2 (all vertices of a level are handled together
// and the next level starts only once the whole level is done; the section
// also shows the wrong levels a search gets without it).  Per level the kernel runs one
// of two steps, chosen identically by every block from global counters:
//
//  top-down (Algorithm "Parallel BFS", Sec. 2.3.2): for every frontier vertex
//    and every neighbour in parallel, an unvisited neighbour is claimed with
//    an atomic OR on the visited bitmap; the winner records parent and level
//    and appends the vertex to the next queue with one atomic per warp.
//    Frontier vertices of degree <= big_degree are expanded 32 at a time by a
//    warp that gathers their adjacency lists as one contiguous stream of
//    edges; larger ones are cut into 128-edge chunks spread over all warps.
//  bottom-up (Beamer, Asanovic, Patterson, SC 2012): every unvisited vertex
//    scans its sorted adjacency list and stops at the first neighbour in the
//    frontier bitmap, which is therefore the smallest-id parent.  Outside
//    canonical mode it first tests its hub (a neighbour of largest degree,
//    built with the graph): a hub in the frontier is a valid parent, found
//    without reading the row, and a row of one entry whose hub is not in the
//    frontier is settled without reading it either.
//
// The switch follows Beamer: top-down -> bottom-up when the frontier's edges
// exceed (edges of unvisited vertices) / alpha, back when the frontier is
// shrinking and smaller than n / beta.  Both steps leave the next frontier as
// a queue and as a bitmap, so switching costs nothing.  In canonical mode the
// parents of vertices claimed top-down are recomputed at the next level as
// their smallest-id neighbour in the previous frontier, which makes the tree
// the unique one the oracle derives from the level array (Sec. 2.3.1).
//
// Memory layout of one search: visited bitmap and a ring of four frontier
// bitmaps (n/8 bytes each, L2-resident at SCALE 26: 8 MB), one int32 queue of
// n entries holding every level's frontier back to back (the BFS order), one
// state byte per vertex (level and parent source, mostly L2-resident: 64 MB at
// SCALE 26), a list of big frontier vertices with their chunk bases, and four
// level control records (ring).  The level and parent outputs are written once,
// by a last pass over all vertices.
#include "common.cuh"
#include "internal.h"

#include <algorithm>
#include <mutex>
#include <string>

namespace gb {
namespace {

constexpr int BFS_THREADS = 512;
constexpr int BIG_CHUNK = 128;      // edges per chunk of a big frontier vertex (one round)
constexpr int BU_LANE_FIRST = 8;    // bottom-up: each lane probes this many neighbours itself
constexpr int BU_WORDS = 2;         // bottom-up hub pass: visited words (or 32-entry list groups) per warp step
constexpr int PBUF = 256;           // per-warp ring of vertices left for the row pass
constexpr int QBUF = 512;           // per-warp buffer of discovered vertices (shared memory)
constexpr int BBUF = 32;            // per-warp buffer of discovered big-degree vertices
// Narrow top-down levels are run by one block (solo_levels): frontiers of at
// most SOLO_Q vertices with at most SOLO_E edges, or SOLO_E_SHORT edges if
// the rows are short (at most SOLO_ROW entries each, one vertex per thread).
// At 4,000 edges of long rows the one block took 20 us longer than the grid.
constexpr int SOLO_Q = 1024;
constexpr int SOLO_E = 1024;
constexpr int SOLO_E_SHORT = 4096;
// The other blocks wait for a whole stretch, which a quarter of the wait limit (ns)
// ends: below SOLO_SHORT_WAIT the clock is read after every level, not every 16th (16
// levels of 25 us, the longest in canonical mode, would leave nothing of such a limit), and
// below SOLO_MIN_WAIT, where one level is a quarter, every level takes the grid.
constexpr uint64_t SOLO_SHORT_WAIT = 1000000, SOLO_MIN_WAIT = 100000;
constexpr int SITE_BFS_BAR = 20;
constexpr int SITE_BFS_LEVELS = 21;

// With GB_CHECKED defined every global index below is tested first; a bad
// one is recorded in the status word (site, index) and the access skipped.
#ifdef GB_CHECKED
#define GB_OK_IDX(st, i, bound, site) \
    ((int64_t)(i) >= 0 && (int64_t)(i) < (int64_t)(bound) \
         ? true : (grid_error((st), GB_ERR_RANGE, (site), (long long)(i)), false))
#else
#define GB_OK_IDX(st, i, bound, site) true
#endif

struct LevelCtl {
    unsigned long long qcnt;  // vertices appended to the next queue
    unsigned long long mf;    // sum of their degrees
    unsigned long long big;   // (count << 32) | chunks of big vertices appended
    unsigned long long pad;
};

struct BigEnt {
    int32_t u;
    uint32_t cbase;
};

// What the block that ran a stretch of narrow levels tells the others.
struct SoloRec {
    long long l;        // level of the frontier it left (in ctl)
    long long qbase;    // start of that frontier in the queue
    long long prev_qn;  // size of the frontier before it
    double mu;          // edges of unvisited vertices, before that frontier's are taken off
};

struct WsHeader {
    GridBarrier bar;
    unsigned done;
    unsigned pad0;
    LevelCtl ctl[4];
    SoloRec solo;
    unsigned long long acc[6];  // edges, touched, reached, nlevels, td, bu
    unsigned long long t0;      // global timer at the end of the init phase
};

struct BfsArgs {
    const int64_t *off;
    const int32_t *col;
    const uint32_t *nz;  // degree >= 1 bitmap
    const int32_t *hub;  // per vertex a neighbour of largest degree (-1: none); null: unused
    int64_t n;
    int64_t nnz;
    int32_t root;
    int32_t *parent;
    int32_t *level;
    uint8_t *st8;  // per vertex: level + 1 (7 bits) and "parent is the hub" (bit 7)
    unsigned *vis;
    unsigned *fb;  // 4 bitmaps of nw words
    int64_t nw;
    int32_t *queue;
    int32_t *ulist;  // per warp a segment of useg entries: the vertices a bottom-up level left open (or null)
    int64_t useg;
    const int32_t *nzl;  // the vertices of degree >= 1, ascending (or null)
    const int2 *hd;         // (hub, min(degree, 65535)) per vertex (set whenever ulist is)
    int64_t nnzv;
    BigEnt *bigq;
    int64_t bigcap;
    WsHeader *hdr;
    DevStatus *st;
    BfsDevStats *stats;
    float alpha, alpha_hub, hub_deg;  // see go_bottom_up
    float beta;
    int big_deg;
    int canonical;
    int vec_out;  // parent, level, hub and the state bytes allow 16-byte vector access
    int vec_col;  // col is 16-byte aligned and padded to a multiple of 4 entries
    uint64_t timeout_ns;
    int solo_q, solo_clock;  // see set_wait
};

// The switch to bottom-up, for a frontier of qn vertices with mf edges, mu edges
// left unvisited.  alpha is the ratio at which it pays for a frontier of
// ordinary vertices.  One of hubs, with HUB_MEAN times the mean degree and more, is
// worth 1.4 times as much (a ratio of at most 64): an open vertex
// then meets the frontier at its first test, its highest-degree
// neighbour, while every edge of a hub costs top-down its atomic whether or not it
// finds a vertex.  SCALE 26, a frontier of 16,304 vertices and 150 M edges (just below 1/14): that
// level 1.68 ms top-down, 0.90 bottom-up, the search 2.32 -> 1.47 ms. Not further: SCALE 24,
// 2,406 vertices with about 1/21, 0.28 ms top-down, 0.38 bottom-up.  Mean us a search over 128
// roots with the factor 1 / 1.2 / 1.4 / 2 / 4: SCALE 20 104.9 / 104.9 / 104.9 / 105.5 / 106.3,
// SCALE 22 162.5 / 161.9 / 161.9 / 162.3 / 166.0, SCALE 24 367.9 / 367.5 / 367.3 / 368.9 / 382.0, SCALE
// 26 1177 / 1155 / 1156 / 1158 / 1201 (slowest root 2227 / 1791 / 1791 / 1895 / 2411).  In canonical
// mode and for a caller's arrays no hub is tested first, but a hub's edges cost top-down
// twice, for the claims and for the smallest parents: us a search over 64 roots with
// the rule / without it, canonical, SCALE 20 122.5 / 122.8, SCALE 22 235.1 / 235.6, SCALE 24
// 618 / 621 (slowest root 849 / 1015); bfs_noalloc, SCALE 20, 153.1 / 154.3.
constexpr float HUB_MEAN = 16.0f;
__device__ __forceinline__ bool go_bottom_up(float mf, float mu, float qn, const BfsArgs &a)
{
    return mf * a.alpha > mu || (mf * a.alpha_hub > mu && mf > qn * a.hub_deg);
}

// The wait limit, and what follows from it for narrow levels: the widest frontier that one
// block takes (none below SOLO_MIN_WAIT), and after which levels it reads the clock.
void set_wait(BfsArgs &a)
{
    a.timeout_ns = timeout_ns();
    a.solo_q = a.timeout_ns >= SOLO_MIN_WAIT ? SOLO_Q : -1;
    a.solo_clock = a.timeout_ns < SOLO_SHORT_WAIT ? 0 : 15;
}

void set_switch(BfsArgs &a, const gb_bfs_options &o)
{
    a.alpha = (float)o.alpha;
    a.alpha_hub = (float)std::max(o.alpha, std::min(1.4 * o.alpha, 64.0));
    a.hub_deg = HUB_MEAN * (float)((double)a.nnz / (double)std::max<int64_t>(a.nnzv > 0 ? a.nnzv : a.n, 1));
    a.beta = (float)o.beta;
}

// The big list is written by other blocks during the previous level: read it
// from L2, never from a possibly stale L1 line.
__device__ __forceinline__ BigEnt load_big(const BigEnt *q, int64_t i)
{
    const unsigned long long r = __ldcg(reinterpret_cast<const unsigned long long *>(q) + i);
    BigEnt b;
    b.u = (int32_t)(r & 0xffffffffull);
    b.cbase = (uint32_t)(r >> 32);
    return b;
}

// Chunks of a big vertex start at 16-byte boundaries of the column array
// (the row start rounded down to a multiple of 4 entries, then every
// BIG_CHUNK entries), so that every lane reads its four entries of a chunk
// with one aligned 16-byte load; a row of deg entries spans at most this
// many such chunks (one may come out empty).
__device__ __forceinline__ unsigned nchunks(int64_t deg)
{
    return (unsigned)((deg + 3 + BIG_CHUNK - 1) / BIG_CHUNK);
}

// The outputs are not written level by level: a search would then rewrite
// scattered parts of almost every 32-byte sector of the two n-entry output
// arrays at every large level, each a read-modify-write in DRAM.  A reached
// vertex records one byte instead (its level + 1, and whether its parent is
// its hub, which the bottom-up hub test then need not store), and the last
// pass writes level and parent of every vertex as whole lines.  A parent
// found any other way is written to the parent output at once (few: the
// top-down claims and the row-pass finds).  Levels from ST_ESC - 1 up are
// written to the level output directly and flagged ST_ESC.
constexpr unsigned ST_HUB = 0x80u;
constexpr unsigned ST_ESC = 0x7fu;

__device__ __forceinline__ void mark_reached(const BfsArgs &a, int64_t v, int lvl, bool via_hub)
{
    unsigned e = (unsigned)lvl + 1u;
    if (e >= ST_ESC) {
        e = ST_ESC;
        a.level[v] = lvl;
    }
    a.st8[v] = (uint8_t)(e | (via_hub ? ST_HUB : 0u));
}

// Discovered vertices are staged per warp in shared memory and moved to the
// global queue with one atomic per flush, so that the level counters see a
// few atomics per warp instead of one per 32 discoveries.  The fill levels
// are warp-uniform registers: every lane adds the same ballot counts, so no
// lane ever reads a count another lane is writing.
struct WarpBuf {
    int32_t q[QBUF];
    unsigned long long b[BBUF];  // v | nchunks << 32
    int32_t pu[PBUF];            // bottom-up: vertices waiting for a row pass
};

// Warp-collective: move the staged queue entries to the next level's queue.
__device__ __forceinline__ void flush_queue(WarpBuf &wb, int &qn, const BfsArgs &a,
                                            LevelCtl *nxt, int64_t qnext_base)
{
    if (qn == 0) return;
    __syncwarp();  // the lanes' buffer writes are visible to the whole warp
    const unsigned lane = lane_id();
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(&nxt->qcnt, (unsigned long long)qn);
    base = __shfl_sync(kFull, base, 0);
    for (int i = lane; i < qn; i += 32)
        if (GB_OK_IDX(a.st, qnext_base + (int64_t)base + i, a.n, 200))
            __stcg(&a.queue[qnext_base + (int64_t)base + i], wb.q[i]);
    __syncwarp();  // every lane has read the buffer before it is refilled
    qn = 0;
}

// Warp-collective: give the staged big vertices their chunk ranges and list them.
__device__ __forceinline__ void flush_big(WarpBuf &wb, int &bn, const BfsArgs &a, LevelCtl *nxt,
                                          int64_t bnext_base)
{
    if (bn == 0) return;
    __syncwarp();
    const unsigned lane = lane_id();
    const unsigned long long e = (int)lane < bn ? wb.b[lane] : 0ull;
    const unsigned nch = (unsigned)(e >> 32);
    const unsigned incl = warp_inclusive_scan(nch);
    const unsigned total = __shfl_sync(kFull, incl, 31);
    unsigned long long p = 0;
    if (lane == 0) p = atomicAdd(&nxt->big, ((unsigned long long)bn << 32) | total);
    p = __shfl_sync(kFull, p, 0);
    if ((int)lane < bn && GB_OK_IDX(a.st, bnext_base + (int64_t)(p >> 32) + lane, a.bigcap, 202)) {
        const unsigned long long cb = (p & 0xffffffffull) + incl - nch;
        __stcg(reinterpret_cast<unsigned long long *>(a.bigq) + bnext_base + (int64_t)(p >> 32) + lane,
               (e & 0xffffffffull) | (cb << 32));
    }
    __syncwarp();
    bn = 0;
}

// Block-collective, at the end of a level: what the warps still hold staged, with
// one atomic per block and list.  Each of 4864 warps (two blocks per SM) took one for
// itself, 1.6 ns apiece on the same address: 8 us a list and level.
struct LevelFlush {
    unsigned q[32];              // staged vertices of every warp, then where they go
    unsigned long long b[32];    // (big vertices << 32) | their chunks, likewise
};
__device__ __forceinline__ void flush_level(LevelFlush &lf, WarpBuf &wb, int &qn, int &bn, int nwarps, const BfsArgs &a,
                                            LevelCtl *nxt, int64_t qnext_base, int64_t bnext_base)
{
    const unsigned lane = lane_id();
    const int warp = threadIdx.x >> 5;
    __syncwarp();
    const unsigned long long e = (int)lane < bn ? wb.b[lane] : 0ull;
    const unsigned nch = (unsigned)(e >> 32);
    const unsigned incl = warp_inclusive_scan(nch);
    if (lane == 31) {
        lf.q[warp] = (unsigned)qn;
        lf.b[warp] = ((unsigned long long)bn << 32) | incl;
    }
    __syncthreads();
    if (warp == 0) {
        const unsigned q = (int)lane < nwarps ? lf.q[lane] : 0u;
        const unsigned long long b = (int)lane < nwarps ? lf.b[lane] : 0ull;
        const unsigned qi = warp_inclusive_scan(q);
        const unsigned long long bi = warp_inclusive_scan(b);
        unsigned long long q0 = 0, b0 = 0;
        if (lane == 31) {
            if (qi) q0 = atomicAdd(&nxt->qcnt, (unsigned long long)qi);
            if (bi) b0 = atomicAdd(&nxt->big, bi);
        }
        q0 = __shfl_sync(kFull, q0, 31);
        b0 = __shfl_sync(kFull, b0, 31);
        lf.q[lane] = (unsigned)q0 + qi - q;  // a level holds at most n < 2^31 vertices
        lf.b[lane] = b0 + bi - b;
    }
    __syncthreads();
    const int64_t q0 = qnext_base + (int64_t)lf.q[warp];
    const unsigned long long p = lf.b[warp];
    for (int i = lane; i < qn; i += 32)
        if (GB_OK_IDX(a.st, q0 + i, a.n, 200)) __stcg(&a.queue[q0 + i], wb.q[i]);
    if ((int)lane < bn && GB_OK_IDX(a.st, bnext_base + (int64_t)(p >> 32) + lane, a.bigcap, 202)) {
        const unsigned long long cb = (p & 0xffffffffull) + incl - nch;
        __stcg(reinterpret_cast<unsigned long long *>(a.bigq) + bnext_base + (int64_t)(p >> 32) + lane,
               (e & 0xffffffffull) | (cb << 32));
    }
    __syncwarp();
    qn = 0;
    bn = 0;
}

// Warp-collective: the lanes with `keep` stay open for the next level.  A
// bottom-up level lists the vertices it leaves open in the warp's own segment
// of the open list (no atomics: the warp owns the segment), and a bottom-up
// level that follows lets the same warp walk that segment instead of its
// words of the visited bitmap, compacting it in place (a vertex is written
// back only after it and every vertex before it were read).
__device__ __forceinline__ void append_open(bool keep, int32_t u, int32_t *seg, int &un)
{
    if (!seg) return;
    const unsigned bal = __ballot_sync(kFull, keep);
    if (keep) __stcg(&seg[un + __popc(bal & lanemask_lt())], u);
    un += __popc(bal);
}

// Warp-collective: set the visited and next-frontier bits of the lanes with
// `on`.  Lanes that hold vertices of the same bitmap word next to each other
// (the lists are in increasing vertex order) form a run; an OR scan within
// the runs gives the last lane of each run the run's bits, and that lane sets
// them with one atomic per bitmap.  Lanes of one word that are not adjacent
// only cost an extra atomic.
__device__ __forceinline__ void set_bits(bool on, int32_t u, unsigned *vis, unsigned *Fn)
{
    const int lane = (int)lane_id();
    const int w = on ? (int)((unsigned)u >> 5) : -1;
    unsigned bits = on ? 1u << (u & 31) : 0u;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned ob = __shfl_up_sync(kFull, bits, d);
        const int ow = __shfl_up_sync(kFull, w, d);
        if (lane >= d && ow == w) bits |= ob;
    }
    const int wnext = __shfl_down_sync(kFull, w, 1);
    if (on && (lane == 31 || wnext != w)) {
        atomicOr(&vis[w], bits);
        atomicOr(&Fn[w], bits);
    }
}

// Warp-collective: the lanes with `won` join the next frontier.
__device__ __forceinline__ void append_next(bool won, int32_t v, int64_t dv, const BfsArgs &a,
                                            WarpBuf &wb, int &qn, int &bn,
                                            unsigned long long &my_mf, LevelCtl *nxt,
                                            int64_t qnext_base, int64_t bnext_base)
{
    const unsigned bal = __ballot_sync(kFull, won);
    if (bal == 0) return;
    const int cnt = __popc(bal);
    if (qn + cnt > QBUF) flush_queue(wb, qn, a, nxt, qnext_base);
    if (won) {
        const int pos = qn + __popc(bal & lanemask_lt());
        if (GB_OK_IDX(a.st, pos, QBUF, 203)) wb.q[pos] = v;
        my_mf += (unsigned long long)dv;
    }
    qn += cnt;
    const bool big = won && dv > a.big_deg;
    const unsigned bb = __ballot_sync(kFull, big);
    if (bb) {
        const int bc = __popc(bb);
        if (bn + bc > BBUF) flush_big(wb, bn, a, nxt, bnext_base);
        if (big) {
            const int pos = bn + __popc(bb & lanemask_lt());
            if (GB_OK_IDX(a.st, pos, BBUF, 204))
                wb.b[pos] = (unsigned long long)(uint32_t)v | ((unsigned long long)nchunks(dv) << 32);
        }
        bn += bc;
    }
}

// Warp-collective top-down visit of TD_E edges per lane (src[t] -> v[t] where
// valid[t]): the visited-bit tests of the TD_E edges are issued together, then
// the claiming atomics together with the candidates' degree loads (a winner
// needs its degree for the next frontier's counters).
constexpr int TD_E = 4;
static_assert(BIG_CHUNK == 32 * TD_E, "a big-vertex chunk is one TD_E-entry group per lane");
__device__ __forceinline__ void td_visit(const bool (&valid)[TD_E], const int32_t (&src)[TD_E],
                                         const int32_t (&v)[TD_E], int l, const BfsArgs &a,
                                         unsigned *Fn, WarpBuf &wb, int &qn, int &bn,
                                         unsigned long long &my_mf, LevelCtl *nxt,
                                         int64_t qnext_base, int64_t bnext_base)
{
    bool cand[TD_E], won[TD_E];
#pragma unroll
    for (int t = 0; t < TD_E; ++t) {
        cand[t] = valid[t] && GB_OK_IDX(a.st, v[t], a.n, 205) &&
                  !((ldcg_u32(&a.vis[(unsigned)v[t] >> 5]) >> (v[t] & 31)) & 1u);
    }
    // the candidates' degrees are loaded with the claims, not after them
    int64_t dv[TD_E];
#pragma unroll
    for (int t = 0; t < TD_E; ++t) dv[t] = cand[t] ? __ldg(&a.off[v[t] + 1]) - __ldg(&a.off[v[t]]) : 0;
#pragma unroll
    for (int t = 0; t < TD_E; ++t) {
        won[t] = false;
        if (cand[t]) {
            const unsigned bit = 1u << (v[t] & 31);
            won[t] = !(atomicOr(&a.vis[(unsigned)v[t] >> 5], bit) & bit);
        }
    }
#pragma unroll
    for (int t = 0; t < TD_E; ++t) {
        if (won[t]) {
            a.parent[v[t]] = src[t];
            mark_reached(a, v[t], l + 1, false);
            atomicOr(&Fn[(unsigned)v[t] >> 5], 1u << (v[t] & 31));
        } else {
            dv[t] = 0;
        }
    }
#pragma unroll
    for (int t = 0; t < TD_E; ++t)
        append_next(won[t], v[t], dv[t], a, wb, qn, bn, my_mf, nxt, qnext_base, bnext_base);
}

// Warp-collective: the row tails [j, e) of the lanes with `open` are scanned
// together.  Each round deals 4 x 32 neighbour slots, an equal share to every
// row still open (consecutive slots of a row are consecutive CSR entries), so
// rows that find their parent leave and the loads of a round are all in
// flight at once.  The first slot of a row whose neighbour is in the frontier
// gives the smallest-id parent.
__device__ __forceinline__ void bu_stream_rows(const BfsArgs &a, const unsigned *F, bool open,
                                               int64_t j, int64_t e, int32_t &found,
                                               unsigned long long &my_edges)
{
    const int lane = (int)lane_id();
    while (true) {
        const bool act = open && found < 0 && j < e;
        const unsigned am = __ballot_sync(kFull, act);
        if (!am) break;
        const int q = 128 / __popc(am);
        const int64_t rem = act ? e - j : 0;
        const int len = (int)(rem < q ? rem : q);
        const int incl = warp_inclusive_scan(len);
        const int total = __shfl_sync(kFull, incl, 31);
        const int excl = incl - len;
        int32_t vv[4];
        unsigned fw[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int k = t * 32 + lane;
            int o = 0;
#pragma unroll
            for (int step = 16; step >= 1; step >>= 1) {
                const int c = o + step;
                if (__shfl_sync(kFull, excl, c) <= k) o = c;
            }
            const int64_t jo = __shfl_sync(kFull, j, o);
            const int eo = __shfl_sync(kFull, excl, o);
            const int64_t pos = jo + (k - eo);
            vv[t] = k < total && GB_OK_IDX(a.st, pos, a.nnz, 218) ? __ldg(&a.col[pos]) : -1;
        }
#pragma unroll
        for (int t = 0; t < 4; ++t)
            fw[t] = vv[t] >= 0 && GB_OK_IDX(a.st, vv[t], a.n, 219) ? ldcg_u32(&F[vv[t] >> 5]) : 0u;
        // each row owner looks for the first hit among its slots, group by group
        int32_t got = -1;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const bool h = vv[t] >= 0 && ((fw[t] >> (vv[t] & 31)) & 1u);
            const unsigned hm = __ballot_sync(kFull, h);
            const int a0 = excl - t * 32, a1 = excl + len - t * 32;
            const int lo = a0 > 0 ? a0 : 0, hi = a1 < 32 ? a1 : 32;
            unsigned seg = 0;
            if (len > 0 && hi > lo) seg = (hi >= 32 ? kFull : ((1u << hi) - 1u)) & ~((1u << lo) - 1u);
            const unsigned mine = hm & seg;
            const int fl = mine ? __ffs(mine) - 1 : 0;
            const int32_t cand = __shfl_sync(kFull, vv[t], fl);
            if (got < 0 && mine) {
                got = cand;
                my_edges += (unsigned long long)(32 * t + fl - excl + 1);
            }
        }
        if (got >= 0) {
            found = got;
        } else {
            my_edges += (unsigned long long)len;
            j += len;
        }
    }
}

// Warp-collective bottom-up row pass over `cnt` (<= 32) vertices of the warp's
// pending ring from position `head`, lane i taking entry head + i: the lane probes the first
// BU_LANE_FIRST neighbours of its row, rows still open are streamed by the
// warp; the first frontier neighbour in row order is the parent.  Entries come
// from several visited words, so the visited and next-frontier bits are set
// with atomics.
__device__ __forceinline__ void bu_row_pass(const BfsArgs &a, const unsigned *F, unsigned *Fn,
                                            int head, int cnt, int l, WarpBuf &wb, int &qn, int &bn,
                                            int32_t *seg, int &un, unsigned long long &my_mf,
                                            unsigned long long &my_edges, LevelCtl *nxt,
                                            int64_t qnext_base, int64_t bnext_base)
{
    const int lane = (int)lane_id();
    __syncwarp();  // the entries, and the commits of their words, are visible to the warp
    const bool act = lane < cnt;
    const int32_t u = act ? wb.pu[(head + lane) & (PBUF - 1)] : 0;
    __syncwarp();  // read before the ring is refilled
    // the offsets were read by this warp in the hub pass: L1 hits
    const int64_t s = act ? __ldg(&a.off[u]) : 0;
    const int32_t d = act ? (int32_t)(__ldg(&a.off[u + 1]) - s) : 0;
    const int32_t la = d < BU_LANE_FIRST ? d : BU_LANE_FIRST;
    int32_t vv[BU_LANE_FIRST];
    unsigned fw[BU_LANE_FIRST];
#pragma unroll
    for (int t = 0; t < BU_LANE_FIRST; ++t)
        vv[t] = t < la && GB_OK_IDX(a.st, s + t, a.nnz, 222) ? __ldg(&a.col[s + t]) : -1;
#pragma unroll
    for (int t = 0; t < BU_LANE_FIRST; ++t)
        fw[t] = vv[t] >= 0 && GB_OK_IDX(a.st, vv[t], a.n, 223) ? ldcg_u32(&F[vv[t] >> 5]) : 0u;
    int hit = -1;
#pragma unroll
    for (int t = 0; t < BU_LANE_FIRST; ++t)
        if (hit < 0 && vv[t] >= 0 && ((fw[t] >> (vv[t] & 31)) & 1u)) hit = t;
    int32_t found = -1;
#pragma unroll
    for (int t = 0; t < BU_LANE_FIRST; ++t)  // select without indexing registers
        if (hit == t) found = vv[t];
    my_edges += (unsigned long long)(hit >= 0 ? hit + 1 : la);
    bu_stream_rows(a, F, act && found < 0 && la < d, s + la, s + d, found, my_edges);
    const bool won = act && found >= 0 && GB_OK_IDX(a.st, u, a.n, 224);
    if (won) {
        a.parent[u] = found;
        mark_reached(a, u, l + 1, false);
        const unsigned bit = 1u << (u & 31);
        atomicOr(&a.vis[(unsigned)u >> 5], bit);
        atomicOr(&Fn[(unsigned)u >> 5], bit);
    }
    append_next(won, u, d, a, wb, qn, bn, my_mf, nxt, qnext_base, bnext_base);
    append_open(act && !won, u, seg, un);  // still no parent: open at the next level
}

// Canonical mode: the vertices claimed top-down at the previous level (queue
// entries [qbase, qbase + qn)) get as parent their smallest-id neighbour in
// that level's frontier Fp, the first one in row order.  32 vertices per warp,
// their rows streamed together, so that a long row (a hub claimed next to the
// root) is scanned by the whole warp rather than by one thread.  Kept out of
// line: the fast path does not carry its code.
__device__ __noinline__ void canonical_rescan(const BfsArgs &a, const unsigned *Fp, int64_t qbase,
                                              int64_t qn, int64_t gwarp, int64_t nwarps)
{
    const int lane = (int)lane_id();
    unsigned long long examined = 0;
    const int rn = rows_per_warp(qn, nwarps);
    for (int64_t i0 = gwarp * rn; i0 < qn; i0 += nwarps * rn) {
        const int64_t i = lane < rn ? i0 + lane : qn;
        int32_t u = 0;
        int64_t s = 0, e = 0;
        if (i < qn && GB_OK_IDX(a.st, qbase + i, a.n, 226)) {
            u = ldcg_i32(&a.queue[qbase + i]);
            if (GB_OK_IDX(a.st, u, a.n, 227)) {
                s = a.off[u];
                e = a.off[u + 1];
            }
        }
        int32_t found = -1;
        bu_stream_rows(a, Fp, i < qn && e > s, s, e, found, examined);
        if (i < qn && found >= 0) a.parent[u] = found;
    }
}

// The same by the other end of the edges: every edge of the previous level's frontier
// (queue entries [qb, qb + qn), big vertices bb.. in nc chunks) once more, each
// neighbour that the level claimed (a bit of F) keeping the least of the frontier
// vertices that reach it.  The choice is by edges: a few vertices next to
// the root claim the hubs, whose rows hold a thousand times as many entries
// (SCALE 26: 7 vertices claimed 159,420 with 1.3 G entries; scanned row by
// row, the longest by one warp, the search took 9.1 ms, by the frontier's edges 1.8), while
// a wide frontier's last claims have short rows.
__device__ __noinline__ void canonical_edges(const BfsArgs &a, const unsigned *F, int64_t qb, int64_t qn, int64_t bb,
                                             int64_t nb, int64_t nc, int64_t gwarp, int64_t nwarps)
{
    const int lane = (int)lane_id();
    const auto edge = [&](int64_t j, int32_t u) {
        if (!GB_OK_IDX(a.st, j, a.nnz, 228)) return;
        const int32_t v = __ldg(&a.col[j]);
        if (!GB_OK_IDX(a.st, v, a.n, 229)) return;
        if (((__ldcg(&F[(unsigned)v >> 5]) >> (v & 31)) & 1u) && ldcg_i32(&a.parent[v]) > u) atomicMin(&a.parent[v], u);
    };
    for (int64_t c = gwarp; c < nc; c += nwarps) {
        int64_t lo = 0, hi = nb;  // largest i with cbase(i) <= c
        while (hi - lo > 1) {
            const int64_t mid = (lo + hi) >> 1;
            if ((int64_t)load_big(a.bigq, bb + mid).cbase <= c) lo = mid;
            else hi = mid;
        }
        const BigEnt be = load_big(a.bigq, bb + lo);
        if (!GB_OK_IDX(a.st, be.u, a.n, 230)) continue;
        const int64_t su = a.off[be.u], eu = a.off[be.u + 1];
        const int64_t cs = (su & ~int64_t(3)) + (c - (int64_t)be.cbase) * BIG_CHUNK;
        const int64_t e = cs + BIG_CHUNK < eu ? cs + BIG_CHUNK : eu;
        for (int64_t j = cs + lane; j < e; j += 32)
            if (j >= su) edge(j, be.u);
    }
    const int rn = rows_per_warp(qn, nwarps);
    for (int64_t i0 = gwarp * rn; i0 < qn; i0 += nwarps * rn) {
        const int64_t i = lane < rn ? i0 + lane : qn;
        int32_t u = 0;
        int64_t s = 0, d = 0;
        if (i < qn && GB_OK_IDX(a.st, qb + i, a.n, 231)) {
            u = ldcg_i32(&a.queue[qb + i]);
            if (!GB_OK_IDX(a.st, u, a.n, 232)) u = 0;
            s = a.off[u];
            d = a.off[u + 1] - s;
            if (d > a.big_deg) d = 0;
        }
        const int64_t incl = warp_inclusive_scan(d);
        const int64_t total = __shfl_sync(kFull, incl, 31);
        const int64_t excl = incl - d;
        for (int64_t b = 0; b < total; b += 32) {
            const int64_t k = b + lane;
            int owner = 0;
#pragma unroll
            for (int step = 16; step >= 1; step >>= 1) {
                const int64_t ex = __shfl_sync(kFull, excl, owner + step);
                if (ex <= k) owner += step;
            }
            const int32_t su = __shfl_sync(kFull, u, owner);
            const int64_t so = __shfl_sync(kFull, s, owner), eo = __shfl_sync(kFull, excl, owner);
            if (k < total) edge(so + (k - eo), su);
        }
    }
}

// Shared memory of solo_levels (laid over the warp buffers, which are empty
// between levels): the frontier being expanded and the one being filled, each
// vertex with its row start and degree, the exclusive prefix of the degrees,
// and a ring of counters (one record being filled, one read, one cleared).
struct SoloBuf {
    int64_t start[2][SOLO_Q];
    int32_t v[2][SOLO_Q];
    int32_t deg[2][SOLO_Q];
    int32_t pre[SOLO_Q];
    struct {
        unsigned long long mf;
        int cnt, dmax, stop;
    } c[3];
    unsigned long long big;
    int wsum[32];
};
static_assert(sizeof(SoloBuf) <= sizeof(WarpBuf) * (BFS_THREADS / 32), "SoloBuf lies over the warp buffers");
static_assert(SOLO_Q == 2 * BFS_THREADS, "two frontier vertices per thread in the prefix sum");

// Block-collective part of a narrow level: TD_E edges per thread (src[t] ->
// v[t], v[t] < 0: none).  An edge's target is claimed on the visited bitmap
// while its offsets are loaded; the winners join the next frontier.  TEST: only
// targets that a plain load shows unvisited are claimed (a line of the L1 may be old,
// which costs an atomic, not a wrong answer): one more memory latency, but one
// SM's loads of scattered words are what a level of some hundred vertices waits for.
template <bool TEST>
__device__ __forceinline__ void solo_visit(const BfsArgs &a, SoloBuf &sb, int nx, int slot, int l, int64_t qnext,
                                           const int32_t (&src)[TD_E], const int32_t (&v)[TD_E],
                                           unsigned long long &mfs, int &dmax)
{
    unsigned old[TD_E];
    int64_t s0[TD_E];
    int32_t dg[TD_E];
#pragma unroll
    for (int t = 0; t < TD_E; ++t) old[t] = v[t] < 0 ? kFull : TEST ? a.vis[(unsigned)v[t] >> 5] : 0u;
    bool cand[TD_E];
#pragma unroll
    for (int t = 0; t < TD_E; ++t) {
        cand[t] = !((old[t] >> (v[t] & 31)) & 1u);
        if (cand[t]) old[t] = atomicOr(&a.vis[(unsigned)v[t] >> 5], 1u << (v[t] & 31));
    }
#pragma unroll
    for (int t = 0; t < TD_E; ++t) {
        s0[t] = cand[t] ? __ldg(&a.off[v[t]]) : 0;
        dg[t] = cand[t] ? (int32_t)(__ldg(&a.off[v[t] + 1]) - s0[t]) : 0;
    }
    int c = 0;
#pragma unroll
    for (int t = 0; t < TD_E; ++t) c += !((old[t] >> (v[t] & 31)) & 1u);
    const int ci = warp_inclusive_scan(c);
    int pos = 0;
    if (lane_id() == 31 && ci) pos = atomicAdd(&sb.c[slot].cnt, ci);
    pos = __shfl_sync(kFull, pos, 31) + ci - c;
#pragma unroll
    for (int t = 0; t < TD_E; ++t) {
        if ((old[t] >> (v[t] & 31)) & 1u) continue;
        a.parent[v[t]] = src[t];
        mark_reached(a, v[t], l + 1, false);
        if (GB_OK_IDX(a.st, qnext + pos, a.n, 243)) __stcg(&a.queue[qnext + pos], v[t]);
        if (pos < SOLO_Q) {
            sb.v[nx][pos] = v[t];
            sb.start[nx][pos] = s0[t];
            sb.deg[nx][pos] = dg[t];
        }
        mfs += (unsigned long long)dg[t];
        dmax = dg[t] > dmax ? dg[t] : dmax;
        ++pos;
    }
}

// The frontier vertex of edge k in the prefix of the degrees (the last one
// whose prefix is <= k).
__device__ __forceinline__ int solo_owner(const SoloBuf &sb, int k)
{
    int o = 0;
#pragma unroll
    for (int step = SOLO_Q / 2; step >= 1; step >>= 1)
        if (sb.pre[o + step] <= k) o += step;
    return o;
}

// Canonical mode, CSR entry j of frontier vertex u at level l: if its target
// was claimed by this level, u is one of its possible parents.
__device__ __forceinline__ void solo_min_parent(const BfsArgs &a, int64_t j, int32_t u, int l)
{
    const int32_t w = GB_OK_IDX(a.st, j, a.nnz, 244) ? __ldg(&a.col[j]) : -1;
    if (w < 0 || !GB_OK_IDX(a.st, w, a.n, 245)) return;
    const unsigned e = __ldcg(&a.st8[w]) & ST_ESC;
    const int lw = e == ST_ESC ? ldcg_i32(&a.level[w]) : (int)e - 1;
    if (lw == l + 1) atomicMin(&a.parent[w], u);
}

// A stretch of narrow top-down levels, run by block 0 alone while the others
// wait at the level barrier.  A level of a few hundred vertices is a chain of
// dependent L2 accesses, not work: with the grid barrier and the global queue
// and counters in that chain it took 7.5-10 us, whatever the frontier's size.
// Here the frontier stays in shared memory with its row starts and degrees (a
// discovered vertex's offsets are loaded beside the atomic that claims it), so
// a level is two round trips to L2 (column, claim) and one block barrier, three where
// the rows are short (their targets are tested before they are claimed).  A
// frontier of short rows is dealt four or eight lanes a row; any other one edge
// by edge, each thread finding its edges' vertices in the prefix of the
// degrees, so that a hub does not hold one warp.  A 997 x 601 mesh (1,233
// levels, frontiers of up to 1,000 vertices): 12.3 -> 5.4 ms, 10.0 -> 4.4 us a
// level; levels of three vertices 2.3 us.
//
// The frontier bitmaps are not kept during the stretch: nothing reads them
// between top-down levels.  Its last frontier's bits are set at the end, in
// the bitmap Fn that is clear now and becomes the next level's.  In canonical
// mode every frontier vertex offers itself as parent of the vertices the
// level claimed (a minimum), so no rescan follows.  The stretch ends when the
// frontier is empty or too wide for it, when the rule asks for bottom-up, or
// after a quarter of the wait limit, so that the waiting blocks stay within it.
// Whether it ends is part of the level's record in the ring, as its counts are: one
// flag for all levels could be set at the next level before a slow warp has read it for
// this one, and the warps would part at the block's barriers.
constexpr int SOLO_ROW = 2 * TD_E;
__device__ __forceinline__ void solo_levels(const BfsArgs &a, SoloBuf &sb, int l, int64_t qbase, int64_t qn,
                                            int64_t bnext_base, double mf, double mu, unsigned *Fn, LevelCtl *nxt)
{
    constexpr int NT = BFS_THREADS;
    const int tid = threadIdx.x;
    const int lane = (int)lane_id();
    const int warp = tid >> 5;
    WsHeader *h = a.hdr;
    const uint64_t t_start = globaltimer_ns();
    for (int i = tid; i < qn; i += NT) {
        int32_t u = ldcg_i32(&a.queue[qbase + i]);
        if (!GB_OK_IDX(a.st, u, a.n, 240)) u = 0;
        const int64_t s0 = a.off[u];
        sb.v[0][i] = u;
        sb.start[0][i] = s0;
        sb.deg[0][i] = (int32_t)(a.off[u + 1] - s0);
    }
    if (tid == 0) {
        sb.c[0].cnt = sb.c[0].dmax = sb.c[0].stop = 0;
        sb.c[0].mf = 0;
        sb.big = 0;
    }
    __syncthreads();
    unsigned long long edges = 0, touched = 0;
    int64_t prev_qn = 0;
    int x = 0;                            // levels of the stretch so far
    int slot = 0;                         // x mod 3: the counters being filled
    int dm = SOLO_ROW + 1;                // the frontier's largest degree (not known of the first)
    for (;;) {
        const int cur = x & 1;
        const int q = (int)qn;
        const int total = (int)mf;
        const int64_t qnext = qbase + qn;
        const int slot1 = slot == 2 ? 0 : slot + 1;
        if (tid == 0) {  // its last readers passed the previous level's barrier
            sb.c[slot1].cnt = sb.c[slot1].dmax = sb.c[slot1].stop = 0;
            sb.c[slot1].mf = 0;
        }
        unsigned long long mfs = 0;
        int dmx = 0;
        const bool by_edge = dm > SOLO_ROW;
        if (!by_edge) {
            // four or eight lanes a row, a lane an entry: a load of the columns touches 8
            // or 4 rows' lines, not 32
            const int gs = dm <= 4 ? 2 : 3;
            const int e = tid & ((1 << gs) - 1), rows = NT >> gs;
            for (int i0 = tid >> gs; i0 - (tid >> gs) < q; i0 += TD_E * rows) {
                int32_t src[TD_E], v[TD_E];
#pragma unroll
                for (int t = 0; t < TD_E; ++t) {
                    const int i = i0 + t * rows;
                    src[t] = i < q ? sb.v[cur][i] : 0;
                    const int d = i < q ? sb.deg[cur][i] : 0;
                    const int64_t j = (i < q ? sb.start[cur][i] : 0) + e;
                    v[t] = e < d && GB_OK_IDX(a.st, j, a.nnz, 241) ? __ldg(&a.col[j]) : -1;
                    if (v[t] >= 0 && !GB_OK_IDX(a.st, v[t], a.n, 242)) v[t] = -1;
                }
                solo_visit<true>(a, sb, cur ^ 1, slot, l, qnext, src, v, mfs, dmx);
            }
        } else {
            // exclusive prefix of the frontier's degrees, two vertices per thread
            // (of the first SOLO_Q / 2)
            const int d0 = 2 * tid < q ? sb.deg[cur][2 * tid] : 0;
            const int d1 = 2 * tid + 1 < q ? sb.deg[cur][2 * tid + 1] : 0;
            const int incl = warp_inclusive_scan(d0 + d1);
            if (lane == 31) sb.wsum[warp] = incl;
            __syncthreads();
            const int ws = lane < NT / 32 ? sb.wsum[lane] : 0;
            const int wi = warp_inclusive_scan(ws);
            const int ex = __shfl_sync(kFull, wi - ws, warp) + incl - d0 - d1;
            if (2 * tid < SOLO_Q) {
                sb.pre[2 * tid] = 2 * tid < q ? ex : 0x7fffffff;
                sb.pre[2 * tid + 1] = 2 * tid + 1 < q ? ex + d0 : 0x7fffffff;
            }
            __syncthreads();
            for (int k0 = 0; k0 < total; k0 += TD_E * NT) {
                int32_t src[TD_E], v[TD_E];
#pragma unroll
                for (int t = 0; t < TD_E; ++t) {
                    const int k = k0 + t * NT + tid;
                    const int o = solo_owner(sb, k);
                    src[t] = sb.v[cur][o];
                    const int64_t j = sb.start[cur][o] + (k - sb.pre[o]);
                    v[t] = k < total && GB_OK_IDX(a.st, j, a.nnz, 241) ? __ldg(&a.col[j]) : -1;
                    if (v[t] >= 0 && !GB_OK_IDX(a.st, v[t], a.n, 242)) v[t] = -1;
                }
                solo_visit<false>(a, sb, cur ^ 1, slot, l, qnext, src, v, mfs, dmx);
            }
        }
        if (__any_sync(kFull, mfs != 0)) {
            // 64-bit degree sum from two 32-bit reductions (each half's sum fits)
            const unsigned lo = __reduce_add_sync(kFull, (unsigned)(mfs & 0x3ffffffu));
            const unsigned hi = __reduce_add_sync(kFull, (unsigned)(mfs >> 26));
            dmx = __reduce_max_sync(kFull, dmx);
            if (lane == 0) {
                atomicAdd(&sb.c[slot].mf, ((unsigned long long)hi << 26) + lo);
                atomicMax(&sb.c[slot].dmax, dmx);
            }
        }
        if (tid == 0) {
            edges += (unsigned long long)total;
            touched += (unsigned long long)q;
            if (l < kStatLevels || (x & a.solo_clock) == a.solo_clock) {
                const uint64_t now = globaltimer_ns();
                if (now - t_start > a.timeout_ns / 4) sb.c[slot].stop = 1;
                if (l < kStatLevels) {
                    a.stats->level_ns[l] = now - h->t0;
                    a.stats->level_frontier[l] = qn;
                    a.stats->level_dir[l] = 1;
                    h->t0 = now;
                }
            }
        }
        __syncthreads();
        if (a.canonical) {
            // smallest-id parents: every edge of the level once more, to the
            // vertices the level claimed (parent writes above are complete)
            for (int k = tid; by_edge && k < total; k += NT) {
                const int o = solo_owner(sb, k);
                solo_min_parent(a, sb.start[cur][o] + (k - sb.pre[o]), sb.v[cur][o], l);
            }
            for (int i = tid; !by_edge && i < q; i += NT)
                for (int t = 0; t < sb.deg[cur][i]; ++t) solo_min_parent(a, sb.start[cur][i] + t, sb.v[cur][i], l);
            __syncthreads();
        }
        const int64_t cnt = sb.c[slot].cnt;
        const unsigned long long nmf = sb.c[slot].mf;
        dm = sb.c[slot].dmax;
        const bool stop = sb.c[slot].stop != 0;
        prev_qn = qn;
        qbase = qnext;
        qn = cnt;
        mf = (double)nmf;
        ++l;
        ++x;
        slot = slot1;
        if (qn == 0 || qn > SOLO_Q || nmf > (unsigned long long)(dm > SOLO_ROW ? SOLO_E : SOLO_E_SHORT) || stop ||
            l > a.n)
            break;
        if (qn > prev_qn && go_bottom_up((float)mf, (float)(mu - mf), (float)qn, a)) break;  // the bottom-up rule, applied by the grid
        mu -= mf;
    }
    // the frontier left: its bits, its big vertices, its counters (the first
    // SOLO_Q vertices are in shared memory)
    const int cur = x & 1;
    for (int64_t i0 = 0; i0 < qn; i0 += TD_E * NT) {
        int32_t u[TD_E];
        int64_t d[TD_E];
#pragma unroll
        for (int t = 0; t < TD_E; ++t) {
            const int64_t i = i0 + t * NT + tid;
            u[t] = i >= qn ? -1 : i < SOLO_Q ? sb.v[cur][i] : ldcg_i32(&a.queue[qbase + i]);
            if (u[t] >= 0 && !GB_OK_IDX(a.st, u[t], a.n, 246)) u[t] = -1;
            if (u[t] >= 0) atomicOr(&Fn[(unsigned)u[t] >> 5], 1u << (u[t] & 31));
        }
        if (dm <= a.big_deg) continue;
#pragma unroll
        for (int t = 0; t < TD_E; ++t) {
            const int64_t i = i0 + t * NT + tid;
            d[t] = u[t] < 0 ? 0 : i < SOLO_Q ? (int64_t)sb.deg[cur][i] : a.off[u[t] + 1] - a.off[u[t]];
        }
#pragma unroll
        for (int t = 0; t < TD_E; ++t) {
            const bool big = d[t] > a.big_deg;
            const unsigned bm = __ballot_sync(kFull, big);
            if (!bm) continue;
            const unsigned nch = big ? nchunks(d[t]) : 0u;
            const unsigned incl = warp_inclusive_scan(nch);
            unsigned long long b = 0;
            if (lane == 31) b = atomicAdd(&sb.big, ((unsigned long long)__popc(bm) << 32) | incl);
            b = __shfl_sync(kFull, b, 31);
            const int64_t at = bnext_base + (int64_t)(b >> 32) + __popc(bm & lanemask_lt());
            if (big && GB_OK_IDX(a.st, at, a.bigcap, 247))
                __stcg(reinterpret_cast<unsigned long long *>(a.bigq) + at,
                       (unsigned long long)(uint32_t)u[t] | (((b & 0xffffffffull) + incl - nch) << 32));
        }
    }
    __syncthreads();
    if (tid == 0) {
        nxt->qcnt = (unsigned long long)qn;
        nxt->mf = (unsigned long long)mf;
        nxt->big = sb.big;
        h->solo.l = l;
        h->solo.qbase = qbase;
        h->solo.prev_qn = prev_qn;
        h->solo.mu = mu;
        atomicAdd(&h->acc[0], edges);
        atomicAdd(&h->acc[1], touched);
        atomicAdd(&h->acc[4], (unsigned long long)x);
    }
    // the barrier that follows returns the buffers to the warps
}

// MINB: the blocks per SM that the register budget is sized for, 2 (64 registers) or 3
// (40 registers, spills, more warps to hide latency).
template <int MINB>
__global__ void __launch_bounds__(BFS_THREADS, MINB) bfs_kernel(BfsArgs a)
{
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t gthreads = (int64_t)gridDim.x * blockDim.x;
    const unsigned lane = lane_id();
    const int64_t gwarp = gtid >> 5;
    const int64_t nwarps = gthreads >> 5;
    const int64_t n = a.n, nw = a.nw;
    WsHeader *h = a.hdr;
    const int32_t root = a.root;
    grid_barrier_begin(&h->bar);
    __shared__ WarpBuf s_wb[BFS_THREADS / 32];
    __shared__ unsigned long long s_mf;
    __shared__ LevelFlush s_lf;
    WarpBuf &wb = s_wb[threadIdx.x >> 5];
    int qn_buf = 0, bn_buf = 0;  // warp-uniform fill levels of wb
    int un_open = 0;             // warp-uniform: vertices in this warp's open-list segment
    if (threadIdx.x == 0) s_mf = 0;
    unsigned long long my_mf = 0;

    // ---- init: bitmaps cleared, the root placed (the outputs are written
    // by the last pass; a vertex's state byte counts only once it is visited)
    for (int64_t w = gtid; w < nw; w += gthreads) {
        const unsigned rb = (w == (root >> 5)) ? 1u << (root & 31) : 0u;
        // isolated vertices (and ids >= n) start as visited: no search reaches
        // them and the bottom-up step need not test them; their outputs stay -1
        a.vis[w] = ~a.nz[w] | rb;
        a.fb[w] = rb;
        a.fb[nw + w] = 0;
        a.fb[2 * nw + w] = 0;
        a.fb[3 * nw + w] = 0;
    }
    if (gtid == 0) {
        const int64_t dr = a.off[root + 1] - a.off[root];
        a.parent[root] = root;
        mark_reached(a, root, 0, false);
        a.queue[0] = root;
        h->ctl[0].qcnt = 1;
        h->ctl[0].mf = (unsigned long long)dr;
        if (dr > a.big_deg) {
            h->ctl[0].big = (1ull << 32) | nchunks(dr);
            BigEnt be;
            be.u = root;
            be.cbase = 0;
            a.bigq[0] = be;
        }
    }
    if (!grid_sync(&h->bar, a.st, a.timeout_ns, SITE_BFS_BAR)) return;
    if (gtid == 0) {
        h->t0 = globaltimer_ns();
        a.stats->init_ns = 0;
    }

    int64_t qbase = 0, bbase = 0, prev_qn = 0;
    double mu = (double)a.nnz;
    bool td = true, prev_td = true;
    bool rescan = false;  // canonical mode: the frontier was claimed by a grid-wide top-down level
    double prev_mf = 0;   // that level's edges and big vertices
    int64_t prev_nb = 0, prev_nc = 0;
    unsigned long long my_edges = 0, my_touched = 0;
    int l = 0;
    // ring position of the level's bitmaps and control record: one step per
    // grid-wide level and per stretch of narrow levels
    for (int p = 0;; ++p, ++l) {
        LevelCtl *cur = &h->ctl[p & 3];
        const int64_t qn = (int64_t)ldcg_u64(&cur->qcnt);
        if (qn == 0) break;
        if (l > n) {
            if (gtid == 0) grid_error(a.st, GB_ERR_TIMEOUT, SITE_BFS_LEVELS, l);
            break;
        }
        const double mf = (double)ldcg_u64(&cur->mf);
        const unsigned long long bigp = ldcg_u64(&cur->big);
        const int64_t nb = (int64_t)(bigp >> 32);
        const int64_t nc = (int64_t)(bigp & 0xffffffffull);
        mu -= mf;
        if (l > 0) {
            if (td) {
                // bottom-up pays while the frontier grows: after its peak, few
                // vertices are unvisited and the ratio alone would send a
                // search of thin last levels over every vertex again
                if (go_bottom_up((float)mf, (float)mu, (float)qn, a) && qn > prev_qn) td = false;
            } else if (qn < prev_qn && (double)qn < (double)n / a.beta) {
                td = true;
            }
        }
        unsigned *F = a.fb + (size_t)(p & 3) * nw;
        unsigned *Fn = a.fb + (size_t)((p + 1) & 3) * nw;
        unsigned *Fz = a.fb + (size_t)((p + 2) & 3) * nw;
        unsigned *Fp = a.fb + (size_t)((p + 3) & 3) * nw;
        LevelCtl *nxt = &h->ctl[(p + 1) & 3];
        const int64_t qnext_base = qbase + qn;
        const int64_t bnext_base = bbase + nb;

        // Clear the bitmap and control record that the next step will fill.
        for (int64_t w = gtid; w < nw; w += gthreads) Fz[w] = 0;
        if (gtid == 0) {
            LevelCtl z = {0, 0, 0, 0};
            h->ctl[(p + 2) & 3] = z;
        }

        // Canonical parents of vertices claimed top-down at level l-1.
        if (rescan) {
            if (prev_mf < mf) canonical_edges(a, F, qbase - prev_qn, prev_qn, bbase - prev_nb, prev_nb, prev_nc, gwarp, nwarps);
            else canonical_rescan(a, Fp, qbase, qn, gwarp, nwarps);
        }

        // Narrow levels: block 0 runs them alone, the others wait.
        if (td && qn <= a.solo_q &&
            (mf <= (double)SOLO_E || (mf <= (double)SOLO_E_SHORT && mf <= 4.0 * (double)qn))) {
            if (blockIdx.x == 0)
                solo_levels(a, reinterpret_cast<SoloBuf &>(s_wb), l, qbase, qn, bnext_base, mf, mu, Fn, nxt);
            if (!grid_sync(&h->bar, a.st, a.timeout_ns, SITE_BFS_BAR)) return;
            l = (int)__ldcg(&h->solo.l) - 1;  // the loop adds one
            qbase = __ldcg(&h->solo.qbase);
            prev_qn = __ldcg(&h->solo.prev_qn);
            mu = __ldcg(&h->solo.mu);
            bbase += nb;
            prev_td = true;
            rescan = false;
            continue;
        }

        if (td) {
            // (a) chunks of big frontier vertices, a contiguous range per warp
            if (nc > 0) {
                const int64_t per = (nc + nwarps - 1) / nwarps;
                const int64_t c0 = gwarp * per;
                const int64_t c1 = c0 + per < nc ? c0 + per : nc;
                if (c0 < c1) {
                    int64_t lo = 0, hi = nb;  // largest i with cbase(i) <= c0
                    while (hi - lo > 1) {
                        const int64_t mid = (lo + hi) >> 1;
                        if ((int64_t)load_big(a.bigq, bbase + mid).cbase <= c0) lo = mid;
                        else hi = mid;
                    }
                    int64_t ow = lo;
                    BigEnt be = load_big(a.bigq, bbase + ow);
                    for (int64_t c = c0; c < c1; ++c) {
                        while (ow + 1 < nb && (int64_t)load_big(a.bigq, bbase + ow + 1).cbase <= c) {
                            ++ow;
                            be = load_big(a.bigq, bbase + ow);
                        }
                        if (!GB_OK_IDX(a.st, be.u, a.n, 206)) continue;
                        const int64_t su = a.off[be.u], eu = a.off[be.u + 1];
                        const int64_t cs = (su & ~int64_t(3)) + (c - (int64_t)be.cbase) * BIG_CHUNK;
                        const int64_t s = su > cs ? su : cs;
                        const int64_t e = cs + BIG_CHUNK < eu ? cs + BIG_CHUNK : eu;
                        if (s >= e) continue;  // the empty chunk a row may end with
                        if (lane == 0) my_edges += (unsigned long long)(e - s);
                        // lane i: entries cs + 4i .. cs + 4i + 3, one 16-byte load when
                        // the column array allows it (the library's own graphs)
                        const int64_t j0 = cs + 4 * (int64_t)lane;
                        bool valid[TD_E];
                        int32_t sv[TD_E], vv[TD_E];
                        if (a.vec_col) {
                            int4 x = make_int4(0, 0, 0, 0);
                            if (j0 < e && GB_OK_IDX(a.st, j0 + 3, col_alloc_entries(a.nnz), 207))
                                x = __ldg(reinterpret_cast<const int4 *>(a.col + j0));
                            vv[0] = x.x;
                            vv[1] = x.y;
                            vv[2] = x.z;
                            vv[3] = x.w;
#pragma unroll
                            for (int t = 0; t < TD_E; ++t) valid[t] = j0 + t >= s && j0 + t < e;
                        } else {
#pragma unroll
                            for (int t = 0; t < TD_E; ++t) {
                                valid[t] = j0 + t >= s && j0 + t < e && GB_OK_IDX(a.st, j0 + t, a.nnz, 207);
                                vv[t] = valid[t] ? __ldg(&a.col[j0 + t]) : 0;
                            }
                        }
#pragma unroll
                        for (int t = 0; t < TD_E; ++t) sv[t] = be.u;
                        td_visit(valid, sv, vv, l, a, Fn, wb, qn_buf, bn_buf, my_mf, nxt,
                                 qnext_base, bnext_base);
                    }
                }
            }
            // (b) the other frontier vertices, up to 32 per warp, edges gathered as one stream
            const int rn = rows_per_warp(qn, nwarps);
            for (int64_t i0 = gwarp * rn; i0 < qn; i0 += nwarps * rn) {
                const int64_t i = (int)lane < rn ? i0 + lane : qn;
                int32_t u = 0;
                int64_t s = 0, d = 0;
                if (i < qn && GB_OK_IDX(a.st, qbase + i, a.n, 208)) {
                    u = ldcg_i32(&a.queue[qbase + i]);
                    if (!GB_OK_IDX(a.st, u, a.n, 209)) u = 0;
                    s = a.off[u];
                    d = a.off[u + 1] - s;
                    if (d > a.big_deg) d = 0;
                }
                const int64_t incl = warp_inclusive_scan(d);
                const int64_t total = __shfl_sync(kFull, incl, 31);
                const int64_t excl = incl - d;
                my_edges += d;
                my_touched += (i < qn);
                for (int64_t b = 0; b < total; b += 32 * TD_E) {
                    bool valid[TD_E];
                    int32_t sv[TD_E], vv[TD_E];
#pragma unroll
                    for (int t = 0; t < TD_E; ++t) {
                        const int64_t k = b + t * 32 + lane;
                        int owner = 0;
#pragma unroll
                        for (int step = 16; step >= 1; step >>= 1) {
                            const int cand = owner + step;
                            const int64_t ex = __shfl_sync(kFull, excl, cand);
                            if (ex <= k) owner = cand;
                        }
                        sv[t] = __shfl_sync(kFull, u, owner);
                        const int64_t so = __shfl_sync(kFull, s, owner);
                        const int64_t eo = __shfl_sync(kFull, excl, owner);
                        valid[t] = k < total && GB_OK_IDX(a.st, so + (k - eo), a.nnz, 210);
                        vv[t] = valid[t] ? __ldg(&a.col[so + (k - eo)]) : 0;
                    }
                    td_visit(valid, sv, vv, l, a, Fn, wb, qn_buf, bn_buf, my_mf, nxt, qnext_base,
                             bnext_base);
                }
            }
        } else {
            // bottom-up.  Hub pass: every open vertex tests its hub (fast mode),
            // a neighbour of largest degree, against the frontier bitmap; a hit
            // is its parent.  The vertices left open queue up in the warp's
            // pending ring, and every 32 of them take a row pass (one vertex per
            // lane), so the row probes run with full warps.  Vertices the row
            // pass leaves open go to the open list.  A bottom-up level that
            // follows another walks that list, 128 vertices per warp step, with
            // no bitmap scan and no visited test (only the lane holding a vertex
            // can visit it now); otherwise the warp walks its words of the
            // visited bitmap, BU_WORDS words (lane i: vertex i of each) per step,
            // and bulk-prefetches the next step's hub entries and row offsets
            // into L2 (16-byte aligned arrays only: the library's own are; a
            // caller's offsets may not be).
            int ph = 0, pt = 0;  // warp-uniform head and tail of the pending ring
            int32_t *seg = a.ulist ? a.ulist + gwarp * a.useg : nullptr;
            const bool from_seg = seg && l > 0 && !prev_td;   // the open list of the previous level
            const bool from_nzl = seg && !from_seg && a.nzl;  // the graph's non-isolated vertices
            // a list walk: this warp's segment (its own entries, in steps of
            // 32 * BU_WORDS), or the non-isolated list (steps strided over the
            // grid, a visited test per entry: top-down levels visited some)
            const int32_t *L = from_seg ? seg : a.nzl;
            const int64_t lcnt = from_seg ? un_open : a.nnzv;
            const int64_t lstart = from_seg ? 0 : gwarp * 32 * BU_WORDS;
            const int64_t lstride = from_seg ? 32 * BU_WORDS : nwarps * 32 * BU_WORDS;
            un_open = 0;
            const bool bulk_pf = !from_seg && !from_nzl && ((reinterpret_cast<uintptr_t>(a.off) |
                                                             reinterpret_cast<uintptr_t>(a.hub)) & 15u) == 0;
            if (from_seg || from_nzl) {
            for (int64_t i0 = lstart; i0 < lcnt; i0 += lstride) {
                int32_t u[BU_WORDS], dg[BU_WORDS], hb[BU_WORDS];
                bool cand[BU_WORDS];
#pragma unroll
                for (int t = 0; t < BU_WORDS; ++t) {
                    const int64_t i = i0 + t * 32 + lane;
                    cand[t] = i < lcnt;
                    u[t] = cand[t] ? ldcg_i32(&L[i]) : 0;
                    cand[t] = cand[t] && GB_OK_IDX(a.st, u[t], a.n, 232);
                }
                unsigned vw[BU_WORDS];
#pragma unroll
                for (int t = 0; t < BU_WORDS; ++t) {
                    vw[t] = cand[t] && from_nzl ? ldcg_u32(&a.vis[(unsigned)u[t] >> 5]) : 0u;
                    // hub and degree in one 8-byte load, not two scattered offsets
                    const int2 x = cand[t] ? __ldg(&a.hd[u[t]]) : make_int2(-1, 0);
                    dg[t] = x.y;
                    hb[t] = a.hub ? x.x : -1;
                }
#pragma unroll
                for (int t = 0; t < BU_WORDS; ++t) {
                    if (dg[t] == 65535)  // saturated: the exact degree from the offsets
                        dg[t] = (int32_t)(__ldg(&a.off[u[t] + 1]) - __ldg(&a.off[u[t]]));
                    if ((vw[t] >> (u[t] & 31)) & 1u) {  // visited by a top-down level
                        cand[t] = false;
                        hb[t] = -1;
                    }
                }
                unsigned fh[BU_WORDS];
#pragma unroll
                for (int t = 0; t < BU_WORDS; ++t)
                    fh[t] = hb[t] >= 0 && GB_OK_IDX(a.st, hb[t], a.n, 233) ? ldcg_u32(&F[hb[t] >> 5]) : 0u;
#pragma unroll
                for (int t = 0; t < BU_WORDS; ++t) {
                    const bool won = hb[t] >= 0 && ((fh[t] >> (hb[t] & 31)) & 1u);
                    my_touched += (unsigned)cand[t];
                    my_edges += (unsigned long long)(hb[t] >= 0);
                    if (won) mark_reached(a, u[t], l + 1, true);
                    set_bits(won, u[t], a.vis, Fn);
                    append_next(won, u[t], dg[t], a, wb, qn_buf, bn_buf, my_mf, nxt, qnext_base, bnext_base);
                    // a row of one entry was settled by the hub test: still open
                    const bool whole = hb[t] >= 0 && dg[t] == 1;
                    append_open(cand[t] && !won && whole, u[t], seg, un_open);
                    const bool pend = cand[t] && !won && !whole;
                    const unsigned pm = __ballot_sync(kFull, pend);
                    if (pend) wb.pu[(pt + __popc(pm & lanemask_lt())) & (PBUF - 1)] = u[t];
                    pt += __popc(pm);
                }
                while (pt - ph >= 32) {
                    bu_row_pass(a, F, Fn, ph, 32, l, wb, qn_buf, bn_buf, seg, un_open, my_mf, my_edges,
                                nxt, qnext_base, bnext_base);
                    ph += 32;
                }
            }
            } else {
            // this warp's words of the visited bitmap, BU_WORDS per step
            for (int64_t w0 = gwarp * BU_WORDS; w0 < nw; w0 += nwarps * BU_WORDS) {
                const int64_t wn = w0 + nwarps * BU_WORDS;
                if (bulk_pf && lane == 0 && (wn + BU_WORDS) * 32 <= n) {
                    if (a.hub) prefetch_l2_bulk(a.hub + wn * 32, BU_WORDS * 32 * sizeof(int32_t));
                    prefetch_l2_bulk(a.off + wn * 32, BU_WORDS * 32 * sizeof(int64_t));
                }
                unsigned vw[BU_WORDS];
                bool any = false;
#pragma unroll
                for (int t = 0; t < BU_WORDS; ++t) {
                    vw[t] = w0 + t < nw ? ldcg_u32(&a.vis[w0 + t]) : kFull;
                    any |= vw[t] != kFull;
                }
                if (!any) continue;
                int32_t dg[BU_WORDS], hb[BU_WORDS];
#pragma unroll
                for (int t = 0; t < BU_WORDS; ++t) {
                    const int64_t u = (w0 + t) * 32 + lane;
                    const bool cand = !((vw[t] >> lane) & 1u) && GB_OK_IDX(a.st, u, a.n, 216);
                    dg[t] = 0;
                    hb[t] = -1;
                    if (cand) {
                        dg[t] = (int32_t)(__ldg(&a.off[u + 1]) - __ldg(&a.off[u]));
                        if (a.hub) hb[t] = __ldg(&a.hub[u]);
                    }
                }
                unsigned fh[BU_WORDS];
#pragma unroll
                for (int t = 0; t < BU_WORDS; ++t)
                    fh[t] = hb[t] >= 0 && GB_OK_IDX(a.st, hb[t], a.n, 220) ? ldcg_u32(&F[hb[t] >> 5]) : 0u;
#pragma unroll
                for (int t = 0; t < BU_WORDS; ++t) {
                    if (vw[t] == kFull) continue;  // a fully visited word (warp-uniform)
                    const int64_t w = w0 + t;
                    const int64_t u = w * 32 + lane;
                    const bool cand = !((vw[t] >> lane) & 1u) && u < n;
                    const int32_t found = hb[t] >= 0 && ((fh[t] >> (hb[t] & 31)) & 1u) ? hb[t] : -1;
                    my_touched += (unsigned)cand;
                    my_edges += (unsigned long long)(hb[t] >= 0);
                    const bool won = found >= 0;
                    if (won) mark_reached(a, u, l + 1, true);
                    // the warp owns word w: commit it with two plain stores
                    const unsigned nm = __ballot_sync(kFull, won);
                    if (nm && lane == 0) {
                        __stcg(&a.vis[w], vw[t] | nm);
                        __stcg(&Fn[w], nm);
                    }
                    append_next(won, (int32_t)u, dg[t], a, wb, qn_buf, bn_buf, my_mf, nxt, qnext_base, bnext_base);
                    // no row pass for an empty row, nor for a row of one entry (its hub)
                    const bool pend = cand && found < 0 && dg[t] > (hb[t] >= 0 ? 1 : 0);
                    const unsigned pm = __ballot_sync(kFull, pend);
                    if (pend) wb.pu[(pt + __popc(pm & lanemask_lt())) & (PBUF - 1)] = (int32_t)u;
                    pt += __popc(pm);
                }
                while (pt - ph >= 32) {
                    bu_row_pass(a, F, Fn, ph, 32, l, wb, qn_buf, bn_buf, seg, un_open, my_mf, my_edges,
                                nxt, qnext_base, bnext_base);
                    ph += 32;
                }
            }
            }
            if (pt > ph)
                bu_row_pass(a, F, Fn, ph, pt - ph, l, wb, qn_buf, bn_buf, seg, un_open, my_mf, my_edges,
                            nxt, qnext_base, bnext_base);
        }
        // end of level: flush the staged vertices and add the block's degree sum
        flush_level(s_lf, wb, qn_buf, bn_buf, BFS_THREADS / 32, a, nxt, qnext_base, bnext_base);
        {
            const unsigned long long t = warp_sum(my_mf);
            my_mf = 0;
            if (lane == 0 && t) atomicAdd(&s_mf, t);
            __syncthreads();
            if (threadIdx.x == 0) {
                if (s_mf) atomicAdd(&nxt->mf, s_mf);
                s_mf = 0;
            }
        }
        prev_td = td;
        rescan = td && a.canonical;
        prev_mf = mf;
        prev_nb = nb;
        prev_nc = nc;
        prev_qn = qn;
        qbase += qn;
        bbase += nb;
        if (gtid == 0) atomicAdd(&h->acc[td ? 4 : 5], 1ull);
        if (!grid_sync(&h->bar, a.st, a.timeout_ns, SITE_BFS_BAR)) return;
        if (gtid == 0 && l < kStatLevels) {
            const uint64_t now = globaltimer_ns();
            a.stats->level_ns[l] = now - h->t0;
            a.stats->level_frontier[l] = qn;
            a.stats->level_dir[l] = td ? 1 : 2;
            h->t0 = now;
        }
    }

    // ---- outputs: level and parent of every vertex, whole lines per warp.
    // Reached = visited and not isolated (isolated vertices start visited),
    // or the root; everyone else gets -1.  The state bytes, parents and
    // escaped levels were written by other blocks before the last barrier.
    // Each lane takes 4 consecutive vertices: one 4-byte load of their state
    // bytes, and the hub and parent entries loaded as 16-byte vectors at the
    // same time (not after the state bytes: one memory round trip per
    // group), so that a warp moves 128 vertices per step.
    if (a.vec_out) {
        for (int64_t g0 = gwarp * 128; g0 < n; g0 += nwarps * 128) {
            const int64_t v0 = g0 + 4 * (int64_t)lane;
            if (v0 + 3 < n) {
                const int64_t w = v0 >> 5;
                const unsigned sh = (unsigned)(v0 & 31);
                const unsigned rbits = ((ldcg_u32(&a.vis[w]) & __ldg(&a.nz[w])) >> sh) & 15u;
                const unsigned sw = __ldcg(reinterpret_cast<const unsigned *>(a.st8 + v0));
                const int4 hv = a.hub ? __ldg(reinterpret_cast<const int4 *>(a.hub + v0)) : make_int4(-1, -1, -1, -1);
                const int4 pv = __ldcg(reinterpret_cast<const int4 *>(a.parent + v0));
                int lv[4], pr[4];
                const int hh[4] = {hv.x, hv.y, hv.z, hv.w};
                const int pp[4] = {pv.x, pv.y, pv.z, pv.w};
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const unsigned b = (sw >> (8 * t)) & 255u;
                    const bool reached = ((rbits >> t) & 1u) || v0 + t == root;
                    lv[t] = -1;
                    pr[t] = -1;
                    if (reached) {
                        lv[t] = (b & ST_ESC) == ST_ESC ? ldcg_i32(&a.level[v0 + t]) : (int32_t)(b & ST_ESC) - 1;
                        pr[t] = (b & ST_HUB) ? hh[t] : pp[t];
                    }
                }
                *reinterpret_cast<int4 *>(a.level + v0) = make_int4(lv[0], lv[1], lv[2], lv[3]);
                *reinterpret_cast<int4 *>(a.parent + v0) = make_int4(pr[0], pr[1], pr[2], pr[3]);
            } else {
                for (int64_t v = v0; v < n && v < v0 + 4; ++v) {
                    const bool reached = ((ldcg_u32(&a.vis[v >> 5]) & __ldg(&a.nz[v >> 5])) >> (v & 31) & 1u) ||
                                         v == root;
                    int32_t lvv = -1, prv = -1;
                    if (reached) {
                        const unsigned b = __ldcg(&a.st8[v]);
                        lvv = (b & ST_ESC) == ST_ESC ? ldcg_i32(&a.level[v]) : (int32_t)(b & ST_ESC) - 1;
                        prv = (b & ST_HUB) ? __ldg(&a.hub[v]) : ldcg_i32(&a.parent[v]);
                    }
                    a.level[v] = lvv;
                    a.parent[v] = prv;
                }
            }
        }
    } else {
        for (int64_t v = gtid; v < n; v += gthreads) {
            const bool reached = ((ldcg_u32(&a.vis[v >> 5]) & __ldg(&a.nz[v >> 5])) >> (v & 31) & 1u) ||
                                 v == root;
            int32_t lvv = -1, prv = -1;
            if (reached) {
                const unsigned b = __ldcg(&a.st8[v]);
                lvv = (b & ST_ESC) == ST_ESC ? ldcg_i32(&a.level[v]) : (int32_t)(b & ST_ESC) - 1;
                prv = (b & ST_HUB) ? __ldg(&a.hub[v]) : ldcg_i32(&a.parent[v]);
            }
            a.level[v] = lvv;
            a.parent[v] = prv;
        }
    }

    // ---- statistics: block partial sums, the last block publishes them
    my_edges = warp_sum(my_edges);
    my_touched = warp_sum(my_touched);
    if (lane == 0) {
        if (my_edges) atomicAdd(&h->acc[0], my_edges);
        if (my_touched) atomicAdd(&h->acc[1], my_touched);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned prev = atomicAdd(&h->done, 1u);
        if (prev == gridDim.x - 1) {
            __threadfence();
            BfsDevStats &s = *a.stats;
            s.nlevels = (unsigned long long)l;
            s.edges_examined = ldcg_u64(&h->acc[0]);
            s.vertices_touched = ldcg_u64(&h->acc[1]);
            s.reached = (unsigned long long)qbase;
            s.td_levels = ldcg_u64(&h->acc[4]);
            s.bu_levels = ldcg_u64(&h->acc[5]);
        }
    }
}

}  // namespace

// The output pass uses 16-byte vector access when every array it touches
// allows it (a caller's outputs may start anywhere).
static int vec_ok(const BfsArgs &a)
{
    const uintptr_t m = reinterpret_cast<uintptr_t>(a.parent) | reinterpret_cast<uintptr_t>(a.level) |
                        reinterpret_cast<uintptr_t>(a.hub) | reinterpret_cast<uintptr_t>(a.st8);
    return (m & 15u) == 0 ? 1 : 0;
}

int bfs_pick_blocks(int num_sms, int minb)
{
    int per_sm = 0;
    const void *k = minb == 2 ? (const void *)bfs_kernel<2> : (const void *)bfs_kernel<3>;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, BFS_THREADS, 0) != cudaSuccess ||
        per_sm < 1)
        per_sm = 1;
    return num_sms * std::min(per_sm, minb);
}

namespace {
// How a search is launched: the kernel and its grid.
struct BfsLaunch {
    const void *kern;
    int blocks;
};

// `cap`: the most blocks the caller grants (0: the whole GPU).  The grid
// follows the graph: every level passes a barrier of all its blocks, which
// costs more than a small graph's work.  us per search of Kronecker graphs
// (edgefactor 16) on 1 / 16 / 64 / 152 / 304 blocks of 512 threads: SCALE 10
// 41 / 42 / 45 / 49 / 63; SCALE 14 92 / 59 / 61 / 67 / 82; SCALE 17 401 / 86 /
// 72 / 77 / 97; SCALE 20 - / 240 / 122 / 107 / 132; SCALE 21 - / 486 / 212 /
// 164 / 174; SCALE 22 - / 936 / 304 / 193 / 184.  From 2^22 vertices the work asks for two blocks' worth
// of warps per SM, whatever the edges: us for eight searches on 152 / 304 blocks of 512 / 152 of
// 1024 threads, SCALE 22 with 46 M entries 1634 / 1521 / 1570, with 122 M 1725 / 1566 / 1598, SCALE 23 with 94 M
// 2308 / 2068 / 2143; SCALE 21 with 60 M 1220 / 1254 / 1332, with 82 M 1039 / 1110 / -. (Blocks of
// 1024 threads halved the barriers' arrivals; they lose since a block
// takes one atomic per list at the end of a level.)
BfsLaunch pick_launch(int64_t n, int64_t nnz, const gb_bfs_options &o, int num_sms, int blocks2, int blocks3, int cap)
{
    constexpr int64_t kPerBlock = int64_t(1) << 15;  // CSR entries per block of a small graph
    constexpr int64_t kWideN = int64_t(1) << 22;
    const int one = std::max(1, std::min(blocks2, num_sms));
    if (o.blocks_per_sm == 3) {
        const int b = cap > 0 ? std::min(cap, blocks3) : blocks3;
        return {(const void *)bfs_kernel<3>, b};
    }
    int b = o.blocks_per_sm == 1 || n < kWideN ? one : blocks2;
    if (cap > 0) b = std::min(b, cap);
    b = (int)std::min<int64_t>(b, std::max<int64_t>(1, (nnz + kPerBlock - 1) / kPerBlock));
    return {(const void *)bfs_kernel<2>, b};
}
}  // namespace

namespace {
// Entries of the open list: every warp of the grid gets a segment for the
// vertices of its bitmap words (it owns BU_WORDS words of every
// nwarps * BU_WORDS), i.e. n rounded up per warp; room for grids of up to
// kOpenMaxWarps warps.
constexpr int64_t kOpenMaxWarps = 8192;
int64_t open_list_cap(int64_t n) { return ((n + 31) / 32) * 32 + kOpenMaxWarps * 32 * BU_WORDS; }

// Segment length per warp for a grid of nwarps warps, or 0 if the list cannot
// hold them (the search then walks the bitmap at every bottom-up level).
int64_t open_list_seg(int64_t n, int64_t nwarps)
{
    const int64_t nw = (n + 31) / 32;
    const int64_t steps = (nw + nwarps * BU_WORDS - 1) / (nwarps * BU_WORDS);
    const int64_t seg = steps * BU_WORDS * 32;
    return seg * nwarps <= open_list_cap(n) ? seg : 0;
}

struct WsLayout {
    size_t off_vis, off_fb, off_q, off_st, off_ul, off_big, total;
    int64_t bigcap;
};
// one buffer: header | visited | 4 frontier bitmaps | queue | state bytes |
// open list | big list
WsLayout ws_layout(const gb_graph *g, int big_deg)
{
    WsLayout L;
    const int64_t n = g->n, nw = (n + 31) / 32;
    L.bigcap = g->nnz / (big_deg + 1) + 2;
    L.off_vis = (sizeof(WsHeader) + 255) & ~size_t(255);
    L.off_fb = L.off_vis + ((nw * 4 + 255) & ~size_t(255));
    L.off_q = L.off_fb + ((4 * nw * 4 + 255) & ~size_t(255));
    L.off_st = L.off_q + ((n * 4 + 255) & ~size_t(255));
    L.off_ul = L.off_st + ((nw * 32 + 255) & ~size_t(255));
    L.off_big = L.off_ul + ((open_list_cap(n) * 4 + 255) & ~size_t(255));
    L.total = L.off_big + L.bigcap * sizeof(BigEnt);
    return L;
}
}  // namespace

size_t bfs_workspace_bytes(const gb_graph *g)
{
    return ws_layout(g, 1).total;  // big_degree 1 is the largest big list
}

gb_status bfs_impl(const gb_graph *g, int64_t root, int32_t *parent, int32_t *level,
                   BfsDevStats *stats, cudaStream_t s, int grid, unsigned char *given_ws)
{
    Context *ctx = context();
    if (!ctx) return GB_ERR_CUDA;
    const gb_bfs_options &o = options();
    const int64_t n = g->n;
    const int64_t nw = (n + 31) / 32;
    const int big_deg = std::max(o.big_degree, 1);
    const WsLayout Lw = ws_layout(g, big_deg);
    const int64_t bigcap = Lw.bigcap;
    const size_t off_vis = Lw.off_vis, off_fb = Lw.off_fb, off_q = Lw.off_q, off_big = Lw.off_big;
    unsigned char *ws = given_ws;
    Scratch tmp(s);
    if (!ws) GB_CUDA(tmp.alloc(&ws, Lw.total));
    GB_CUDA(cudaMemsetAsync(ws, 0, sizeof(WsHeader), s));
    BfsArgs a;
    a.off = g->off;
    a.col = g->col;
    a.nz = g->nz;
    // the hub test finds some parent, not the smallest-id one
    a.hub = o.canonical_parents ? nullptr : g->hub;
    a.n = n;
    a.nnz = g->nnz;
    a.root = (int32_t)root;
    a.parent = parent;
    a.level = level;
    a.hdr = reinterpret_cast<WsHeader *>(ws);
    a.vis = reinterpret_cast<unsigned *>(ws + off_vis);
    a.fb = reinterpret_cast<unsigned *>(ws + off_fb);
    a.nw = nw;
    a.queue = reinterpret_cast<int32_t *>(ws + off_q);
    a.st8 = ws + Lw.off_st;
    a.ulist = reinterpret_cast<int32_t *>(ws + Lw.off_ul);
    a.nzl = g->nzl;
    a.nnzv = g->nnzv;
    a.hd = g->hd;
    a.bigq = reinterpret_cast<BigEnt *>(ws + off_big);
    a.bigcap = bigcap;
    a.st = ctx->status;
    a.stats = stats;
    set_switch(a, o);
    a.big_deg = big_deg;
    a.canonical = o.canonical_parents;
    a.vec_out = vec_ok(a);
    a.vec_col = (reinterpret_cast<uintptr_t>(a.col) & 15u) == 0;  // allocated with col_alloc_entries
    set_wait(a);
    void *args[] = {&a};
    const BfsLaunch L = pick_launch(n, g->nnz, o, ctx->num_sms, ctx->bfs_blocks2, ctx->bfs_blocks, grid);
    a.useg = open_list_seg(n, (int64_t)L.blocks * (BFS_THREADS / 32));
    if (a.useg == 0 || !a.hd) a.ulist = nullptr;  // the list walks read hd
    GB_CUDA(cudaLaunchCooperativeKernel(L.kern, dim3(L.blocks), dim3(BFS_THREADS), args, 0, s));
    note_launch();
    return GB_OK;
}

}  // namespace gb

// ---------------------------------------------------------------------------
// bfs_noalloc: the single-source BFS kernel above, for callers that cannot
// allocate device memory.  Its scratch lives in one file-scope device array
// sized for graphs of up to 2^20 vertices; nothing here calls cudaMalloc,
// cudaMallocAsync or cudaFree.
// ---------------------------------------------------------------------------
namespace gb {
namespace {

constexpr int64_t kNaMaxN = int64_t(1) << 20;      // largest graph (vertices)
constexpr int64_t kNaWords = kNaMaxN / 32;
constexpr int64_t kNaBigCap = kNaMaxN + 2;         // a vertex enters the big list at most once
constexpr size_t kNaHdr = 0;
constexpr size_t kNaVis = 1024;
constexpr size_t kNaFb = kNaVis + kNaWords * 4;
constexpr size_t kNaNz = kNaFb + 4 * kNaWords * 4;
constexpr size_t kNaQueue = kNaNz + kNaWords * 4;
constexpr size_t kNaSt = kNaQueue + kNaMaxN * 4;
constexpr size_t kNaBig = kNaSt + kNaMaxN;
constexpr size_t kNaStatus = kNaBig + kNaBigCap * sizeof(BigEnt);
constexpr size_t kNaStats = kNaStatus + 256;
constexpr size_t kNaBytes = kNaStats + ((sizeof(BfsDevStats) + 255) & ~size_t(255));
static_assert(sizeof(WsHeader) <= kNaVis - kNaHdr, "header region too small");
static_assert(sizeof(DevStatus) <= 256, "status region too small");

// Shared by every call on a device; the last call's contents stay behind.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaBytes];

// Bit v of word v/32: row v is not empty (computed into the scratch).
__global__ void na_nz_kernel(const int64_t *__restrict__ off, int64_t n, uint32_t *__restrict__ nz,
                             int64_t nw)
{
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t stride = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const unsigned lane = threadIdx.x & 31u;
    for (int64_t w = gw; w < nw; w += stride) {
        const int64_t v = w * 32 + lane;
        const bool has = v < n && off[v + 1] > off[v];
        const unsigned b = __ballot_sync(kFull, has);
        if (lane == 0) nz[w] = b;
    }
}

struct NoAllocDevice {
    bool ready = false;
    unsigned char *scratch = nullptr;  // device address of g_noalloc_scratch
    int num_sms = 0;
    int blocks = 0;
};
std::mutex g_na_mu;
NoAllocDevice g_na[64];

}  // namespace

gb_status bfs_noalloc_impl(const int64_t *off, const int32_t *col, int64_t n, int64_t nnz,
                           int64_t root, int32_t *parent, int32_t *level, cudaStream_t s)
{
    if (!off || !parent || !level || (nnz > 0 && !col) || n < 1 || nnz < 0) {
        set_error("bfs_noalloc: need off, parent, level (and col when nnz > 0), n >= 1");
        return GB_ERR_INVALID;
    }
    if (n > kNaMaxN) {
        set_error("bfs_noalloc: the graph has more than 2^20 vertices, the size of the "
                  "built-in scratch; use bfs() instead");
        return GB_ERR_RANGE;
    }
    if (root < 0 || root >= n) {
        set_error("bfs_noalloc: root outside [0, n)");
        return GB_ERR_RANGE;
    }
    int dev = 0;
    GB_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) {
        set_error("bfs_noalloc: device index above 63");
        return GB_ERR_INVALID;
    }
    NoAllocDevice d;
    {
        // One-time set-up per device, with that device current: the device
        // address of the scratch array and the cooperative grid size.
        std::lock_guard<std::mutex> lk(g_na_mu);
        if (!g_na[dev].ready) {
            NoAllocDevice nd;
            GB_CUDA(cudaGetSymbolAddress((void **)&nd.scratch, g_noalloc_scratch));
            GB_CUDA(cudaDeviceGetAttribute(&nd.num_sms, cudaDevAttrMultiProcessorCount, dev));
            int per_sm = 0;
            GB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bfs_kernel<2>,
                                                                  BFS_THREADS, 0));
            nd.blocks = nd.num_sms * std::max(1, std::min(per_sm, 2));
            nd.ready = true;
            g_na[dev] = nd;
        }
        d = g_na[dev];
    }
    const gb_bfs_options &o = options();
    const int64_t nw = (n + 31) / 32;
    unsigned char *ws = d.scratch;
    // The header (barrier, level counters) and the status word must start at zero.
    GB_CUDA(cudaMemsetAsync(ws + kNaHdr, 0, sizeof(WsHeader), s));
    GB_CUDA(cudaMemsetAsync(ws + kNaStatus, 0, sizeof(DevStatus), s));
    na_nz_kernel<<<d.num_sms * 4, 256, 0, s>>>(off, n, reinterpret_cast<uint32_t *>(ws + kNaNz), nw);
    note_launch();
    GB_CUDA(cudaGetLastError());
    BfsArgs a;
    a.off = off;
    a.col = col;
    a.nz = reinterpret_cast<const uint32_t *>(ws + kNaNz);
    a.hub = nullptr;
    a.n = n;
    a.nnz = nnz;
    a.root = (int32_t)root;
    a.parent = parent;
    a.level = level;
    a.hdr = reinterpret_cast<WsHeader *>(ws + kNaHdr);
    a.vis = reinterpret_cast<unsigned *>(ws + kNaVis);
    a.fb = reinterpret_cast<unsigned *>(ws + kNaFb);
    a.nw = nw;
    a.queue = reinterpret_cast<int32_t *>(ws + kNaQueue);
    a.st8 = ws + kNaSt;
    a.ulist = nullptr;  // no open list: every bottom-up level walks the bitmap
    a.useg = 0;
    a.nzl = nullptr;
    a.nnzv = 0;
    a.hd = nullptr;
    a.bigq = reinterpret_cast<BigEnt *>(ws + kNaBig);
    a.bigcap = kNaBigCap;
    a.st = reinterpret_cast<DevStatus *>(ws + kNaStatus);
    a.stats = reinterpret_cast<BfsDevStats *>(ws + kNaStats);
    set_switch(a, o);
    a.big_deg = std::max(o.big_degree, 1);
    a.canonical = o.canonical_parents;
    a.vec_out = vec_ok(a);
    a.vec_col = 0;  // a caller's columns: neither alignment nor padding is known
    set_wait(a);
    void *args[] = {&a};
    // the scratch holds no open list, so any grid will do; one block per SM at most
    gb_bfs_options one = o;
    one.blocks_per_sm = 1;
    const BfsLaunch L = pick_launch(n, nnz, one, d.num_sms, d.blocks, d.blocks, 0);
    GB_CUDA(cudaLaunchCooperativeKernel(L.kern, dim3(L.blocks), dim3(BFS_THREADS), args, 0, s));
    note_launch();
    DevStatus hst;
    GB_CUDA(cudaMemcpyAsync(&hst, ws + kNaStatus, sizeof(hst), cudaMemcpyDeviceToHost, s));
    GB_CUDA(cudaStreamSynchronize(s));
    if (hst.code != 0) {
        set_error("bfs_noalloc: device status " + std::to_string(hst.code) + " at site " +
                  std::to_string(hst.where));
        return (gb_status)hst.code;
    }
    return GB_OK;
}

}  // namespace gb

extern "C" gb_status bfs_noalloc(const int64_t *off, const int32_t *col, int64_t n, int64_t nnz,
                                 int64_t root, int32_t *parent, int32_t *level, gb_stream s)
{
    try {
        return gb::bfs_noalloc_impl(off, col, n, nnz, root, parent, level,
                                    reinterpret_cast<cudaStream_t>(s));
    } catch (...) {
        gb::set_error("bfs_noalloc: internal error");
        return GB_ERR_INVALID;
    }
}
