// Kernel 1's sort by buckets (Sec. 2.2 builds the CSR from the edges in sorted
// order): most significant digits first, the last ones in shared memory.
//
//   0. one read of the tuples counts the symmetric keys (u << S | v), both
//      directions of every tuple but self-loops, by their top digit (at most 10
//      bits); a scan gives every bucket its place, and a second read of the
//      tuples writes the keys to their buckets;
//   1. from about 2 M keys up the buckets are split once more by the next digit.  What
//      is left of a key then fits 32 bits (64 with a weight), so from here on
//      an entry moves 4 bytes, not 8;
//   2. buckets longer than CAP keys (rows of high degree) are split by a further
//      digit, as many bits as their length asks for;
//   3. every bucket of at most CAP keys is sorted by one block in shared memory, by
//      counting (count_sort below).  Repeated entries are marked, the kept ones
//      counted per 4096 positions, and the first position of every row in the
//      bucket's key range recorded.  What is still too long then (columns crowded
//      in a part of their range) is split again, from the highest bit that its
//      keys differ in, until nothing is (split_rest): every such split parts
//      a bucket's keys, and one whose keys do not differ is a repeated pair, which
//      needs no sort;
//   4. a scan of those counts, then one pass that drops the marked entries and
//      one that turns the row positions into offsets.
//
// Why not the LSD sort of sort.cu: an LSD pass has to be stable, so every key
// is ranked among its warp's with a ballot per digit bit and every tile waits for
// the ones before it, and all key bits take part: 6 passes of 16 bytes a key at
// SCALE 26, each at a quarter of the copy bandwidth.  A bucket's order does
// not matter until its last sort, so a rank here is the return value of
// one shared-memory atomic, a tile's place one global atomic per digit, and
// three quarters of the key's bits never need a pass of their own.
//
// SCALE 26 (1.07 G tuples), whole kernel 1: 125.7 ms by the LSD sort, 54.5 ms by
// buckets; SCALE 22 with weights (least weight per pair and weight-ordered rows): 48 -> 7.3 ms.
// SCALE 20 with the vertices as the generator's quadrants number them, whose long rows
// crowd at low columns: 1.92 and 1.46 ms (renumbered at random: 1.88 and 1.11).
#include "bucket.h"

#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace gb {
namespace {

constexpr int BK_BITS = 10;  // largest digit
constexpr int BK_BINS = 1 << BK_BITS;
constexpr int BK_THREADS = 512;
constexpr int BK_ITEMS = 16;
constexpr int BK_TILE = BK_THREADS * BK_ITEMS;  // keys per tile: 8 per bin of the widest digit
constexpr int BK_MEAN = 2048;                   // keys a bucket holds on average after step 1
constexpr int BK_CAP = 4096;                    // longest bucket sorted in shared memory
constexpr int BK_SPLIT = 1024;                  // mean length aimed at by the extra splits
constexpr int BK_GROUP = 2048;                  // and how many keys' pieces are taken together
static_assert(2 * BK_GROUP <= BK_CAP, "a group ends within BK_GROUP keys after the next border");
constexpr int BK_ROWBITS = 9;                   // most rows of a bucket, as bits
constexpr int SC_THREADS = 256;  // of the scans of a split's pieces
constexpr int SC_WARPS = SC_THREADS / 32;
constexpr int LF_THREADS = 256;
constexpr int LF_WARPS = LF_THREADS / 32;
constexpr int WBITS = 25;  // bits of a weight in units of 2^-24
constexpr int POS_TILE = 4096;
constexpr int SITE_BK_POS = 16;

// A bucket: its place, its length, and which keys it holds.  Of its stored keys
// the lowest `pr >> 56` bits count, the bits above them are `prefix` (its lowest 56 bits;
// (row, weight, column) keys may have more, whose rows the sort does not ask for); of those
// key ranges of 2^rem keys it holds the `span` ones from `lo` on.
struct BkDesc {
    uint32_t start, count;
    uint64_t pr;  // prefix | bits << 56
    uint32_t lo;
    uint16_t span, rem;
};
constexpr uint64_t kPrefixMask = (uint64_t(1) << 56) - 1;
__device__ __forceinline__ uint64_t desc_pr(uint64_t prefix, int rem)
{
    return (prefix & kPrefixMask) | ((uint64_t)rem << 56);
}
__device__ __forceinline__ int desc_bits(uint64_t pr) { return (int)(pr >> 56); }
__device__ __forceinline__ uint64_t desc_prefix(uint64_t pr) { return pr & kPrefixMask; }
__device__ __forceinline__ BkDesc whole_desc(uint32_t start, uint32_t count, uint64_t prefix, int rem)
{
    BkDesc d;
    d.start = start;
    d.count = count;
    d.pr = desc_pr(prefix, rem);
    d.lo = 0;
    d.span = 1;
    d.rem = (uint16_t)rem;
    return d;
}

// A bucket to be split by `bits` bits at `shift`: its pieces are entries
// gbase.. of the level's counts and cursors.
struct BkSeg {
    uint32_t start, count, gbase;
    uint16_t bits, shift;
    uint64_t pr;
    unsigned long long differ;  // the bits that its keys differ in (split_rest)
};

struct BkCtl {
    unsigned nseg, ntile, npiece, ndesc, overflow, pad[3];  // overflow: pieces too long for a sort
};

__device__ __forceinline__ uint64_t low_mask(int bits)
{
    return bits >= 64 ? ~uint64_t(0) : (uint64_t(1) << bits) - 1;
}

// ---- step 0 ---------------------------------------------------------------

// A tuple's endpoints, and whether it takes part (in range, no self-loop).
__device__ __forceinline__ bool tuple_ok(int64_t u, int64_t v, int64_t n)
{
    return u >= 0 && u < n && v >= 0 && v < n && u != v;
}

__global__ void __launch_bounds__(BK_THREADS) bk_hist0_kernel(const int64_t *__restrict__ edges, int64_t m,
                                                              int scale, int p0, unsigned *__restrict__ cnt,
                                                              DevStatus *st)
{
    __shared__ unsigned s_h[BK_BINS];
    for (int i = threadIdx.x; i < BK_BINS; i += BK_THREADS) s_h[i] = 0;
    __syncthreads();
    const int64_t n = int64_t(1) << scale;
    const int sh = 2 * scale - p0;
    const int64_t stride = (int64_t)gridDim.x * BK_THREADS;
    constexpr int U = 8;  // loads in flight per thread
    for (int64_t e0 = (int64_t)blockIdx.x * BK_THREADS + threadIdx.x; e0 < m; e0 += U * stride) {
        int64_t u[U], v[U];
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const int64_t e = e0 + j * stride;
            u[j] = e < m ? __ldcs(edges + e) : 0;
            v[j] = e < m ? __ldcs(edges + m + e) : 0;
        }
#pragma unroll
        for (int j = 0; j < U; ++j) {
            if (u[j] < 0 || u[j] >= n || v[j] < 0 || v[j] >= n) {
                record_error(st, GB_ERR_RANGE, SITE_K1_RANGE, (long long)(e0 + j * stride));
            } else if (u[j] != v[j]) {
                atomicAdd(&s_h[(unsigned)((((uint64_t)u[j] << scale) | (uint64_t)v[j]) >> sh)], 1u);
                atomicAdd(&s_h[(unsigned)((((uint64_t)v[j] << scale) | (uint64_t)u[j]) >> sh)], 1u);
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < (1 << p0); i += BK_THREADS)
        if (s_h[i]) atomicAdd(&cnt[i], s_h[i]);
}

// Exclusive scan of up to BK_BINS bin counts by one block of SC_THREADS.
__device__ __forceinline__ void scan_bins(const unsigned *cnt, int nb, unsigned *excl4, unsigned *s_w)
{
    const int i0 = threadIdx.x * 4;
    unsigned c[4], t = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        c[j] = i0 + j < nb ? cnt[i0 + j] : 0u;
        t += c[j];
    }
    const unsigned incl = warp_inclusive_scan(t);
    if ((threadIdx.x & 31) == 31) s_w[threadIdx.x >> 5] = incl;
    __syncthreads();
    unsigned run = incl - t;
    for (int w = 0; w < (int)(threadIdx.x >> 5); ++w) run += s_w[w];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        excl4[j] = run;
        run += c[j];
    }
    __syncthreads();
}
static_assert(SC_THREADS * 4 == BK_BINS, "scan_bins: four bins a thread");

// The pieces of every listed bucket: places, cursors, descriptors.  One block a
// bucket.  grouped: neighbouring pieces are taken together, those that start in
// the same BK_GROUP keys, so that the next sort gets buckets of a useful length
// (a piece longer than BK_GROUP stays alone); a group's keys count from the split
// bucket's prefix, whose bits they still hold.
__global__ void __launch_bounds__(SC_THREADS) bk_scan_kernel(const BkSeg *__restrict__ segs, BkCtl *__restrict__ ctl,
                                                             int grouped, const unsigned *__restrict__ cnt,
                                                             unsigned *__restrict__ cursor,
                                                             BkDesc *__restrict__ desc)
{
    __shared__ unsigned s_w[SC_WARPS], s_ex[BK_BINS + 1], s_base;
    __shared__ uint16_t s_first[BK_BINS];
    const unsigned nseg = ctl->nseg;
    for (unsigned q = blockIdx.x; q < nseg; q += gridDim.x) {
        const BkSeg sg = segs[q];
        const int nb = 1 << sg.bits;
        unsigned ex[4];
        scan_bins(cnt + sg.gbase, nb, ex, s_w);
        const int rem = desc_bits(sg.pr) - sg.bits;
        const uint64_t pre = desc_prefix(sg.pr) << sg.bits;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int i = threadIdx.x * 4 + j;
            if (i >= nb) break;
            s_ex[i] = ex[j];
            cursor[sg.gbase + i] = sg.start + ex[j];
        }
        if (threadIdx.x == 0) s_ex[nb] = sg.count;
        __syncthreads();
        if (!grouped) {
            for (int i = threadIdx.x; i < nb; i += SC_THREADS)
                desc[sg.gbase + i] = whole_desc(sg.start + s_ex[i], s_ex[i + 1] - s_ex[i], pre | (uint64_t)i, rem);
        } else {
            unsigned first = 0, nf = 0;  // bit j: piece 4 t + j opens a group
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int i = threadIdx.x * 4 + j;
                if (i >= nb) break;
                const bool f = i == 0 || s_ex[i + 1] - s_ex[i] > (unsigned)BK_GROUP ||
                               s_ex[i] - s_ex[i - 1] > (unsigned)BK_GROUP ||
                               s_ex[i] / BK_GROUP != s_ex[i - 1] / BK_GROUP;
                first |= (unsigned)f << j;
                nf += f;
            }
            const unsigned incl = warp_inclusive_scan(nf);
            if ((threadIdx.x & 31) == 31) s_w[threadIdx.x >> 5] = incl;
            __syncthreads();
            unsigned g = incl - nf, total = 0;
            for (int w = 0; w < SC_WARPS; ++w) {
                if (w < (int)(threadIdx.x >> 5)) g += s_w[w];
                total += s_w[w];
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if ((first >> j) & 1u) s_first[g++] = (uint16_t)(threadIdx.x * 4 + j);
            if (threadIdx.x == 0) s_base = atomicAdd(&ctl->ndesc, total);
            __syncthreads();
            for (unsigned k = threadIdx.x; k < total; k += SC_THREADS) {
                const int i = s_first[k], e = k + 1 < total ? (int)s_first[k + 1] : nb;
                BkDesc d;
                if (e == i + 1) {
                    d = whole_desc(sg.start + s_ex[i], s_ex[e] - s_ex[i], pre | (uint64_t)i, rem);
                } else {
                    d.start = sg.start + s_ex[i];
                    d.count = s_ex[e] - s_ex[i];
                    d.pr = sg.pr;
                    d.lo = (uint32_t)i;
                    d.span = (uint16_t)(e - i);
                    d.rem = (uint16_t)rem;
                }
                desc[s_base + k] = d;
            }
        }
        __syncthreads();
    }
}

// Step 0's buckets: one segment over all keys, its total to *total.
__global__ void __launch_bounds__(SC_THREADS) bk_scan0_kernel(const unsigned *__restrict__ cnt, int p0, int rem,
                                                              unsigned *__restrict__ cursor,
                                                              BkDesc *__restrict__ desc, unsigned *__restrict__ total)
{
    __shared__ unsigned s_w[SC_WARPS];
    unsigned ex[4];
    const int nb = 1 << p0;
    scan_bins(cnt, nb, ex, s_w);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int i = threadIdx.x * 4 + j;
        if (i >= nb) break;
        desc[i] = whole_desc(ex[j], cnt[i], (uint64_t)i, rem);
        cursor[i] = ex[j];
        if (i == nb - 1) *total = ex[j] + cnt[i];
    }
}

// Shared memory of one partition tile: the keys in bin order, each bin's first
// place in the tile, and what to add to a place for its position in the output.
template <typename KOUT, bool BINS>
struct PartShared {
    static constexpr int keys_bytes = BK_TILE * (int)sizeof(KOUT);
    static constexpr int bytes = keys_bytes + 2 * BK_BINS * 4 + (BINS ? BK_TILE * 2 : 0);
};

// The tile's keys (bin[j] < 0: none) to their bins' next places in `out`.
// BINS: the digit is not part of the stored key, so it is kept beside it.
template <typename KOUT, bool BINS>
__device__ __forceinline__ void part_tile(const KOUT (&k)[BK_ITEMS], int (&bin)[BK_ITEMS], int nb, int shift,
                                          unsigned *__restrict__ cursor, KOUT *__restrict__ out, unsigned limit,
                                          unsigned char *smem, unsigned *s_w, DevStatus *st)
{
    KOUT *s_keys = reinterpret_cast<KOUT *>(smem);
    unsigned *s_excl = reinterpret_cast<unsigned *>(smem + PartShared<KOUT, BINS>::keys_bytes);
    unsigned *s_dst = s_excl + BK_BINS;
    uint16_t *s_bin = reinterpret_cast<uint16_t *>(s_dst + BK_BINS);
    const int tid = threadIdx.x;
    s_excl[2 * tid] = 0;
    s_excl[2 * tid + 1] = 0;
    __syncthreads();
    // a key's rank among its bin's keys of the tile, any order
#pragma unroll
    for (int j = 0; j < BK_ITEMS; ++j)
        if (bin[j] >= 0) bin[j] |= (int)(atomicAdd(&s_excl[bin[j]], 1u) << BK_BITS);
    __syncthreads();
    const unsigned c0 = s_excl[2 * tid], c1 = s_excl[2 * tid + 1];
    unsigned g0 = 0, g1 = 0;
    if (c0) g0 = atomicAdd(&cursor[2 * tid], c0);
    if (c1) g1 = atomicAdd(&cursor[2 * tid + 1], c1);
    const unsigned incl = warp_inclusive_scan(c0 + c1);
    if ((tid & 31) == 31) s_w[tid >> 5] = incl;
    __syncthreads();
    unsigned ex = incl - c0 - c1, total = 0;
#pragma unroll
    for (int w = 0; w < BK_THREADS / 32; ++w) {
        const unsigned c = s_w[w];
        if (w < (tid >> 5)) ex += c;
        total += c;
    }
    s_excl[2 * tid] = ex;
    s_excl[2 * tid + 1] = ex + c0;
    s_dst[2 * tid] = g0 - ex;
    s_dst[2 * tid + 1] = g1 - (ex + c0);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < BK_ITEMS; ++j) {
        if (bin[j] >= 0) {
            const int b = bin[j] & (BK_BINS - 1);
            const unsigned pos = s_excl[b] + ((unsigned)bin[j] >> BK_BITS);
            s_keys[pos] = k[j];
            if (BINS) s_bin[pos] = (uint16_t)b;
        }
    }
    __syncthreads();
    for (unsigned i = tid; i < total; i += BK_THREADS) {
        const KOUT x = s_keys[i];
        const int b = BINS ? (int)s_bin[i] : (int)(x >> shift) & (nb - 1);
        const unsigned o = s_dst[b] + i;
        if (o < limit) out[o] = x;
        else record_error(st, GB_ERR_RANGE, SITE_BK_POS, o);
    }
}

// Both directions of every tuple to the buckets of their top digit.  WEIGHTED:
// the weight's 25 bits below the key.  A stored key keeps the bits that its type
// holds: all of them where 2S bits fit, else those below the digit.
template <typename KOUT, bool WEIGHTED, bool BINS>
__global__ void __launch_bounds__(BK_THREADS, 2) bk_part0_kernel(const int64_t *__restrict__ edges,
                                                              const float *__restrict__ wrow, int64_t m, int scale,
                                                              int p0, unsigned *__restrict__ cursor,
                                                              KOUT *__restrict__ out, unsigned limit, DevStatus *st)
{
    extern __shared__ __align__(16) unsigned char bk_dyn[];
    __shared__ unsigned s_w[BK_THREADS / 32];
    const int64_t n = int64_t(1) << scale;
    const int sh = 2 * scale - p0;
    constexpr int TUP = BK_TILE / 2;
    const int64_t ntile = (m + TUP - 1) / TUP;
    for (int64_t t = blockIdx.x; t < ntile; t += gridDim.x) {
        KOUT k[BK_ITEMS];
        int bin[BK_ITEMS];
        int64_t u[BK_ITEMS / 2], v[BK_ITEMS / 2];
        float w[BK_ITEMS / 2];
#pragma unroll
        for (int j = 0; j < BK_ITEMS / 2; ++j) {
            const int64_t e = t * TUP + j * BK_THREADS + threadIdx.x;
            u[j] = e < m ? __ldcs(edges + e) : 0;
            v[j] = e < m ? __ldcs(edges + m + e) : 0;
            if (WEIGHTED) w[j] = e < m ? __ldcs(wrow + e) : 1.0f;
        }
#pragma unroll
        for (int j = 0; j < BK_ITEMS / 2; ++j) {
            const bool ok = tuple_ok(u[j], v[j], n);
            uint64_t a = ((uint64_t)u[j] << scale) | (uint64_t)v[j];
            uint64_t b = ((uint64_t)v[j] << scale) | (uint64_t)u[j];
            bin[2 * j] = ok ? (int)(a >> sh) : -1;
            bin[2 * j + 1] = ok ? (int)(b >> sh) : -1;
            if (WEIGHTED) {
                uint32_t wu = weight_units(w[j]);
                if (wu == 0u) {
                    record_error(st, GB_ERR_RANGE, SITE_SP_W, (long long)(t * TUP + j * BK_THREADS + threadIdx.x));
                    wu = 1u;
                }
                a = ((a & low_mask(sh)) << WBITS) | wu;
                b = ((b & low_mask(sh)) << WBITS) | wu;
            }
            k[2 * j] = (KOUT)a;
            k[2 * j + 1] = (KOUT)b;
        }
        part_tile<KOUT, BINS>(k, bin, 1 << p0, sh, cursor, out, limit, bk_dyn, s_w, st);
        __syncthreads();
    }
}

// ---- steps 1 and 2: splitting listed buckets ------------------------------

// Lists the buckets to split and the tiles that cover them.  forced > 0: all of
// them by that many bits, the pieces of bucket i at i << forced; else those
// longer than BK_CAP.  BY_LENGTH: down to single rows (`field` bits hold what is not the
// row) and from there by as many bits as bring a row of the bucket's length to
// BK_SPLIT keys: long buckets are long by one row as a rule, and bits of the row
// do not split it.  BY_DIFFERENCE: by bits that bk_digit_kernel chooses.  low: bits
// that do not tell entries apart.
constexpr int BY_LENGTH = 0, BY_DIFFERENCE = -1;
// Bits that bring `count` keys to BK_SPLIT a piece, if they spread evenly.
__device__ __forceinline__ int split_bits(unsigned count)
{
    const unsigned want = (count - 1) / BK_SPLIT + 1;  // rounded up; a sum could pass 2^32
    return 32 - __clz(want - 1);
}

__global__ void bk_list_kernel(const BkDesc *__restrict__ desc, const unsigned *__restrict__ ndesc_dev, unsigned ndesc,
                               int forced, int field, int low, BkSeg *__restrict__ segs, uint2 *__restrict__ tiles,
                               BkCtl *__restrict__ ctl)
{
    const unsigned nd = ndesc_dev ? *ndesc_dev : ndesc;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < nd; i += gridDim.x * blockDim.x) {
        const BkDesc d = desc[i];
        const int rem = desc_bits(d.pr);
        int bits = 0;
        unsigned gbase = 0, q;
        if (forced > 0) {
            bits = forced;
            gbase = i << forced;
            q = i;
            if (i == 0) ctl->nseg = nd;
        } else {
            if (d.count <= (unsigned)BK_CAP || rem <= low) continue;
            if (forced == BY_LENGTH) {
                bits = split_bits(d.count) + max(0, rem - field);
                bits = min(min(bits, BK_BITS), rem - low);
                gbase = atomicAdd(&ctl->npiece, 1u << bits);
            }
            q = atomicAdd(&ctl->nseg, 1u);
        }
        BkSeg sg;
        sg.start = d.start;
        sg.count = d.count;
        sg.gbase = gbase;
        sg.bits = (uint16_t)bits;
        sg.shift = (uint16_t)(rem - bits);
        sg.pr = d.pr;
        sg.differ = 0;
        segs[q] = sg;
        const unsigned nt = d.count ? (d.count - 1) / BK_TILE + 1 : 0u;
        const unsigned t0 = atomicAdd(&ctl->ntile, nt);
        for (unsigned t = 0; t < nt; ++t) tiles[t0 + t] = make_uint2(q, t);
    }
}

// The bits in which the keys of every listed bucket differ from its first.  A block a tile.
template <typename K>
__global__ void __launch_bounds__(BK_THREADS) bk_differ_kernel(const K *__restrict__ keys, BkSeg *__restrict__ segs,
                                                               const uint2 *__restrict__ tiles,
                                                               const BkCtl *__restrict__ ctl)
{
    const unsigned nt = ctl->ntile;
    for (unsigned t = blockIdx.x; t < nt; t += gridDim.x) {
        const uint2 tl = tiles[t];
        const uint32_t start = segs[tl.x].start, count = segs[tl.x].count;
        const K first = keys[start];
        const unsigned o0 = tl.y * BK_TILE, left = count - o0;
        uint64_t d = 0;
#pragma unroll
        for (int j = 0; j < BK_ITEMS; ++j) {
            const unsigned i = j * BK_THREADS + threadIdx.x;
            if (i < left) d |= (uint64_t)(keys[start + o0 + i] ^ first);
        }
        const unsigned lo = __reduce_or_sync(kFull, (unsigned)d), hi = __reduce_or_sync(kFull, (unsigned)(d >> 32));
        if ((threadIdx.x & 31) == 0 && (lo | hi)) atomicOr(&segs[tl.x].differ, ((unsigned long long)hi << 32) | lo);
    }
}

// The digit of every listed bucket: from the highest bit that its keys differ in, eight
// times as many pieces as its length asks for (a first split by length
// left it crowded), none if only the bits that do not count differ.  What its keys share above the
// digit goes into its prefix; rawoff (if given): the rows that begin in the part of its
// key range left out so are empty, and lie before or after all its keys.
template <typename K>
__global__ void bk_digit_kernel(const K *__restrict__ keys, BkSeg *__restrict__ segs, BkCtl *__restrict__ ctl, int low,
                                int scale, unsigned *__restrict__ rawoff)
{
    const unsigned nseg = ctl->nseg;
    for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < nseg; q += gridDim.x * blockDim.x) {
        BkSeg sg = segs[q];
        const int rem = desc_bits(sg.pr);
        const unsigned long long differ = sg.differ & low_mask(rem) & ~low_mask(low);
        const int top = differ ? 64 - __clzll((long long)differ) : low;
        const int bits = min(min(split_bits(sg.count) + 3, BK_BITS), top - low);
        const uint64_t old = desc_prefix(sg.pr);
        const uint64_t pre = (old << (rem - top)) | (((uint64_t)keys[sg.start] & low_mask(rem)) >> top);
        if (rawoff) {  // a key counts the pairs (u, v) from here on
            const uint64_t vmask = low_mask(scale);
            const uint64_t lo = old << (rem - low), hi = lo + (uint64_t(1) << (rem - low));
            const uint64_t nlo = pre << (top - low), nhi = nlo + (uint64_t(1) << (top - low));
            for (uint64_t r = (lo + vmask) >> scale; r < (hi + vmask) >> scale; ++r) {
                if (r << scale <= nlo) rawoff[r] = sg.start;
                else if (r << scale >= nhi) rawoff[r] = sg.start + sg.count;
            }
        }
        sg.pr = desc_pr(pre, top);
        sg.bits = (uint16_t)bits;
        sg.shift = (uint16_t)(top - bits);
        sg.gbase = atomicAdd(&ctl->npiece, 1u << bits);
        segs[q] = sg;
    }
}

// Digit counts of the listed buckets.  A block takes a run of the tile list and
// adds its counts to global memory when the bucket changes.
template <typename KIN>
__global__ void __launch_bounds__(BK_THREADS) bk_hist_kernel(const KIN *__restrict__ keys, const BkSeg *__restrict__ segs,
                                                             const uint2 *__restrict__ tiles,
                                                             const BkCtl *__restrict__ ctl, unsigned *__restrict__ cnt)
{
    __shared__ unsigned s_h[BK_BINS];
    const unsigned nt = ctl->ntile;
    const unsigned per = (nt + gridDim.x - 1) / gridDim.x;
    const unsigned t0 = blockIdx.x * per, t1 = min(nt, t0 + per);
    if (t0 >= t1) return;
    for (int i = threadIdx.x; i < BK_BINS; i += BK_THREADS) s_h[i] = 0;
    __syncthreads();
    unsigned cur = tiles[t0].x;
    BkSeg sg = segs[cur];
    for (unsigned t = t0; t < t1; ++t) {
        const uint2 tl = tiles[t];
        if (tl.x != cur) {
            __syncthreads();
            for (int i = threadIdx.x; i < (1 << sg.bits); i += BK_THREADS) {
                if (s_h[i]) atomicAdd(&cnt[sg.gbase + i], s_h[i]);
                s_h[i] = 0;
            }
            __syncthreads();
            cur = tl.x;
            sg = segs[cur];
        }
        const unsigned o0 = tl.y * BK_TILE;
        const unsigned left = sg.count - o0;
        const unsigned dm = (1u << sg.bits) - 1u;
        const KIN *src = keys + sg.start + o0;
        KIN k[BK_ITEMS];
#pragma unroll
        for (int j = 0; j < BK_ITEMS; ++j) {
            const unsigned i = j * BK_THREADS + threadIdx.x;
            k[j] = i < left ? src[i] : 0;
        }
#pragma unroll
        for (int j = 0; j < BK_ITEMS; ++j)
            if (j * BK_THREADS + threadIdx.x < left) atomicAdd(&s_h[(unsigned)(k[j] >> sg.shift) & dm], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < (1 << sg.bits); i += BK_THREADS)
        if (s_h[i]) atomicAdd(&cnt[sg.gbase + i], s_h[i]);
}

template <typename KIN, typename KOUT>
__global__ void __launch_bounds__(BK_THREADS, 2) bk_part_kernel(const KIN *__restrict__ keys, const BkSeg *__restrict__ segs,
                                                             const uint2 *__restrict__ tiles,
                                                             const BkCtl *__restrict__ ctl,
                                                             unsigned *__restrict__ cursor, KOUT *__restrict__ out,
                                                             unsigned limit, DevStatus *st)
{
    constexpr bool BINS = sizeof(KIN) != sizeof(KOUT);  // the digit lies above the stored bits
    extern __shared__ __align__(16) unsigned char bk_dyn[];
    __shared__ unsigned s_w[BK_THREADS / 32];
    const unsigned nt = ctl->ntile;
    for (unsigned t = blockIdx.x; t < nt; t += gridDim.x) {
        const uint2 tl = tiles[t];
        const BkSeg sg = segs[tl.x];
        const unsigned o0 = tl.y * BK_TILE;
        const unsigned left = sg.count - o0;
        const int dm = (1 << sg.bits) - 1;
        const KIN *src = keys + sg.start + o0;
        KOUT k[BK_ITEMS];
        int bin[BK_ITEMS];
#pragma unroll
        for (int j = 0; j < BK_ITEMS; ++j) {
            const unsigned i = j * BK_THREADS + threadIdx.x;
            const KIN x = i < left ? src[i] : 0;
            bin[j] = i < left ? (int)(x >> sg.shift) & dm : -1;
            k[j] = (KOUT)x;
        }
        part_tile<KOUT, BINS>(k, bin, 1 << sg.bits, sg.shift, cursor + sg.gbase, out, limit, bk_dyn, s_w, st);
        __syncthreads();
    }
}

// ---- step 3: sorting a bucket in shared memory ----------------------------

// Places are spread by one word in 33, so that lanes I keys apart do not share a bank.
__device__ __forceinline__ int lf_pad(int i) { return i + (i >> 5); }

template <typename K>
__device__ __forceinline__ void cmp_swap(K &a, K &b)
{
    const K lo = a < b ? a : b, hi = a < b ? b : a;
    a = lo;
    b = hi;
}

// By comparisons: sorts the bucket's n <= 256 * I keys into s (places through lf_pad).
template <typename K, int I>
__device__ __noinline__ void merge_sort(const K *src, int n, K kmask, K base_key, K *s)
{
    const int tid = threadIdx.x, lane = tid & 31, base = (tid >> 5) * 32 * I;
    if (base < n) {
        K x[I];
#pragma unroll
        for (int j = 0; j < I; ++j) {
            const int i = base + j * 32 + lane;
            x[j] = i < n ? (src[i] & kmask) - base_key : (K)~(K)0;
        }
        // bitonic network over places lane * I + j, every comparison ascending:
        // a merge of two runs starts by comparing mirrored places
#pragma unroll
        for (int k = 2; k <= I; k <<= 1) {
#pragma unroll
            for (int j = 0; j < I; ++j)
                if ((j ^ (k - 1)) > j) cmp_swap(x[j], x[j ^ (k - 1)]);
#pragma unroll
            for (int d = k >> 2; d > 0; d >>= 1)
#pragma unroll
                for (int j = 0; j < I; ++j)
                    if ((j ^ d) > j) cmp_swap(x[j], x[j ^ d]);
        }
#pragma unroll
        for (int ml = 2; ml <= 32; ml <<= 1) {
            const bool low = !(lane & (ml >> 1));
#pragma unroll
            for (int j = 0; j < I / 2; ++j) {
                const K y0 = __shfl_xor_sync(kFull, x[I - 1 - j], ml - 1);
                const K y1 = __shfl_xor_sync(kFull, x[j], ml - 1);
                x[j] = low ? min(x[j], y0) : max(x[j], y0);
                x[I - 1 - j] = low ? min(x[I - 1 - j], y1) : max(x[I - 1 - j], y1);
            }
#pragma unroll
            for (int d = ml >> 2; d > 0; d >>= 1) {
                const bool lo2 = !(lane & d);
#pragma unroll
                for (int j = 0; j < I; ++j) {
                    const K y = __shfl_xor_sync(kFull, x[j], d);
                    x[j] = lo2 ? min(x[j], y) : max(x[j], y);
                }
            }
#pragma unroll
            for (int d = I >> 1; d > 0; d >>= 1)
#pragma unroll
                for (int j = 0; j < I; ++j)
                    if ((j ^ d) > j) cmp_swap(x[j], x[j ^ d]);
        }
#pragma unroll
        for (int j = 0; j < I; ++j) s[lf_pad(base + lane * I + j)] = x[j];
    }
    __syncthreads();
    // runs of L merged in pairs: a thread finds where its I outputs begin in
    // the two runs by bisection (merge path) and merges them one by one
    for (int L = 32 * I; L < n; L <<= 1) {
        const int t0 = tid * I;
        K o[I];
        if (t0 < n) {
            const int a0 = t0 & ~(2 * L - 1), b0 = a0 + L;
            const int la = min(L, n - a0), lb = max(0, min(L, n - b0));
            const int diag = t0 - a0;
            int lo = max(0, diag - lb), hi = min(diag, la);
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (s[lf_pad(a0 + mid)] <= s[lf_pad(b0 + diag - 1 - mid)]) lo = mid + 1;
                else hi = mid;
            }
            int ia = a0 + lo, ib = b0 + diag - lo;
            const int ea = a0 + la, eb = b0 + lb;
            K ka = ia < ea ? s[lf_pad(ia)] : (K)~(K)0;
            K kb = ib < eb ? s[lf_pad(ib)] : (K)~(K)0;
#pragma unroll
            for (int j = 0; j < I; ++j) {
                const bool ta = ib >= eb || (ia < ea && ka <= kb);
                o[j] = ta ? ka : kb;
                const int nx = ta ? ++ia : ++ib;
                const K f = nx < (ta ? ea : eb) ? s[lf_pad(nx)] : (K)~(K)0;
                if (ta) ka = f;
                else kb = f;
            }
        }
        __syncthreads();
        if (t0 < n) {
#pragma unroll
            for (int j = 0; j < I; ++j) s[lf_pad(t0 + j)] = o[j];
        }
        __syncthreads();
    }
}

constexpr int LF_ROWS = 1 << BK_ROWBITS;
constexpr int LF_BINS = 4096;   // places shared out among the rows, about one or two a key
// Keys read per key for the ranks above which a bucket is sorted by comparisons
// instead (evenly spread columns read two; comparing costs as much as about 60).
constexpr int LF_CROWD = 64;

constexpr int LF_PLACES = BK_CAP + BK_CAP / 32;

struct LeafShared {
    alignas(16) unsigned bins[LF_BINS + LF_ROWS + 4];
    unsigned row[LF_ROWS];  // entries, then first place | places << 16
    unsigned w[LF_WARPS];
    unsigned crowd;  // keys that the ranks will read
};

struct LeafArgs {
    const BkDesc *desc, *desc2;  // two lists of buckets: ndesc of them, read from src,
    unsigned ndesc;
    const unsigned *ndesc2;      // and *ndesc2 pieces of the longer ones, read from src2
    int scale;
    BkCtl *ctl2;           // its overflow counts the pieces too long for a sort here
    unsigned *tile_cnt;    // kept entries per POS_TILE positions
    unsigned *rawoff;      // [n + 1] first position of every row
    uint2 *wadj;           // MODE 2
};

// A bucket as the sort sees it: keys relative to the first key of the row that the
// bucket's range begins in.
template <typename K>
struct Leaf {
    uint32_t start;
    int n;
    K kmask, kbase;
    int field, fbits;  // bits below the row; those that a key of this bucket uses
    int nrows;
    uint64_t uv0;      // (u, v) of relative key 0
    uint64_t r0, r1;   // rows whose first possible key lies in the bucket's range
};

// MODE 0: entries (u, v); the column with bit 31 set for a repeat goes to dst.
// MODE 1: entries (u, v, w): column, mark and weight as one 64-bit word; of
//         entries with the same (u, v) the one of least weight is kept.
// MODE 2: entries (u, w, v) of finished rows: (column, weight) pairs to wadj.
template <typename K, int MODE>
__device__ __forceinline__ void leaf_put(const LeafArgs &a, const Leaf<K> &lf, K *dst, uint32_t pos, K k, bool keep)
{
    constexpr int LOW = MODE == 1 ? WBITS : 0;
    // the column lies in the low 32 bits of (u, v)
    const uint32_t c = ((uint32_t)lf.uv0 + (uint32_t)(k >> LOW)) & (uint32_t)low_mask(a.scale);
    if (MODE == 0) {
        dst[pos] = (K)(c | (keep ? 0u : 0x80000000u));
    } else if (MODE == 1) {
        dst[pos] = (K)(((uint64_t)(c | (keep ? 0u : 0x80000000u)) << 32) | ((uint64_t)k & ((1u << WBITS) - 1)));
    } else {
        a.wadj[pos] = make_uint2(c, (uint32_t)((lf.uv0 + (uint64_t)k) >> a.scale) & ((1u << WBITS) - 1));
    }
}

// Adds a bucket's kept entries, ca before and cb after its first border of POS_TILE positions.
__device__ __forceinline__ void leaf_count(const LeafArgs &a, uint32_t start, unsigned ca, unsigned cb)
{
    ca = __reduce_add_sync(kFull, ca);
    cb = __reduce_add_sync(kFull, cb);
    if ((threadIdx.x & 31) == 0 && ca) atomicAdd(&a.tile_cnt[start / POS_TILE], ca);
    if ((threadIdx.x & 31) == 0 && cb) atomicAdd(&a.tile_cnt[start / POS_TILE + 1], cb);
}

// The bucket's keys by counting.  Every row gets places in proportion to
// its entries, a key's place is its column scaled to its row's places, and
// within a place (one or two keys where columns spread evenly, as they do in a
// graph with shuffled numbers) a key's rank is the number of lesser ones, found by
// reading them all.  No comparison network, no stable pass: three shared atomics
// a key, one exchange through shared memory, and about five keys read for the rank by the
// slowest lane of a warp.  A repeat is a key with an equal one before it in its
// place, and a row's first position is the start of its first place.  The keys are
// read from memory (the L1 from the second time on) by each of the three first loops
// instead of being held in registers: unrolled over up to 16 registers in three
// sizes the kernel did not fit the instruction cache and waited for it half
// of its time.  false: the places are too crowded (columns close together, or
// many copies) and nothing is written.
template <typename K, int MODE>
__device__ __forceinline__ bool count_sort(const LeafArgs &a, const Leaf<K> &lf, const K *src, K *dst, K *s, LeafShared &sh)
{
    constexpr int LOW = MODE == 1 ? WBITS : 0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = lf.n;
    int nb = 256;
    while (nb < n) nb <<= 1;  // at most LF_BINS
    // 16 leading bits of the field place a key in its row (the weight, last, takes no part)
    const int vb = lf.fbits - LOW;
    const int rsh = lf.field, dsh = LOW + max(0, vb - 16), ush = max(0, 16 - vb);
    const K fmask = (K)low_mask(lf.fbits);
    const bool rows = lf.nrows > 1;
    const int total_max = nb + (rows ? lf.nrows : 0);
    for (int i = tid; i <= total_max >> 2; i += LF_THREADS) reinterpret_cast<uint4 *>(sh.bins)[i] = make_uint4(0, 0, 0, 0);
    if (rows)
        for (int i = tid; i < lf.nrows; i += LF_THREADS) sh.row[i] = 0;
    if (tid == 0) sh.crowd = 0;
    __syncthreads();
    const auto load = [&](int i) { return (src[lf.start + i] & lf.kmask) - lf.kbase; };
    int total = nb;
    if (rows) {
#pragma unroll 4
        for (int i = tid; i < n; i += LF_THREADS) atomicAdd(&sh.row[(unsigned)(load(i) >> rsh)], 1u);
        __syncthreads();
        constexpr int RP = LF_ROWS / LF_THREADS;
        unsigned c[RP], t = 0;
#pragma unroll
        for (int j = 0; j < RP; ++j) {
            const int r = tid * RP + j;
            const unsigned e = r < lf.nrows ? sh.row[r] : 0u;
            c[j] = e ? (e * (unsigned)nb + (unsigned)n - 1u) / (unsigned)n : 0u;  // nb and e at most 4096
            t += c[j];
        }
        const unsigned incl = warp_inclusive_scan(t);
        if (lane == 31) sh.w[warp] = incl;
        __syncthreads();
        unsigned run = incl - t;
        total = 0;
#pragma unroll
        for (int w = 0; w < LF_WARPS; ++w) {
            if (w < warp) run += sh.w[w];
            total += (int)sh.w[w];
        }
#pragma unroll
        for (int j = 0; j < RP; ++j) {
            const int r = tid * RP + j;
            if (r < lf.nrows) sh.row[r] = run | (c[j] << 16);
            run += c[j];
        }
        __syncthreads();
    }
    const auto place = [&](K k) -> unsigned {
        const unsigned t = (unsigned)((k & fmask) >> dsh) << ush;
        const unsigned ri = rows ? sh.row[(unsigned)(k >> rsh)] : (unsigned)nb << 16;
        return (ri & 0xffffu) + ((t * (ri >> 16)) >> 16);
    };
    // bins[b + 1] counts place b, then holds where its next key goes, at last its end
#pragma unroll 4
    for (int i = tid; i < n; i += LF_THREADS) atomicAdd(&sh.bins[place(load(i)) + 1], 1u);
    __syncthreads();
    {  // exclusive scan of the places, each thread a run of them
        const int per = ((total + LF_THREADS - 1) / LF_THREADS) | 1;  // odd: a warp's runs start in 32 banks
        const int i0 = 1 + tid * per, i1 = min(total + 1, i0 + per);
        unsigned t = 0, reads = 0;
        for (int i = i0; i < i1; ++i) {
            const unsigned c = sh.bins[i];
            t += c;
            reads += c * c;
        }
        const unsigned incl = warp_inclusive_scan(t);
        if (lane == 31) sh.w[warp] = incl;
        reads = __reduce_add_sync(kFull, reads);
        if (lane == 0) atomicAdd(&sh.crowd, reads);
        __syncthreads();
        unsigned run = incl - t;
#pragma unroll
        for (int w = 0; w < LF_WARPS; ++w)
            if (w < warp) run += sh.w[w];
        for (int i = i0; i < i1; ++i) {
            const unsigned c = sh.bins[i];
            sh.bins[i] = run;
            run += c;
        }
    }
    __syncthreads();
    if (sh.crowd > (unsigned)(LF_CROWD * n)) return false;
#pragma unroll 4
    for (int i = tid; i < n; i += LF_THREADS) {
        const K k = load(i);
        s[atomicAdd(&sh.bins[place(k) + 1], 1u)] = k;
    }
    __syncthreads();
    if (MODE != 2) {
        const uint64_t ra = lf.uv0 >> a.scale;
        for (uint64_t q = lf.r0 + tid; q < lf.r1; q += LF_THREADS)
            a.rawoff[q] = lf.start + (rows ? sh.bins[sh.row[q - ra] & 0xffffu] : 0u);
    }
    unsigned ca = 0, cb = 0;
    const unsigned border = POS_TILE - (lf.start & (POS_TILE - 1));
    for (int i = tid; i < n; i += LF_THREADS) {
        const K k = s[i];
        const unsigned b = place(k);
        const unsigned p0 = sh.bins[b], p1 = sh.bins[b + 1];
        unsigned rank = 0;
        bool keep = true;
#pragma unroll 2
        for (unsigned p = p0; p < p1; ++p) {
            const K o = s[p];
            const bool less = o < k || (o == k && p < (unsigned)i);
            rank += less;
            if (MODE != 2) keep = keep && !(less && (o >> LOW) == (k >> LOW));
        }
        const unsigned pos = p0 + rank;
        leaf_put<K, MODE>(a, lf, dst, lf.start + pos, k, keep);
        ca += keep && pos < border;
        cb += keep && pos >= border;
    }
    if (MODE != 2) leaf_count(a, lf.start, ca, cb);
    return true;
}

template <typename K, int MODE>
__global__ void __launch_bounds__(LF_THREADS, sizeof(K) == 4 ? 6 : 4) bk_leaf_kernel(LeafArgs a, const K *src1, const K *src2, K *dst)
{
    extern __shared__ __align__(16) unsigned char lf_dyn[];
    K *s = reinterpret_cast<K *>(lf_dyn);
    LeafShared &sh = *reinterpret_cast<LeafShared *>(lf_dyn + LF_PLACES * sizeof(K));
    __shared__ unsigned long long s_min;
    const unsigned nd = a.ndesc + *a.ndesc2;
    constexpr int LOW = MODE == 1 ? WBITS : 0;  // bits that do not tell entries apart
    const uint64_t vmask = low_mask(a.scale);
    const int tid = threadIdx.x;
    for (unsigned q = blockIdx.x; q < nd; q += gridDim.x) {
        const bool piece = q >= a.ndesc;
        const BkDesc d = piece ? a.desc2[q - a.ndesc] : a.desc[q];
        const K *src = piece ? src2 : src1;
        const int bits = desc_bits(d.pr), rem = d.rem;
        const bool big = d.count > (unsigned)BK_CAP;
        if (big && rem > LOW) {
            if (piece && tid == 0) atomicAdd(&a.ctl2->overflow, 1u);
            continue;
        }
        Leaf<K> lf;
        lf.start = d.start;
        lf.n = (int)d.count;
        lf.field = a.scale + (MODE ? WBITS : 0);
        lf.kmask = (K)low_mask(bits);
        // range [lo, hi) of keys below the prefix, counted from the start of lo's row
        const uint64_t lo = (uint64_t)d.lo << rem, base = bits > lf.field ? lo & ~low_mask(lf.field) : 0;
        const uint64_t last = lo - base + ((uint64_t)d.span << rem) - 1;  // span << rem is at most 2^bits
        lf.kbase = (K)base;
        lf.nrows = bits > lf.field ? (int)(last >> lf.field) + 1 : 1;
        lf.fbits = lf.nrows > 1 ? lf.field : 64 - __clzll((long long)last);
        const uint64_t pre = desc_prefix(d.pr) << (bits - LOW);
        lf.uv0 = pre + (base >> LOW);
        const uint64_t first_uv = pre + (lo >> LOW);
        lf.r0 = (first_uv + vmask) >> a.scale;
        lf.r1 = (first_uv + ((uint64_t)d.span << (rem - LOW)) + vmask) >> a.scale;
        if (big) {
            // one (u, v) repeated: nothing to sort, only the least weight to find
            if (tid == 0) s_min = ~0ull;
            __syncthreads();
            unsigned long long mn = ~0ull;
            for (unsigned i = tid; i < d.count; i += LF_THREADS)
                mn = min(mn, (unsigned long long)((src[d.start + i] & lf.kmask) - lf.kbase));
            atomicMin(&s_min, mn);
            __syncthreads();
            if (MODE != 2) {
                for (uint64_t r = lf.r0 + tid; r < lf.r1; r += LF_THREADS) a.rawoff[r] = d.start;
                for (unsigned i = tid; i < d.count; i += LF_THREADS)
                    leaf_put<K, MODE>(a, lf, dst, d.start + i, (K)s_min, i == 0);
                leaf_count(a, d.start, tid == 0, 0);
            }
            __syncthreads();
            continue;
        }
        const int n = lf.n;
        const bool ok = count_sort<K, MODE>(a, lf, src, dst, s, sh);
        if (!ok) {
            merge_sort<K, 16>(src + d.start, n, lf.kmask, lf.kbase, s);
            if (MODE != 2) {
                for (uint64_t r = lf.r0 + tid; r < lf.r1; r += LF_THREADS) {
                    const uint64_t first = (r << a.scale) - lf.uv0;  // least key of row r
                    int b = 0, e = n;
                    while (b < e) {
                        const int mid = (b + e) >> 1;
                        if ((uint64_t)(s[lf_pad(mid)] >> LOW) < first) b = mid + 1;
                        else e = mid;
                    }
                    a.rawoff[r] = d.start + b;
                }
            }
            unsigned ca = 0, cb = 0;
            const unsigned border = POS_TILE - (d.start & (POS_TILE - 1));
            for (int i = tid; i < n; i += LF_THREADS) {
                const K k = s[lf_pad(i)];
                const bool keep = i == 0 || (s[lf_pad(i - 1)] >> LOW) != (k >> LOW);
                leaf_put<K, MODE>(a, lf, dst, d.start + i, k, keep);
                ca += keep && (unsigned)i < border;
                cb += keep && (unsigned)i >= border;
            }
            if (MODE != 2) leaf_count(a, d.start, ca, cb);
        }
        __syncthreads();
    }
}

// ---- step 4 ---------------------------------------------------------------

constexpr int PS_THREADS = 1024;
constexpr int PS_ITEMS = 4;
constexpr int PS_CHUNK = PS_THREADS * PS_ITEMS;  // tile counts per block

__global__ void __launch_bounds__(PS_THREADS) bk_possum_kernel(const unsigned *__restrict__ cnt, unsigned nt,
                                                               unsigned *__restrict__ sums)
{
    __shared__ unsigned s_w[PS_THREADS / 32];
    unsigned t = 0;
#pragma unroll
    for (int j = 0; j < PS_ITEMS; ++j) {
        const unsigned i = blockIdx.x * PS_CHUNK + j * PS_THREADS + threadIdx.x;
        if (i < nt) t += cnt[i];
    }
    t = __reduce_add_sync(kFull, t);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x < 32) {
        t = __reduce_add_sync(kFull, s_w[threadIdx.x]);
        if (threadIdx.x == 0) sums[blockIdx.x] = t;
    }
}

// What the host reads once the entries are sorted.
struct BkResult {
    unsigned nnz, overflow;
    DevStatus status;
};

// base[i] = kept entries before tile i; their total, how many pieces are left that
// need a further split, and the device status to *res.
__global__ void __launch_bounds__(PS_THREADS) bk_posscan_kernel(const unsigned *__restrict__ cnt, unsigned nt,
                                                                const unsigned *__restrict__ sums,
                                                                unsigned *__restrict__ base,
                                                                const BkCtl *__restrict__ ctl, const DevStatus *st,
                                                                BkResult *__restrict__ res)
{
    __shared__ unsigned s_w[PS_THREADS / 32], s_b[PS_THREADS / 32];
    unsigned before = 0;
    for (unsigned b = threadIdx.x; b < blockIdx.x; b += PS_THREADS) before += sums[b];
    before = __reduce_add_sync(kFull, before);
    const unsigned i0 = blockIdx.x * PS_CHUNK + threadIdx.x * PS_ITEMS;
    unsigned c[PS_ITEMS], t = 0;
#pragma unroll
    for (int j = 0; j < PS_ITEMS; ++j) {
        c[j] = i0 + j < nt ? cnt[i0 + j] : 0u;
        t += c[j];
    }
    const unsigned incl = warp_inclusive_scan(t);
    if ((threadIdx.x & 31) == 31) s_w[threadIdx.x >> 5] = incl;
    if ((threadIdx.x & 31) == 0) s_b[threadIdx.x >> 5] = before;
    __syncthreads();
    unsigned run = incl - t;
    for (int w = 0; w < PS_THREADS / 32; ++w) {
        run += s_b[w];
        if (w < (int)(threadIdx.x >> 5)) run += s_w[w];
    }
#pragma unroll
    for (int j = 0; j < PS_ITEMS; ++j) {
        if (i0 + j < nt) base[i0 + j] = run;
        run += c[j];
        if (i0 + j + 1 == nt) {
            res->nnz = run;
            res->overflow = ctl->overflow;
            res->status = *st;
        }
    }
}

// The kept entries of every tile to their columns (and weights); for every 32
// positions which are kept and how many before them, for the row offsets.
constexpr int CP_THREADS = 256;
constexpr int CP_ROUNDS = POS_TILE / CP_THREADS;  // 16 positions a lane
template <typename K>
__global__ void __launch_bounds__(CP_THREADS) bk_compact_kernel(const K *__restrict__ ent, const unsigned *__restrict__ total_p,
                                                                const unsigned *__restrict__ base,
                                                                int32_t *__restrict__ col, uint32_t *__restrict__ wgt,
                                                                uint2 *__restrict__ kept, unsigned nnz, DevStatus *st)
{
    __shared__ unsigned s_w[CP_THREADS / 32];
    const unsigned total = *total_p;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned t0 = blockIdx.x * (unsigned)POS_TILE;
    if (t0 >= total) return;
    const unsigned w0 = t0 + warp * (32 * CP_ROUNDS);
    K x[CP_ROUNDS];
#pragma unroll
    for (int j = 0; j < CP_ROUNDS; ++j) {
        const unsigned i = w0 + 32 * j + lane;
        x[j] = i < total ? ent[i] : (K)~(K)0;  // past the end: marked as dropped
    }
    unsigned mk[CP_ROUNDS], c = 0;
#pragma unroll
    for (int j = 0; j < CP_ROUNDS; ++j) {
        const uint32_t cv = sizeof(K) == 8 ? (uint32_t)((uint64_t)x[j] >> 32) : (uint32_t)x[j];
        mk[j] = __ballot_sync(kFull, !(cv & 0x80000000u));
        c += __popc(mk[j]);
    }
    if (lane == 0) s_w[warp] = c;
    __syncthreads();
    unsigned pos = base[blockIdx.x];
    for (int w = 0; w < warp; ++w) pos += s_w[w];
#pragma unroll
    for (int j = 0; j < CP_ROUNDS; ++j) {
        if (lane == j) kept[(w0 >> 5) + j] = make_uint2(mk[j], pos);
        if ((mk[j] >> lane) & 1u) {
            const unsigned o = pos + __popc(mk[j] & lanemask_lt());
            if (o < nnz) {
                if (sizeof(K) == 8) {
                    col[o] = (int32_t)((uint64_t)x[j] >> 32);
                    wgt[o] = (uint32_t)x[j];
                } else {
                    col[o] = (int32_t)x[j];
                }
            } else {
                record_error(st, GB_ERR_RANGE, SITE_BK_POS + 1, o);
            }
        }
        pos += __popc(mk[j]);
    }
}

__global__ void bk_off_kernel(const unsigned *__restrict__ rawoff, const uint2 *__restrict__ kept,
                              const unsigned *__restrict__ total_p, int64_t n, int64_t nnz, int64_t *__restrict__ off)
{
    const unsigned total = *total_p;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r <= n; r += stride) {
        const unsigned p = r < n ? rawoff[r] : total;
        int64_t o = nnz;
        if (p < total) {
            const uint2 k = kept[p >> 5];
            o = (int64_t)k.y + __popc(k.x & ((1u << (p & 31)) - 1u));
        }
        off[r] = o;
    }
}

// ---- the weight-ordered rows ------------------------------------------------

// Buckets of 2^q whole rows of a finished CSR.
__global__ void bk_rows_kernel(const int64_t *__restrict__ off, int64_t n, int q, int rem, unsigned nd,
                               BkDesc *__restrict__ desc)
{
    for (unsigned g = blockIdx.x * blockDim.x + threadIdx.x; g < nd; g += gridDim.x * blockDim.x) {
        const int64_t r0 = (int64_t)g << q, r1 = min((int64_t)n, r0 + (int64_t(1) << q));
        desc[g] = whole_desc((uint32_t)off[r0], (uint32_t)(off[r1] - off[r0]), g, rem);
    }
}

// The row that holds entry i, among rows [lo, hi] of which it is one.
__device__ __forceinline__ int64_t row_of(const int64_t *__restrict__ off, int64_t lo, int64_t hi, int64_t i)
{
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (off[mid + 1] <= i) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// Key (row's low q bits, weight, column) of every entry.  A warp takes 512
// entries, whatever rows they belong to, bisects the offsets for the first and
// last row and each entry among those.
constexpr int RK_ROUNDS = 16;
__global__ void bk_rowkeys_kernel(const int64_t *__restrict__ off, const int32_t *__restrict__ col,
                                  const uint32_t *__restrict__ wgt, int64_t n, int64_t nnz, int scale, int q,
                                  uint64_t *__restrict__ keys)
{
    const unsigned lane = threadIdx.x & 31u;
    const int64_t gwarp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const uint64_t qmask = (uint64_t(1) << q) - 1;
    for (int64_t e0 = gwarp * (32 * RK_ROUNDS); e0 < nnz; e0 += nwarps * (32 * RK_ROUNDS)) {
        const int64_t e1 = min(nnz, e0 + 32 * RK_ROUNDS) - 1;
        const int64_t rr = row_of(off, 0, n - 1, lane == 0 ? e0 : e1);
        const int64_t r0 = __shfl_sync(kFull, rr, 0), r1 = __shfl_sync(kFull, rr, 1);
#pragma unroll 4
        for (int j = 0; j < RK_ROUNDS; ++j) {
            const int64_t i = e0 + 32 * j + lane;
            if (i <= e1)
                keys[i] = ((((uint64_t)row_of(off, r0, r1, i) & qmask) << WBITS | (uint64_t)wgt[i]) << scale) |
                          (uint64_t)(uint32_t)col[i];
        }
    }
}

// ---- host -------------------------------------------------------------------

template <typename Kern>
cudaError_t smem_limit(Kern k, int bytes)
{
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

int ceil_log2(uint64_t x)
{
    int b = 0;
    while ((uint64_t(1) << b) < x) ++b;
    return b;
}

// One split of the listed buckets: list, count, place, move.
struct Level {
    BkSeg *segs = nullptr;
    uint2 *tiles = nullptr;
    unsigned *cnt = nullptr, *cursor = nullptr;
    BkDesc *desc = nullptr;
    BkCtl *ctl = nullptr;
};

// rawoff: BY_DIFFERENCE only.
template <typename KIN, typename KOUT>
gb_status split(Context *ctx, const Level &lv, const BkDesc *desc, const unsigned *ndesc_dev, unsigned ndesc, int forced,
                int field, int low, int64_t nk, const KIN *in, KOUT *out, cudaStream_t s, int scale = 0,
                unsigned *rawoff = nullptr)
{
    const int sms = ctx->num_sms;
    const int64_t most = ndesc_dev ? nk / (BK_SPLIT / 2) + 2 : (int64_t)ndesc;
    const int lb = (int)std::max<int64_t>(1, std::min<int64_t>((most + 255) / 256, sms * 4));
    bk_list_kernel<<<lb, 256, 0, s>>>(desc, ndesc_dev, ndesc, forced, field, low, lv.segs, lv.tiles, lv.ctl);
    const int64_t tiles = nk / BK_TILE + 1 + (forced > 0 ? (int64_t)ndesc : nk / BK_CAP);
    const int hb = (int)std::min<int64_t>(tiles, sms * 4), pb = (int)std::min<int64_t>(tiles, sms * 2);
    const int64_t nseg = forced > 0 ? (int64_t)ndesc : nk / BK_CAP + 1;
    if (forced == BY_DIFFERENCE) {
        bk_differ_kernel<KIN><<<hb, BK_THREADS, 0, s>>>(in, lv.segs, lv.tiles, lv.ctl);
        bk_digit_kernel<KIN><<<(int)std::min<int64_t>((nseg + 255) / 256, sms * 4), 256, 0, s>>>(in, lv.segs, lv.ctl, low,
                                                                                             scale, rawoff);
        note_launch(2);
    }
    bk_hist_kernel<KIN><<<hb, BK_THREADS, 0, s>>>(in, lv.segs, lv.tiles, lv.ctl, lv.cnt);
    bk_scan_kernel<<<(int)std::min<int64_t>(nseg, sms * 8), SC_THREADS, 0, s>>>(
        lv.segs, lv.ctl, forced <= 0, lv.cnt, lv.cursor, lv.desc);
    constexpr int smem = PartShared<KOUT, sizeof(KIN) != sizeof(KOUT)>::bytes;
    GB_CUDA(smem_limit(bk_part_kernel<KIN, KOUT>, smem));
    bk_part_kernel<KIN, KOUT><<<pb, BK_THREADS, smem, s>>>(in, lv.segs, lv.tiles, lv.ctl, lv.cursor, out, (unsigned)nk,
                                                           ctx->status);
    note_launch(4);
    GB_CUDA(cudaGetLastError());
    return GB_OK;
}

template <typename K, int MODE>
gb_status leaves(Context *ctx, const LeafArgs &a, int64_t most, const K *src, const K *src2, K *dst, cudaStream_t s)
{
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(most, (int64_t)ctx->num_sms * 32));
    constexpr int smem = LF_PLACES * (int)sizeof(K) + (int)sizeof(LeafShared);
    GB_CUDA(smem_limit(bk_leaf_kernel<K, MODE>, smem));
    bk_leaf_kernel<K, MODE><<<grid, LF_THREADS, smem, s>>>(a, src, src2, dst);
    note_launch();
    GB_CUDA(cudaGetLastError());
    return GB_OK;
}

// Device memory carved from one block, zeroed part first.
struct Arena {
    size_t used = 0;
    size_t take(size_t bytes)
    {
        const size_t o = used;
        used = (used + bytes + 255) & ~size_t(255);
        return o;
    }
};

// Most pieces of a split of buckets longer than BK_CAP among nk keys, the rows
// of a bucket numbered by `rowbits` bits: two per BK_SPLIT keys and row, BK_BINS a bucket.
int64_t split_pieces(int64_t nk, int rowbits)
{
    const int64_t by_rows = (nk / (BK_SPLIT / 2) + 2) << std::max(0, std::min(rowbits, BK_BITS));
    return std::min(by_rows, (nk / BK_CAP + 1) * BK_BINS);
}

struct LevelPlan {
    size_t ctl, cnt, segs, tiles, cursor, desc;
};

LevelPlan plan_zeroed(Arena &a, int64_t pieces)
{
    LevelPlan p{};
    p.ctl = a.take(sizeof(BkCtl));
    p.cnt = a.take((size_t)pieces * 4);
    return p;
}

void plan_rest(Arena &a, LevelPlan &p, int64_t nseg, int64_t tiles, int64_t pieces, int64_t descs)
{
    p.segs = a.take((size_t)nseg * sizeof(BkSeg));
    p.tiles = a.take((size_t)tiles * sizeof(uint2));
    p.cursor = a.take((size_t)pieces * 4);
    p.desc = a.take((size_t)descs * sizeof(BkDesc));
}

Level level_at(unsigned char *b, const LevelPlan &p)
{
    Level l;
    l.ctl = reinterpret_cast<BkCtl *>(b + p.ctl);
    l.cnt = reinterpret_cast<unsigned *>(b + p.cnt);
    l.segs = reinterpret_cast<BkSeg *>(b + p.segs);
    l.tiles = reinterpret_cast<uint2 *>(b + p.tiles);
    l.cursor = reinterpret_cast<unsigned *>(b + p.cursor);
    l.desc = reinterpret_cast<BkDesc *>(b + p.desc);
    return l;
}

// What the sorts of `from`'s pieces left because it was too long, `left` pieces with
// their keys in ka: split from the bits they differ in and sorted into kb, until nothing is left.
// Every turn a piece gives up at least the bit that parts its keys, so there are at most 64.
// look(ctl, &left): waits for the stream and reads ctl's overflow.
// Why by the bits that differ: splits at fixed digits took 10 bits whether or not keys
// differed in them, gave up after two, and the LSD sort began anew (SCALE 20 as
// drawn 3.1 ms, now 1.46; unit weights beside a row of 10^5, whose weight bits are all
// equal, 6.6 ms, now 3.2).  Where length alone asks for a second split (more than 2^10
// pieces of one bucket) a turn costs 10 to 20 us more than a third fixed digit did, for its
// two launches more.
template <typename K, int MODE, typename Look>
gb_status split_rest(Context *ctx, LeafArgs la, Level from, unsigned left, int low, int64_t nk, K *ka, K *kb,
                     Look look, cudaStream_t s)
{
    const int64_t desc_x = nk / (BK_SPLIT / 2) + 2;  // as many descriptors as `from` has
    Scratch tmp(s);
    unsigned char *prev = nullptr;
    K *in = ka, *out = kb;
    for (int turn = 0; left; ++turn) {
        if (turn == 64) {
            set_error("kernel 1: a bucket that no digit splits");
            return GB_ERR_CUDA;
        }
        // bk_digit_kernel takes less than 1/64 as many pieces as keys
        const int64_t pieces = std::min<int64_t>(nk / 64 + 8, (int64_t)left << BK_BITS);
        Arena ar;
        LevelPlan p = plan_zeroed(ar, pieces);
        const size_t zeroed = ar.used;
        plan_rest(ar, p, left, nk / BK_TILE + 1 + left, pieces, desc_x);
        unsigned char *ws = nullptr;
        GB_CUDA(tmp.alloc(&ws, ar.used));
        GB_CUDA(cudaMemsetAsync(ws, 0, zeroed, s));
        const Level lv = level_at(ws, p);
        gb_status rc = split<K, K>(ctx, lv, from.desc, &from.ctl->ndesc, 0, BY_DIFFERENCE, 0, low, nk, in, out, s, la.scale,
                                   la.rawoff);
        if (rc != GB_OK) return rc;
        la.ndesc = 0;
        la.desc2 = lv.desc;
        la.ndesc2 = &lv.ctl->ndesc;
        la.ctl2 = lv.ctl;
        rc = leaves<K, MODE>(ctx, la, desc_x, out, out, kb, s);
        if (rc != GB_OK) return rc;
        rc = look(lv.ctl, &left);
        if (rc != GB_OK) return rc;
        if (prev) GB_CUDA(tmp.drop(prev));
        prev = ws;
        from = lv;
        std::swap(in, out);
        note_split();
    }
    return GB_OK;
}

// Steps 0-4 for one key type.
template <typename K, bool WEIGHTED>
gb_status build(const int64_t *edges, const float *w, int64_t m, int scale, const BucketPlan &bp, gb_graph *g,
                cudaStream_t s)
{
    constexpr int MODE = WEIGHTED ? 1 : 0;
    constexpr int LOW = WEIGHTED ? WBITS : 0;
    Context *ctx = context();
    const int field = scale + LOW;  // bits of an entry below its row
    const int64_t nk = 2 * m, n = int64_t(1) << scale;
    const int sms = ctx->num_sms;
    const int total_bits = bp.p0 + bp.p1;
    const int64_t npos = (nk + POS_TILE - 1) / POS_TILE;
    const int64_t n0 = int64_t(1) << bp.p0, n1 = int64_t(1) << total_bits;
    const int rowbits = std::max(0, scale - total_bits);  // of a bucket after step 1
    const int64_t seg_x = nk / BK_CAP + 1, desc_x = nk / (BK_SPLIT / 2) + 2, tile_x = nk / BK_TILE + 1 + seg_x;
    const int64_t piece2 = split_pieces(nk, rowbits);

    Arena ar;
    const size_t o_cnt0 = ar.take(BK_BINS * 4);
    const size_t o_total = ar.take(16);
    const size_t o_pos = ar.take((size_t)npos * 4 + 4);
    LevelPlan l1{};
    if (bp.p1) l1 = plan_zeroed(ar, n1);
    LevelPlan l2 = plan_zeroed(ar, piece2);
    const size_t zeroed = ar.used;
    const size_t o_cur0 = ar.take(BK_BINS * 4);
    const size_t o_desc0 = ar.take(BK_BINS * sizeof(BkDesc));
    const size_t o_base = ar.take((size_t)npos * 4);
    const size_t o_res = ar.take(sizeof(BkResult));
    const size_t o_sums = ar.take((size_t)(npos / PS_CHUNK + 1) * 4);
    const size_t o_raw = ar.take((size_t)(n + 1) * 4);
    const size_t o_kept = ar.take((size_t)npos * (POS_TILE / 32) * sizeof(uint2));
    if (bp.p1) plan_rest(ar, l1, n0, nk / BK_TILE + 1 + n0, n1, n1);
    plan_rest(ar, l2, seg_x, tile_x, piece2, desc_x);

    const size_t o_kb = ar.take((size_t)nk * sizeof(K));
    const size_t o_ka = ar.take((size_t)nk * (bp.p1 ? sizeof(uint64_t) : sizeof(K)));
    // all in one block: a build that repeats gets the same one from the pool, where blocks
    // of several sizes, freed and taken between the graphs' arrays, made the pool
    // map memory anew (SCALE 26: 54.3 to 59.1 ms in turns, so 54.2 to 54.5)
    Scratch tmp(s);
    unsigned char *ws = nullptr;
    GB_CUDA(tmp.alloc(&ws, ar.used));
    K *kb = reinterpret_cast<K *>(ws + o_kb);  // entries after step 1
    K *ka = reinterpret_cast<K *>(ws + o_ka);  // a second buffer for the splits,
    uint64_t *k0 = reinterpret_cast<uint64_t *>(ws + o_ka);  // before them the entries after step 0, where step 1 follows
    GB_CUDA(cudaMemsetAsync(ws, 0, zeroed, s));
    unsigned *cnt0 = reinterpret_cast<unsigned *>(ws + o_cnt0), *cur0 = reinterpret_cast<unsigned *>(ws + o_cur0);
    unsigned *total = reinterpret_cast<unsigned *>(ws + o_total);
    BkDesc *desc0 = reinterpret_cast<BkDesc *>(ws + o_desc0);

    // step 0
    const int64_t hthreads = (m + BK_THREADS * 8 - 1) / (BK_THREADS * 8);
    bk_hist0_kernel<<<(int)std::max<int64_t>(1, std::min<int64_t>(hthreads, sms * 4)), BK_THREADS, 0, s>>>(
        edges, m, scale, bp.p0, cnt0, ctx->status);
    const int rem0 = 2 * scale + LOW - bp.p0;
    bk_scan0_kernel<<<1, SC_THREADS, 0, s>>>(cnt0, bp.p0, rem0, cur0, desc0, total);
    const int64_t tiles0 = (nk + BK_TILE - 1) / BK_TILE;
    const int pb = (int)std::min<int64_t>(tiles0, sms * 2);
    const unsigned limit = (unsigned)nk;
    if (bp.p1 || WEIGHTED) {
        // 64-bit keys; an unweighted one keeps its digit
        constexpr int smem = PartShared<uint64_t, WEIGHTED>::bytes;
        GB_CUDA(smem_limit(bk_part0_kernel<uint64_t, WEIGHTED, WEIGHTED>, smem));
        bk_part0_kernel<uint64_t, WEIGHTED, WEIGHTED><<<pb, BK_THREADS, smem, s>>>(
            edges, w, m, scale, bp.p0, cur0, bp.p1 ? k0 : reinterpret_cast<uint64_t *>(kb), limit, ctx->status);
    } else {
        constexpr int smem = PartShared<uint32_t, true>::bytes;
        GB_CUDA(smem_limit(bk_part0_kernel<uint32_t, false, true>, smem));
        bk_part0_kernel<uint32_t, false, true><<<pb, BK_THREADS, smem, s>>>(
            edges, nullptr, m, scale, bp.p0, cur0, reinterpret_cast<uint32_t *>(kb), limit, ctx->status);
    }
    note_launch(3);
    GB_CUDA(cudaGetLastError());
    // step 1
    gb_status rc;
    const BkDesc *leaf_desc = desc0;
    if (bp.p1) {
        const Level lv = level_at(ws, l1);
        rc = split<uint64_t, K>(ctx, lv, desc0, nullptr, (unsigned)n0, bp.p1, field, LOW, nk, k0, kb, s);
        if (rc != GB_OK) return rc;
        leaf_desc = lv.desc;
    }
    // steps 2 and 3: the buckets of at most BK_CAP keys, and the pieces of the longer
    // ones, moved to ka and sorted back into their places in kb
    const Level lv2 = level_at(ws, l2);
    LeafArgs la{};
    la.desc = leaf_desc;
    la.ndesc = (unsigned)n1;
    la.desc2 = lv2.desc;
    la.ndesc2 = &lv2.ctl->ndesc;
    la.ctl2 = lv2.ctl;
    la.scale = scale;
    la.tile_cnt = reinterpret_cast<unsigned *>(ws + o_pos);
    la.rawoff = reinterpret_cast<unsigned *>(ws + o_raw);
    rc = split<K, K>(ctx, lv2, leaf_desc, nullptr, (unsigned)n1, BY_LENGTH, field, LOW, nk, kb, ka, s);
    if (rc != GB_OK) return rc;
    rc = leaves<K, MODE>(ctx, la, n1 + desc_x, kb, ka, kb, s);
    if (rc != GB_OK) return rc;
    // step 4
    unsigned *sums = reinterpret_cast<unsigned *>(ws + o_sums), *base = reinterpret_cast<unsigned *>(ws + o_base);
    BkResult *res = reinterpret_cast<BkResult *>(ws + o_res);
    const unsigned psb = (unsigned)((npos + PS_CHUNK - 1) / PS_CHUNK);
    BkResult hr;
    const auto positions = [&](const BkCtl *ctl, unsigned *left) -> gb_status {
        bk_possum_kernel<<<psb, PS_THREADS, 0, s>>>(la.tile_cnt, (unsigned)npos, sums);
        bk_posscan_kernel<<<psb, PS_THREADS, 0, s>>>(la.tile_cnt, (unsigned)npos, sums, base, ctl, ctx->status, res);
        note_launch(2);
        GB_CUDA(cudaGetLastError());
        GB_CUDA(cudaMemcpyAsync(&hr, res, sizeof(hr), cudaMemcpyDeviceToHost, s));
        GB_CUDA(cudaStreamSynchronize(s));
        *left = hr.status.code == 0 ? hr.overflow : 0;  // an error: no further work on these keys
        return GB_OK;
    };
    unsigned left = 0;
    rc = positions(lv2.ctl, &left);
    if (rc == GB_OK) rc = split_rest<K, MODE>(ctx, la, lv2, left, LOW, nk, ka, kb, positions, s);
    if (rc != GB_OK) return rc;
    const DevStatus &hst = hr.status;
    const unsigned nnz = hr.nnz;
    if (hst.code != 0) {
        GB_CUDA(cudaMemsetAsync(ctx->status, 0, sizeof(DevStatus), s));
        set_error(hst.code != GB_ERR_RANGE      ? "graph_build_csr: device error during the build"
                  : hst.where == SITE_SP_W      ? "graph_build_csr_weighted: a weight outside (0, 1]"
                  : hst.where == SITE_K1_RANGE  ? "graph_build_csr: an edge endpoint is outside [0, 2^scale)"
                                                : "graph_build_csr: device error during the build");
        return (gb_status)hst.code;
    }
    g->nnz = (int64_t)nnz;
    GB_CUDA(gb::dmalloc_async(&g->off, (n + 1) * sizeof(int64_t), s));
    GB_CUDA(gb::dmalloc_async(&g->col, col_alloc_entries(g->nnz) * sizeof(int32_t), s));
    if (WEIGHTED) GB_CUDA(gb::dmalloc_async(&g->wgt, std::max<int64_t>(g->nnz, 4) * sizeof(uint32_t), s));
    uint2 *kept = reinterpret_cast<uint2 *>(ws + o_kept);
    bk_compact_kernel<K><<<(unsigned)npos, CP_THREADS, 0, s>>>(kb, total, base, g->col, g->wgt, kept, nnz, ctx->status);
    bk_off_kernel<<<(int)std::min<int64_t>((n + 256) / 256, sms * 16), 256, 0, s>>>(la.rawoff, kept, total, n, g->nnz,
                                                                                  g->off);
    note_launch(2);
    GB_CUDA(cudaGetLastError());
    return build_graph_aux(g, s);
}

}  // namespace

bool bucket_plan(int64_t m, int scale, bool weighted, BucketPlan *out)
{
    const int64_t nk = 2 * m;
    if (m < 1 || nk >= (int64_t(1) << 32)) return false;  // positions are 32-bit
    const int low = weighted ? WBITS : 0, kbits = weighted ? 64 : 32;
    int p = std::max(2 * scale + low - kbits, ceil_log2((uint64_t)((nk + BK_MEAN - 1) / BK_MEAN)));
    p = std::max(p, scale - BK_ROWBITS);
    p = std::max(1, std::min(p, 2 * scale));
    if (p > 2 * BK_BITS) {
        if (2 * scale + low - 2 * BK_BITS > kbits) return false;  // SCALE 27 and more: the rest would not fit
        p = 2 * BK_BITS;
    }
    BucketPlan b{};
    if (p <= BK_BITS) {
        b.p0 = p;
    } else {
        b.p0 = std::max((p + 1) / 2, 2 * scale + low - 64);
        if (b.p0 > BK_BITS) return false;  // a weighted key does not fit 64 bits below the first digit
        b.p1 = p - b.p0;                   // p > BK_BITS >= p0
    }
    *out = b;
    return true;
}

gb_status bucket_build(const int64_t *edges, const float *w, int64_t m, int scale, const BucketPlan &plan, gb_graph *g,
                       cudaStream_t s)
{
    note_build(plan.p1 ? 2 : 1);
    return w ? build<uint64_t, true>(edges, w, m, scale, plan, g, s)
             : build<uint32_t, false>(edges, nullptr, m, scale, plan, g, s);
}

bool bucket_order_fits(int64_t nnz) { return nnz >= 1 && nnz < (int64_t(1) << 32); }

gb_status bucket_weight_order(const gb_graph *g, uint2 *wadj, cudaStream_t s)
{
    Context *ctx = context();
    const int64_t nnz = g->nnz, n = g->n;
    // 2^q rows a bucket, BK_MEAN entries on average
    int q = 0;
    while (q < BK_ROWBITS && q + 1 < g->scale && (nnz >> (g->scale - q - 1)) <= BK_MEAN && q + 1 + WBITS + g->scale <= 60) ++q;
    const int field = WBITS + g->scale, rem = q + field;
    const unsigned nd = (unsigned)((n + (int64_t(1) << q) - 1) >> q);
    const int64_t seg_x = nnz / BK_CAP + 1, desc_x = nnz / (BK_SPLIT / 2) + 2, tile_x = nnz / BK_TILE + 1 + seg_x;
    const int64_t piece2 = split_pieces(nnz, q);
    Arena ar;
    LevelPlan l2 = plan_zeroed(ar, piece2);
    const size_t zeroed = ar.used;
    const size_t o_desc = ar.take((size_t)nd * sizeof(BkDesc));
    plan_rest(ar, l2, seg_x, tile_x, piece2, desc_x);
    const size_t o_ka = ar.take((size_t)nnz * 8), o_kb = ar.take((size_t)nnz * 8);
    Scratch tmp(s);
    unsigned char *ws = nullptr;
    GB_CUDA(tmp.alloc(&ws, ar.used));
    uint64_t *ka = reinterpret_cast<uint64_t *>(ws + o_ka), *kb = reinterpret_cast<uint64_t *>(ws + o_kb);
    GB_CUDA(cudaMemsetAsync(ws, 0, zeroed, s));
    BkDesc *desc = reinterpret_cast<BkDesc *>(ws + o_desc);
    const Level lv2 = level_at(ws, l2);
    bk_rows_kernel<<<(int)std::min<int64_t>((nd + 255) / 256, ctx->num_sms * 8), 256, 0, s>>>(g->off, n, q, rem, nd, desc);
    bk_rowkeys_kernel<<<ctx->num_sms * 8, 256, 0, s>>>(g->off, g->col, g->wgt, n, nnz, g->scale, q, kb);
    note_launch(2);
    GB_CUDA(cudaGetLastError());
    LeafArgs la{};
    la.desc = desc;
    la.ndesc = nd;
    la.desc2 = lv2.desc;
    la.ndesc2 = &lv2.ctl->ndesc;
    la.ctl2 = lv2.ctl;
    la.scale = g->scale;
    la.wadj = wadj;
    gb_status rc = split<uint64_t, uint64_t>(ctx, lv2, desc, nullptr, nd, BY_LENGTH, field, 0, nnz, kb, ka, s);
    if (rc != GB_OK) return rc;
    rc = leaves<uint64_t, 2>(ctx, la, nd + desc_x, kb, ka, kb, s);
    if (rc != GB_OK) return rc;
    const auto look = [&](const BkCtl *ctl, unsigned *left) -> gb_status {
        GB_CUDA(cudaMemcpyAsync(left, &ctl->overflow, sizeof(*left), cudaMemcpyDeviceToHost, s));
        GB_CUDA(cudaStreamSynchronize(s));
        return GB_OK;
    };
    unsigned left = 0;
    rc = look(lv2.ctl, &left);
    return rc == GB_OK ? split_rest<uint64_t, 2>(ctx, la, lv2, left, 0, nnz, ka, kb, look, s) : rc;
}

}  // namespace gb
